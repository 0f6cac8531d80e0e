// V(t)^dag psi projections (Eq. 1, Eq. 3) on the tensor cores, FP64-accurate.
//
// Per timeslice t the projection is the complex contraction
//   coeff[j][t][alpha][k] = sum_{kappa = (m, c)} conj(V_t[k][kappa]) psi_j(m, t, alpha, c),
// rows r = (j, alpha), columns k, contraction over kappa (3 L^3).  Written in real
// arithmetic with the contraction index kappa2 = 2 kappa + (0 re, 1 im):
//   A[r][kappa2]           = (re psi, im psi)
//   B[k][kappa2]           = (re v, im v)        -> re coeff
//   B[N + k][kappa2]       = (-im v, re v)       -> im coeff
//
// Split-precision scheme (in the family of Ozaki's error-free splitting): every
// row of A and of B is cut into chunks of 128 complex kappa; within a chunk each
// real x is written with the chunk's exponent e (|x| < 2^e) as
//   x = 2^(e - 7) sum_{i=0..5} d_i 256^-i  (+ a remainder below 2^(e - 48)),
// with signed digits |d_i| <= 128, exact in bf16 (8-bit significand).  The product of
// two values is sum_{i,j} d_i d'_j 2^(ex + ey - 14 - 8 (i + j)); the pairs with
// i + j <= 5 are kept (21 of 36), grouped by class c = i + j (6 classes).  A class sum
// over one chunk is an integer below (c + 1) 256 128^2 = (c + 1) 2^22: up to class 3 the
// tensor core's FP32 accumulation of the bf16 products is exact.  In the last two a sum
// whose digits are all large and of one sign passes 2^24, where an accumulation loses up
// to 2 units: in class 4 (units of 2^-32) the last 16 of 80, 2^-49 of the largest chunk sum
// 2^22, in class 5 (units of 2^-40) the last 32 of 96, 2^-56 of it.  Each class is scaled by
// its power of two and added to a double-float (hi, lo) accumulator.  The result carries
// about 47 bits: relative to max |x| of a chunk the digits lose 2^-48.
// (Digits of 6 bits, 8 per value, need 36 products and a third more digit traffic.)
//
// Kernels: k_slice_psi / k_slice_modes write the digits as bf16 in the tensor
// core's canonical K-major layout (8-row x 16-byte core matrices), one 8 KB /
// 4 KB tile per digit, per 32 reals of kappa2 and per 128 rows / 64 columns;
// k_proj_mma streams them with cp.async.bulk into a three-stage shared-memory
// ring and issues tcgen05.mma into six TMEM class accumulators (6 x 64 columns).  The
// digit tiles of B are adjacent, so they read as one operand of N = 64 x digits: digit i
// of A against digits 0 .. 5 - i of B lands in classes i .. 5 at once, 8 instructions
// (N up to 256) per 16 reals instead of 21, with A read from shared memory 8 times.
// Eight epilogue warps read the classes after every chunk.
#include "common.cuh"
#include "tc.cuh"

#include <cuda_bf16.h>

namespace {

constexpr int S = 6;                   // digits per value
constexpr int NCLS = S;                // classes c = i + j = 0 .. 5
constexpr int CK = 128;                // complex kappa per chunk
constexpr int KB = 32;                 // reals of kappa2 per pipeline stage (two MMA K-steps)
constexpr int NBK = 2 * CK / KB;       // stages per chunk
constexpr int TM = 128;                // tile rows (j, alpha)
constexpr int TN = 64;                 // tile columns: 32 modes x (re, im)
constexpr int A_TILE = TM * KB * 2;    // bytes of one digit tile of A
constexpr int B_TILE = TN * KB * 2;
constexpr int SBO = (KB / 8) * 128;    // 8-row group stride inside a tile
constexpr int LBO = 128;               // K-adjacent core matrices
constexpr int STAGE_A = S * A_TILE, STAGE_B = S * B_TILE;
constexpr int EXP_BYTES = (TM + TN) * 4;
constexpr int NST = 3;                 // ring stages
constexpr int SMEM_BYTES = NST * (STAGE_A + STAGE_B) + 2 * EXP_BYTES;
constexpr long WAIT_LIMIT = 1l << 22;

// Digits by integer arithmetic on the FP64 bits (FP64 arithmetic is scarce on this
// GPU).  exp_above: e with |x| < 2^e (zero and denormals: kExpZero, below every
// normal exponent).  fixed47: X = round(x 2^(47 - e)), |X| <= 2^47.  Balanced base-256
// digits X = sum_{i=0..5} d_i 256^(5 - i): the bytes of X + 128 (256^6 - 1) / 255, less
// 128 (d_0, the part above bit 40, may reach 128), so x = 2^(e - 7) sum_i d_i 256^-i up
// to the rounding of X.
constexpr int kExpZero = -1100;
__device__ __forceinline__ int exp_above(double x) {
  const int E = (int)((__double_as_longlong(x) >> 52) & 0x7FF);
  return E == 0 ? kExpZero : E - 1023 + 1;
}
__device__ __forceinline__ long long fixed47(double x, int e) {
  const long long b = __double_as_longlong(x);
  const int E = (int)((b >> 52) & 0x7FF);
  if (E == 0) return 0;
  const long long M = (b & 0xFFFFFFFFFFFFFll) | (1ll << 52);
  const int k = e + 5 - (E - 1023);            // >= 6 since E - 1023 < e
  const long long X = k >= 62 ? 0 : ((M + (1ll << (k - 1))) >> k);
  return b < 0 ? -X : X;
}
__device__ __forceinline__ void digits(double x, int e, float (&d)[S]) {
  const unsigned long long Y = (unsigned long long)(fixed47(x, e) + 0x808080808080ll);
  const uint32_t lo = (uint32_t)Y, hi = (uint32_t)(Y >> 32);     // hi: bytes 4 and 5 (with its carry)
  d[0] = (float)((int)(hi >> 8) - 128);
  // byte b as the float 2^23 + b, less 2^23 + 128
  d[1] = __uint_as_float(__byte_perm(hi, 0x4B000000u, 0x7440)) - 8388736.f;
#pragma unroll
  for (int i = 2; i < S; i++) d[i] = __uint_as_float(__byte_perm(lo, 0x4B000000u, 0x7440 + 5 - i)) - 8388736.f;
}

// 2^e as a float (exact for -126 <= e <= 127, 0 below)
__device__ __forceinline__ float pow2f(int e) {
  return e < -126 ? 0.f : (e > 127 ? __int_as_float(0x7f800000) : __int_as_float((e + 127) << 23));
}

// one 16-byte core-matrix row of a digit tile: 8 bf16
__device__ __forceinline__ uint4 pack8(const float (&v)[8]) {
  uint32_t w[4];
#pragma unroll
  for (int q = 0; q < 4; q++) {
    __nv_bfloat162 h = __floats2bfloat162_rn(v[2 * q], v[2 * q + 1]);
    w[q] = *(uint32_t*)&h;
  }
  return make_uint4(w[0], w[1], w[2], w[3]);
}

// The slicers: one warp per (timeslice, chunk, group of 8 rows).  Lane = row % 8 + 8 core:
// in step b (a 32-real K-block of the chunk) a lane holds the 8 reals of one core-matrix
// row, so that every digit of the group leaves as one contiguous 512-byte store (the
// tile's four core matrices of these rows).  The chunk is read twice, first for the rows'
// exponents; the second pass finds it in L1.  (With a row per warp the digits left as
// 16-byte pieces of separate sectors: 2.3 ms for 40 right-hand sides on 16^3 x 32, now
// 0.66 ms: 2.5 GB read or written.)
// load(kappa): the complex value of this lane's row, zero beyond the operand.
template <class Load>
__device__ __forceinline__ int group_exponent(const Load& load, int kappa0) {
  int ex = kExpZero;
#pragma unroll 2
  for (int b = 0; b < NBK; b++)
#pragma unroll
    for (int u = 0; u < 4; u++) {
      const double2 v = load(kappa0 + b * (KB / 2) + u);
      ex = max(ex, max(exp_above(v.x), exp_above(v.y)));
    }
  ex = max(ex, __shfl_xor_sync(0xffffffffu, ex, 8));
  return max(ex, __shfl_xor_sync(0xffffffffu, ex, 16));
}

// A digits of right-hand sides: row 4 j + alpha, element kappa = (m, c) of psi_j; rows
// of padding (j >= nrhs) and kappa >= K are zero.
struct PsiRows {
  const double2* psi;          // of this row's right-hand side, spin and timeslice; null: padding
  int K;
  __device__ __forceinline__ double2 operator()(int kappa) const {
    if (!psi || kappa >= K) return make_double2(0, 0);
    const int m = kappa / 3;
    return __ldg(psi + (size_t)m * 12 + (kappa - 3 * m));
  }
};
// A digits of a generic complex source: element kappa of the row at p[kappa sk]
struct GenRows {
  const double2* p;
  size_t sk;
  int K;
  __device__ __forceinline__ double2 operator()(int kappa) const {
    return p && kappa < K ? __ldg(p + (size_t)kappa * sk) : make_double2(0, 0);
  }
};

template <class Load>
__device__ __forceinline__ void slice_rows(const Load& load, int tl, int row, int ql, int q, int Qg, int RT,
                                           uint8_t* As, int* eA, int* eAmax) {
  const int lane = threadIdx.x & 31, kc = lane >> 3, rt = row / TM, rr = row % TM;
  const int kappa0 = q * CK + 4 * kc;
  const int e = group_exponent(load, kappa0);
  if (kc == 0) {
    eA[((size_t)(tl * RT + rt) * Qg + ql) * TM + rr] = e;
    atomicMax(eAmax + (size_t)tl * RT * TM + row, e);
  }
  uint8_t* out = As + (((size_t)(tl * RT + rt) * Qg + ql) * NBK * S) * A_TILE + (size_t)(rr / 8) * SBO + lane * 16;
#pragma unroll 1
  for (int b = 0; b < NBK; b++) {
    float d[8][S];
#pragma unroll
    for (int u = 0; u < 4; u++) {
      const double2 v = load(kappa0 + b * (KB / 2) + u);
      digits(v.x, e, d[2 * u]);
      digits(v.y, e, d[2 * u + 1]);
    }
#pragma unroll
    for (int s = 0; s < S; s++) {
      float v[8];
#pragma unroll
      for (int u = 0; u < 8; u++) v[u] = d[u][s];
      *(uint4*)(out + (size_t)(b * S + s) * A_TILE) = pack8(v);
    }
  }
}

__global__ void __launch_bounds__(128) k_slice_psi(const double2* __restrict__ psi, size_t stride_sites, int site_t0,
                                                   int Vs, int Tg, int nrhs, int K, int q0, int Qg, int RT,
                                                   uint8_t* As, int* eA, int* eAmax) {
  const long wg = ((long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  if (wg >= (long)Tg * RT * (TM / 8) * Qg) return;
  const int ql = (int)(wg % Qg);
  const long rest = wg / Qg;
  const int grp = (int)(rest % (RT * (TM / 8))), tl = (int)(rest / (RT * (TM / 8)));
  const int row = 8 * grp + (threadIdx.x & 7), j = row >> 2;
  PsiRows load{nullptr, K};
  if (j < nrhs) load.psi = psi + ((size_t)j * stride_sites + (size_t)(site_t0 + tl) * Vs) * 12 + (row & 3) * 3;
  slice_rows(load, tl, row, ql, q0 + ql, Qg, RT, As, eA, eAmax);
}

// row r of timeslice t, element kappa at src[t st + r sr + kappa sk]; rows >= R are zero
__global__ void __launch_bounds__(128) k_slice_agen(const double2* __restrict__ src, size_t st, size_t sr, size_t sk,
                                                    int Tg, int R, int K, int q0, int Qg, int RT, uint8_t* As, int* eA,
                                                    int* eAmax) {
  const long wg = ((long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  if (wg >= (long)Tg * RT * (TM / 8) * Qg) return;
  const int ql = (int)(wg % Qg);
  const long rest = wg / Qg;
  const int grp = (int)(rest % (RT * (TM / 8))), tl = (int)(rest / (RT * (TM / 8)));
  const int row = 8 * grp + (threadIdx.x & 7);
  const GenRows load{row < R ? src + (size_t)tl * st + (size_t)row * sr : nullptr, sk, K};
  slice_rows(load, tl, row, ql, q0 + ql, Qg, RT, As, eA, eAmax);
}

// B digits: mode k = 32 mb + kk is row kk (re coefficient: re v, im v) and row 32 + kk
// (im coefficient: -im v, re v) of its block.  VT is [t][kappa][k] (mode fastest).
__global__ void __launch_bounds__(128) k_slice_modes(const double2* __restrict__ VT, int N, int K, int Tg, int q0,
                                                     int Qg, int MB, uint8_t* Bs, int* eB, int* eBmax,
                                                     int conj_in = 0) {
  const long wg = ((long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31, kc = lane >> 3;
  if (wg >= (long)Tg * MB * 4 * Qg) return;
  const int grp = (int)(wg & 3);
  const long rest0 = wg >> 2;
  const int ql = (int)(rest0 % Qg);
  const long rest = rest0 / Qg;
  const int mb = (int)(rest % MB), tl = (int)(rest / MB);
  const int kk = 8 * grp + (lane & 7), k = mb * 32 + kk;
  const GenRows load{k < N ? VT + (size_t)tl * K * N + k : nullptr, (size_t)N, K};
  const int kappa0 = (q0 + ql) * CK + 4 * kc;
  const int e = group_exponent(load, kappa0);
  if (kc == 0) {
    eB[((size_t)(tl * MB + mb) * Qg + ql) * TN + kk] = e;
    eB[((size_t)(tl * MB + mb) * Qg + ql) * TN + 32 + kk] = e;
    atomicMax(eBmax + (size_t)(tl * MB + mb) * TN + kk, e);
    atomicMax(eBmax + (size_t)(tl * MB + mb) * TN + 32 + kk, e);
  }
  uint8_t* out = Bs + (((size_t)(tl * MB + mb) * Qg + ql) * NBK * S) * B_TILE + (size_t)grp * SBO + lane * 16;
#pragma unroll 1
  for (int b = 0; b < NBK; b++) {
    float d[8][S];
#pragma unroll
    for (int u = 0; u < 4; u++) {
      const double2 v = load(kappa0 + b * (KB / 2) + u);
      digits(v.x, e, d[2 * u]);
      digits(conj_in ? -v.y : v.y, e, d[2 * u + 1]);
    }
#pragma unroll
    for (int s = 0; s < S; s++) {
      float v[8], w[8];
#pragma unroll
      for (int u = 0; u < 4; u++) {
        v[2 * u] = d[2 * u][s];
        v[2 * u + 1] = d[2 * u + 1][s];
        w[2 * u] = -d[2 * u + 1][s];
        w[2 * u + 1] = d[2 * u][s];
      }
      *(uint4*)(out + (size_t)(b * S + s) * B_TILE) = pack8(v);
      *(uint4*)(out + (size_t)(b * S + s) * B_TILE + 4 * SBO) = pack8(w);
    }
  }
}

__global__ void k_fill_int(int* p, size_t n, int v) {
  const size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e < n) p[e] = v;
}

// Tile (row block rt, mode block mb, timeslice tl) over a share of the group's chunks.
// Bound by the MMAs (8192 FLOP per clock and SM) and, not overlapped with them, the
// epilogue's reading of the six classes after every chunk (two class sets do not fit
// in TMEM).  40 right-hand sides, 32 modes, 16^3 x 32: 2.76 ms with 36 products of 6-bit
// digits in N = 64 instructions on 64 blocks; 1.49 ms with 21 products of 8-bit digits;
// 0.53 ms with the digits of B side by side and 7 blocks per tile (chunk_split).
// Warp 0: bulk copies; warp 1: TMEM and MMAs; warps 2..9: epilogue (warp w reads
// TMEM lanes 32 (w % 4) .. + 31 and columns 32 ((w - 2) / 4) .. + 31).
__global__ void __launch_bounds__(320, 1) k_proj_mma(const uint8_t* __restrict__ As, const uint8_t* __restrict__ Bs,
                                                     const int* __restrict__ eA, const int* __restrict__ eB,
                                                     const int* __restrict__ eAmax, const int* __restrict__ eBmax,
                                                     int Qg, int RT, int MB, int R, int N, int Tsel, int ksplit,
                                                     int accumulate, double* coeff, size_t part_stride, int* err,
                                                     int omode = 0) {
  extern __shared__ __align__(1024) uint8_t smem[];
  __shared__ __align__(8) uint64_t full[NST], empty[NST], accf, acce, drain;
  __shared__ uint32_t tbase;
  __shared__ int abort_flag;
  __shared__ int ref_b[TN];     // reference exponents of the tile's columns
  const auto sA = [&](int st) { return smem + st * STAGE_A; };
  const auto sB = [&](int st) { return smem + NST * STAGE_A + st * STAGE_B; };
  const auto sE = [&](int q) { return (int*)(smem + NST * (STAGE_A + STAGE_B) + (q & 1) * EXP_BYTES); };
  const int rt = blockIdx.x, mb = blockIdx.y, tl = blockIdx.z / ksplit, part = blockIdx.z - tl * ksplit;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // this block's chunks: qb .. qb + nq - 1 of the group's Qg
  const int qb = (int)((long)Qg * part / ksplit), nq = (int)((long)Qg * (part + 1) / ksplit) - qb;
  const int nstages = nq * NBK;

  if (threadIdx.x == 0) {
    for (int s = 0; s < NST; s++) {
      tc::mbar_init(&full[s], 1);
      tc::mbar_init(&empty[s], 1);
    }
    tc::mbar_init(&accf, 1);
    tc::mbar_init(&acce, 8);
    tc::mbar_init(&drain, 1);
    abort_flag = 0;
    tc::mbar_fence_init();
  }
  if (threadIdx.x < TN) ref_b[threadIdx.x] = eBmax[(size_t)(tl * MB + mb) * TN + threadIdx.x];
  if (warp == 1) tc::tmem_alloc(&tbase, 512);
  tc::fence_before();
  __syncthreads();
  tc::fence_after();
  const uint32_t tmem = tbase;

  if (warp == 0) {
    // ---- producer ----
    if (lane == 0) {
      int issued = 0;
      for (int it = 0; it < nstages; it++) {
        if (abort_flag) break;
        const int st = it % NST, use = it / NST;
        if (it >= NST && !tc::mbar_wait(&empty[st], (use - 1) & 1, WAIT_LIMIT)) {
          abort_flag = 1;
          atomicExch(err, 1);
          break;
        }
        const int ql = it / NBK, b = it % NBK, qg = qb + ql;
        const size_t ta = (((size_t)(tl * RT + rt) * Qg + qg) * NBK + b) * S;
        const size_t tb = (((size_t)(tl * MB + mb) * Qg + qg) * NBK + b) * S;
        const uint32_t bytes = STAGE_A + STAGE_B + (b == 0 ? EXP_BYTES : 0);
        tc::mbar_arrive_expect_tx(&full[st], bytes);
        tc::bulk_g2s(sA(st), As + ta * A_TILE, STAGE_A, &full[st]);
        tc::bulk_g2s(sB(st), Bs + tb * B_TILE, STAGE_B, &full[st]);
        if (b == 0) {
          tc::bulk_g2s(sE(ql), eA + ((size_t)(tl * RT + rt) * Qg + qg) * TM, TM * 4, &full[st]);
          tc::bulk_g2s(sE(ql) + TM, eB + ((size_t)(tl * MB + mb) * Qg + qg) * TN, TN * 4, &full[st]);
        }
        issued = it + 1;
      }
      // copies still in flight land before the shared memory is given up
      for (int it = issued - NST < 0 ? 0 : issued - NST; it < issued; it++)
        tc::mbar_wait(&full[it % NST], (it / NST) & 1, WAIT_LIMIT);
    }
  } else if (warp == 1) {
    // ---- MMA issue ----
    if (lane == 0) {
      for (int it = 0; it < nstages; it++) {
        const int st = it % NST, use = it / NST;
        const int ql = it / NBK, b = it % NBK;
        if (abort_flag) break;
        if (b == 0 && ql > 0 && !tc::mbar_wait(&acce, (ql - 1) & 1, WAIT_LIMIT)) {
          abort_flag = 1;
          atomicExch(err, 1);
          break;
        }
        if (!tc::mbar_wait(&full[st], use & 1, WAIT_LIMIT)) {
          abort_flag = 1;
          atomicExch(err, 1);
          break;
        }
        tc::fence_after();
        const uint32_t a0 = tc::smem_addr(sA(st)), b0 = tc::smem_addr(sB(st));
#pragma unroll
        for (int ks = 0; ks < KB / 16; ks++)
#pragma unroll
          for (int i = 0; i < S; i++) {
            // digit i of A against digits j0 .. j0 + nd - 1 of B: classes i + j0 .. (the
            // digit tiles of B follow one another at eight SBO strides)
            const uint64_t ad = tc::smem_desc(a0 + i * A_TILE + ks * 256, LBO, SBO);
#pragma unroll
            for (int j0 = 0; j0 < S - i; j0 += 4) {
              const int nd = S - i - j0 < 4 ? S - i - j0 : 4;
              const uint64_t bd = tc::smem_desc(b0 + j0 * B_TILE + ks * 256, LBO, SBO);
              const uint32_t acc = (b == 0 && ks == 0 && i == 0) ? 0u : 1u;
              tc::mma_bf16(tmem + (i + j0) * TN, ad, bd, tc::idesc_bf16_f32(TM, nd * TN), acc);
            }
          }
        tc::mma_commit(&empty[st]);                   // the stage may be refilled
        if (b == NBK - 1) tc::mma_commit(&accf);      // chunk complete: classes ready
      }
      // every MMA issued has completed before TMEM is read for the last time / freed
      tc::mma_commit(&drain);
      tc::mbar_wait(&drain, 0, WAIT_LIMIT);
    }
  } else {
    // ---- epilogue: double-float accumulation of the scaled class sums ----
    const int quarter = warp & 3, half = (warp - 2) >> 2;
    const int row = quarter * 32 + lane;
    // reference exponents of the row and the columns: the float accumulator holds the
    // sum relative to 2^(ra + rb), restored in FP64 at the end
    const int ra = eAmax[(size_t)tl * RT * TM + rt * TM + row];
    const int* rb = ref_b + half * 32;
    float hi[32], lo[32];
#pragma unroll
    for (int n = 0; n < 32; n++) hi[n] = lo[n] = 0.f;
    for (int ql = 0; ql < nq; ql++) {
      if (!tc::mbar_wait(&accf, ql & 1, WAIT_LIMIT)) {
        abort_flag = 1;
        atomicExch(err, 1);
        break;
      }
      tc::fence_after();
      const int ea = sE(ql)[row];
      const int* eb = sE(ql) + TM + half * 32;
      float sc[32];
#pragma unroll
      for (int n = 0; n < 32; n++) sc[n] = pow2f((ea - ra) + (eb[n] - rb[n]) - 14);
#pragma unroll 1
      for (int c = 0; c < NCLS; c++) {
        uint32_t r[32];
        tc::tmem_ld32(tmem + ((uint32_t)(quarter * 32) << 16) + c * TN + half * 32, r);
        tc::tmem_wait_ld();
        const float w = __int_as_float((127 - 8 * c) << 23);      // 2^(-8 c)
#pragma unroll
        for (int n = 0; n < 32; n++) {
          const float v = (__uint_as_float(r[n]) * w) * sc[n];    // powers of two: exact
          const float s = hi[n] + v;
          const float bp = s - hi[n];
          lo[n] += (hi[n] - (s - bp)) + (v - bp);
          hi[n] = s;
        }
      }
      tc::fence_before();
      __syncwarp();
      if (lane == 0) tc::mbar_arrive(&acce);
    }
    const int grow = rt * TM + row;
    if (!abort_flag && grow < R) {
      const int j = grow / 4, alpha = grow % 4;
#pragma unroll
      for (int n = 0; n < 32; n++) {
        const int k = mb * 32 + n;
        if (k >= N) break;
        // omode 0: coeff[j][t][alpha][k]; 1: out[t][k][row]; 2: out[t][row][k]
        const size_t idx = omode == 0 ? (((size_t)j * Tsel + tl) * 4 + alpha) * N + k
                           : omode == 1 ? ((size_t)tl * N + k) * R + grow
                                        : ((size_t)tl * R + grow) * N + k;
        double* o = coeff + part * part_stride + 2 * idx + half;
        const double v = ldexp((double)hi[n] + (double)lo[n], ra + rb[n]);
        *o = accumulate ? *o + v : v;
      }
    }
  }
  tc::fence_before();
  __syncthreads();
  if (warp == 1) {
    tc::fence_after();
    tc::tmem_dealloc(tmem, 512);
  }
}

// out = sum of the ks partial results, in their order
__global__ void k_sum_parts(const double* __restrict__ part, size_t n, int ks, double* out) {
  const size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= n) return;
  double s = part[e];
  for (int k = 1; k < ks; k++) s += part[(size_t)k * n + e];
  out[e] = s;
}

// blocks that share one output tile by splitting its chunks: enough that the tiles fill
// the SMs (one block each) without a nearly empty last wave, at least 8 chunks per block
// (its pipeline's start and end cost about two)
int chunk_split(long tiles, int Q) {
  int best = 1;
  double cost = 1e300;
  for (int ks = 1; ks <= 16 && Q / ks >= 8; ks++) {
    const long waves = (tiles * ks + 151) / 152;
    const double c = (double)waves * ((Q + ks - 1) / ks + 2);
    if (c < 0.97 * cost) { cost = c; best = ks; }
  }
  return best;
}

}  // namespace

// How run_products works: chunk groups, blocks per tile and the bytes of its work buffers
struct Plan {
  int Q, RT, MB, Qg, ks;
  size_t a, b, e, p;             // WS_TC_A, WS_TC_B, WS_TC_E, WS_TC_P
};
static Plan make_plan(const dlma_ctx* ctx, int T, int R, int N, int K, size_t out_count) {
  Plan P;
  P.Q = (K + CK - 1) / CK;
  P.RT = (R + TM - 1) / TM;
  P.MB = (N + 31) / 32;
  // digit bytes per chunk of every timeslice: A (RT tiles of rows) and B (MB tiles of modes)
  const size_t per_chunk = (size_t)T * NBK * S * ((size_t)P.RT * A_TILE + (size_t)P.MB * B_TILE);
  size_t budget = (size_t)4 << 30;
  if (ctx->memcap) budget = std::min(budget, (size_t)ctx->memcap / 4);
  P.Qg = (int)std::max<size_t>(1, std::min<size_t>((size_t)P.Q, budget / per_chunk));
  P.Qg = (P.Q + (P.Q + P.Qg - 1) / P.Qg - 1) / ((P.Q + P.Qg - 1) / P.Qg);       // equal groups
  P.ks = chunk_split((long)T * P.RT * P.MB, P.Qg);
  // the partial results keep to a quarter of a memory cap, like the digits
  if (ctx->memcap) P.ks = (int)std::max<size_t>(1, std::min<size_t>(P.ks, ctx->memcap / 4 / (out_count * 16)));
  P.a = (size_t)T * P.RT * P.Qg * NBK * S * A_TILE;
  P.b = (size_t)T * P.MB * P.Qg * NBK * S * B_TILE;
  P.e = (size_t)T * (P.Qg + 1) * (P.RT * TM + P.MB * TN) * sizeof(int);
  P.p = P.ks > 1 ? (size_t)P.ks * out_count * 16 : 0;
  return P;
}

// Shared by the projection and the eigensolver's block products: digit buffers, the
// chunk groups and the products; slice_a launches the row slicer.
template <class SliceA>
static dlma_status run_products(dlma_ctx* ctx, int T, int R, int N, int K, const double2* b_src, int b_conj, int omode,
                                double2* out, size_t out_count, const char* what, const SliceA& slice_a) {
  const Plan P = make_plan(ctx, T, R, N, K, out_count);
  const int Q = P.Q, RT = P.RT, MB = P.MB, Qg = P.Qg, ks = P.ks;
  uint8_t *As, *Bs;
  int *eA, *eB;
  TRY(workT(ctx, WS_TC_A, P.a, &As));
  TRY(workT(ctx, WS_TC_B, P.b, &Bs));
  TRY(workT(ctx, WS_TC_E, P.e / sizeof(int), &eA));
  eB = eA + (size_t)T * Qg * RT * TM;
  int* eAmax = eB + (size_t)T * Qg * MB * TN;
  int* eBmax = eAmax + (size_t)T * RT * TM;
  const size_t nref = (size_t)T * (RT * TM + MB * TN);
  double* parts = (double*)out;
  if (ks > 1) TRY(workT(ctx, WS_TC_P, P.p / sizeof(double), &parts));
  int* err = ctx->flag + 8;
  CU(cudaMemsetAsync(err, 0, sizeof(int), ctx->stream));
  static bool attr_set[64] = {false};
  if (ctx->device >= 0 && ctx->device < 64 && !attr_set[ctx->device]) {
    CU(cudaFuncSetAttribute(k_proj_mma, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_BYTES));
    attr_set[ctx->device] = true;
  }
  for (int q0 = 0; q0 < Q; q0 += Qg) {
    const int qn = std::min(Qg, Q - q0);
    const int kq = std::min(ks, qn);        // the last group may hold fewer chunks
    const long wa = (long)T * RT * (TM / 8) * qn, wb = (long)T * MB * 4 * qn;
    k_fill_int<<<(unsigned)((nref + 255) / 256), 256, 0, ctx->stream>>>(eAmax, nref, kExpZero);
    CHECK_LAUNCH();
    slice_a((unsigned)((wa + 3) / 4), q0, qn, RT, As, eA, eAmax);
    CHECK_LAUNCH();
    k_slice_modes<<<(unsigned)((wb + 3) / 4), 128, 0, ctx->stream>>>(b_src, N, K, T, q0, qn, MB, Bs, eB, eBmax, b_conj);
    CHECK_LAUNCH();
    // partial results beyond this group's kq keep their sums of the earlier groups
    k_proj_mma<<<dim3(RT, MB, T * kq), 320, SMEM_BYTES, ctx->stream>>>(As, Bs, eA, eB, eAmax, eBmax, qn, RT, MB, R, N, T,
                                                                      kq, q0 > 0 ? 1 : 0, parts, 2 * out_count, err,
                                                                      omode);
    CHECK_LAUNCH();
  }
  if (ks > 1) {
    k_sum_parts<<<(unsigned)((2 * out_count + 255) / 256), 256, 0, ctx->stream>>>(parts, 2 * out_count, ks, (double*)out);
    CHECK_LAUNCH();
  }
  int h = 0;
  CU(cudaMemcpyAsync(&h, err, sizeof(int), cudaMemcpyDeviceToHost, ctx->stream));
  CU(cudaStreamSynchronize(ctx->stream));
  if (h) return set_err(ctx, DLMA_ERR_CUDA, "%s: a pipeline wait timed out", what);
  return DLMA_OK;
}

// coeff[j][Tsel][4][N] = V^dag psi on the tensor cores (see the top of the file);
// VT [Tsel][3 Vs][N] (mode fastest), psi canonical with stride_sites per rhs,
// timeslices site_t0 .. site_t0 + Tsel - 1.  The digit buffers are bounded: the
// chunks of kappa run in groups whose results accumulate in FP64 in coeff.
dlma_status project_tc(dlma_ctx* ctx, const double2* VT, int N, int Tsel, const double* psi, size_t stride_sites,
                       int site_t0, int nrhs, double2* coeff) {
  const int Vs = ctx->g.Vs, K = 3 * Vs;
  return run_products(ctx, Tsel, 4 * nrhs, N, K, VT, 0, 0, coeff, (size_t)nrhs * Tsel * 4 * N,
                      "tensor-core projection",
                      [&](unsigned nb, int q0, int qn, int RT, uint8_t* As, int* eA, int* eAmax) {
                        k_slice_psi<<<nb, 128, 0, ctx->stream>>>((const double2*)psi, stride_sites, site_t0, Vs, Tsel,
                                                                 nrhs, K, q0, qn, RT, As, eA, eAmax);
                      });
}

// bytes of the digit buffers of R rows, N modes and one chunk on T timeslices (the least
// that run_products works with)
size_t tc_min_bytes(int R, int N, int T) {
  return (size_t)T * NBK * S * ((size_t)((R + TM - 1) / TM) * A_TILE + (size_t)((N + 31) / 32) * B_TILE);
}

// device memory that the products below of n x m blocks on T timeslices (Gram matrices and
// rotations) add to the work buffers held
size_t tc_block_bytes(const dlma_ctx* ctx, int n, int m, int T) {
  const Plan G = make_plan(ctx, T, m, m, n, (size_t)T * m * m), Z = make_plan(ctx, T, n, m, m, (size_t)T * n * m);
  const auto grow = [&](int slot, size_t g, size_t z) {
    const size_t need = std::max(g, z), held = ctx->wb[slot].bytes;
    return need > held ? need - held : 0;
  };
  return grow(WS_TC_A, G.a, Z.a) + grow(WS_TC_B, G.b, Z.b) + grow(WS_TC_E, G.e, Z.e) + grow(WS_TC_P, G.p, Z.p);
}

// Block products of the eigensolver's FP64 phase on the tensor cores, with the same
// FP64-accurate digit scheme.  For every timeslice t:
//   out[t] (omode 1: [N][R], omode 2: [R][N]) holds sum_kappa conj(B_k(kappa)) A_r(kappa)
// with A_r(kappa) = a_src[t a_st + r a_sr + kappa a_sk] (R rows, K long) and
// B_k(kappa) = b_src[(t K + kappa) N + k] (conjugated first when b_conj).
dlma_status tc_block_product(dlma_ctx* ctx, int omode, const double2* a_src, size_t a_st, size_t a_sr, size_t a_sk,
                             int R, const double2* b_src, int b_conj, int N, int K, int T, double2* out) {
  if (omode != 1 && omode != 2) return set_err(ctx, DLMA_ERR_INVALID_ARG, "tc_block_product mode");
  return run_products(ctx, T, R, N, K, b_src, b_conj, omode, out, (size_t)T * R * N, "tensor-core block product",
                      [&](unsigned nb, int q0, int qn, int RT, uint8_t* As, int* eA, int* eAmax) {
                        k_slice_agen<<<nb, 128, 0, ctx->stream>>>(a_src, a_st, a_sr, a_sk, T, R, K, q0, qn, RT, As, eA,
                                                                  eAmax);
                      });
}
