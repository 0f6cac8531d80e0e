// Spatial covariant Laplacian of Eq. 1 and its low modes, batched over
// timeslices.
//
//   (lap v)(m, t) = -6 v(m) + sum_{j=1..3} [U_j(m,t) v(m+j) + U_j(m-j,t)^dag v(m-j)]
//
// The modes are the N lowest eigenpairs of A = -lap(t) (spectrum in [0, 12]) on
// every timeslice at once, by Chebyshev-filtered subspace iteration on a block
// of m = N + buffer vectors per timeslice.  Each iteration filters the block
// with a degree-d Chebyshev polynomial of A that damps [cut, 12] and then
// diagonalises it per timeslice (Rayleigh-Ritz):
//   G = Y^dag Y, H = Y^dag (A Y)  ->  G = Q diag(g) Q^dag, S = Q g^-1/2,
//   S^dag H S = Z diag(theta) Z^dag,  X <- Y S Z,  A X <- (A Y) S Z,
// with the small m x m eigenproblems solved by parallel cyclic Jacobi in the
// block's precision (smalleig.cuh; one CTA per timeslice).
//
// Precision: phase A runs the whole iteration in FP32 until the residuals reach
// ~1e-5.  Phase B keeps X, A X and the Rayleigh-Ritz in FP64 but still filters
// in FP32, on the residual: with R = A X - X Theta and the filter's scalar
// recurrence s_k(theta), p_k(A) X = X s_k(Theta) + E_k where
//   E_{k+1} = a_k A E_k + b_k E_k + c_k E_{k-1} + a_k R s_k(Theta),  E_0 = 0,
// so the FP32 rounding only touches the (small) E, and Y = X + E_d / s_d (the
// filtered block with every column divided by its own s_d, so that the Gram
// matrix stays well conditioned) is formed in FP64.  Stops when every wanted
// pair has ||A x - theta x|| <= tol max(theta, 1).  For tol >= 1e-11 the FP64
// blocks' Gram matrices and rotations compute in double-float (~46 bits,
// dfloat.cuh) on the FP32 units or, for large blocks, with the split-digit
// products of tcproj.cu on the tensor cores; the matvec and the small problems
// stay FP64.
//
// Block layout (row-major per timeslice): element (t, row r = 3 site + colour,
// column j) of a batch of Tn timeslices at (t * 3 Vs + r) * m + j, so a warp
// reads consecutive columns of one site (coalesced) and shares its links.
#include "common.cuh"
#include "dfloat.cuh"
#include "smalleig.cuh"
#include <algorithm>
#include <math.h>

namespace {

__device__ __forceinline__ void load_link3(const double2* __restrict__ U, int k, size_t s, size_t V, Cx<double> u[3][3]) {
#pragma unroll
  for (int q = 0; q < 9; q++) {
    double2 e = __ldg(U + ((size_t)k * 9 + q) * V + s);
    u[q / 3][q % 3] = cx<double>(e.x, e.y);
  }
}
// all 18 reals: the load is shared by the columns of a site, rebuilding the third row
// would cost each thread 24 operations
__device__ __forceinline__ void load_link3(const float4* __restrict__ U, int k, size_t s, size_t V, Cx<float> u[3][3]) {
#pragma unroll
  for (int q = 0; q < 5; q++) {
    const float4 e = __ldg(U + ((size_t)k * 5 + q) * V + s);
    u[(2 * q) / 3][(2 * q) % 3] = cx<float>(e.x, e.y);
    if (2 * q + 1 < 9) u[(2 * q + 1) / 3][(2 * q + 1) % 3] = cx<float>(e.z, e.w);
  }
}

// NC adjacent complex entries starting at p (16-byte aligned when NC is even): FP32
// pairs move as one 128-bit access
template <int NC>
__device__ __forceinline__ void ld_cols(const Cx<float>* __restrict__ p, Cx<float> (&v)[NC]) {
#pragma unroll
  for (int c = 0; c < NC; c += 2) {
    const float4 e = *(const float4*)(p + c);
    v[c] = cx<float>(e.x, e.y);
    v[c + 1] = cx<float>(e.z, e.w);
  }
}
template <int NC>
__device__ __forceinline__ void st_cols(Cx<float>* p, const Cx<float> (&v)[NC]) {
#pragma unroll
  for (int c = 0; c < NC; c += 2) *(float4*)(p + c) = make_float4(v[c].re, v[c].im, v[c + 1].re, v[c + 1].im);
}
// storage (R) <-> arithmetic (A) precision: A = R, or A = df for FP64 storage (the
// double-float arithmetic of the FP64 phase, see dfloat.cuh)
template <class A, class R> __device__ __forceinline__ Cx<A> to_a(Cx<R> v) { return cx<A>((A)v.re, (A)v.im); }
template <class R, class A> __device__ __forceinline__ Cx<R> to_s(Cx<A> v) { return cx<R>((R)v.re, (R)v.im); }

// out = A in, A = 6 - hopping = -lap, in FP64: one thread per (site, column); the block is
// [t][site][colour][m].  Bound by FP64 arithmetic (about 250 instructions per entry).
__global__ void __launch_bounds__(256, 2) k_lap(Geom g, int t0, int Tn, int m, const double2* __restrict__ U,
                                                const Cx<double>* __restrict__ in, Cx<double>* __restrict__ out) {
  // 32-bit index arithmetic (the host keeps Tn Vs m below 2^31): 64-bit divisions
  // would cost more than the stencil's arithmetic
  const unsigned e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= (unsigned)Tn * (unsigned)g.Vs * (unsigned)m) return;
  const unsigned sl = e / (unsigned)m;
  const int j0 = (int)(e - sl * (unsigned)m);
  const int tl = (int)(sl / (unsigned)g.Vs);
  const int ms = (int)(sl - (unsigned)tl * (unsigned)g.Vs);
  const size_t rowbase = (size_t)tl * g.Vs;
  const int yz = ms / g.L, x = ms - yz * g.L, z = yz / g.L, y = yz - z * g.L;
  const size_t s = (size_t)(t0 + tl) * g.Vs + ms;
  Cx<double> h[3];
#pragma unroll
  for (int a = 0; a < 3; a++) h[a] = cx<double>(0, 0);
#pragma unroll
  for (int k = 0; k < 3; k++) {
    int xf = x, yf = y, zf = z, xb = x, yb = y, zb = z;
    if (k == 0) { xf = x + 1 == g.L ? 0 : x + 1; xb = x == 0 ? g.L - 1 : x - 1; }
    else if (k == 1) { yf = y + 1 == g.L ? 0 : y + 1; yb = y == 0 ? g.L - 1 : y - 1; }
    else { zf = z + 1 == g.L ? 0 : z + 1; zb = z == 0 ? g.L - 1 : z - 1; }
    const int mf = xf + g.L * (yf + g.L * zf), mb = xb + g.L * (yb + g.L * zb);
    Cx<double> uf[3][3], ub[3][3], vf[3], vb[3];
    load_link3(U, k, s, (size_t)g.V, uf);
    load_link3(U, k, (size_t)(t0 + tl) * g.Vs + mb, (size_t)g.V, ub);
#pragma unroll
    for (int a = 0; a < 3; a++) {
      vf[a] = in[((rowbase + mf) * 3 + a) * m + j0];
      vb[a] = in[((rowbase + mb) * 3 + a) * m + j0];
    }
#pragma unroll
    for (int a = 0; a < 3; a++)
#pragma unroll
      for (int b = 0; b < 3; b++) {
        fma_acc(h[a], uf[a][b], vf[b]);
        fma_conj_acc(h[a], ub[b][a], vb[b]);
      }
  }
#pragma unroll
  for (int a = 0; a < 3; a++) {
    const size_t e3 = ((rowbase + ms) * 3 + a) * m + j0;
    const Cx<double> v = in[e3];
    out[e3] = cx<double>(fma(6.0, v.re, -h[a].re), fma(6.0, v.im, -h[a].im));
  }
}

// FP32: out = alpha_t (A in) + beta_t in + gamma_t prev + alpha_t s[t][j] rin (prev and rin
// may be nullptr).
// Two columns per thread (m is even, so a pair is 16-byte aligned), marching along z: a
// thread keeps its column's sites z, z + 1 and the backward product U_z(z)^dag v(z) in
// registers, so every value is loaded once along z and each z link once; a block covers a
// patch of px x py sites of a plane, whose x and y neighbours meet in L1.  The plain form
// (k_lap: a row of sites per block) moved 6.5 vectors per application from L2 to the SMs
// (0.215 ms for a block of 16^3 x 32 with 64 columns, 2.12 for 24^3 x 48 with 128); this
// one moves about 3.5 and takes 0.184 and 1.68 ms, bound by instruction issue (some 560
// per site and column pair; DRAM floor 0.09, 0.92).  With 12-real links, whose third row
// each thread rebuilds, and separate sums per direction it took 0.196 and 1.87.
// Block: pw column pairs x (px py) sites; grid: (patches of a plane x z segments x column
// groups, timeslices).
struct LapTiling {
  int pw, px, py, groups, nx, ny, nz, zlen;
};
__global__ void __launch_bounds__(256, 2) k_lap_z(Geom g, int t0, int m, LapTiling L, const float4* __restrict__ U,
                                                  const Cx<float>* __restrict__ in, const Cx<float>* __restrict__ prev,
                                                  const Cx<float>* __restrict__ rin, const double* __restrict__ scol,
                                                  Cx<float>* __restrict__ out, const double* __restrict__ coef) {
  const int tl = blockIdx.y;
  int b = blockIdx.x;
  const int grp = b % L.groups;
  b /= L.groups;
  const int bx = b % L.nx;
  b /= L.nx;
  const int by = b % L.ny, bz = b / L.ny;
  const int site = threadIdx.x / L.pw, pair = grp * L.pw + (threadIdx.x - site * L.pw);
  const int x = bx * L.px + site % L.px, y = by * L.py + site / L.px;
  if (site >= L.px * L.py || x >= g.L || y >= g.L || 2 * pair >= m) return;
  const int z0 = bz * L.zlen, z1 = min(g.L, z0 + L.zlen);
  const int j0 = 2 * pair, plane = g.L * g.L;
  const float alpha = (float)coef[3 * tl], gamma = (float)coef[3 * tl + 2];
  const size_t row0 = (size_t)tl * g.Vs;                   // first site of the block's timeslice
  const size_t s0 = (size_t)(t0 + tl) * g.Vs;              // ... and of the links'
  const int xf = x + 1 == g.L ? 0 : x + 1, xb = x == 0 ? g.L - 1 : x - 1;
  const int yf = y + 1 == g.L ? 0 : y + 1, yb = y == 0 ? g.L - 1 : y - 1;
  const int o = x + g.L * y, oxb = xb + g.L * y, oyb = x + g.L * yb;
  const int nbr[4] = {xf + g.L * y, oxb, x + g.L * yf, oyb};
  float fr0 = 0, fr1 = 0;
  if (rin) {
    fr0 = alpha * (float)scol[(size_t)tl * m + j0];
    fr1 = alpha * (float)scol[(size_t)tl * m + j0 + 1];
  }
  const auto load = [&](const Cx<float>* p, int ms, Cx<float>(&v)[3][2]) {
#pragma unroll
    for (int a = 0; a < 3; a++) ld_cols<2>(p + ((row0 + ms) * 3 + a) * m + j0, v[a]);
  };
  // w += U v, w += U^dag v
  const auto mul = [&](const Cx<float>(&u)[3][3], const Cx<float>(&v)[3][2], Cx<float>(&w)[3][2]) {
#pragma unroll
    for (int a = 0; a < 3; a++)
#pragma unroll
      for (int c = 0; c < 2; c++)
#pragma unroll
        for (int q = 0; q < 3; q++) fma_acc(w[a][c], u[a][q], v[q][c]);
  };
  const auto dag_mul = [&](const Cx<float>(&u)[3][3], const Cx<float>(&v)[3][2], Cx<float>(&w)[3][2]) {
#pragma unroll
    for (int a = 0; a < 3; a++)
#pragma unroll
      for (int c = 0; c < 2; c++)
#pragma unroll
        for (int q = 0; q < 3; q++) fma_conj_acc(w[a][c], u[q][a], v[q][c]);
  };
  const float b6 = (float)(6.0 * coef[3 * tl] + coef[3 * tl + 1]);
  // hop: the sum of the six hopping terms, started with the backward z one
  Cx<float> cur[3][2], hop[3][2];
#pragma unroll
  for (int a = 0; a < 3; a++) hop[a][0] = hop[a][1] = cx<float>(0, 0);
  {
    const int zb = z0 == 0 ? g.L - 1 : z0 - 1;
    Cx<float> u[3][3], v[3][2];
    load_link3(U, 2, s0 + o + (size_t)plane * zb, (size_t)g.V, u);
    load(in, o + plane * zb, v);
    dag_mul(u, v, hop);
    load(in, o + plane * z0, cur);
  }
  for (int z = z0; z < z1; z++) {
    const int zo = plane * z, zf = plane * (z + 1 == g.L ? 0 : z + 1);
    Cx<float> nxt[3][2], wz[3][2];
    load(in, o + zf, nxt);
    {
      Cx<float> u[3][3];
      load_link3(U, 2, s0 + o + zo, (size_t)g.V, u);
      mul(u, nxt, hop);
#pragma unroll
      for (int a = 0; a < 3; a++) wz[a][0] = wz[a][1] = cx<float>(0, 0);
      dag_mul(u, cur, wz);
    }
#pragma unroll
    for (int k = 0; k < 2; k++) {
      Cx<float> u[3][3], v[3][2];
      load_link3(U, k, s0 + o + zo, (size_t)g.V, u);
      load(in, nbr[2 * k] + zo, v);
      mul(u, v, hop);
      load_link3(U, k, s0 + (k == 0 ? oxb : oyb) + zo, (size_t)g.V, u);
      load(in, nbr[2 * k + 1] + zo, v);
      dag_mul(u, v, hop);
    }
#pragma unroll
    for (int a = 0; a < 3; a++) {
      const size_t idx = ((row0 + o + zo) * 3 + a) * m + j0;
      Cx<float> r[2];
#pragma unroll
      for (int c = 0; c < 2; c++) r[c] = b6 * cur[a][c];
      if (prev) {
        Cx<float> pv[2];
        ld_cols<2>(prev + idx, pv);
#pragma unroll
        for (int c = 0; c < 2; c++) r[c] = add_s(r[c], gamma, pv[c]);
      }
      if (rin) {
        Cx<float> rv[2];
        ld_cols<2>(rin + idx, rv);
        r[0] = add_s(r[0], fr0, rv[0]);
        r[1] = add_s(r[1], fr1, rv[1]);
      }
#pragma unroll
      for (int c = 0; c < 2; c++) r[c] = add_s(r[c], -alpha, hop[a][c]);
      st_cols<2>(out + idx, r);
#pragma unroll
      for (int c = 0; c < 2; c++) {
        cur[a][c] = nxt[a][c];
        hop[a][c] = wz[a][c];
      }
    }
  }
}

// tiling of k_lap_z: at most 32 column pairs per block; the patch that loads the fewest
// halo sites and idle threads; z segments of at least 4 planes so that the grid fills the
// GPU a few times, or the length whose waves of blocks (two resident per SM) march the
// fewest planes, a segment costing its planes and about 1.5 more at its ends, where that
// saves more than the 4 % to which this count is good.  Filter and FP64 stencil of one
// eigensolve, ms: 6^3 x 20 (80 blocks without segments, 2 planes for 6) 1.85 -> 1.49,
// 24^3 x 26 (780, 8 for 12) 72.2 -> 68.3, 16^3 x 12 (192, 6 for 4) 10.6 -> 10.3; 14^3 x 22
// (308) keeps 5 planes: the count puts 7 ahead by 2 %, the clock behind by 12 %.
static LapTiling lap_tiling(int L, int m, int Tn) {
  LapTiling best{};
  const int mg = m / 2, groups = (mg + 31) / 32, pw = (mg + groups - 1) / groups;
  double cost = 1e300;
  for (int px = 1; px <= 8; px++)
    for (int py = 1; py <= px; py++) {
      if (px * py * pw > 256) continue;
      const int nx = (L + px - 1) / px, ny = (L + py - 1) / py;
      const double loads = (double)(px * py + 2 * px + 2 * py) * nx * ny, threads = 256.0 / pw * nx * ny;
      const double c = loads + threads;
      if (c < cost) {
        cost = c;
        best = LapTiling{pw, px, py, groups, nx, ny, 1, L};
      }
    }
  const long blocks = (long)best.nx * best.ny * groups * Tn;
  const auto planes = [&](int zlen) { return (double)((blocks * ((L + zlen - 1) / zlen) + 303) / 304) * (zlen + 1.5); };
  const int fill = (int)std::max<long>(1, std::min<long>(L / 4, (4 * 304 + blocks - 1) / blocks));
  int zmin = L;
  for (int zlen = L - 1; zlen >= 1; zlen--)
    if (planes(zlen) < planes(zmin)) zmin = zlen;
  best.zlen = (L + fill - 1) / fill;
  if (planes(zmin) < 0.96 * planes(best.zlen)) best.zlen = zmin;
  best.nz = (L + best.zlen - 1) / best.zlen;
  return best;
}

// Gram partials: part[t][split][i][j] = sum_{k in chunk} conj(X_t[k][i]) Y_t[k][j]
// herm: the product is hermitian (X^dag X, or Y^dag A Y with A hermitian): only the
// tiles on and above the diagonal are computed, k_gram_reduce mirrors the rest
constexpr int GT = 32, GKS = 32;
template <class R, class A>
__global__ void __launch_bounds__(256) k_gram(const Cx<R>* __restrict__ X, const Cx<R>* __restrict__ Y, int n, int m,
                                              int nsplit, int herm, double2* part) {
  __shared__ Cx<A> xs[GKS][GT + 1];
  __shared__ Cx<A> ys[GKS][GT + 1];
  const int tiles_j = (m + GT - 1) / GT;
  int ti = blockIdx.x / tiles_j, tj = blockIdx.x % tiles_j;
  if (herm) {                 // blockIdx.x enumerates the pairs ti <= tj row by row
    int b = blockIdx.x;
    ti = 0;
    while (b >= tiles_j - ti) { b -= tiles_j - ti; ti++; }
    tj = ti + b;
  }
  const int i0 = ti * GT, j0 = tj * GT;
  const int split = blockIdx.y, t = blockIdx.z;
  const int chunk = (n + nsplit - 1) / nsplit;
  const int k0 = split * chunk, k1 = min(n, k0 + chunk);
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4, tid = threadIdx.x;
  const Cx<R>* Xt = X + (size_t)t * n * m;
  const Cx<R>* Yt = Y + (size_t)t * n * m;
  Cx<A> acc[2][2];
#pragma unroll
  for (int a = 0; a < 2; a++)
#pragma unroll
    for (int b = 0; b < 2; b++) acc[a][b] = cx<A>(0, 0);
  for (int kb = k0; kb < k1; kb += GKS) {
#pragma unroll
    for (int q = 0; q < (GKS * GT) / 256; q++) {
      const int e = tid + 256 * q;
      const int r = e / GT, c = e % GT;
      const int k = kb + r;
      Cx<R> vx = cx<R>(0, 0), vy = cx<R>(0, 0);
      if (k < k1) {
        if (i0 + c < m) vx = Xt[(size_t)k * m + i0 + c];
        if (j0 + c < m) vy = Yt[(size_t)k * m + j0 + c];
      }
      xs[r][c] = to_a<A>(vx);
      ys[r][c] = to_a<A>(vy);
    }
    __syncthreads();
#pragma unroll 8
    for (int r = 0; r < GKS; r++) {
      const Cx<A> x0 = xs[r][ty], x1 = xs[r][ty + 16], y0 = ys[r][tx], y1 = ys[r][tx + 16];
      fma_conj_acc(acc[0][0], x0, y0);
      fma_conj_acc(acc[0][1], x0, y1);
      fma_conj_acc(acc[1][0], x1, y0);
      fma_conj_acc(acc[1][1], x1, y1);
    }
    __syncthreads();
  }
#pragma unroll
  for (int a = 0; a < 2; a++)
#pragma unroll
    for (int b = 0; b < 2; b++) {
      const int i = i0 + ty + 16 * a, j = j0 + tx + 16 * b;
      if (i < m && j < m)
        part[(((size_t)t * nsplit + split) * m + i) * m + j] = make_double2((double)acc[a][b].re, (double)acc[a][b].im);
    }
}

// FP32 blocks: 64 x 64 output tiles, 4 x 4 entries per thread, so that 64 multiply-adds
// share four 128-bit shared loads (32 x 32 tiles with 2 x 2 entries were bound by shared
// memory: 6.8 ms for 24^3 x 48 with 128 columns, now 3.9; FP32 floor 2.6).  The next
// slab of 16 rows is loaded into registers while the current one is used.
constexpr int FT = 64, FK = 16;
__device__ __forceinline__ void ld4(const Cx<float>* __restrict__ p, bool on, int room, Cx<float> (&v)[4]) {
#pragma unroll
  for (int h = 0; h < 2; h++) {
    const float4 e = on && 2 * h < room ? __ldg((const float4*)(p + 2 * h)) : make_float4(0, 0, 0, 0);
    v[2 * h] = cx<float>(e.x, e.y);
    v[2 * h + 1] = cx<float>(e.z, e.w);
  }
}
__device__ __forceinline__ void sh4(const Cx<float>* p, Cx<float> (&v)[4]) {
#pragma unroll
  for (int h = 0; h < 2; h++) {
    const float4 e = *(const float4*)(p + 2 * h);
    v[2 * h] = cx<float>(e.x, e.y);
    v[2 * h + 1] = cx<float>(e.z, e.w);
  }
}
__device__ __forceinline__ void st4(Cx<float>* p, const Cx<float> (&v)[4]) {
#pragma unroll
  for (int h = 0; h < 2; h++)
    *(float4*)(p + 2 * h) = make_float4(v[2 * h].re, v[2 * h].im, v[2 * h + 1].re, v[2 * h + 1].im);
}
__global__ void __launch_bounds__(256) k_gram_f(const Cx<float>* __restrict__ X, const Cx<float>* __restrict__ Y, int n,
                                                int m, int nsplit, int herm, double2* part) {
  __shared__ __align__(16) Cx<float> xs[2][FK][FT], ys[2][FK][FT];
  const int tiles_j = (m + FT - 1) / FT;
  int ti = blockIdx.x / tiles_j, tj = blockIdx.x % tiles_j;
  if (herm) {                 // blockIdx.x enumerates the pairs ti <= tj row by row
    int b = blockIdx.x;
    ti = 0;
    while (b >= tiles_j - ti) { b -= tiles_j - ti; ti++; }
    tj = ti + b;
  }
  const int i0 = ti * FT, j0 = tj * FT;
  const int split = blockIdx.y, t = blockIdx.z;
  const int chunk = (n + nsplit - 1) / nsplit;
  const int k0 = split * chunk, k1 = min(n, k0 + chunk);
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  const Cx<float>* Xt = X + (size_t)t * n * m + i0 + 4 * tx;
  const Cx<float>* Yt = Y + (size_t)t * n * m + j0 + 4 * tx;
  const int rx = m - i0 - 4 * tx, ry = m - j0 - 4 * tx;     // columns left (m is even)
  Cx<float> acc[4][4];
#pragma unroll
  for (int a = 0; a < 4; a++)
#pragma unroll
    for (int b = 0; b < 4; b++) acc[a][b] = cx<float>(0, 0);
  Cx<float> vx[4], vy[4];
  ld4(Xt + (size_t)(k0 + ty) * m, k0 + ty < k1, rx, vx);
  ld4(Yt + (size_t)(k0 + ty) * m, k0 + ty < k1, ry, vy);
  for (int kb = k0, st = 0; kb < k1; kb += FK, st ^= 1) {
    st4(&xs[st][ty][4 * tx], vx);
    st4(&ys[st][ty][4 * tx], vy);
    __syncthreads();
    const int kn = kb + FK + ty;
    ld4(Xt + (size_t)kn * m, kn < k1, rx, vx);
    ld4(Yt + (size_t)kn * m, kn < k1, ry, vy);
#pragma unroll
    for (int r = 0; r < FK; r++) {
      Cx<float> xv[4], yv[4];
      sh4(&xs[st][r][4 * ty], xv);
      sh4(&ys[st][r][4 * tx], yv);
#pragma unroll
      for (int a = 0; a < 4; a++)
#pragma unroll
        for (int b = 0; b < 4; b++) fma_conj_acc(acc[a][b], xv[a], yv[b]);
    }
  }
#pragma unroll
  for (int a = 0; a < 4; a++)
#pragma unroll
    for (int b = 0; b < 4; b++) {
      const int i = i0 + 4 * ty + a, j = j0 + 4 * tx + b;
      if (i < m && j < m)
        part[(((size_t)t * nsplit + split) * m + i) * m + j] = make_double2((double)acc[a][b].re, (double)acc[a][b].im);
    }
}

__global__ void k_gram_reduce(const double2* part, int nsplit, int m, int Tn, int herm, int tile, double2* G) {
  const size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  const size_t per = (size_t)m * m;
  if (e >= per * Tn) return;
  const size_t t = e / per;
  const int i = (int)((e % per) / m), j = (int)(e % m);
  const bool mirror = herm && (i / tile) > (j / tile);    // tile below the diagonal: conj of (j, i)
  const size_t ij = mirror ? (size_t)j * m + i : (size_t)i * m + j;
  double2 s = make_double2(0, 0);
  for (int q = 0; q < nsplit; q++) {
    const double2 v = part[(t * nsplit + q) * per + ij];
    s.x += v.x;
    s.y += v.y;
  }
  if (mirror) s.y = -s.y;
  G[e] = s;
}

// rotation Z_t = X_t C_t (X_t n x m row-major, C_t m x m row-major FP64); 64 x 64 output tiles
constexpr int RT = 64, RL = 16;
template <class R, class A>
__global__ void __launch_bounds__(256) k_rotate(const Cx<R>* __restrict__ X, const double2* __restrict__ Cm, int n,
                                                int m, Cx<R>* __restrict__ Z) {
  __shared__ Cx<A> xs[RT][RL + 1];
  __shared__ Cx<A> cs[RL][RT + 1];
  const int t = blockIdx.z, k0 = blockIdx.x * RT, j0 = blockIdx.y * RT;
  const int tid = threadIdx.x, tr = tid >> 4, tc = tid & 15;
  const Cx<R>* Xt = X + (size_t)t * n * m;
  const double2* C = Cm + (size_t)t * m * m;
  Cx<A> acc[4][4];
#pragma unroll
  for (int a = 0; a < 4; a++)
#pragma unroll
    for (int b = 0; b < 4; b++) acc[a][b] = cx<A>(0, 0);
  for (int l0 = 0; l0 < m; l0 += RL) {
#pragma unroll
    for (int q = 0; q < (RT * RL) / 256; q++) {
      const int e = tid + 256 * q;
      const int r = e / RL, c = e % RL;
      const int k = k0 + r, l = l0 + c;
      xs[r][c] = (k < n && l < m) ? to_a<A>(Xt[(size_t)k * m + l]) : cx<A>(0, 0);
      const int r2 = e / RT, c2 = e % RT;
      const int l2 = l0 + r2, j2 = j0 + c2;
      double2 cv = (l2 < m && j2 < m) ? C[(size_t)l2 * m + j2] : make_double2(0, 0);
      cs[r2][c2] = cx<A>((A)cv.x, (A)cv.y);
    }
    __syncthreads();
#pragma unroll
    for (int l = 0; l < RL; l++) {
      Cx<A> xv[4], cv[4];
#pragma unroll
      for (int a = 0; a < 4; a++) xv[a] = xs[tr + 16 * a][l];
#pragma unroll
      for (int b = 0; b < 4; b++) cv[b] = cs[l][tc + 16 * b];
#pragma unroll
      for (int a = 0; a < 4; a++)
#pragma unroll
        for (int b = 0; b < 4; b++) fma_acc(acc[a][b], xv[a], cv[b]);
    }
    __syncthreads();
  }
  Cx<R>* Zt = Z + (size_t)t * n * m;
#pragma unroll
  for (int a = 0; a < 4; a++)
#pragma unroll
    for (int b = 0; b < 4; b++) {
      const int k = k0 + tr + 16 * a, j = j0 + tc + 16 * b;
      if (k < n && j < m) Zt[(size_t)k * m + j] = to_s<R>(acc[a][b]);
    }
}

// FP32 blocks: the same 64 x 64 tiles as k_gram_f (5.95 ms for 24^3 x 48 with 128 columns
// with scalar shared loads and C converted from FP64 at every use, now 5.2; FP32 floor 3.5)
__global__ void __launch_bounds__(256) k_rotate_f(const Cx<float>* __restrict__ X, const Cx<float>* __restrict__ Cm,
                                                  int n, int m, Cx<float>* __restrict__ Z) {
  __shared__ __align__(16) Cx<float> xs[2][FK][FT + 2], cs[2][FK][FT];     // xs transposed: [l][k]
  const int t = blockIdx.z, k0 = blockIdx.x * FT, j0 = blockIdx.y * FT;
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  const int xr = threadIdx.x >> 2, xl = (threadIdx.x & 3) * 4;             // this thread's row and columns of X
  const Cx<float>* Xt = X + ((size_t)t * n + k0 + xr) * m + xl;
  const Cx<float>* C = Cm + (size_t)t * m * m + j0 + 4 * tx;
  const bool xon = k0 + xr < n;
  Cx<float> acc[4][4];
#pragma unroll
  for (int a = 0; a < 4; a++)
#pragma unroll
    for (int b = 0; b < 4; b++) acc[a][b] = cx<float>(0, 0);
  Cx<float> vx[4], vc[4];
  const auto fetch = [&](int l0) {
    ld4(Xt + l0, xon, m - l0 - xl, vx);
    ld4(C + (size_t)(l0 + ty) * m, l0 + ty < m, m - j0 - 4 * tx, vc);
  };
  fetch(0);
  for (int l0 = 0, st = 0; l0 < m; l0 += FK, st ^= 1) {
#pragma unroll
    for (int q = 0; q < 4; q++) xs[st][xl + q][xr] = vx[q];
    st4(&cs[st][ty][4 * tx], vc);
    __syncthreads();
    fetch(l0 + FK);
#pragma unroll
    for (int l = 0; l < FK; l++) {
      Cx<float> xv[4], cv[4];
      sh4(&xs[st][l][4 * ty], xv);
      sh4(&cs[st][l][4 * tx], cv);
#pragma unroll
      for (int a = 0; a < 4; a++)
#pragma unroll
        for (int b = 0; b < 4; b++) fma_acc(acc[a][b], xv[a], cv[b]);
    }
  }
#pragma unroll
  for (int a = 0; a < 4; a++) {
    const int k = k0 + 4 * ty + a;
    if (k >= n) continue;
    Cx<float>* z = Z + ((size_t)t * n + k) * m + j0 + 4 * tx;
#pragma unroll
    for (int h = 0; h < 2; h++)
      if (j0 + 4 * tx + 2 * h < m)
        *(float4*)(z + 2 * h) = make_float4(acc[a][2 * h].re, acc[a][2 * h].im, acc[a][2 * h + 1].re,
                                            acc[a][2 * h + 1].im);
  }
}

// residual norms res[t][j] = ||W_j - theta_j X_j||; optionally R = W - X Theta stored in
// FP32.  Bound by memory: the rows of a timeslice are shared out over blockIdx.z (one
// block per 32 columns and timeslice kept 64 of 152 SMs busy: 0.51 ms for an FP32 block
// of 16^3 x 32, 64 columns, now
// 0.07), with the partial sums in part[t][z][j].
constexpr int kResidSplit = 24;
template <class R>
__global__ void __launch_bounds__(256) k_resid(const Cx<R>* __restrict__ X, const Cx<R>* __restrict__ W,
                                               const double* __restrict__ theta, int n, int m, double* part,
                                               Cx<float>* Rout) {
  const int t = blockIdx.y;
  const int j = blockIdx.x * 32 + (threadIdx.x & 31), lane = threadIdx.x >> 5;
  const int chunk = (n + gridDim.z - 1) / gridDim.z, k0 = blockIdx.z * chunk, k1 = min(n, k0 + chunk);
  R s = 0;   // in the block's precision (FP64 arithmetic is scarce next to an FP32 block)
  if (j < m) {
    const R th = (R)theta[(size_t)t * m + j];
    const size_t base = (size_t)t * n * m;
#pragma unroll 4
    for (int k = k0 + lane; k < k1; k += 8) {
      const size_t idx = base + (size_t)k * m + j;
      const Cx<R> w = W[idx], x = X[idx];
      const R dx = w.re - th * x.re, dy = w.im - th * x.im;
      s += dx * dx + dy * dy;
      if (Rout) Rout[idx] = cx<float>((float)dx, (float)dy);
    }
  }
  __shared__ double red[8][33];
  red[lane][threadIdx.x & 31] = (double)s;
  __syncthreads();
  if (lane == 0 && j < m) {
    double tot = 0;
    for (int q = 0; q < 8; q++) tot += red[q][threadIdx.x];
    part[((size_t)t * gridDim.z + blockIdx.z) * m + j] = tot;
  }
}
__global__ void k_resid_sum(const double* __restrict__ part, int splits, int m, int total, double* res) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= total) return;
  const int t = e / m, j = e - t * m;
  double s = 0;
  for (int z = 0; z < splits; z++) s += part[((size_t)t * splits + z) * m + j];
  res[e] = sqrt(s);
}

// Y64 = X64 + E32 / s[t][j]  (phase B filter output, column j divided by s_d(theta_j)).
// The division leaves the span, and so the Rayleigh-Ritz, unchanged, but keeps the
// columns of Y at unit scale: X s_d + E has columns from 1 down to 1 / rho, whose
// Gram matrix (condition number up to rho^2) would limit the FP64 Ritz vectors
// near the cut to a few 1e-10.  s_d(theta) >= 1 / rho > 0 on [theta_0, cut].
__global__ void k_combine(const Cx<double>* __restrict__ X, const Cx<float>* __restrict__ E,
                          const double* __restrict__ scol, size_t nm, int m, size_t total, Cx<double>* Y) {
  const size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= total) return;
  const unsigned e32 = (unsigned)e;           // total < 2^31 (checked with the block)
  const int j = (int)(e32 % (unsigned)m);
  const unsigned t = e32 / (unsigned)nm;
  const double sj = scol[t * m + j];
  const Cx<float> ev = E[e];
  const Cx<double> ed = cx<double>((double)ev.re, (double)ev.im);
  // a vanishing s_d (possible only when the cut is pushed below 12 on a block that
  // spans nearly the whole timeslice) keeps the unscaled column
  Y[e] = fabs(sj) > 1e-280 ? X[e] + (1.0 / sj) * ed : sj * X[e] + ed;
}

// first step of phase B's filter: out = alpha_t s[t][j] rin
__global__ void k_filter_start(const Cx<float>* __restrict__ rin, const double* __restrict__ scol,
                               const double* __restrict__ coef, size_t nm, int m, size_t total, Cx<float>* out) {
  const size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= total) return;
  const unsigned e32 = (unsigned)e;
  const unsigned t = e32 / (unsigned)nm;
  out[e] = ((float)coef[3 * t] * (float)scol[t * m + e32 % (unsigned)m]) * rin[e];
}

template <class A, class B> __global__ void k_convert_block(const Cx<A>* in, Cx<B>* out, size_t total) {
  const size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e < total) out[e] = cx<B>((B)in[e].re, (B)in[e].im);
}

// counter-based start vectors: splitmix64 of (seed, index) -> two uniforms in (-1, 1)
__device__ __forceinline__ uint64_t splitmix64(uint64_t z) {
  z += 0x9e3779b97f4a7c15ULL;
  z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ULL;
  z = (z ^ (z >> 27)) * 0x94d049bb133111ebULL;
  return z ^ (z >> 31);
}
__global__ void k_random(Cx<float>* X, size_t count, uint64_t seed) {
  const size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= count) return;
  const uint64_t h = splitmix64(seed ^ splitmix64(e));
  const double a = (double)(h >> 11) * (1.0 / 9007199254740992.0) * 2.0 - 1.0;
  const uint64_t h2 = splitmix64(h);
  const double b = (double)(h2 >> 11) * (1.0 / 9007199254740992.0) * 2.0 - 1.0;
  X[e] = cx<float>((float)a, (float)b);
}

// columns whose Ritz value is marked dropped (>= 1e299) get fresh random entries
template <class R>
__global__ void k_refill(Cx<R>* X, const double* theta, int n, int m, size_t total, uint64_t seed) {
  const size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= total) return;
  const int j = e % m;
  const size_t t = e / ((size_t)n * m);
  if (theta[t * m + j] < 1e299) return;
  const uint64_t h = splitmix64(seed ^ splitmix64(e));
  const uint64_t h2 = splitmix64(h);
  X[e] = cx<R>((R)((double)(h >> 11) * (2.0 / 9007199254740992.0) - 1.0),
               (R)((double)(h2 >> 11) * (2.0 / 9007199254740992.0) - 1.0));
}

// first N columns of the block -> out [Tn][N][Vs][3] (cache_layout: [N][T][Vs][3] at timeslice t0 + t)
__global__ void k_extract(const Cx<double>* X, int n, int Tn, int m, int N, double2* out, int cache_layout, int T,
                          int t0) {
  const size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  const size_t total = (size_t)N * Tn * n;
  if (e >= total) return;
  const size_t r = e % n;
  const size_t rest = e / n;
  const int k = rest % N;
  const int t = rest / N;
  const Cx<double> v = X[((size_t)t * n + r) * m + k];
  const size_t o = cache_layout ? ((size_t)k * T + t0 + t) * n + r : ((size_t)t * N + k) * n + r;
  out[o] = make_double2(v.re, v.im);
}

// the original per-vector layout ([nvec][V][3]) for dlma_apply_laplacian
__global__ void k_lap_canonical(Geom g, const double2* __restrict__ U3, const double2* __restrict__ in, double2* out,
                                int nvec) {
  const int s = blockIdx.x * blockDim.x + threadIdx.x;
  const int j = blockIdx.y;
  if (s >= g.V || j >= nvec) return;
  const int x = s % g.L, y = (s / g.L) % g.L, z = (s / (g.L * g.L)) % g.L, t = s / g.Vs;
  const Coord c{x, y, z, t};
  const double2* v = in + (size_t)j * g.V * 3;
  Cx<double> acc[3];
  for (int a = 0; a < 3; a++) {
    const double2 e = v[(size_t)s * 3 + a];
    acc[a] = cx<double>(-6.0 * e.x, -6.0 * e.y);
  }
  for (int k = 0; k < 3; k++) {
    const int nf = nbr_lex(g, c, k + 1, +1), nb = nbr_lex(g, c, k + 1, -1);
    for (int a = 0; a < 3; a++)
      for (int b = 0; b < 3; b++) {
        const double2 uf = U3[((size_t)k * 9 + a * 3 + b) * g.V + s];
        const double2 ub = U3[((size_t)k * 9 + b * 3 + a) * g.V + nb];
        const double2 vf = v[(size_t)nf * 3 + b], vb = v[(size_t)nb * 3 + b];
        fma_acc(acc[a], cx<double>(uf.x, uf.y), cx<double>(vf.x, vf.y));
        fma_conj_acc(acc[a], cx<double>(ub.x, ub.y), cx<double>(vb.x, vb.y));
      }
  }
  double2* o = out + (size_t)j * g.V * 3;
  for (int a = 0; a < 3; a++) o[(size_t)s * 3 + a] = make_double2(acc[a].re, acc[a].im);
}

}  // namespace

// ---------------------------------------------------------------------------
struct Eig {
  dlma_ctx* ctx;
  int t0, Tn, N, m, n, nsplit, nsplit_f, degree;   // row splits of the Gram products, FP64 and FP32 blocks
  int df = 0;   // phase B: Gram matrices and rotations in double-float (tol >= 1e-11)
  int tc = 0;   // phase B: Gram matrices and rotations on the tensor cores (tcproj.cu)
  size_t blk;                    // m * Tn * n complex entries per block
  Cx<float> *F0, *F1, *F2, *F3;  // FP32 blocks
  Cx<double> *D0, *D1, *D2;      // FP64 blocks
  double2 *G, *H, *C, *part, *gwork;
  double *theta, *res, *coef, *scol;
  const double* plain;           // coefficients of the plain operator: coef slot `degree`
  int* dropped;                  // [0] dropped directions of the last small_rr, [1 + 2t + {0,1}] Jacobi sweeps
  bool refilled = false;         // the last fetch refilled dropped columns
  PhaseTimer* pt = nullptr;      // phases: kPhMatvec, kPhOrtho, kPhHost
  double drop_rel;
  uint64_t refill_seed;
  std::vector<double> th, rs;
};

// timing slots of dlma_laplacian_eigs (Table 2's split of the eigensolver time):
// Laplacian applications, orthogonalisation (Gram matrices, small eigenproblems,
// rotations, residuals, block conversions), host-side steps and transfers
constexpr int kPhMatvec = 3, kPhOrtho = 4, kPhHost = 5;
static inline void phase(Eig& E, int p) {
  if (E.pt) E.pt->enter(p);
}

// one step of the FP32 filter (k_lap_z): out = alpha (A in) + beta in + gamma prev +
// alpha s rin, two columns per thread (m is even: one 128-bit access per pair)
static dlma_status lap_filter(Eig& E, const Cx<float>* in, const Cx<float>* prev, const Cx<float>* rin,
                              const double* scol, Cx<float>* out, const double* coef) {
  dlma_ctx* ctx = E.ctx;
  phase(E, kPhMatvec);
  const LapTiling t = lap_tiling(ctx->g.L, E.m, E.Tn);
  k_lap_z<<<dim3((unsigned)(t.nx * t.ny * t.nz * t.groups), E.Tn), 256, 0, ctx->stream>>>(
      ctx->g, E.t0, E.m, t, ctx->U3f, in, prev, rin, scol, out, coef);
  CHECK_LAUNCH();
  return DLMA_OK;
}
// out = A in.  FP32: a filter step with the coefficients of the plain operator.  FP64 is
// bound by its arithmetic and takes one column per thread (a double-float matvec, 170
// registers and a split of every loaded value, was slower).
static dlma_status lap(Eig& E, const Cx<float>* in, Cx<float>* out) {
  return lap_filter(E, in, nullptr, nullptr, nullptr, out, E.plain);
}
static dlma_status lap(Eig& E, const Cx<double>* in, Cx<double>* out) {
  dlma_ctx* ctx = E.ctx;
  phase(E, kPhMatvec);
  k_lap<<<(unsigned)((E.blk / 3 + 255) / 256), 256, 0, ctx->stream>>>(ctx->g, E.t0, E.Tn, E.m, ctx->U3, in, out);
  CHECK_LAUNCH();
  return DLMA_OK;
}

// whether a tensor-core product found no memory for its digits: their buffers are given
// back and double-float takes this product and the following ones
static bool no_digits(Eig& E, dlma_status st) {
  if (st != DLMA_ERR_OOM) return false;
  E.tc = 0;
  cudaStreamSynchronize(E.ctx->stream);
  for (int s : {WS_TC_A, WS_TC_B, WS_TC_E, WS_TC_P}) work_free(E.ctx, s);
  return true;
}

// out = X^dag Y per timeslice; herm = 1 when the result is hermitian by construction
template <class R> static dlma_status gram(Eig& E, const Cx<R>* X, const Cx<R>* Y, double2* out, int herm) {
  dlma_ctx* ctx = E.ctx;
  const int tj = (E.m + GT - 1) / GT;
  const int tiles = herm ? tj * (tj + 1) / 2 : tj * tj;
  phase(E, kPhOrtho);
  const dim3 grid(tiles, E.nsplit, E.Tn);
  if constexpr (sizeof(R) == 8) {
    if (E.tc) {   // G[t][i][j] = sum_k conj(X[k][i]) Y[k][j]: rows = columns of Y, modes = columns of X
      const dlma_status st = tc_block_product(ctx, 1, (const double2*)Y, (size_t)E.n * E.m, 1, (size_t)E.m, E.m,
                                              (const double2*)X, 0, E.m, E.n, E.Tn, out);
      if (!no_digits(E, st)) return st;
    }
    if (E.df) k_gram<R, df><<<grid, 256, 0, ctx->stream>>>(X, Y, E.n, E.m, E.nsplit, herm, E.part);
    else k_gram<R, R><<<grid, 256, 0, ctx->stream>>>(X, Y, E.n, E.m, E.nsplit, herm, E.part);
  } else {
    const int tf = (E.m + FT - 1) / FT;
    k_gram_f<<<dim3(herm ? tf * (tf + 1) / 2 : tf * tf, E.nsplit_f, E.Tn), 256, 0, ctx->stream>>>(
        X, Y, E.n, E.m, E.nsplit_f, herm, E.part);
  }
  CHECK_LAUNCH();
  const size_t tot = (size_t)E.m * E.m * E.Tn;
  const bool f32 = sizeof(R) == 4;
  k_gram_reduce<<<(unsigned)((tot + 255) / 256), 256, 0, ctx->stream>>>(E.part, f32 ? E.nsplit_f : E.nsplit, E.m, E.Tn,
                                                                       herm, f32 ? FT : GT, out);
  CHECK_LAUNCH();
  return DLMA_OK;
}

template <class R> static dlma_status rotate(Eig& E, const Cx<R>* X, Cx<R>* Z) {
  dlma_ctx* ctx = E.ctx;
  phase(E, kPhOrtho);
  const dim3 grid((E.n + RT - 1) / RT, (E.m + RT - 1) / RT, E.Tn);
  if constexpr (sizeof(R) == 8) {
    if (E.tc) {   // Z[t][k][j] = sum_l X[k][l] C[l][j]: rows = rows of X, modes = conj of the columns of C
      const dlma_status st = tc_block_product(ctx, 2, (const double2*)X, (size_t)E.n * E.m, (size_t)E.m, 1, E.n, E.C, 1,
                                              E.m, E.m, E.Tn, (double2*)Z);
      if (!no_digits(E, st)) return st;
    }
    if (E.df) k_rotate<R, df><<<grid, 256, 0, ctx->stream>>>(X, E.C, E.n, E.m, Z);
    else k_rotate<R, R><<<grid, 256, 0, ctx->stream>>>(X, E.C, E.n, E.m, Z);
  } else {
    // C in FP32 first, into the Gram partials' area (a conversion per use would occupy the
    // FP64 pipe for half of the kernel's time)
    const size_t mmt = (size_t)E.m * E.m * E.Tn;
    Cx<float>* Cf = (Cx<float>*)E.part;
    k_convert_block<double, float><<<(unsigned)((mmt + 255) / 256), 256, 0, ctx->stream>>>((const Cx<double>*)E.C, Cf, mmt);
    CHECK_LAUNCH();
    k_rotate_f<<<dim3((E.n + FT - 1) / FT, (E.m + FT - 1) / FT, E.Tn), 256, 0, ctx->stream>>>(X, Cf, E.n, E.m, Z);
  }
  CHECK_LAUNCH();
  return DLMA_OK;
}

// small Rayleigh-Ritz problems in precision T (float in phase A, double in phase B).
// The orthonormalisation tries the Cholesky route first in both phases; a pivot
// below the precision's floor (an ill-conditioned Gram matrix, as the unscaled
// phase-A block can have) falls back to the Jacobi route inside the kernel.
template <class T> static dlma_status small_rr(Eig& E) {
  dlma_ctx* ctx = E.ctx;
  size_t sm = 0;
  const int place = small_rr_place<T>(E.m, &sm);
  phase(E, kPhOrtho);
  if (sm) CU(cudaFuncSetAttribute(k_small_rr<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm));
  CU(cudaMemsetAsync(E.dropped, 0, sizeof(int), ctx->stream));
  const int chol = 1;
  k_small_rr<T><<<E.Tn, 1024, sm, ctx->stream>>>(E.G, E.H, E.m, E.C, E.theta, (Cx<T>*)E.gwork, place, E.dropped,
                                                 E.drop_rel, chol);
  CHECK_LAUNCH();
  return DLMA_OK;
}

template <class R> static dlma_status resid(Eig& E, const Cx<R>* X, const Cx<R>* W, Cx<float>* Rout) {
  dlma_ctx* ctx = E.ctx;
  phase(E, kPhOrtho);
  // partial sums in the Gram partials' work area, which holds 2 m^2 doubles per timeslice
  const int splits = std::max(1, std::min(std::min(kResidSplit, E.n / 64), 2 * E.m));
  k_resid<R><<<dim3((E.m + 31) / 32, E.Tn, splits), 256, 0, ctx->stream>>>(X, W, E.theta, E.n, E.m, (double*)E.part,
                                                                          Rout);
  CHECK_LAUNCH();
  k_resid_sum<<<(E.m * E.Tn + 127) / 128, 128, 0, ctx->stream>>>((const double*)E.part, splits, E.m, E.m * E.Tn, E.res);
  CHECK_LAUNCH();
  return DLMA_OK;
}

// Rayleigh-Ritz of the block Y: W = A Y, then X <- Y C, AX <- W C, residuals (and R = AX - X Theta in FP32)
template <class R>
static dlma_status rayleigh_ritz(Eig& E, Cx<R>* Y, Cx<R>* W, Cx<R>* Xout, Cx<R>* AXout, Cx<float>* Rout) {
  TRY(lap(E, Y, W));
  TRY(gram<R>(E, Y, Y, E.G, 1));
  TRY(gram<R>(E, Y, W, E.H, 1));
  TRY(small_rr<R>(E));
  TRY(rotate<R>(E, Y, Xout));
  TRY(rotate<R>(E, W, AXout));
  return resid<R>(E, Xout, AXout, Rout);
}

// fetch theta / residuals; returns the worst relative residual over the wanted pairs.
// Dropped directions (buffer columns that fell below the block's rounding level)
// are refilled with random entries in X and get the largest finite Ritz value of
// their timeslice on the host, so the filter's cut stays finite.
template <class R> static dlma_status fetch(Eig& E, double* worst, Cx<R>* X) {
  dlma_ctx* ctx = E.ctx;
  const size_t cnt = (size_t)E.m * E.Tn;
  phase(E, kPhHost);
  CU(cudaMemcpyAsync(E.th.data(), E.theta, sizeof(double) * cnt, cudaMemcpyDeviceToHost, ctx->stream));
  CU(cudaMemcpyAsync(E.rs.data(), E.res, sizeof(double) * cnt, cudaMemcpyDeviceToHost, ctx->stream));
  int hdrop = 0;
  CU(cudaMemcpyAsync(&hdrop, E.dropped, sizeof(int), cudaMemcpyDeviceToHost, ctx->stream));
  CU(cudaStreamSynchronize(ctx->stream));
  if (E.pt) E.pt->collect();
  E.refilled = hdrop != 0;
  if (hdrop) {
    phase(E, kPhOrtho);
    k_refill<R><<<(unsigned)((E.blk + 255) / 256), 256, 0, ctx->stream>>>(X, E.theta, E.n, E.m, E.blk,
                                                                         E.refill_seed++);
    CHECK_LAUNCH();
    for (int t = 0; t < E.Tn; t++) {
      double mx = 0;
      for (int j = 0; j < E.m; j++) {
        const double v = E.th[(size_t)t * E.m + j];
        if (v < 1e299) mx = std::max(mx, v);
      }
      for (int j = 0; j < E.m; j++) {
        double& v = E.th[(size_t)t * E.m + j];
        if (v >= 1e299) { v = mx; E.rs[(size_t)t * E.m + j] = 1.0; }
      }
    }
  }
  double w = 0;
  for (int t = 0; t < E.Tn; t++)
    for (int k = 0; k < E.N; k++) {
      const double r = E.rs[(size_t)t * E.m + k] / std::max(1.0, fabs(E.th[(size_t)t * E.m + k]));
      if (!(r == r)) return set_err(ctx, DLMA_ERR_NONFINITE, "NaN in the eigensolver");
      w = std::max(w, r);
    }
  *worst = w;
  return DLMA_OK;
}

// largest degree (<= dmax) whose amplification across [theta_0, cut] stays below rho on every timeslice
static int safe_degree(const Eig& E, double rho, int dmax) {
  int d = dmax;
  for (int t = 0; t < E.Tn; t++) {
    double a = E.th[(size_t)t * E.m + E.m - 1], a0 = E.th[(size_t)t * E.m];
    const double b = 12.0;
    if (a >= b) a = 0.5 * (a0 + b);
    const double e = 0.5 * (b - a), c = 0.5 * (b + a);
    const double x0 = (c - a0) / e;
    if (x0 > 1.0) d = std::min(d, (int)(acosh(rho) / acosh(x0)));
  }
  return std::max(d, 2);
}

// Chebyshev coefficients of every step (scaled three-term recurrence damping [cut_t, 12],
// normalised at lam0_t): slot 0 = first step, slot k-1 = step k; slot `degree` = plain A.
// With s_k(theta) (the scalar recurrence at each Ritz value) when scol != nullptr.
static void cheb_coefficients(Eig& E, int d, std::vector<double>& hc, std::vector<double>* hs) {
  const int Tn = E.Tn, m = E.m;
  hc.assign((size_t)(E.degree + 1) * 3 * Tn, 0.0);
  if (hs) hs->assign((size_t)(E.degree + 1) * Tn * m, 0.0);
  for (int t = 0; t < Tn; t++) {
    double a = E.th[(size_t)t * m + m - 1], a0 = E.th[(size_t)t * m];
    const double b = 12.0;
    if (a >= b) a = 0.5 * (a0 + b);
    const double e = 0.5 * (b - a), c = 0.5 * (b + a);
    double sigma = e / (a0 - c);
    const double tau = 2.0 / sigma;
    double* c0 = &hc[3 * t];
    c0[0] = sigma / e;
    c0[1] = -c * sigma / e;
    c0[2] = 0.0;
    std::vector<double> sp(m, 1.0), sc(m);
    for (int j = 0; j < m; j++) sc[j] = c0[0] * E.th[(size_t)t * m + j] + c0[1];
    if (hs) {
      for (int j = 0; j < m; j++) (*hs)[(size_t)t * m + j] = 1.0;                    // s_0
      for (int j = 0; j < m; j++) (*hs)[(size_t)Tn * m + (size_t)t * m + j] = sc[j];  // s_1
    }
    for (int k = 2; k <= d; k++) {
      const double sn = 1.0 / (tau - sigma);
      double* ck = &hc[(size_t)(k - 1) * 3 * Tn + 3 * t];
      ck[0] = 2.0 * sn / e;
      ck[1] = -2.0 * c * sn / e;
      ck[2] = -sigma * sn;
      sigma = sn;
      for (int j = 0; j < m; j++) {
        const double th = E.th[(size_t)t * m + j];
        const double nv = ck[0] * th * sc[j] + ck[1] * sc[j] + ck[2] * sp[j];
        sp[j] = sc[j];
        sc[j] = nv;
        if (hs) (*hs)[(size_t)k * Tn * m + (size_t)t * m + j] = nv;
      }
    }
    double* cd = &hc[(size_t)E.degree * 3 * Tn + 3 * t];   // slot of the plain A application
    cd[0] = 1;
    cd[1] = 0;
    cd[2] = 0;
  }
}

// Whether phase B's products take the tensor cores instead of double-float: from 5e7
// complex multiply-adds (n m^2 Tn) on, where they are faster (eigensolve, double-float
// against tensor cores: 110 and 96 ms on 16^3 x 32 with 64 columns, 2e9; 1277 and 957 ms
// on 24^3 x 48 with 128; equal at 2.5e7, 8^3 x 16 with 32), as far as the modes come out
// no less orthonormal.  The digits' error is that of a chunk's largest entry whatever the
// size, rms of V^dag V - 1 4e-15 ... 6e-15; double-float's grows with the rows per sum,
// n / nsplit: 3.7e-15 at 375 rows (10^3 x 18, 40 columns), 4.6e-15 at 1263 (20^3 x 8, 48),
// 5.9e-15 at 1365 (16^3 x 16, 64), 9.3e-15 at 3072 (16^3 x 32, 64), either side of 5e-15
// between 860 and 1270.  (The eigenvalues come out to an rms of 6e-15 ... 1e-14 with
// double-float and 2e-15 ... 8e-15 with the digits, both far below any tol.)  From 4e9
// multiply-adds on always.
static bool tc_products(int n, int m, int Tn, int nsplit) {
  const double macs = (double)n * m * m * Tn;
  return macs >= 4.0e9 || (macs >= 5.0e7 && n >= 1300 * nsplit);
}

static dlma_status eig_batch(dlma_ctx* ctx, int t0, int Tn, int N, double tol, double* lam_out,
                             Cx<double>** Xres, int* m_out, int* iters_out, PhaseTimer* pt) {
  Eig E;
  E.ctx = ctx;
  E.pt = pt;
  E.t0 = t0;
  E.Tn = Tn;
  E.N = N;
  E.n = 3 * ctx->g.Vs;
  int buf = std::max(16, std::min(N, 64));
  int m = N + buf;
  m += m & 1;
  if (m > E.n) m = E.n - (E.n & 1);
  if (m < N) return set_err(ctx, DLMA_ERR_INVALID_ARG, "N too large for the timeslice");
  if (m > kSmallMaxM - 2)
    return set_err(ctx, DLMA_ERR_INVALID_ARG, "N + buffer above the eigensolver's limit of %d", kSmallMaxM - 2);
  E.m = m;
  E.degree = 40;            // largest filter degree (phase B); phase A stays below 20
  E.blk = (size_t)m * Tn * E.n;
  if (E.blk >= (1ull << 31)) return set_err(ctx, DLMA_ERR_INVALID_ARG, "eigensolver block above 2^31 entries");
  E.nsplit = std::max(1, std::min(64, (4 * 152) / std::max(1, Tn * ((m + GT - 1) / GT) * ((m + GT - 1) / GT))));
  E.nsplit = std::min(E.nsplit, std::max(1, E.n / 256));
  {
    const int tf = (m + FT - 1) / FT;
    E.nsplit_f = std::max(1, std::min(64, (4 * 152) / std::max(1, Tn * tf * (tf + 1) / 2)));
    E.nsplit_f = std::min(E.nsplit_f, std::max(1, E.n / 256));
  }
  TRY(workT(ctx, WS_EIG_X, E.blk * 2, &E.F0));
  E.F1 = E.F0 + E.blk;
  TRY(workT(ctx, WS_EIG_Y, E.blk * 2, &E.F2));
  E.F3 = E.F2 + E.blk;
  TRY(workT(ctx, WS_EIG_Y2, E.blk, &E.D0));
  TRY(workT(ctx, WS_EIG_W, E.blk * 2, &E.D1));
  E.D2 = E.D1 + E.blk;
  const size_t mm = (size_t)m * m;
  TRY(workT(ctx, WS_EIG_G, 3 * mm * Tn, &E.G));
  E.H = E.G + mm * Tn;
  E.C = E.H + mm * Tn;
  TRY(workT(ctx, WS_EIG_PART, (size_t)std::max(E.nsplit, E.nsplit_f) * mm * Tn, &E.part));
  TRY(workT(ctx, WS_EIG_S, 3 * (size_t)m * (m + 1) * Tn, &E.gwork));
  const int d = E.degree;
  double* aux;
  const size_t ncoef = (size_t)(d + 1) * 3 * Tn, nscol = (size_t)(d + 1) * Tn * m;
  TRY(workT(ctx, WS_EIG_AUX, 2 * (size_t)m * Tn + ncoef + nscol + Tn + 16, &aux));
  E.theta = aux;
  E.res = aux + (size_t)m * Tn;
  E.coef = E.res + (size_t)m * Tn;
  E.scol = E.coef + ncoef;
  E.dropped = (int*)(E.scol + nscol);
  E.th.resize((size_t)m * Tn);
  E.rs.resize((size_t)m * Tn);
  E.drop_rel = 1e-10;
  E.refill_seed = 0x7e11ULL + (uint64_t)t0;
  std::vector<double> hc, hs;
  // plain A for the Rayleigh-Ritz W = A Y: coefficient slot d
  hc.assign(ncoef, 0.0);
  for (int t = 0; t < Tn; t++) hc[(size_t)d * 3 * Tn + 3 * t] = 1.0;
  phase(E, kPhHost);
  CU(cudaMemcpyAsync(E.coef, hc.data(), sizeof(double) * ncoef, cudaMemcpyHostToDevice, ctx->stream));
  E.plain = E.coef + (size_t)d * 3 * Tn;

  // ---- phase A: FP32 ----
  phase(E, kPhOrtho);
  k_random<<<(unsigned)((E.blk + 255) / 256), 256, 0, ctx->stream>>>(E.F1, E.blk, 0x5eed2022ULL + (uint64_t)t0 * 7919ULL);
  CHECK_LAUNCH();
  // three FP32 blocks rotate: p3[0] = Ritz vectors X, p3[1], p3[2] free; F3 holds A X
  Cx<float>* p3[3] = {E.F0, E.F1, E.F2};
  TRY(rayleigh_ritz<float>(E, p3[1], p3[2], p3[0], E.F3, nullptr));
  double worst = 1;
  int it = 0;
  const int maxA = 60, maxB = 40;
  const double switch_tol = std::max(tol, 3e-6);
  double prev_worst = 1e300;
  E.drop_rel = 1e-10;       // FP32 block: Gram eigenvalues below ~1e-10 gmax are rounding noise
  for (; it < maxA; it++) {
    TRY(fetch<float>(E, &worst, p3[0]));
    if (worst <= switch_tol) break;
    // single precision has stopped paying off: hand over to the FP64 phase
    if (it >= 3 && worst > 0.5 * prev_worst) break;
    prev_worst = worst;
    // FP32 filter: keep the amplification across [theta_0, cut] below ~300 so the
    // filtered block stays resolvable in single precision
    const int dA = safe_degree(E, 300.0, 20);
    cheb_coefficients(E, dA, hc, nullptr);
    phase(E, kPhHost);
    CU(cudaMemcpyAsync(E.coef, hc.data(), sizeof(double) * ncoef, cudaMemcpyHostToDevice, ctx->stream));
    Cx<float>*prev = p3[0], *cur = p3[1], *nxt = p3[2];
    TRY(lap_filter(E, prev, nullptr, nullptr, nullptr, cur, E.coef));
    for (int k = 2; k <= dA; k++) {
      TRY(lap_filter(E, cur, prev, nullptr, nullptr, nxt, E.coef + (size_t)(k - 1) * 3 * Tn));
      Cx<float>* t = prev;
      prev = cur;
      cur = nxt;
      nxt = t;
    }
    // cur holds the filtered block; prev and nxt are free (one of them held X)
    TRY(rayleigh_ritz<float>(E, cur, prev, nxt, E.F3, nullptr));
    p3[0] = nxt;
    p3[1] = cur;
    p3[2] = prev;
  }
  Cx<float>* X = p3[0];
  // ---- phase B: FP64 Ritz vectors, FP32 residual-driven filter ----
  // The FP64 blocks' Gram matrices and rotations run in double-float on the FP32
  // units when the tolerance leaves room for its ~2^-46 rounding.
  E.df = ctx->df_eigs && tol >= 1e-11;
  // (and large ones on the tensor cores; DLMA_EIGS_TC=1 / 0 forces either)
  E.tc = E.df && tc_products(E.n, E.m, E.Tn, E.nsplit);
  // the rotation's digits (every row of the block) have to fit a memory cap, and all of
  // them (up to 4 GB) the device beside the modes to come (cached, and on their way out)
  if (ctx->memcap && tc_min_bytes(E.n, E.m, E.Tn) > ctx->memcap) E.tc = 0;
  if (E.tc) {
    size_t freeb = 0, totb = 0;
    CU(cudaMemGetInfo(&freeb, &totb));
    const size_t modes = 2 * (size_t)N * ctx->g.T * E.n * sizeof(double2);
    if (tc_block_bytes(ctx, E.n, E.m, E.Tn) + modes > freeb - freeb / 64) E.tc = 0;
  }
  if (const char* e = getenv("DLMA_EIGS_TC")) E.tc = E.df && atoi(e) == 1;
  Cx<double> *X64 = E.D0, *W64 = E.D1, *Y64 = E.D2;
  // phase A's last Ritz pairs were not fetched, or hold refilled (random) columns
  const bool rr_first = E.refilled || it >= maxA;
  phase(E, kPhOrtho);
  k_convert_block<float, double><<<(unsigned)((E.blk + 255) / 256), 256, 0, ctx->stream>>>(X, rr_first ? Y64 : X64,
                                                                                           E.blk);
  CHECK_LAUNCH();
  Cx<float>* R32 = E.F3;   // residual R = AX - X Theta
  Cx<float>* Ebuf[3];
  {
    int q = 0;
    Cx<float>* all[4] = {E.F0, E.F1, E.F2, E.F3};
    for (int i = 0; i < 4; i++)
      if (all[i] != R32) Ebuf[q++] = all[i];
  }
  // The filter below needs only R32 = A X - X Theta for the current X and Theta, which
  // hold for phase A's Ritz pairs as they stand: X64 = X, Y64 = A X64, R32.  After a
  // refill the block is first re-diagonalised in FP64.
  E.drop_rel = 1e-24;
  if (rr_first) {
    TRY(rayleigh_ritz<double>(E, Y64, W64, X64, Y64, R32));
  } else {
    TRY(lap(E, X64, Y64));
    TRY(resid<double>(E, X64, Y64, R32));
  }
  bool conv = false;
  int itB = 0;
  int dB = d;
  for (; itB < maxB; itB++) {
    TRY(fetch<double>(E, &worst, X64));
    if (worst <= tol) { conv = true; break; }
    dB = safe_degree(E, 1e6, d);
    cheb_coefficients(E, dB, hc, &hs);
    phase(E, kPhHost);
    CU(cudaMemcpyAsync(E.coef, hc.data(), sizeof(double) * ncoef, cudaMemcpyHostToDevice, ctx->stream));
    CU(cudaMemcpyAsync(E.scol, hs.data(), sizeof(double) * nscol, cudaMemcpyHostToDevice, ctx->stream));
    // E_1 = a_1 R s_0 ; E_{k+1} = a_k A E_k + b_k E_k + c_k E_{k-1} + a_k R s_k
    Cx<float>*em = nullptr, *ec = Ebuf[0], *en = Ebuf[1], *spare = Ebuf[2];
    phase(E, kPhMatvec);
    k_filter_start<<<(unsigned)((E.blk + 255) / 256), 256, 0, ctx->stream>>>(R32, E.scol, E.coef, (size_t)E.n * m, m,
                                                                             E.blk, ec);
    CHECK_LAUNCH();
    for (int k = 2; k <= dB; k++) {
      TRY(lap_filter(E, ec, em, R32, E.scol + (size_t)(k - 1) * Tn * m, en, E.coef + (size_t)(k - 1) * 3 * Tn));
      Cx<float>* t = em ? em : spare;
      em = ec;
      ec = en;
      en = t;
    }
    // Y = (X s_d + E_d) / s_d column by column
    phase(E, kPhOrtho);
    k_combine<<<(unsigned)((E.blk + 255) / 256), 256, 0, ctx->stream>>>(X64, ec, E.scol + (size_t)dB * Tn * m,
                                                                        (size_t)E.n * m, m, E.blk, Y64);
    CHECK_LAUNCH();
    // Rayleigh-Ritz of Y64: W64 = A Y64; X64 <- Y64 C; AX into W... (use X64 as output: Y64 and W64 are inputs)
    TRY(lap(E, Y64, W64));
    TRY(gram<double>(E, Y64, Y64, E.G, 1));
    TRY(gram<double>(E, Y64, W64, E.H, 1));
    TRY(small_rr<double>(E));
    TRY(rotate<double>(E, Y64, X64));
    // A X afresh in FP64: W C by the same product would add that one's rounding (some 1e-13
    // of |W|) to the residual (24^3 x 48, 128 columns: 30 ms; a tensor-core product 12 ms)
    TRY(lap(E, X64, Y64));
    TRY(resid<double>(E, X64, Y64, R32));
  }
  if (!conv) {
    TRY(fetch<double>(E, &worst, X64));
    conv = worst <= tol;
  }
  if (!conv)
    return set_err(ctx, DLMA_ERR_NOT_CONVERGED, "eigensolver at %.3g, not %.3g, after %d + %d iterations", worst, tol,
                   it, itB);
  for (int t = 0; t < Tn; t++)
    for (int k = 0; k < N; k++) lam_out[(size_t)t * N + k] = E.th[(size_t)t * m + k];
  *Xres = X64;
  *m_out = m;
  if (iters_out) { iters_out[0] = it; iters_out[1] = itB; }
  return DLMA_OK;
}

extern "C" dlma_status dlma_apply_laplacian(dlma_ctx* ctx, const double* in, double* out, int nvec, dlma_mem mem) {
  if (!ctx) return DLMA_ERR_INVALID_ARG;
  if (!ctx->have_gauge) return set_err(ctx, DLMA_ERR_STATE, "no gauge field");
  if (!in || !out || nvec < 1) return set_err(ctx, DLMA_ERR_INVALID_ARG, "bad argument");
  CU(cudaSetDevice(ctx->device));
  const size_t bytes = (size_t)nvec * ctx->g.V * 3 * 16;
  const double* din;
  TRY(copy_in(ctx, WS_IN, in, bytes, mem, &din));
  double* dout = out;
  if (mem == DLMA_MEM_HOST) TRY(workT(ctx, WS_OUT, bytes / 8, &dout));
  dim3 grid((ctx->g.V + 127) / 128, nvec);
  k_lap_canonical<<<grid, 128, 0, ctx->stream>>>(ctx->g, ctx->U3, (const double2*)din, (double2*)dout, nvec);
  CHECK_LAUNCH();
  TRY(copy_out(ctx, out, dout, bytes, mem));
  CU(cudaStreamSynchronize(ctx->stream));
  return DLMA_OK;
}

extern "C" dlma_status dlma_laplacian_eigs(dlma_ctx* ctx, int t, int N, double tol, double* evals, double* evecs,
                                           dlma_mem mem) {
  if (!ctx) return DLMA_ERR_INVALID_ARG;
  if (!ctx->have_gauge) return set_err(ctx, DLMA_ERR_STATE, "no gauge field");
  if (!evals || N < 1 || t < -1 || t >= ctx->g.T || !(tol > 0) || N > 3 * ctx->g.Vs / 2)
    return set_err(ctx, DLMA_ERR_INVALID_ARG, "bad argument to dlma_laplacian_eigs");
  CU(cudaSetDevice(ctx->device));
  const int t0 = t < 0 ? 0 : t, Tn = t < 0 ? ctx->g.T : 1;
  const int n = 3 * ctx->g.Vs;
  cudaEvent_t e0, e1;
  CU(cudaEventCreate(&e0));
  CU(cudaEventCreate(&e1));
  CU(cudaEventRecord(e0, ctx->stream));
  Cx<double>* X = nullptr;
  int m = 0, iters[2] = {0, 0};
  PhaseTimer pt(ctx->stream);
  pt.enter(kPhHost);
  dlma_status st = eig_batch(ctx, t0, Tn, N, tol, evals, &X, &m, iters, &pt);
  if (st != DLMA_OK) {
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    return st;
  }
  pt.enter(kPhHost);
  ctx->eig_gen++;
  if (ctx->eig_N != N || !ctx->eig_V) {
    if (ctx->eig_V) cudaFree(ctx->eig_V);
    ctx->eig_V = nullptr;
    ctx->eig_N = 0;
    CU(cudaMalloc(&ctx->eig_V, (size_t)N * ctx->g.T * n * sizeof(double2)));
    ctx->eig_lam.assign((size_t)N * ctx->g.T, 0.0);
    ctx->eig_have.assign(ctx->g.T, 0);
    ctx->eig_N = N;
  }
  const size_t tot = (size_t)N * Tn * n;
  k_extract<<<(unsigned)((tot + 255) / 256), 256, 0, ctx->stream>>>(X, n, Tn, m, N, ctx->eig_V, 1, ctx->g.T, t0);
  CHECK_LAUNCH();
  for (int tt = 0; tt < Tn; tt++) {
    ctx->eig_have[t0 + tt] = 1;
    for (int k = 0; k < N; k++) ctx->eig_lam[(size_t)(t0 + tt) * N + k] = evals[(size_t)tt * N + k];
  }
  if (evecs) {
    const size_t bytes = tot * sizeof(double2);
    double2* dst = (double2*)evecs;
    if (mem == DLMA_MEM_HOST) TRY(workT(ctx, WS_OUT, tot, &dst));
    k_extract<<<(unsigned)((tot + 255) / 256), 256, 0, ctx->stream>>>(X, n, Tn, m, N, dst, 0, ctx->g.T, t0);
    CHECK_LAUNCH();
    if (mem == DLMA_MEM_HOST) TRY(copy_out(ctx, evecs, (const double*)dst, bytes, mem));
  }
  CU(cudaEventRecord(e1, ctx->stream));
  CU(cudaStreamSynchronize(ctx->stream));
  pt.mark(-1);
  CU(cudaStreamSynchronize(ctx->stream));
  pt.collect();
  float ms = 0;
  cudaEventElapsedTime(&ms, e0, e1);
  for (int i = 0; i < kTimingSlots; i++) ctx->timing[i] = 0;
  ctx->timing[0] = ms;
  ctx->timing[1] = iters[0];
  ctx->timing[2] = iters[1];
  ctx->timing[kPhMatvec] = pt.acc[kPhMatvec];
  ctx->timing[kPhOrtho] = pt.acc[kPhOrtho];
  ctx->timing[kPhHost] = pt.acc[kPhHost];
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  return DLMA_OK;
}
