// FP64 stencil for few (site, right-hand side) pairs: the work of one pair is split
// over 16 threads.
//
// What bounds it: the FP64 pipe of one SM sub-partition takes 64 cycles per warp
// instruction (2 lanes per clock and SM), and k_hop's one thread per pair issues about
// 1180 of them in a row, 38 us however small the lattice, on as many of the 608
// sub-partitions as there are warps: a 4^3 x 8 lattice with one vector fills 8.  Here
//   1. 16 threads per pair = 8 directions x 2 projected spins: one 3 x 3 product each,
//   2. 12 threads per pair = spin x colour: the sum over directions, then the rows of
//      the site matrices (clover, inverse clover),
// meeting in shared memory: about 100 FP64 instructions deep, 41 warp instructions per
// pair against k_hop's 37, so k_hop stays ahead once every sub-partition has a warp of
// its own (kHopSplitPairs).  Measured, one Schur application on 4^3 x 8: 87 -> 20 us with
// one vector, 87 -> 28 us with 12 (12 us at the FP64 rate; the rest is the latency of two
// dependent loads and two barriers per launch).  Signs, factors +-i and the conjugations are integer
// operations on the operands, not FP64 ones.
//
// Fields are read and written in k_hop's layout or, for the operator calls on user
// arrays, in the canonical one (Field::lay), which saves the packing launches.
#pragma once
#include "fieldio.cuh"

constexpr int kSplitSites = 8;              // sites per block (16 threads each)

// element k of the spinor at compressed index i of parity p
struct SplitView {
  double2* p = nullptr;
  size_t rhs = 0;                           // double2 units per right-hand side
  int lay = 0;
};
__device__ __forceinline__ size_t split_site(const Geom& g, int lay, int par, int i) {
  if (lay == kLayInternal) return (size_t)i;
  if (lay == kLayHalf) return (size_t)i * 12;
  const int r = (2 * i) / g.L, y = r % g.L, z = (r / g.L) % g.L, t = r / (g.L * g.L);
  return ((size_t)2 * i + ((y + z + t + par) & 1)) * 12;
}

struct SplitArgs {
  Geom g;
  int p_out, nrhs, ntiles, site0, nsites;
  SplitView in, own, out;
  const double2 *U, *Kown, *Kout;           // K: at parity p_out
  double s;
  int hop, g5_in, g5_hop, own_op, kout;     // own_op: 0 none, 1 identity, 2 Kown
  const int* active;
  const int4* nbr;
  double* norm_part;
  double2 *cg_x, *cg_r;
  const double2* cg_p;
  const double* cg_alpha;
};

__device__ __forceinline__ double flip_if(double x, int neg) {
  return __hiloint2double(__double2hiint(x) ^ (neg ? (int)0x80000000 : 0), __double2loint(x));
}
// +-v or +-i v
__device__ __forceinline__ Cx<double> unit_mul(Cx<double> v, int imag, int neg) {
  return cx<double>(flip_if(imag ? v.im : v.re, neg ^ imag), flip_if(imag ? v.re : v.im, neg));
}
// row r (0..5) of a packed hermitian 6 x 6 block (see pack_block in ctx.cu): the load,
// issued before the hopping term so that its latency is hidden, and the product with v
__device__ __forceinline__ void load_row(const double2* __restrict__ K, int Vh, int i, int ch, int r, Cx<double> m[6]) {
  const double2* k = K + (size_t)18 * ch * Vh + i;
#pragma unroll
  for (int c = 0; c < 6; c++) {
    const int hi = r > c ? r : c, lo = r > c ? c : r;
    const double2 l = __ldg(k + (size_t)(r == c ? r >> 1 : 3 + (hi * (hi - 1)) / 2 + lo) * Vh);
    m[c] = r == c ? cx<double>((r & 1) ? l.y : l.x, 0.0) : cx<double>(l.x, flip_if(l.y, r < c));
  }
}
// (r's own, real entry multiplies no imaginary parts: 0 x Inf would be NaN)
__device__ __forceinline__ Cx<double> row_mul(const Cx<double> m[6], const Cx<double> v[6], int r) {
  Cx<double> s = cx<double>(0, 0);
#pragma unroll
  for (int c = 0; c < 6; c++) {
    const double xr = c == r ? 0.0 : v[c].re, xi = c == r ? 0.0 : v[c].im;
    s.re = fma(-m[c].im, xi, fma(m[c].re, v[c].re, s.re));
    s.im = fma(m[c].im, xr, fma(m[c].re, v[c].im, s.im));
  }
  return s;
}

__global__ void __launch_bounds__(16 * kSplitSites) k_hop_split(SplitArgs a) {
  const Geom g = a.g;
  const int j = blockIdx.x / a.ntiles, tile = blockIdx.x - j * a.ntiles;
  if (a.active && !a.active[j]) return;     // the whole block
  const int sl = threadIdx.x >> 4, q = threadIdx.x & 15;
  const int il = tile * kSplitSites + sl;
  const bool on = il < a.nsites;
  int i = a.site0 + il;
  if (i >= g.Vh) i -= g.Vh;
  __shared__ double2 W[kSplitSites][16][3];
  __shared__ double2 Rs[kSplitSites][12];
  // step 2: 12 threads per site, in three full warps
  const int s2 = threadIdx.x / 12, q2 = threadIdx.x - 12 * s2;
  const int sp = q2 / 3, c = q2 - 3 * sp, ch = sp >> 1, row = (sp & 1) * 3 + c;
  const int il2 = tile * kSplitSites + s2;
  const bool work = s2 < kSplitSites && il2 < a.nsites;
  int i2 = a.site0 + il2;
  if (i2 >= g.Vh) i2 -= g.Vh;
  Cx<double> ko[6], ow[6];
  if (work && a.own_op) {
    const double2* o = a.own.p + (size_t)j * a.own.rhs + split_site(g, a.own.lay, a.p_out, i2);
    const size_t cs = a.own.lay == kLayInternal ? (size_t)g.Vh : 1;
#pragma unroll
    for (int r = 0; r < 6; r++) {
      const double2 e = o[(size_t)(6 * ch + r) * cs];
      ow[r] = cx<double>(e.x, e.y);
    }
    if (a.own_op == 2) load_row(a.Kown, g.Vh, i2, ch, row, ko);
  }
  if (work && a.kout) load_row(a.Kout, g.Vh, i2, ch, row, ko);
  if (a.hop && on) {
    // 1. one direction and one projected spin: w = U (psi_s + coef psi_k), or U^dag
    const int d = q >> 1, h = q & 1, mu = d >> 1, bwd = d & 1;
    const int raw = __ldg((const int*)(a.nbr + ((size_t)a.p_out * 2 + (d >> 2)) * g.Vh + i) + (d & 3));
    const int n = raw & 0x7fffffff;
    // (1 -+ g_mu): partner spin, +-1 or +-i
    const int k = 2 + ((mu == 0 || mu == 3) ? h : 1 - h);
    const int imag = mu == 1 || mu == 3;
    const int neg = bwd ^ (mu >= 2 ? h : 0) ^ a.g5_in;
    const double2* src = a.in.p + (size_t)j * a.in.rhs + split_site(g, a.in.lay, 1 - a.p_out, n);
    const size_t cs = a.in.lay == kLayInternal ? (size_t)g.Vh : 1;
    const double2* u = a.U + (size_t)((bwd ? 1 - a.p_out : a.p_out) * 4 + mu) * 9 * g.Vh + (bwd ? n : i);
    Cx<double> v[3], m[3][3];
#pragma unroll
    for (int c = 0; c < 3; c++) {
      const double2 x = __ldg(src + (size_t)(3 * h + c) * cs), y = __ldg(src + (size_t)(3 * k + c) * cs);
      v[c] = cx<double>(x.x, x.y) + unit_mul(cx<double>(y.x, y.y), imag, neg);
#pragma unroll
      for (int b = 0; b < 3; b++) {
        const double2 e = __ldg(u + (size_t)(bwd ? 3 * b + c : 3 * c + b) * g.Vh);
        m[c][b] = cx<double>(e.x, flip_if(e.y, bwd));
      }
    }
#pragma unroll
    for (int c = 0; c < 3; c++) {
      Cx<double> w = m[c][0] * v[0];
      fma_acc(w, m[c][1], v[1]);
      fma_acc(w, m[c][2], v[2]);
      // antiperiodic time: bit 31 of the neighbour word
      W[sl][q][c] = make_double2(flip_if(w.re, raw < 0), flip_if(w.im, raw < 0));
    }
  }
  __syncthreads();
  // 2. one spin-colour row: sum over the directions
  Cx<double> res = cx<double>(0, 0);
  if (work && a.hop) {
#pragma unroll
    for (int d = 0; d < 8; d++) {
      const int mu = d >> 1, bwd = d & 1;
      // spins 2, 3 of (1 -+ g_mu) from the projected ones: the entry of row sp of -+g_mu
      const int up = sp < 2;
      const int h = up ? sp : ((mu == 0 || mu == 3) ? sp - 2 : 3 - sp);
      const int imag = !up && (mu == 1 || mu == 3);
      const int neg = !up && (mu == 0 ? bwd : mu == 1 ? 1 - bwd : (bwd ^ (sp == 2)));
      const double2 w = W[s2][2 * d + h][c];
      res = res + unit_mul(cx<double>(w.x, w.y), imag, neg);
    }
    const double f = flip_if(-0.5 * a.s, a.g5_hop && sp >= 2);
    res = f * res;
  }
  if (work && a.own_op) {
    Cx<double> t = cx<double>(0, 0);
    if (a.own_op == 2) t = row_mul(ko, ow, row);
    else {
#pragma unroll
      for (int r = 0; r < 6; r++)
        if (r == row) t = ow[r];
    }
    res = res + t;
  }
  if (a.kout) {
    if (work) Rs[s2][q2] = make_double2(res.re, res.im);
    __syncthreads();
    if (work) {
      Cx<double> v[6];
#pragma unroll
      for (int r = 0; r < 6; r++) v[r] = cx<double>(Rs[s2][6 * ch + r].x, Rs[s2][6 * ch + r].y);
      res = row_mul(ko, v, row);
    }
  }
  double nrm = 0;
  if (work) {
    if (a.cg_x) {                            // the CG update of k_hop's epilogue
      const size_t o = ((size_t)12 * j + q2) * g.Vh + i2;
      const double al = a.cg_alpha[j];
      double2 x = a.cg_x[o], r = a.cg_r[o];
      const double2 p = a.cg_p[o];
      x.x += al * p.x; x.y += al * p.y;
      r.x -= al * res.re; r.y -= al * res.im;
      a.cg_x[o] = x;
      a.cg_r[o] = r;
      nrm = r.x * r.x + r.y * r.y;
    } else {
      double2* o = a.out.p + (size_t)j * a.out.rhs + split_site(g, a.out.lay, a.p_out, i2);
      o[(size_t)q2 * (a.out.lay == kLayInternal ? (size_t)g.Vh : 1)] = make_double2(res.re, res.im);
      nrm = norm2(res);
    }
  }
  if (a.norm_part) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) nrm += __shfl_down_sync(0xffffffffu, nrm, o);
    __shared__ double red[kSplitSites / 2];
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = nrm;
    __syncthreads();
    if (threadIdx.x == 0) {
      double t = 0;
#pragma unroll
      for (int w = 0; w < kSplitSites / 2; w++) t += red[w];
      a.norm_part[(size_t)j * a.ntiles + tile] = t;
    }
  }
}
