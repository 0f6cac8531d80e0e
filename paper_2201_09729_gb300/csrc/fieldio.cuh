// Field I/O shared by the stencil and the solver: one spinor per (site, rhs)
// in the internal even-odd SoA layouts (see Field in common.cuh).
#pragma once
#include "common.cuh"

// R: vector arithmetic, S: links and clover, lanes: right-hand sides per vector
template <int P> struct PT { typedef float R; typedef float S; static constexpr int lanes = 1; };
template <> struct PT<DLMA_FP64> { typedef double R; typedef double S; static constexpr int lanes = 1; };
template <> struct PT<kFP32x2> { typedef f2 R; typedef float S; static constexpr int lanes = 2; };

template <class R> struct Spinor { Cx<R> c[4][3]; };

// per-rhs values of vector j: one value, or the pair's two (an empty partner reads the first)
__device__ __forceinline__ float lane_get(f2 v, int q) { return q ? v.y : v.x; }
__device__ __forceinline__ float lane_get(float v, int) { return v; }
__device__ __forceinline__ double lane_get(double v, int) { return v; }
template <int P> __device__ __forceinline__ typename PT<P>::R lane_pack(double a, double b) {
  if constexpr (P == kFP32x2) return f2((float)a, (float)b);
  else return (typename PT<P>::R)a;
}
// right-hand side of lane q of vector j, and whether it is there and on (mask may be null)
template <int P> __device__ __forceinline__ int lane_rhs(int j, int q, int nrhs) {
  const int r = PT<P>::lanes * j + q;
  return r < nrhs ? r : nrhs - 1;
}
template <int P> __device__ __forceinline__ bool lane_on(int j, int q, int nrhs, const int* mask) {
  const int r = PT<P>::lanes * j + q;
  return r < nrhs && (!mask || mask[r] != 0);
}
template <int P> __device__ __forceinline__ bool vec_on(int j, int nrhs, const int* mask) {
  bool on = lane_on<P>(j, 0, nrhs, mask);
  if constexpr (PT<P>::lanes == 2) on = on || lane_on<P>(j, 1, nrhs, mask);
  return on;
}

template <int P>
__device__ __forceinline__ Spinor<typename PT<P>::R> load_spinor(const void* __restrict__ base,
                                                                 const float* __restrict__ scale, int Vh, int i) {
  typedef typename PT<P>::R R;
  Spinor<R> s;
  if constexpr (P == DLMA_FP64) {
    const double2* b = (const double2*)base;
#pragma unroll
    for (int k = 0; k < 12; k++) {
      double2 v = __ldg(b + (size_t)k * Vh + i);
      s.c[k / 3][k % 3] = cx<R>((R)v.x, (R)v.y);
    }
  } else if constexpr (P == kFP32x2) {
    const float4* b = (const float4*)base;
#pragma unroll
    for (int k = 0; k < 12; k++) {
      const float4 v = __ldg(b + (size_t)k * Vh + i);
      s.c[k / 3][k % 3] = cx<R>(f2(v.x, v.y), f2(v.z, v.w));
    }
  } else if constexpr (P == DLMA_FP32) {
    const float4* b = (const float4*)base;
#pragma unroll
    for (int q = 0; q < 6; q++) {
      float4 v = __ldg(b + (size_t)q * Vh + i);
      s.c[(2 * q) / 3][(2 * q) % 3] = cx<R>(v.x, v.y);
      s.c[(2 * q + 1) / 3][(2 * q + 1) % 3] = cx<R>(v.z, v.w);
    }
  } else {
    const uint4* b = (const uint4*)base;
    float sc = __ldg(scale + i);
#pragma unroll
    for (int q = 0; q < 3; q++) {
      uint4 v = __ldg(b + (size_t)q * Vh + i);
      unsigned w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
      for (int r = 0; r < 4; r++) {
        float2 f = __half22float2(*(__half2*)&w[r]);
        int k = 4 * q + r;
        s.c[k / 3][k % 3] = cx<R>(f.x * sc, f.y * sc);
      }
    }
  }
  return s;
}

template <int P>
__device__ __forceinline__ void store_spinor(void* base, float* scale, int Vh, int i,
                                             const Spinor<typename PT<P>::R>& s) {
  if constexpr (P == DLMA_FP64) {
    double2* b = (double2*)base;
#pragma unroll
    for (int k = 0; k < 12; k++) b[(size_t)k * Vh + i] = make_double2(s.c[k / 3][k % 3].re, s.c[k / 3][k % 3].im);
  } else if constexpr (P == kFP32x2) {
    float4* b = (float4*)base;
#pragma unroll
    for (int k = 0; k < 12; k++) {
      const Cx<f2> v = s.c[k / 3][k % 3];
      b[(size_t)k * Vh + i] = make_float4(v.re.x, v.re.y, v.im.x, v.im.y);
    }
  } else if constexpr (P == DLMA_FP32) {
    float4* b = (float4*)base;
#pragma unroll
    for (int q = 0; q < 6; q++) {
      Cx<float> a0 = cx<float>((float)s.c[(2 * q) / 3][(2 * q) % 3].re, (float)s.c[(2 * q) / 3][(2 * q) % 3].im);
      Cx<float> a1 = cx<float>((float)s.c[(2 * q + 1) / 3][(2 * q + 1) % 3].re,
                               (float)s.c[(2 * q + 1) / 3][(2 * q + 1) % 3].im);
      b[(size_t)q * Vh + i] = make_float4(a0.re, a0.im, a1.re, a1.im);
    }
  } else {
    float m = 0.f;
#pragma unroll
    for (int k = 0; k < 12; k++)
      m = fmaxf(m, fmaxf(fabsf((float)s.c[k / 3][k % 3].re), fabsf((float)s.c[k / 3][k % 3].im)));
    // sites below 1e-30 (down to float denormals, whose reciprocal overflows) are flushed to zero
    if (!(m > 1e-30f)) m = 0.f;
    const float inv = m > 0.f ? 1.f / m : 0.f;
    uint4* b = (uint4*)base;
#pragma unroll
    for (int q = 0; q < 3; q++) {
      unsigned w[4];
#pragma unroll
      for (int r = 0; r < 4; r++) {
        int k = 4 * q + r;
        __half2 h = __floats2half2_rn((float)s.c[k / 3][k % 3].re * inv, (float)s.c[k / 3][k % 3].im * inv);
        w[r] = *(unsigned*)&h;
      }
      b[(size_t)q * Vh + i] = make_uint4(w[0], w[1], w[2], w[3]);
    }
    scale[i] = m;
  }
}


// component k (3 spin + colour) of an FP64 or FP32 vector: the kernels that stream many
// vectors go through them component by component, which keeps few registers alive
template <int P>
__device__ __forceinline__ Cx<typename PT<P>::R> load_comp(const void* __restrict__ base, int Vh, int i, int k) {
  if constexpr (P == kFP32x2) {
    const float4 v = __ldg((const float4*)base + (size_t)k * Vh + i);
    return cx<f2>(f2(v.x, v.y), f2(v.z, v.w));
  } else if constexpr (P == DLMA_FP32) {
    const float2 v = __ldg((const float2*)base + ((size_t)(k >> 1) * Vh + i) * 2 + (k & 1));
    return cx<float>(v.x, v.y);
  } else {
    const double2 v = __ldg((const double2*)base + (size_t)k * Vh + i);
    return cx<double>(v.x, v.y);
  }
}
template <int P>
__device__ __forceinline__ void store_comp(void* base, int Vh, int i, int k, Cx<typename PT<P>::R> v) {
  if constexpr (P == kFP32x2)
    ((float4*)base)[(size_t)k * Vh + i] = make_float4(v.re.x, v.re.y, v.im.x, v.im.y);
  else if constexpr (P == DLMA_FP32)
    ((float2*)base)[((size_t)(k >> 1) * Vh + i) * 2 + (k & 1)] = make_float2(v.re, v.im);
  else
    ((double2*)base)[(size_t)k * Vh + i] = make_double2(v.re, v.im);
}

// components 4 g .. 4 g + 3
template <int P>
__device__ __forceinline__ void load_comp4(const void* __restrict__ base, int Vh, int i, int g,
                                           Cx<typename PT<P>::R> (&v)[4]) {
  if constexpr (P == DLMA_FP32) {
#pragma unroll
    for (int h = 0; h < 2; h++) {
      const float4 e = __ldg((const float4*)base + (size_t)(2 * g + h) * Vh + i);
      v[2 * h] = cx<float>(e.x, e.y);
      v[2 * h + 1] = cx<float>(e.z, e.w);
    }
  } else {
#pragma unroll
    for (int k = 0; k < 4; k++) v[k] = load_comp<P>(base, Vh, i, 4 * g + k);
  }
}
template <int P>
__device__ __forceinline__ void store_comp4(void* base, int Vh, int i, int g, const Cx<typename PT<P>::R> (&v)[4]) {
  if constexpr (P == DLMA_FP32) {
#pragma unroll
    for (int h = 0; h < 2; h++)
      ((float4*)base)[(size_t)(2 * g + h) * Vh + i] =
          make_float4(v[2 * h].re, v[2 * h].im, v[2 * h + 1].re, v[2 * h + 1].im);
  } else {
#pragma unroll
    for (int k = 0; k < 4; k++) store_comp<P>(base, Vh, i, 4 * g + k, v[k]);
  }
}
