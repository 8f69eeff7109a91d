// Explicitly rounded arithmetic of the LU kernels in T = float / double,
// rounding to the storage format F, and what the panels of the two LUs
// (lu_panel.cuh: a cluster, lu_cta.cuh: one block) share.
#pragma once

#include <climits>
#include <cstring>

#include "common.cuh"

namespace msir {

template <typename T> __device__ __forceinline__ T mul_rn(T a, T b);
template <> __device__ __forceinline__ float mul_rn<float>(float a, float b) { return __fmul_rn(a, b); }
template <> __device__ __forceinline__ double mul_rn<double>(double a, double b) { return __dmul_rn(a, b); }
template <typename T> __device__ __forceinline__ T sub_rn(T a, T b);
template <> __device__ __forceinline__ float sub_rn<float>(float a, float b) { return __fsub_rn(a, b); }
template <> __device__ __forceinline__ double sub_rn<double>(double a, double b) { return __dsub_rn(a, b); }
template <typename T> __device__ __forceinline__ T div_rn(T a, T b);
template <> __device__ __forceinline__ float div_rn<float>(float a, float b) { return __fdiv_rn(a, b); }
template <> __device__ __forceinline__ double div_rn<double>(double a, double b) { return __ddiv_rn(a, b); }
template <typename T> __device__ __forceinline__ T fma_rn(T a, T b, T c);
template <> __device__ __forceinline__ float fma_rn<float>(float a, float b, float c) { return __fmaf_rn(a, b, c); }
template <> __device__ __forceinline__ double fma_rn<double>(double a, double b, double c) { return __fma_rn(a, b, c); }

template <typename F> __device__ __forceinline__ F store_rn(typename Fmt<F>::T v);
template <> __device__ __forceinline__ __half store_rn<__half>(float v) { return __float2half_rn(v); }
template <> __device__ __forceinline__ __nv_bfloat16 store_rn<__nv_bfloat16>(float v) {
  return __float2bfloat16_rn(v);
}
template <> __device__ __forceinline__ float store_rn<float>(float v) { return v; }
template <> __device__ __forceinline__ double store_rn<double>(double v) { return v; }

// Panel width limit per arithmetic precision (also the register arrays).
template <typename T> struct PanelNB { static constexpr int v = 32; };
template <> struct PanelNB<double> { static constexpr int v = 16; };

// Pivot order: larger |a| first; NaN only if nothing else; equal magnitudes
// -> smaller row index.
// Pivot keys: monotone in |a|, 0 for "no candidate", 1 for NaN (chosen only
// if nothing else is left), else the bits of |a| plus 2 (the bits of a
// non-negative IEEE number order like its value).
template <typename T> struct PivKey;
template <> struct PivKey<float> {
  using K = unsigned;
  static __device__ __forceinline__ K of(float v) {
    const unsigned b = __float_as_uint(v) & 0x7fffffffu;
    return b > 0x7f800000u ? 1u : b + 2u;
  }
};
template <> struct PivKey<double> {
  using K = unsigned long long;
  static __device__ __forceinline__ K of(double v) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(v) & 0x7fffffffffffffffull;
    return b > 0x7ff0000000000000ull ? 1ull : b + 2ull;
  }
};
// Largest key of the warp and the smallest index among the lanes holding it.
__device__ __forceinline__ void warp_argmax(unsigned& key, int& i) {
  const unsigned mk = __reduce_max_sync(0xffffffffu, key);
  i = __reduce_min_sync(0xffffffffu, key == mk ? i : INT_MAX);
  key = mk;
}
__device__ __forceinline__ void warp_argmax(unsigned long long& key, int& i) {
  const unsigned hi = (unsigned)(key >> 32);
  const unsigned mh = __reduce_max_sync(0xffffffffu, hi);
  const unsigned ml = __reduce_max_sync(0xffffffffu, hi == mh ? (unsigned)key : 0u);
  const unsigned long long mk = ((unsigned long long)mh << 32) | ml;
  i = __reduce_min_sync(0xffffffffu, key == mk ? i : INT_MAX);
  key = mk;
}

// N consecutive values of T in 16-byte loads / stores (16-byte aligned).
template <typename T, int N>
__device__ __forceinline__ void ld_vec(const T* p, T (&v)[N]) {
  constexpr int E = 16 / (int)sizeof(T);
  static_assert(N % E == 0, "whole 16-byte loads");
#pragma unroll
  for (int m = 0; m < N / E; ++m) {
    const uint4 u = reinterpret_cast<const uint4*>(p)[m];
    memcpy(&v[m * E], &u, 16);
  }
}
template <typename T, int N>
__device__ __forceinline__ void st_vec(T* p, const T (&v)[N]) {
  constexpr int E = 16 / (int)sizeof(T);
  static_assert(N % E == 0, "whole 16-byte stores");
#pragma unroll
  for (int m = 0; m < N / E; ++m) {
    uint4 u;
    memcpy(&u, &v[m * E], 16);
    reinterpret_cast<uint4*>(p)[m] = u;
  }
}

// One step of applying the interchange (j, q) to the position of a row.
__device__ __forceinline__ int swap_step(int pos, int j, int q) { return pos == j ? q : (pos == q ? j : pos); }

}  // namespace msir
