// Inverses of the 64x64 diagonal blocks of packed LU factors, formed by the
// refinement kernels when a solve first needs them (refine_impl.cuh).
//
// The inverse X of one triangular block is built by doubling: the 8x8
// diagonal blocks by substitution on the columns of the identity (one thread
// per column), then 16, 32 and 64 from halves,
//   L:  X21 = -X22 (L21 X11)        U:  X12 = -X11 (U12 X22),
// two small products per step with every element a sum of its own, so that
// all 256 threads work and only 2 x 3 barriers separate the products.
//
// Arithmetic (AR): sums of products are compensated (every product's and
// addition's rounding error is kept in a second word, Ogita, Rump and
// Oishi's Dot2, with the low words of pair operands added), results are
// unevaluated pairs h + l:
//   ArFF  pairs of fp32 (about 2^-46 per operation, all work on the fp32
//         pipe): for fp32 solves, whose inverse is the pair rounded to fp32,
//         while the block's condition (inv_cond_below) leaves some 2^-30 of
//         that, as it does for LU factors; other blocks take ArDD;
//   ArDD  pairs of fp64 (about 2^-104): for fp64 solves (the high word) and
//         double-double ones.
#pragma once

#include "common.cuh"

namespace msir {

constexpr int kIB = 64;
constexpr int kInvThreads = 256;
constexpr int kXld = kIB + 1;
// B (64 x 65), Xh, Xl (64 x 65), Th, Tl (32 x 33), reciprocals (2 x 64)
constexpr size_t kInvValues = 3 * kIB * kXld + 2 * (kIB / 2) * (kIB / 2 + 1) + 2 * kIB;
constexpr size_t kInvSmem = sizeof(double) * kInvValues;

// fp32 value nearest to hi + lo (normalised dd): fl32(hi) unless hi is an
// exact tie between two fp32 neighbours, in which case lo decides.
__device__ __forceinline__ float dd_to_f32(double hi, double lo) {
  const float r = __double2float_rn(hi);
  const double rd = (double)r;
  const double d = hi - rd;  // exact
  if (d == 0.0 || lo == 0.0 || !isfinite(rd)) return r;
  const float o = nextafterf(r, d > 0.0 ? INFINITY : -INFINITY);
  if ((double)o - rd != 2.0 * d) return r;  // not a tie
  return ((lo > 0.0) == (d > 0.0)) ? o : r;
}

struct ArFF {
  using S = float;
  struct V { float h, l; };
  using Acc = ff_t;
  static __device__ __forceinline__ Acc zero() { return ff_t{0.0f, 0.0f}; }
  static __device__ __forceinline__ Acc add(Acc a, float p, float e) {
    float s, r;
    two_sum_f(a.s, p, s, r);
    return ff_t{s, __fadd_rn(a.c, __fadd_rn(r, e))};
  }
  // acc + f x, and acc + x y
  static __device__ __forceinline__ Acc term(S f, V x, Acc a) {
    const float p = __fmul_rn(f, x.h);
    return add(a, p, __fmaf_rn(f, x.l, __fmaf_rn(f, x.h, -p)));
  }
  static __device__ __forceinline__ Acc term(V x, V y, Acc a) {
    const float p = __fmul_rn(x.h, y.h);
    return add(a, p, __fmaf_rn(x.l, y.h, __fmaf_rn(x.h, y.l, __fmaf_rn(x.h, y.h, -p))));
  }
  static __device__ __forceinline__ V fin(Acc a) {
    float s, e;
    two_sum_f(a.s, a.c, s, e);
    return V{s, e};
  }
  static __device__ __forceinline__ V neg(V x) { return V{-x.h, -x.l}; }
  static __device__ __forceinline__ V recip(S d) {
    const float q = __fdiv_rn(1.0f, d);
    return V{q, __fdiv_rn(__fmaf_rn(-q, d, 1.0f), d)};
  }
};
struct ArDD {
  using S = double;
  struct V { double h, l; };
  struct Acc { double s, c; };
  static __device__ __forceinline__ Acc zero() { return Acc{0.0, 0.0}; }
  static __device__ __forceinline__ Acc add(Acc a, double p, double e) {
    const dd_t t = two_sum_ord(a.s, p);
    return Acc{t.hi, __dadd_rn(a.c, __dadd_rn(t.lo, e))};
  }
  static __device__ __forceinline__ Acc term(S f, V x, Acc a) {
    const double p = __dmul_rn(f, x.h);
    return add(a, p, __fma_rn(f, x.l, __fma_rn(f, x.h, -p)));
  }
  static __device__ __forceinline__ Acc term(V x, V y, Acc a) {
    const double p = __dmul_rn(x.h, y.h);
    return add(a, p, __fma_rn(x.l, y.h, __fma_rn(x.h, y.l, __fma_rn(x.h, y.h, -p))));
  }
  static __device__ __forceinline__ V fin(Acc a) {
    const dd_t t = two_sum(a.s, a.c);
    return V{t.hi, t.lo};
  }
  static __device__ __forceinline__ V neg(V x) { return V{-x.h, -x.l}; }
  static __device__ __forceinline__ V recip(S d) {
    const dd_t q = dd_div_d(dd_t{1.0, 0.0}, d);
    return V{q.hi, q.lo};
  }
};

// One doubling step: the off-diagonal h x h blocks of the inverses of the
// 2h x 2h diagonal blocks.  A thread takes CNT elements that share a factor:
// neighbouring columns in the first product, neighbouring rows in the second
// (zeros outside the triangles are part of the sums where ranges are shared).
template <typename AR, int h>
__device__ __forceinline__ void inv_double(bool lower, const typename AR::S* B, typename AR::S* Xh,
                                           typename AR::S* Xl, typename AR::S* Th, typename AR::S* Tl) {
  using V = typename AR::V;
  using Acc = typename AR::Acc;
  constexpr int kPairs = kIB / (2 * h);
  constexpr int CNT = kPairs * h * h / kInvThreads;  // 1, 2, 4 for h = 8, 16, 32
  constexpr int ldt = kIB / 2 + 1;
  const int tid = threadIdx.x;
  const int fast = tid % h;
  // pair the short and the long sums on each scheduler (warps w and w + 4)
  const int warp = tid >> 5;
  const int grp = h == 32 ? (warp < 4 ? warp : 11 - warp) : tid / h;
  {
    // T = L21 X11 (k >= j) or U12 X22 (k <= j); i = fast, j = j0 .. j0 + CNT - 1
    const int j0 = (grp * CNT) % h, p = grp * CNT / h, o = p * 2 * h;
    const int xo = lower ? o : o + h, bo = lower ? o + h : o;
    Acc acc[CNT];
#pragma unroll
    for (int q = 0; q < CNT; ++q) acc[q] = AR::zero();
    const int k0 = lower ? j0 : 0, k1 = lower ? h : j0 + CNT;
    for (int k = k0; k < k1; ++k) {
      const typename AR::S b = B[(bo + fast) * kXld + xo + k];
#pragma unroll
      for (int q = 0; q < CNT; ++q) {
        const int e = (xo + k) * kXld + xo + j0 + q;
        acc[q] = AR::term(b, V{Xh[e], Xl[e]}, acc[q]);
      }
    }
#pragma unroll
    for (int q = 0; q < CNT; ++q) {
      const V v = AR::fin(acc[q]);
      Th[(p * h + fast) * ldt + j0 + q] = v.h;
      Tl[(p * h + fast) * ldt + j0 + q] = v.l;
    }
  }
  __syncthreads();
  {
    // X21 = -X22 T (k <= i) or X12 = -X11 T (k >= i); j = fast, rows i0 ..
    const int i0 = (grp * CNT) % h, p = grp * CNT / h, o = p * 2 * h;
    const int ro = lower ? o + h : o, co = lower ? o : o + h;  // rows and columns of the result
    Acc acc[CNT];
#pragma unroll
    for (int q = 0; q < CNT; ++q) acc[q] = AR::zero();
    const int k0 = lower ? 0 : i0, k1 = lower ? i0 + CNT : h;
    for (int k = k0; k < k1; ++k) {
      const V t = V{Th[(p * h + k) * ldt + fast], Tl[(p * h + k) * ldt + fast]};
#pragma unroll
      for (int q = 0; q < CNT; ++q) {
        const int e = (ro + i0 + q) * kXld + ro + k;
        acc[q] = AR::term(V{Xh[e], Xl[e]}, t, acc[q]);
      }
    }
#pragma unroll
    for (int q = 0; q < CNT; ++q) {
      const V v = AR::neg(AR::fin(acc[q]));
      const int e = (ro + i0 + q) * kXld + co + fast;
      Xh[e] = v.h;
      Xl[e] = v.l;
    }
  }
  __syncthreads();
}

// Inverse of the 64x64 triangle staged in sm (B, identity-padded; unit
// diagonal if lower) into Xh + Xl (row stride kXld), by one block of
// kInvThreads threads; sm holds kInvValues values.  B is complete (barrier)
// on entry, X on return.
template <typename AR>
__device__ __forceinline__ void inv_triangle(bool lower, typename AR::S* sm) {
  using S = typename AR::S;
  using V = typename AR::V;
  const S* B = sm;
  S* Xh = sm + kIB * kXld;
  S* Xl = Xh + kIB * kXld;
  S* Th = Xl + kIB * kXld;
  S* Tl = Th + (kIB / 2) * (kIB / 2 + 1);
  S* rh = Tl + (kIB / 2) * (kIB / 2 + 1);
  S* rl = rh + kIB;
  const int tid = threadIdx.x;
  if (tid < kIB) {
    const V r = lower ? V{(S)1, (S)0} : AR::recip(B[tid * kXld + tid]);
    rh[tid] = r.h;
    rl[tid] = r.l;
  }
  for (int e = tid; e < kIB * kXld; e += kInvThreads) Xh[e] = Xl[e] = (S)0;
  __syncthreads();
  if (tid < kIB) {
    // 8x8 diagonal blocks: column c of block o, rows in the order of the
    // substitution (x is zero outside the triangle)
    constexpr int b = 8;
    const int o = tid / b * b, c = tid % b;
    V x[b];
#pragma unroll
    for (int s = 0; s < b; ++s) {
      // row s of the substitution: i = s (L) or b - 1 - s (U)
      typename AR::Acc acc = AR::zero();
      const int i = lower ? s : b - 1 - s;
#pragma unroll
      for (int q = 0; q < s; ++q) {
        const int k = lower ? q : b - 1 - q;
        acc = AR::term(B[(o + i) * kXld + o + k], x[q], acc);
      }
      V v = AR::neg(AR::fin(acc));
      if (i == c) v = V{(S)1, (S)0};
      if (!lower) v = AR::fin(AR::term(v, V{rh[o + i], rl[o + i]}, AR::zero()));
      x[s] = v;
      Xh[(o + i) * kXld + o + c] = v.h;
      Xl[(o + i) * kXld + o + c] = v.l;
    }
  }
  __syncthreads();
  inv_double<AR, 8>(lower, B, Xh, Xl, Th, Tl);
  inv_double<AR, 16>(lower, B, Xh, Xl, Th, Tl);
  inv_double<AR, 32>(lower, B, Xh, Xl, Th, Tl);
}

// |A||B| of two 64x64 arrays of row stride kXld, four by four elements a
// thread.
__device__ __forceinline__ void abs_product(const float* A, const float* B, float (&c)[4][4]) {
  const int i0 = (threadIdx.x >> 4) * 4, j0 = (threadIdx.x & 15) * 4;
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) c[i][j] = 0.0f;
  for (int k = 0; k < kIB; ++k)
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j)
        c[i][j] = __fmaf_rn(fabsf(A[(i0 + i) * kXld + k]), fabsf(B[k * kXld + j0 + j]), c[i][j]);
}

// Whether the pairs' inverse X of the triangle B in sm (inv_triangle's
// arrangement, twice kInvValues values) is good to 2^-46 `limit` of itself:
// its error is 2^-46 |X||B||X|.  First by Skeel's condition number
// max_i (|X||B|e)_i, which bounds that and does not see how the rows are
// scaled, but grows with the scaling of the columns; where it is above the
// limit, by the largest element of a column of |X||B||X| relative to that of
// X.  False if X is not finite.
static __device__ __noinline__ bool inv_cond_below(float* sm, float limit) {
  const float* X = sm + kIB * kXld;
  float* sum = sm + kInvValues - kIB;  // (the reciprocals' low words are no longer read)
  const int row = threadIdx.x >> 2, part = threadIdx.x & 3;
  float s = 0.0f;
  for (int k = part; k < kIB; k += 4) s += fabsf(sm[row * kXld + k]);
  s += __shfl_xor_sync(0xffffffffu, s, 1);
  s += __shfl_xor_sync(0xffffffffu, s, 2);
  if (part == 0) sum[row] = s;
  __syncthreads();
  float v = 0.0f;
  for (int k = part; k < kIB; k += 4) v += fabsf(X[row * kXld + k]) * sum[k];
  v += __shfl_xor_sync(0xffffffffu, v, 1);
  v += __shfl_xor_sync(0xffffffffu, v, 2);
  if (__syncthreads_and(v <= limit)) return true;
  float* W = sm + kInvValues;
  int* top = (int*)(W + kIB * kXld);  // columns' largest elements of X, then of |X||B||X| (bits order like values)
  const int i0 = (threadIdx.x >> 4) * 4, j0 = (threadIdx.x & 15) * 4;
  float c[4][4];
  abs_product(sm, X, c);
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) W[(i0 + i) * kXld + j0 + j] = c[i][j];
  if (threadIdx.x < 2 * kIB) top[threadIdx.x] = 0;
  __syncthreads();
  abs_product(X, W, c);
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    int x = 0, y = 0;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      x = max(x, __float_as_int(fabsf(X[(i0 + i) * kXld + j0 + j])));
      y = max(y, __float_as_int(c[i][j]));
    }
    atomicMax(top + j0 + j, x);
    atomicMax(top + kIB + j0 + j, y);
  }
  __syncthreads();
  const int q = threadIdx.x & (kIB - 1);
  return __syncthreads_and(__int_as_float(top[kIB + q]) <= limit * __int_as_float(top[q])) != 0;
}

// Diagonal block b of triangle `lower` (get(i, k): the packed factor's entry
// (64 b + i, 64 b + k)) into sm; entries outside the n - 64 b rows and
// columns of a ragged last block are those of the identity.
template <typename S, typename Get>
__device__ __forceinline__ void inv_load(S* sm, int n, int b, bool lower, Get get) {
  const int nr = min(kIB, n - b * kIB);
  for (int idx = threadIdx.x; idx < kIB * kIB; idx += kInvThreads) {
    const int i = idx / kIB, k = idx % kIB;
    S v = (S)(i == k ? 1 : 0);
    if (i < nr && k < nr && (lower ? k < i : k >= i)) v = (S)get(i, k);
    sm[i * kXld + k] = v;
  }
  __syncthreads();
}

}  // namespace msir
