// What goes into an LU and what its pivots mean, for the kernels of the
// single-system path (ingest.cu) and the batched engine (batched_impl.cuh).
#pragma once

#include <cstring>
#include <type_traits>

#include "common.cuh"

namespace msir {

// One working-precision entry in the factor format.  16-bit formats round
// from fp32, so an fp32 entry needs no way through fp64.
template <typename F, typename U0>
__device__ __forceinline__ F narrow(U0 v) {
  if constexpr (std::is_same<U0, float>::value && sizeof(F) <= 4) return from_t<F>(v);
  else return from_d<F>((double)v);
}

// Entries j .. j + kFactorVec - 1 (those below n) of row i in the factor
// format: fl_f(a_ij), or fl_f(fl_32(mu R_i a_ij S_j)) with scalings.  Rows
// start on 16-byte boundaries and j is a multiple of kFactorVec; what lies
// past column n is not written.
constexpr int kFactorVec = 8;
template <typename U0, typename F>
__device__ __forceinline__ void factor_piece(const U0* row, int i, int j, int n, F* out_row, const double* R,
                                             const double* S, double mu) {
  const U0* src = row + j;
  F* dst = out_row + j;
  auto entry = [&](U0 a, int e) {
    if (!R) return narrow<F>(a);
    const double v = (double)a;
    return from_d<F>(v * R[i] * S[j + e] * mu);
  };
  if (j + kFactorVec <= n) {
    constexpr int kIn = kFactorVec * (int)sizeof(U0) / 16, kOut = kFactorVec * (int)sizeof(F) / 16;
    uint4 in[kIn], out[kOut];
    U0 a[kFactorVec];
    F f[kFactorVec];
#pragma unroll
    for (int q = 0; q < kIn; ++q) in[q] = ((const uint4*)src)[q];
    memcpy(a, in, sizeof(in));
#pragma unroll
    for (int e = 0; e < kFactorVec; ++e) f[e] = entry(a[e], e);
    memcpy(out, f, sizeof(out));
#pragma unroll
    for (int q = 0; q < kOut; ++q) ((uint4*)dst)[q] = out[q];
  } else {
    for (int e = 0; j + e < n; ++e) dst[e] = entry(src[e], e);
  }
}

// Permutation of LAPACK-style interchanges, (P A)[i] = A[perm[i]], by one
// block.  The interchanges are sequential, but runs of them can be applied
// side by side: one warp per run starts from the identity (16-bit labels in
// shared memory), one of its lanes applying the run's interchanges, and the
// runs' permutations are chained.  sm: n (4 + 2 runs) bytes, at least runs
// warps.  (One thread for all of them took 0.31 ms at n = 8192: about 75
// cycles each.)
constexpr int kPermRuns = 8;
static __device__ void perm_of_pivots(const int* ipiv, int n, int* perm, int runs, int* sm) {
  int* si = sm;
  unsigned short* lab = (unsigned short*)(sm + n);
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    si[i] = ipiv[i];
    for (int q = 0; q < runs; ++q) lab[(size_t)q * n + i] = (unsigned short)i;
  }
  __syncthreads();
  const int run = threadIdx.x >> 5, per = (n + runs - 1) / runs;
  if (run < runs && (threadIdx.x & 31) == 0) {
    unsigned short* l = lab + (size_t)run * n;
    for (int j = run * per; j < min((run + 1) * per, n); ++j) {
      const int p = si[j];
      if (p != j) {
        const unsigned short t = l[j];
        l[j] = l[p];
        l[p] = t;
      }
    }
  }
  __syncthreads();
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    int v = i;
    for (int q = runs - 1; q >= 0; --q) v = lab[(size_t)q * n + v];
    perm[i] = v;
  }
  __syncthreads();
}

}  // namespace msir
