// LU factorisation by one thread block, for the batched engine's small
// systems (n <= kCtaLuMax): Algorithm 4's first step, A = LU by blocked
// right-looking GEPP in u_f (Sec. 1), with the rounding points of the
// library's multi-kernel LU:
//
//  * the matrix is held in u_f storage between steps;
//  * a panel of nb columns is widened to the arithmetic precision T (fp32
//    for u_f <= fp32, fp64 for u_f = fp64) and factored column by column:
//    pivot = largest |a_ij| (ties to the smallest row, NaN never chosen
//    unless every candidate is NaN), full panel rows swapped, the column
//    below divided by the pivot, the trailing panel columns updated with a
//    rounded product and a rounded difference; a zero pivot is recorded and
//    skipped; the panel is stored back in u_f;
//  * interchanges reach the other columns of the outer block, U12 =
//    L11^{-1} A12 by forward substitution in T (rounded product, rounded
//    difference, ascending), stored in u_f;
//  * trailing updates: per element a fused multiply-add chain in T over the
//    K products in ascending order from zero, then one rounded difference
//    and the u_f store.  Two-level blocking: panels of nb inside outer
//    blocks of nbo columns.
//
// For u_f = fp32 / fp64 this is the oracle's model operation for operation.
// The bf16 / fp16 outer update (K = nbo), which the multi-kernel LU runs on
// the tensor cores with fp32 accumulation in an order the hardware does not
// fix, is here the ascending fp32 chain.
//
// How the block does it:
//  * panel: the register panel of lu_panel.cuh without a cluster.  A thread
//    keeps one or two rows, carries their positions instead of moving them,
//    one barrier a column; the columns are stored to the rows' old places,
//    and the rows that changed place (at most 2 nb) then move as a whole,
//    16 bytes at a time through shared memory, which is the interchange of
//    every other column too (none of them is read in between);
//  * substitution: a thread per column, 32 unknowns in registers at a time;
//  * update: 64 x 64 tiles, 4 x 4 elements a thread, operands in shared
//    memory.
// Bound by the latency of the panel's columns and the substitution's chains,
// 8 warps on an SM.  n = 511, fp16, one block: 7.0 ms with the panel, the
// interchanges and the substitution element by element through shared and
// global memory, 2.5 ms so.
#pragma once

#include <type_traits>

#include "common.cuh"
#include "lu_arith.cuh"

namespace msir {

constexpr int kCtaLuMax = 512;    // largest n the batched engine factors in one block
constexpr int kCtaLuThreads = 256;
constexpr int kCtaLuWarps = kCtaLuThreads / 32;

// arithmetic precision of a u_f factorisation
template <typename F> using LuT = typename Fmt<F>::T;

// Shared memory: the panel's candidates and lists, then one area for the
// phases in turn: moved rows, the substitution (two diagonal blocks and the
// block between them, 32 parked unknowns a thread), the update's tiles.
struct CtaLuHead {
  unsigned char stage[2 * kCtaLuWarps * 128];  // candidate rows of the warps
  unsigned long long key[2][kCtaLuWarps];
  int idx[2][kCtaLuWarps];
  int piv[32];
  int from[64], to[64];  // rows that change place
  int cnt, info, nonfinite, pad;
};
constexpr int kCtaLuHead = (sizeof(CtaLuHead) + 127) / 128 * 128;
constexpr int kCtaMoveBytes = 65536;
constexpr int kCtaTriLd = 36, kCtaTileLd = 68;
template <typename F>
constexpr size_t cta_lu_smem() {
  const size_t trsm = (2 * 32 * kCtaTriLd + 32 * 32 + 32 * kCtaLuThreads) * sizeof(LuT<F>);
  const size_t upd = 2 * 64 * kCtaTileLd * sizeof(LuT<F>);
  const size_t m = trsm > upd ? trsm : upd;
  return kCtaLuHead + (m > kCtaMoveBytes ? m : kCtaMoveBytes);
}

// Factor the panel A[kk.., kk..kk+w) (m = n - kk <= RPT * kCtaLuThreads
// rows).  Its columns go back to the rows' old places; h lists the rows that
// change place.
template <typename F, int RPT>
__device__ __noinline__ void cta_panel(F* A, int lda, int n, int kk, int w, int* ipiv, CtaLuHead* h) {
  using T = LuT<F>;
  using PK = PivKey<T>;
  using K = typename PK::K;
  constexpr int NBM = PanelNB<T>::v, CH = 8, NCH = NBM / CH, NW = kCtaLuWarps;
  static_assert(NBM * sizeof(T) == 128, "candidate row");
  const int m = n - kk, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const bool al = (kk & (CH - 1)) == 0;  // rows of the panel start on 16-byte boundaries
  T row[RPT][NBM];
  int pos[RPT];
#pragma unroll
  for (int q = 0; q < RPT; ++q) {
    const int li = tid + q * kCtaLuThreads;
    pos[q] = li < m ? li : -1;
    const F* src = A + (size_t)(kk + (li < m ? li : 0)) * lda + kk;
    if (li < m && w == NBM && al) {
      F e[NBM];
      ld_vec<F, NBM>(src, e);
#pragma unroll
      for (int c = 0; c < NBM; ++c) row[q][c] = (T)to_f(e[c]);
    } else {
#pragma unroll
      for (int c = 0; c < NBM; ++c) row[q][c] = (li < m && c < w) ? (T)to_f(src[c]) : (T)0;
    }
  }
  if (tid == 0) h->cnt = 0;
  int nf = 0;
  for (int jc = 0; jc < NCH && jc * CH < w; ++jc) {
    const int gmax = NCH - jc;  // registers 0 .. NBM - 1 hold columns CH jc ..
#pragma unroll
    for (int jj = 0; jj < CH; ++jj) {
      const int j = jc * CH + jj;
      if (j < w) {
        const int buf = jj & 1;
        K key = 0;
        int p = INT_MAX;
#pragma unroll
        for (int q = 0; q < RPT; ++q) {
          const K kq = pos[q] >= j ? PK::of(row[q][jj]) : (K)0;
          const bool b = kq > key || (kq == key && kq != 0 && pos[q] < p);
          key = b ? kq : key;
          p = b ? pos[q] : p;
        }
        warp_argmax(key, p);
        T* st = (T*)(h->stage + (buf * NW + warp) * 128);
#pragma unroll
        for (int q = 0; q < RPT; ++q)
          if (pos[q] == p) {
#pragma unroll
            for (int g = 0; g < NCH; ++g)
              if (g < gmax) {
                T v[CH];
#pragma unroll
                for (int c = 0; c < CH; ++c) v[c] = row[q][g * CH + c];
                st_vec<T, CH>(st + g * CH, v);
              }
          }
        if (lane == 0) {
          h->key[buf][warp] = key;
          h->idx[buf][warp] = p;
        }
        __syncthreads();
        // every warp reduces the warps' candidates (one barrier a column: the
        // buffers alternate)
        key = lane < NW ? (K)h->key[buf][lane & (NW - 1)] : (K)0;
        p = lane < NW ? h->idx[buf][lane & (NW - 1)] : INT_MAX;
        const int mine = p;
        warp_argmax(key, p);
        const int own = __ffs(__ballot_sync(0xffffffffu, lane < NW && mine == p)) - 1;
        const T* prow = (const T*)(h->stage + (buf * NW + own) * 128);
        const T piv = prow[jj];
        if (tid == 0) {
          h->piv[j] = p;
          if (piv == (T)0 && h->info == 0) h->info = kk + j + 1;
        }
        bool upd[RPT];
        bool any = false;
#pragma unroll
        for (int q = 0; q < RPT; ++q) {
          pos[q] = swap_step(pos[q], j, p);
          upd[q] = pos[q] > j && piv != (T)0;
          any |= upd[q];
        }
        if (any) {
          T l[RPT];
#pragma unroll
          for (int q = 0; q < RPT; ++q) {
            l[q] = div_rn(row[q][jj], piv);
            if (upd[q]) row[q][jj] = l[q];
          }
#pragma unroll
          for (int g = 0; g < NCH; ++g)
            if (g < gmax) {
              T u[CH];
              ld_vec<T, CH>(prow + g * CH, u);
#pragma unroll
              for (int q = 0; q < RPT; ++q)
                if (upd[q]) {
#pragma unroll
                  for (int c = 0; c < CH; ++c)
                    if (g > 0 || c > jj) row[q][g * CH + c] = sub_rn(row[q][g * CH + c], mul_rn(l[q], u[c]));
                }
            }
        }
      }
    }
    // the chunk's columns are final: stored in F, registers shifted down
#pragma unroll
    for (int q = 0; q < RPT; ++q) {
      const int li = tid + q * kCtaLuThreads;
      if (li < m) {
        F* dst = A + (size_t)(kk + li) * lda + kk + jc * CH;
        F e[CH];
#pragma unroll
        for (int c = 0; c < CH; ++c) e[c] = store_rn<F>(row[q][c]);
        if (al && jc * CH + CH <= w) {
#pragma unroll
          for (int c = 0; c < CH; ++c)
            if (!isfinite(to_f(e[c]))) nf = 1;
          st_vec<F, CH>(dst, e);
        } else {
#pragma unroll
          for (int c = 0; c < CH; ++c)
            if (jc * CH + c < w) {
              if (!isfinite(to_f(e[c]))) nf = 1;
              dst[c] = e[c];
            }
        }
      }
#pragma unroll
      for (int c = 0; c + CH < NBM; ++c) row[q][c] = row[q][c + CH];
    }
  }
  if (nf) h->nonfinite = 1;
#pragma unroll
  for (int q = 0; q < RPT; ++q) {
    const int li = tid + q * kCtaLuThreads;
    if (li < m && pos[q] != li) {
      const int e = atomicAdd(&h->cnt, 1);
      if (e < 64) {  // an interchange moves two rows: 2 w at most
        h->from[e] = kk + li;
        h->to[e] = kk + pos[q];
      }
    }
  }
  __syncthreads();
  if (tid < w) ipiv[kk + tid] = kk + h->piv[tid];
}

// The listed rows to their new places, all n columns (rows start on 16-byte
// boundaries; the vector that holds column n - 1 ends inside the row).
template <typename F>
__device__ void cta_move_rows(F* A, int lda, int n, const CtaLuHead* h, unsigned char* sm) {
  const int cnt = h->cnt, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (cnt == 0) return;
  constexpr int E = 16 / (int)sizeof(F);
  const int nv = (n + E - 1) / E, cap = kCtaMoveBytes / 16 / cnt;  // vectors per row and pass
  uint4* st = (uint4*)sm;
  for (int v0 = 0; v0 < nv; v0 += cap) {
    const int cv = min(cap, nv - v0);
    for (int r = warp; r < cnt; r += kCtaLuWarps) {
      const uint4* src = (const uint4*)(A + (size_t)h->from[r] * lda) + v0;
      for (int v = lane; v < cv; v += 32) st[r * cap + v] = src[v];
    }
    __syncthreads();
    for (int r = warp; r < cnt; r += kCtaLuWarps) {
      uint4* dst = (uint4*)(A + (size_t)h->to[r] * lda) + v0;
      for (int v = lane; v < cv; v += 32) dst[v] = st[r * cap + v];
    }
    __syncthreads();
  }
}

// x <- L^{-1} x for a unit lower triangle of 32 rows, Lt[m][i] its columns
// (zero outside): each x_i takes its terms in ascending order.
template <typename T>
__device__ __forceinline__ void tri_solve32(T (&x)[32], const T* Lt) {
#pragma unroll
  for (int m = 0; m < 31; ++m) {
#pragma unroll
    for (int g = 0; g < 8; ++g)
      if (4 * g + 3 > m) {
        T l[4];
        ld_vec<T, 4>(Lt + m * kCtaTriLd + 4 * g, l);
#pragma unroll
        for (int e = 0; e < 4; ++e)
          if (4 * g + e > m) x[4 * g + e] = sub_rn(x[4 * g + e], mul_rn(l[e], x[m]));
      }
  }
}

// U12 = L11^{-1} A12 for rows r0 .. r0+w-1 (w <= 64), columns [c0, c1), in T
// with the stored unit lower L11; stored in u_f.
template <typename F>
__device__ __noinline__ void cta_trsm(F* A, int lda, int r0, int w, int c0, int c1, CtaLuHead* h,
                                      unsigned char* sm) {
  using T = LuT<F>;
  if (c1 <= c0) return;
  const int tid = threadIdx.x;
  T* Lt = (T*)sm;                       // two diagonal blocks, transposed
  T* Lr = Lt + 2 * 32 * kCtaTriLd;      // rows 32 .. 63 of columns 0 .. 31
  T* Y = Lr + 32 * 32 + tid;            // this thread's parked unknowns
  for (int e = tid; e < 32 * 32; e += kCtaLuThreads) {
    const int i = e / 32, m = e % 32;
    const F* src = A + (size_t)r0 * lda + r0;
    Lt[m * kCtaTriLd + i] = (m < i && i < w) ? (T)to_f(src[(size_t)i * lda + m]) : (T)0;
    if (w > 32) {
      const bool in = 32 + i < w;
      Lt[(32 + m) * kCtaTriLd + i] = (m < i && in) ? (T)to_f(src[(size_t)(32 + i) * lda + 32 + m]) : (T)0;
      Lr[i * 32 + m] = in ? (T)to_f(src[(size_t)(32 + i) * lda + m]) : (T)0;
    }
  }
  __syncthreads();
  int bad = 0;
  for (int c = c0 + tid; c < c1; c += kCtaLuThreads) {
    F* col = A + (size_t)r0 * lda + c;
    auto put = [&](int i, T v) {
      const F f = store_rn<F>(v);
      bad |= !isfinite(to_f(f));
      col[(size_t)i * lda] = f;
    };
    T x[32];
#pragma unroll
    for (int i = 0; i < 32; ++i) x[i] = i < w ? (T)to_f(col[(size_t)i * lda]) : (T)0;
    tri_solve32<T>(x, Lt);
#pragma unroll
    for (int i = 0; i < 32; ++i)
      if (i < w) put(i, x[i]);
    if (w > 32) {
      for (int i = 32; i < w; i += 4) {
        T v[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) v[q] = i + q < w ? (T)to_f(col[(size_t)(i + q) * lda]) : (T)0;
#pragma unroll
        for (int m = 0; m < 32; m += 4) {
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            T l[4];
            ld_vec<T, 4>(Lr + (i - 32 + q) * 32 + m, l);
#pragma unroll
            for (int e = 0; e < 4; ++e) v[q] = sub_rn(v[q], mul_rn(l[e], x[m + e]));
          }
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) Y[(i - 32 + q) * kCtaLuThreads] = v[q];
      }
#pragma unroll
      for (int i = 0; i < 32; ++i) x[i] = 32 + i < w ? Y[i * kCtaLuThreads] : (T)0;
      tri_solve32<T>(x, Lt + 32 * kCtaTriLd);
#pragma unroll
      for (int i = 0; i < 32; ++i)
        if (32 + i < w) put(32 + i, x[i]);
    }
  }
  if (bad) h->nonfinite = 1;
  __syncthreads();
}

// C = A[r0+w.., c0..c1) <- fl_f(fl_T(C - L21 U12)), w <= 64 products per
// element as an ascending fused multiply-add chain in T.
template <typename F>
__device__ __noinline__ void cta_update(F* A, int lda, int n, int r0, int w, int c0, int c1, CtaLuHead* h,
                                        unsigned char* sm) {
  using T = LuT<F>;
  const int rb = r0 + w;
  if (c1 <= c0 || rb >= n) return;
  constexpr int LD = kCtaTileLd;
  T* Ls = (T*)sm;        // [k][row]
  T* Us = Ls + 64 * LD;  // [k][column]
  const int tid = threadIdx.x, tr = (tid >> 4) * 4, tc = (tid & 15) * 4;
  const bool al = (c0 & 3) == 0;
  int bad = 0;
  for (int j0 = c0; j0 < c1; j0 += 64) {
    __syncthreads();  // the previous tile's operands are no longer read
    for (int e = tid; e < w * 64; e += kCtaLuThreads) {
      const int k = e / 64, j = e % 64;
      Us[k * LD + j] = j0 + j < c1 ? (T)to_f(A[(size_t)(r0 + k) * lda + j0 + j]) : (T)0;
    }
    for (int i0 = rb; i0 < n; i0 += 64) {
      if (i0 > rb) __syncthreads();
#pragma unroll 8
      for (int e = tid; e < 64 * 64; e += kCtaLuThreads) {
        const int i = e / 64, k = e % 64;
        if (k < w) Ls[k * LD + i] = i0 + i < n ? (T)to_f(A[(size_t)(i0 + i) * lda + r0 + k]) : (T)0;
      }
      const int j = j0 + tc;
      const bool vec = al && j + 4 <= c1;
      F cur[4][4];
#pragma unroll
      for (int a = 0; a < 4; ++a) {
        const F* pc = A + (size_t)min(i0 + tr + a, n - 1) * lda + j;
        if (vec) {
          if constexpr (sizeof(F) == 2) {
            const uint2 t = *(const uint2*)pc;
            memcpy(cur[a], &t, 8);
          } else {
            ld_vec<F, 4>(pc, cur[a]);
          }
        } else {
#pragma unroll
          for (int b = 0; b < 4; ++b)
            if (j + b < c1) cur[a][b] = pc[b];
        }
      }
      __syncthreads();
      T acc[4][4];
#pragma unroll
      for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) acc[a][b] = (T)0;
#pragma unroll 4
      for (int k = 0; k < w; ++k) {
        T l[4], u[4];
        ld_vec<T, 4>(Ls + k * LD + tr, l);
        ld_vec<T, 4>(Us + k * LD + tc, u);
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
          for (int b = 0; b < 4; ++b) acc[a][b] = fma_rn(l[a], u[b], acc[a][b]);
      }
#pragma unroll
      for (int a = 0; a < 4; ++a) {
        if (i0 + tr + a < n) {
          F* pc = A + (size_t)(i0 + tr + a) * lda + j;
          F f[4];
#pragma unroll
          for (int b = 0; b < 4; ++b)
            if (j + b < c1) {
              f[b] = store_rn<F>(sub_rn((T)to_f(cur[a][b]), acc[a][b]));
              bad |= !isfinite(to_f(f[b]));
            }
          if (vec) {
            if constexpr (sizeof(F) == 2) {
              uint2 t;
              memcpy(&t, f, 8);
              *(uint2*)pc = t;
            } else {
              st_vec<F, 4>(pc, f);
            }
          } else {
#pragma unroll
            for (int b = 0; b < 4; ++b)
              if (j + b < c1) pc[b] = f[b];
          }
        }
      }
    }
  }
  if (bad) h->nonfinite = 1;
  __syncthreads();
}

// The whole factorisation.  ipiv: LAPACK-style global rows (0-based).
// info: 1-based first zero pivot (0: none); nonfinite: a stored value is
// Inf or NaN.  Every thread of the block calls it; smem holds
// cta_lu_smem<F>() bytes; rows of A start on 16-byte boundaries and lda
// covers n rounded up to 16 bytes.  nbo <= 64; wider panels than 32 columns
// (fp64: 16) are split.
template <typename F>
__device__ void cta_lu(F* A, int lda, int n, int nb, int nbo, int* ipiv, int* info_out, int* nonfinite_out,
                       unsigned char* smem) {
  nb = min(nb, PanelNB<LuT<F>>::v);  // the panel's registers
  CtaLuHead* h = (CtaLuHead*)smem;
  unsigned char* sm = smem + kCtaLuHead;
  if (threadIdx.x == 0) {
    h->info = 0;
    h->nonfinite = 0;
  }
  __syncthreads();
  for (int k = 0; k < n; k += nbo) {
    const int W = min(nbo, n - k);
    for (int kk = k; kk < k + W; kk += nb) {
      const int w = min(nb, k + W - kk);
      if (n - kk <= kCtaLuThreads) cta_panel<F, 1>(A, lda, n, kk, w, ipiv, h);
      else cta_panel<F, 2>(A, lda, n, kk, w, ipiv, h);
      cta_move_rows<F>(A, lda, n, h, sm);
      __syncthreads();
      cta_trsm<F>(A, lda, kk, w, kk + w, k + W, h, sm);
      cta_update<F>(A, lda, n, kk, w, kk + w, k + W, h, sm);
    }
    cta_trsm<F>(A, lda, k, W, k + W, n, h, sm);
    cta_update<F>(A, lda, n, k, W, k + W, n, h, sm);
  }
  if (threadIdx.x == 0) {
    *info_out = h->info;
    *nonfinite_out = h->nonfinite;
  }
  __syncthreads();
}

}  // namespace msir
