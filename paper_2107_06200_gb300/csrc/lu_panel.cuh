// lu_outer_panel: the panel of the blocked right-looking GEPP (Algorithm 4,
// first step; partial pivoting as in Sec. 1; see lu.cu for the whole).  One
// translation unit per storage format instantiates it (lu_panel_*.cu).
#pragma once

#include <cooperative_groups.h>
#include <climits>
#include <cstring>

#include "common.cuh"
#include "kernels.h"
#include "lu_arith.cuh"

namespace cg = cooperative_groups;

namespace msir {

// ------------------------------------------------------------------ panel

// Optional section timers (rank 0, thread 0): 0 column loop, 4 panel store
// + permutation map, 5 inner interchanges + substitution, 6 inner update,
// 7 panel load.
// They add up in shared memory and reach a.tdbg once, at the kernel's end,
// so that the measurement keeps global-memory round trips off the loop.
#define PT_BEGIN(id) unsigned long long _t##id = (a.tdbg && rank == 0 && tid == 0) ? gtimer() : 0
#define PT_END(id) \
  if (a.tdbg && rank == 0 && tid == 0) s_tacc[id] += gtimer() - _t##id

// Pivot exchange between the CTAs of a cluster: each sends its candidate's
// row (kCandRow bytes) and key / position (16 bytes) into a slot of every
// CTA's shared memory by asynchronous stores that count their bytes on the
// receiver's mbarrier, so a column's exchange is one message and one wait
// (no cluster barrier, whose release waits for all earlier stores).
constexpr int kCandRow = 128;              // NBM values of T
constexpr int kCandBytes = kPanelCandBytes;
static_assert(kCandBytes == kCandRow + 16, "candidate slot");
__device__ __forceinline__ unsigned sm_addr(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }
__device__ __forceinline__ unsigned sm_peer(unsigned addr, int rank) {
  unsigned r;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
__device__ __forceinline__ void st_async16(unsigned addr, uint4 v, unsigned mbar) {
  asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v4.b32 [%0], {%1, %2, %3, %4}, [%5];" ::"r"(addr),
               "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w), "r"(mbar)
               : "memory");
}
__device__ __forceinline__ bool cand_try_wait(unsigned mbar, unsigned parity) {
  unsigned ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(mbar), "r"(parity)
      : "memory");
  return ok != 0;
}
// Bounded wait for a column's candidates.  When it runs out the error is
// recorded and *dead set: the block goes through the remaining columns of
// the panel without waiting (its peers still get a message per column), and
// the cluster leaves together at the panel's end.
static __device__ __noinline__ void cand_wait_slow(unsigned mbar, unsigned parity, volatile int* dead, int* err) {
  const unsigned long long t0 = gtimer();
  while (!cand_try_wait(mbar, parity)) {
    if (*dead) return;
    if (gtimer() - t0 > kWaitTimeoutNs) {
      record_timeout(err, 3, (int)parity, (int)threadIdx.x, 0);
      *dead = 1;
      return;
    }
  }
}

// The column loop is a chain: a pivot search over all rows, one exchange
// across the cluster, one rank-1 update, w times per panel.  What bounds it
// is the latency of each link and the instructions that every warp issues
// beside the update, so
//   * a thread keeps its row of the panel in registers: the rank-1 update
//     loads only the pivot row, 16 bytes at a time and the same address on
//     every lane;
//   * rows are not moved: each carries its position in the pivoted order,
//     an interchange changes two positions, and the row that leaves reaches
//     the others with the pivot candidate.  Values, order and rounding of
//     every operation are those of the interchanged panel;
//   * the pivot search of a column is one warp reduction on integer keys,
//     one block barrier and one message per CTA; with a single CTA no
//     message at all.
// Columns run in chunks of 8 whose registers are then shifted down, so that
// the loop body is 8 columns long (it stays in the instruction cache) and
// every register index is known at compile time.
//
// Measured (n = 8192, fp16, all 256 panels): column loop 16.3 -> 8.1 ms (1.0
// us per column on 16 CTAs; 0.45 us on a single CTA), stores and maps 2.9 ->
// 0.5, inner updates 2.7 -> 2.1, loads 1.4 -> 0.3, against the panel held in
// shared memory with a cluster barrier per column.
template <typename F, int NT, int RPT>
__global__ void __launch_bounds__(NT, 1) lu_outer_panel(PanelArgs a) {
  using T = typename Fmt<F>::T;
  using PK = PivKey<T>;
  using K = typename PK::K;
  constexpr int NBM = PanelNB<T>::v;
  constexpr int CH = 8;         // columns per chunk
  constexpr int NCH = NBM / CH;
  constexpr int NW = NT / 32;
  static_assert(NBM * sizeof(T) == kCandRow, "candidate row");
  // more than three rows per thread do not fit in registers: such panels
  // (more than 24576 rows on 16 CTAs) keep them in local memory, rows one at a time
  constexpr int kUnrollRows = RPT <= 3 ? RPT : 1;
  cg::cluster_group cl = cg::this_cluster();
  const int C = (int)cl.num_blocks();
  const int rank = (int)cl.block_rank();
  const int tid = threadIdx.x;
  const int lane = tid & 31, warp = tid >> 5;
  F* A = (F*)a.A;
  const int lda = a.lda, n = a.n, k = a.k, W = a.W, nb = a.nb;
  const int ldp = nb + 1;        // the last value of a row of P holds the row's final position
  const int ldu = (W + 7) & ~7;  // U12 rows start on 16-byte boundaries

  extern __shared__ __align__(16) unsigned char smem_raw[];
  unsigned char* cand = smem_raw;                             // [2][16][kCandBytes] candidates of the cluster
  T* stage = (T*)(cand + 2 * 16 * kCandBytes);                // [2][NW][NBM] candidate rows of the warps
  T* L11t = stage + 2 * NW * NBM;                             // NBM x NBM, transposed
  T* U12 = L11t + NBM * NBM;                                  // NBM x ldu
  T* P = U12 + (size_t)NBM * ldu;                             // R_cap x ldp
  int* opiv = (int*)(P + (size_t)a.R_cap * ldp);              // [W] pivots of the outer block, relative to k
  int* mpos = opiv + W;                                       // inner map positions [2*NBM]
  int* mval = mpos + 2 * NBM;                                 // inner map sources
  __shared__ __align__(16) K s_key[2][NW];
  __shared__ __align__(16) int s_idx[2][NW];
  __shared__ __align__(8) unsigned long long s_bar[2];        // mbarriers of the candidate slots
  __shared__ int s_piv[32];
  __shared__ int s_cnt, s_nf;
  __shared__ volatile int s_dead;
  __shared__ unsigned long long s_tacc[8];

  if (tid == 0) {
    s_nf = 0;
    s_dead = 0;
    for (int b = 0; b < 2; ++b)
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(sm_addr(&s_bar[b])) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (tid < 8) s_tacc[tid] = 0;
  // identity until a panel's pivots are known (the consumers of the pivots
  // stay in range if the kernel leaves early)
  for (int s = tid; s < W; s += NT) {
    opiv[s] = s;
    if (rank == 0) a.ipiv[k + s] = k + s;
  }
  const unsigned bar0 = sm_addr(&s_bar[0]);
  unsigned parity = 0;  // bit b: parity of the next phase of s_bar[b]
  cl.sync();

  for (int kk = k; kk < k + W; kk += nb) {
    const int w = min(nb, k + W - kk);
    const int m = n - kk;
    const int R = (m + C - 1) / C;
    const int my0 = rank * R;
    const int nloc = max(0, min(m, my0 + R) - my0);

    PT_BEGIN(7);
    T row[RPT][NBM];
    int pos[RPT];  // position in the pivoted order; -1: no row
#pragma unroll(kUnrollRows)
    for (int q = 0; q < RPT; ++q) {
      const int li = tid + q * NT;
      pos[q] = li < nloc ? my0 + li : -1;
      const F* src = A + (size_t)(kk + my0 + (li < nloc ? li : 0)) * lda + kk;
      if (li < nloc && w == NBM) {
        // kk is a multiple of nb = NBM and lda of 64: 16-byte aligned
        F e[NBM];
        ld_vec<F, NBM>(src, e);
#pragma unroll
        for (int c = 0; c < NBM; ++c) row[q][c] = (T)to_f(e[c]);
      } else {
#pragma unroll
        for (int c = 0; c < NBM; ++c) row[q][c] = (li < nloc && c < w) ? (T)to_f(src[c]) : (T)0;
      }
    }
    PT_END(7);

    PT_BEGIN(0);
    int nf = 0;
    for (int jc = 0; jc < NCH && jc * CH < w; ++jc) {
      // registers 0 .. NBM - 1 hold columns CH jc ..; groups of CH up to gmax
      const int gmax = NCH - jc;
#pragma unroll
      for (int jj = 0; jj < CH; ++jj) {
        const int j = jc * CH + jj;
        if (j < w) {
          constexpr int kBufMask = 1;
          const int buf = jj & kBufMask;
          // pivot candidate of the warp among rows at positions >= j
          K key = 0;
          int p = INT_MAX;
#pragma unroll(kUnrollRows)
          for (int q = 0; q < RPT; ++q) {
            const K kq = pos[q] >= j ? PK::of(row[q][jj]) : (K)0;
            const bool b = kq > key || (kq == key && kq != 0 && pos[q] < p);
            key = b ? kq : key;
            p = b ? pos[q] : p;
          }
          warp_argmax(key, p);
          T* st = stage + (buf * NW + warp) * NBM;
#pragma unroll(kUnrollRows)
          for (int q = 0; q < RPT; ++q) {
            if (pos[q] == p) {  // one lane (none if the warp has no candidate)
#pragma unroll
              for (int g = 0; g < NCH; ++g)
                if (g < gmax) {
                  T v[CH];
#pragma unroll
                  for (int c = 0; c < CH; ++c) v[c] = row[q][g * CH + c];
                  st_vec<T, CH>(st + g * CH, v);
                }
            }
          }
          if (lane == 0) {
            s_key[buf][warp] = key;
            s_idx[buf][warp] = p;
            if (tid == 0 && C > 1)
              asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar0 + 8 * buf),
                           "r"(C * kCandBytes)
                           : "memory");
          }
          __syncthreads();
          // every warp reduces the warps' candidates
          int own = 0;
          if constexpr (NW <= 4) {
            key = s_key[buf][0];
            p = s_idx[buf][0];
#pragma unroll
            for (int v = 1; v < NW; ++v) {
              const K kv = s_key[buf][v];
              const int pv = s_idx[buf][v];
              const bool b = kv > key || (kv == key && pv < p);
              key = b ? kv : key;
              p = b ? pv : p;
              own = b ? v : own;
            }
          } else {
            key = lane < NW ? s_key[buf][lane & (NW - 1)] : (K)0;
            p = lane < NW ? s_idx[buf][lane & (NW - 1)] : INT_MAX;
            const int mine = p;
            warp_argmax(key, p);
            own = __ffs(__ballot_sync(0xffffffffu, lane < NW && mine == p)) - 1;
          }
          const T* prow = stage + (buf * NW + own) * NBM;
          if (C > 1) {
            // the CTA's candidate to every CTA of the cluster: lanes 0-7 the
            // row, lane 8 its key and position
            if (lane <= kCandRow / 16) {
              uint4 v;
              if (lane < kCandRow / 16) v = reinterpret_cast<const uint4*>(prow)[lane];
              else v = make_uint4((unsigned)key, (unsigned)((unsigned long long)key >> 32), (unsigned)p, 0u);
              const unsigned dst = sm_addr(cand + (buf * 16 + rank) * kCandBytes + lane * 16);
              for (int d = warp; d < C; d += NW) st_async16(sm_peer(dst, d), v, sm_peer(bar0 + 8 * buf, d));
            }
            if (!s_dead) {
              const unsigned par = (parity >> buf) & 1u;
              int tries = 0;
              while (!cand_try_wait(bar0 + 8 * buf, par))
                if (++tries >= 64) {
                  cand_wait_slow(bar0 + 8 * buf, par, &s_dead, a.err);
                  break;
                }
            }
            parity ^= 1u << buf;
            const uint4 meta =
                *reinterpret_cast<const uint4*>(cand + (buf * 16 + (lane < C ? lane : 0)) * kCandBytes + kCandRow);
            if constexpr (sizeof(K) == 4) key = meta.x;
            else key = ((unsigned long long)meta.y << 32) | meta.x;
            p = (int)meta.z;
            if (lane >= C) { key = 0; p = INT_MAX; }
            const int theirs = p;
            warp_argmax(key, p);
            own = __ffs(__ballot_sync(0xffffffffu, theirs == p)) - 1;
            prow = reinterpret_cast<const T*>(cand + (buf * 16 + (own & 15)) * kCandBytes);
            if ((unsigned)p >= (unsigned)m) p = j;  // only after a wait that ran out
          }
          if (tid == 0) s_piv[j] = p;
          const T piv = prow[jj];
          if (piv == (T)0 && rank == 0 && tid == 0) atomicCAS(a.info, 0, kk + j + 1);
          bool upd[RPT];
          bool any = false;
#pragma unroll(kUnrollRows)
          for (int q = 0; q < RPT; ++q) {
            pos[q] = swap_step(pos[q], j, p);
            upd[q] = pos[q] > j && piv != (T)0;
            any |= upd[q];
          }
          if (any) {
            // rows that are not updated (above the diagonal, or none) subtract
            // zero times the pivot row, which may hold Inf or NaN: they are
            // excluded by selects on the result
            T l[RPT];
#pragma unroll(kUnrollRows)
            for (int q = 0; q < RPT; ++q) {
              l[q] = div_rn(row[q][jj], piv);
              if (upd[q]) row[q][jj] = l[q];
            }
#pragma unroll
            for (int g = 0; g < NCH; ++g)
              if (g < gmax) {
                T u[CH];
                ld_vec<T, CH>(prow + g * CH, u);
#pragma unroll(kUnrollRows)
                for (int q = 0; q < RPT; ++q)
                  if (upd[q]) {
#pragma unroll
                    for (int c = 0; c < CH; ++c)
                      if (g > 0 || c > jj) row[q][g * CH + c] = sub_rn(row[q][g * CH + c], mul_rn(l[q], u[c]));
                  }
              }
          }
          // no barrier here: the candidate buffers alternate, and a buffer is
          // written again only after the next column's barrier and messages
        }
      }
      // the chunk's columns are final: rounded to F into P, registers shifted
#pragma unroll(kUnrollRows)
      for (int q = 0; q < RPT; ++q) {
        const int li = tid + q * NT;
        if (li < nloc) {
#pragma unroll
          for (int c = 0; c < CH; ++c)
            if (jc * CH + c < w) {
              const F v = store_rn<F>(row[q][c]);
              P[li * ldp + jc * CH + c] = (T)to_f(v);
              if (!isfinite(to_f(v))) nf = 1;
            }
        }
#pragma unroll
        for (int c = 0; c + CH < NBM; ++c) row[q][c] = row[q][c + CH];
      }
    }
    PT_END(0);

    // store the panel, each row at its final position, and record its pivots
    PT_BEGIN(4);
#pragma unroll(kUnrollRows)
    for (int q = 0; q < RPT; ++q) {
      const int li = tid + q * NT;
      if (li >= nloc) continue;
      memcpy(&P[li * ldp + nb], &pos[q], sizeof(int));
      if ((unsigned)pos[q] >= (unsigned)m) continue;
      F* dst = A + (size_t)(kk + pos[q]) * lda + kk;
      if (w == NBM) {
        // a row segment of NBM values starts on a 16-byte boundary; the
        // values of P are values of F, so this rounding is exact
        F e[NBM];
#pragma unroll
        for (int c = 0; c < NBM; ++c) e[c] = store_rn<F>(P[li * ldp + c]);
        st_vec<F, NBM>(dst, e);
      } else {
        for (int c = 0; c < w; ++c) dst[c] = store_rn<F>(P[li * ldp + c]);
      }
    }
    if (nf) s_nf = 1;
    __syncthreads();  // s_piv complete
    if (rank == 0 && tid < w) a.ipiv[kk + tid] = kk + s_piv[tid];
    if (tid < w) opiv[kk - k + tid] = kk - k + s_piv[tid];

    // composite permutation of this panel's interchanges (positions relative
    // to kk; positions < w are slots 0 .. w-1): the interchanges only move
    // the rows 0 .. w-1 and the pivots, so each of these (two per lane) is
    // followed through the w interchanges to where it ends
    if (warp == 0) {
      const int pj = lane < w ? s_piv[lane] : -1 - lane;
      const unsigned same = __match_any_sync(0xffffffffu, pj);
      const bool has0 = lane < w, has1 = lane < w && pj >= w && __ffs(same) - 1 == lane;
      int e0 = lane, e1 = pj;
      for (int j = 0; j < w; ++j) {
        const int q = s_piv[j];
        e0 = swap_step(e0, j, q);
        e1 = swap_step(e1, j, q);
      }
      const unsigned out0 = __ballot_sync(0xffffffffu, has0 && e0 >= w);
      const unsigned out1 = __ballot_sync(0xffffffffu, has1 && e1 >= w);
      const unsigned below = (1u << lane) - 1u;
      if (has0) {
        const int s = e0 < w ? e0 : w + __popc(out0 & below);
        mpos[s] = e0;
        mval[s] = lane;
      }
      if (has1) {
        const int s = e1 < w ? e1 : w + __popc(out0) + __popc(out1 & below);
        mpos[s] = e1;
        mval[s] = pj;
      }
      if (lane == 0) s_cnt = w + __popc(out0) + __popc(out1);
    }
    if (s_dead && tid < C) *cl.map_shared_rank((int*)&s_dead, tid) = 1;
    cl.sync();  // panel values visible to the whole cluster
    if (s_dead) break;  // the same on every CTA
    PT_END(4);
    PT_BEGIN(5);

    // inner interchanges on [k, kk) and [kk+w, k+W), then U12 = L11^{-1} A12
    // for [kk+w, k+W): a warp takes columns g and g + the number of warps,
    // whose loads and substitution steps overlap
    const int nleft = kk - k, nright = k + W - kk - w;
    if (nright > 0) {
      for (int i = warp; i < w; i += NW)  // L11t[c][i] = L[i][c]
        if (lane < w) L11t[lane * NBM + i] = (T)to_f(A[(size_t)(kk + i) * lda + kk + lane]);
    }
    __syncthreads();
    const int cnt = s_cnt;
    const int i0 = lane < cnt ? kk + mval[lane] : kk, i1 = lane + 32 < cnt ? kk + mval[lane + 32] : kk;
    const int o0 = lane < cnt ? kk + mpos[lane] : kk, o1 = lane + 32 < cnt ? kk + mpos[lane + 32] : kk;
    for (int g0 = rank * NW + warp; g0 < nleft + nright; g0 += 2 * C * NW) {
      int c[2];
      T x[2], v1[2];
      bool right[2], has[2];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int g = g0 + h * C * NW;
        has[h] = g < nleft + nright;
        c[h] = g < nleft ? k + g : kk + w + (has[h] ? g - nleft : 0);
        right[h] = has[h] && g >= nleft;
        // slots lane and lane + 32
        x[h] = (has[h] && lane < cnt) ? (T)to_f(A[(size_t)i0 * lda + c[h]]) : (T)0;
        v1[h] = (has[h] && lane + 32 < cnt) ? (T)to_f(A[(size_t)i1 * lda + c[h]]) : (T)0;
      }
      __syncwarp();
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        if (has[h] && lane >= w && lane < cnt) A[(size_t)o0 * lda + c[h]] = store_rn<F>(x[h]);
        if (has[h] && lane + 32 >= w && lane + 32 < cnt) A[(size_t)o1 * lda + c[h]] = store_rn<F>(v1[h]);
      }
      if (right[0] || right[1]) {
        for (int mm = 0; mm < w - 1; ++mm) {
          const T l = L11t[mm * NBM + (lane & (NBM - 1))];
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            const T xm = __shfl_sync(0xffffffffu, x[h], mm);
            if (right[h] && lane > mm && lane < w) x[h] = sub_rn(x[h], mul_rn(l, xm));
          }
        }
      }
#pragma unroll
      for (int h = 0; h < 2; ++h)
        if (has[h] && lane < w) {
          const F v = store_rn<F>(x[h]);
          A[(size_t)(kk + lane) * lda + c[h]] = v;
          if (right[h] && !isfinite(to_f(v))) s_nf = 1;
        }
    }
    cl.sync();
    PT_END(5);
    PT_BEGIN(6);

    // inner update of this CTA's rows below the diagonal block:
    // A[kk+pos][kk+w+c] <- fl(A - sum_mm L[pos][mm] U12[mm][c]), L from P,
    // the sum an ascending fused multiply-add chain from zero per element.
    // A warp takes 8 TR rows x 4 TC columns, a thread TR x TC of them (row
    // stride 8: a warp's scalar loads of P fall in different banks); C is
    // loaded before the products.
    if (nright > 0) {
      constexpr int TR = sizeof(T) == 8 || NT > 256 ? 4 : 8, TC = 8;
      for (int i = warp; i < w; i += NW)
        for (int c = lane; c < ldu; c += 32)
          U12[i * ldu + c] = c < nright ? (T)to_f(A[(size_t)(kk + i) * lda + kk + w + c]) : (T)0;
      __syncthreads();
      const int tiles_c = (nright + 4 * TC - 1) / (4 * TC), tiles_r = (nloc + 8 * TR - 1) / (8 * TR);
      const bool vec = ((kk + w) * (int)sizeof(F)) % 16 == 0;  // C rows 16-byte aligned
      const int ri = lane >> 2, ci = lane & 3;
      for (int t = warp; t < tiles_r * tiles_c; t += NW) {
        const int r0 = (t / tiles_c) * 8 * TR + ri, c0 = (t % tiles_c) * 4 * TC + ci * TC;
        if (c0 >= nright) continue;  // no warp-wide operation follows
        const bool full = vec && c0 + TC <= nright;
        F* dst[TR];
        const T* lp[TR];
        F e[TR][TC];
#pragma unroll
        for (int r = 0; r < TR; ++r) {
          const int li = r0 + 8 * r;
          lp[r] = P + (size_t)min(li, nloc - 1) * ldp;
          int ps;
          memcpy(&ps, lp[r] + nb, sizeof(int));
          dst[r] = li < nloc && ps >= w ? A + (size_t)(kk + ps) * lda + kk + w + c0 : nullptr;
          if (dst[r]) {
            if (full) {
              ld_vec<F, TC>(dst[r], e[r]);
            } else {
#pragma unroll
              for (int c = 0; c < TC; ++c)
                if (c0 + c < nright) e[r][c] = dst[r][c];
            }
          }
        }
        T acc[TR][TC];
#pragma unroll
        for (int r = 0; r < TR; ++r)
#pragma unroll
          for (int c = 0; c < TC; ++c) acc[r][c] = (T)0;
#pragma unroll 2
        for (int mm = 0; mm < w; ++mm) {
          T l[TR], u[TC];
          ld_vec<T, TC>(U12 + mm * ldu + c0, u);
#pragma unroll
          for (int r = 0; r < TR; ++r) l[r] = lp[r][mm];
#pragma unroll
          for (int r = 0; r < TR; ++r)
#pragma unroll
            for (int c = 0; c < TC; ++c) acc[r][c] = fma_rn(l[r], u[c], acc[r][c]);
        }
#pragma unroll
        for (int r = 0; r < TR; ++r) {
          if (!dst[r]) continue;
          if (full) {
#pragma unroll
            for (int c = 0; c < TC; ++c) e[r][c] = store_rn<F>(sub_rn((T)to_f(e[r][c]), acc[r][c]));
            st_vec<F, TC>(dst[r], e[r]);
          } else {
#pragma unroll
            for (int c = 0; c < TC; ++c)
              if (c0 + c < nright) dst[r][c] = store_rn<F>(sub_rn((T)to_f(e[r][c]), acc[r][c]));
          }
        }
      }
    }
    cl.sync();
    PT_END(6);
  }

  if (tid == 0 && s_nf) atomicExch(a.nonfinite, 1);
  if (a.tdbg && rank == 0 && tid < 8) a.tdbg[tid] += s_tacc[tid];
  // the outer block's composite permutation, the same way: row s (a row of
  // the block, or a pivot outside it) followed through all W interchanges
  if (rank == 0) {
    if (tid == 0) s_cnt = W;
    __syncthreads();
    for (int t = tid; t < 2 * W; t += NT) {
      const int src = t < W ? t : opiv[t - W];
      bool has = t < W || src >= W;
      int e = src;
      for (int j = 0; j < W; ++j) {
        const int q = opiv[j];
        if (t >= W && j < t - W && q == src) has = false;  // an earlier pivot is the same row
        e = swap_step(e, j, q);
      }
      if (has) {
        const int s = e < W ? e : atomicAdd(&s_cnt, 1);
        a.map_pos[s] = e;
        a.map_val[s] = src;
      }
    }
    __syncthreads();
    if (tid == 0) *a.map_cnt = s_cnt;
  }
  if (s_dead) {
    // messages of peers may still be on their way to this CTA
    const unsigned long long t0 = gtimer();
    while (gtimer() - t0 < 1000000ull) __nanosleep(1000);
    cl.sync();
  }
}

template <typename F, int NT, int RPT>
static cudaError_t launch_panel_rpt(const PanelArgs& a, int C, cudaStream_t st) {
  size_t smem = panel_smem_bytes(Fmt<F>::code, a.R_cap, a.nb, a.W);
  cudaError_t e = cudaFuncSetAttribute(lu_outer_panel<F, NT, RPT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)smem);
  if (e != cudaSuccess) return e;
  if (C > 8) {
    e = cudaFuncSetAttribute(lu_outer_panel<F, NT, RPT>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return e;
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(C, 1, 1);
  cfg.blockDim = dim3(NT, 1, 1);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = C;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, lu_outer_panel<F, NT, RPT>, a);
}

// One row per thread up to 512 rows per CTA (8192 rows on 16 CTAs), with as
// few warps as hold them; more rows per thread beyond.  Measured (column
// loop of a whole n = 8192 fp16 LU, 512 rows per CTA): 512 threads of one
// row 8.1 ms, 256 of two 9.9, 128 of four 13.0: the warps share the fetched
// instructions and hide each other's latencies, which more rows per thread
// do not make up for.
template <typename F>
static cudaError_t launch_panel_t(const PanelArgs& a, int C, cudaStream_t st) {
  const int R = a.R_cap;
  if (R <= 128) return launch_panel_rpt<F, 128, 1>(a, C, st);
  if (R <= 256) return launch_panel_rpt<F, 256, 1>(a, C, st);
  if (R <= 512) return launch_panel_rpt<F, 512, 1>(a, C, st);
  if (R <= 1024) return launch_panel_rpt<F, 512, 2>(a, C, st);
  if (R <= 1536) return launch_panel_rpt<F, 512, 3>(a, C, st);
  if (R <= 6144) return launch_panel_rpt<F, 512, 12>(a, C, st);
  return cudaErrorInvalidValue;
}

}  // namespace msir
