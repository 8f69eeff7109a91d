// Blocked right-looking GEPP in the factorisation precision u_f
// (Algorithm 4, first step; partial pivoting as in Sec. 1).
//
// The matrix lives in device memory in its storage format F (bf16, fp16,
// fp32 or fp64), row-major with leading dimension lda.  Arithmetic of the
// panel and of the triangular solves is carried out in T = fp32 (fp64 when
// F is fp64), with every product and every difference explicitly rounded,
// so those steps are bit-for-bit reproducible; values are rounded back to F
// when they are stored.  Two-level blocking: outer blocks of W = nbo
// columns, factored as panels of nb columns.
//
//   lu_outer_panel      (lu_panel.cuh) one thread-block cluster factors an (n-k) x W outer
//                       block: for each nb-column panel, the pivot search,
//                       interchange, scaling and rank-1 updates run with the
//                       panel in registers; each CTA sends its pivot
//                       candidate and that row to every CTA of the cluster
//                       by asynchronous stores that an mbarrier counts, so a
//                       column costs one message and one wait per CTA and no
//                       cluster barrier.  The inner interchanges,
//                       substitution and update of the outer block follow.
//   lu_outer_swap_trsm  applies the outer block's interchanges to the other
//                       columns, forms U12 = L11^{-1} A12 by substitution and
//                       (for the tensor-core update) writes U12^T.
//   lu_update_simt      A22 <- fl_F(fl_T(A22 - L21 U12)) for fp32/fp64
//                       factors (the bf16/fp16 update is in lu_tc.cu).
#include <cstring>
#include <type_traits>

#include "common.cuh"
#include "kernels.h"
#include "lu_arith.cuh"

namespace msir {

// ------------------------------------------------- outer swaps and TRSM

// Leading dimension of L in shared memory: rows fall in different banks when
// a warp reads a column, and rows of 16-bit values start on a 32-bit word.
__host__ __device__ inline int trsm_ldl(int W, int fsize) { return fsize == 2 ? (W + 1) / 2 * 2 + 2 : W + 1; }

// The substitution U12 = L11^{-1} A12 is a chain of W steps per column.  It
// runs in blocks of 32 rows: within a block a warp takes four columns with
// one row per lane (the solved value of a step reaches the other rows by a
// shuffle, four independent chains hide its latency), then every row below
// subtracts the block's 32 products in ascending order.  Each element sees
// the same rounded products and differences in the same order as in a
// row-by-row substitution, with two block barriers per 32 rows instead of
// one per row.
template <typename F>
__global__ void __launch_bounds__(256) lu_outer_swap_trsm(SwapTrsmArgs a) {
  using T = typename Fmt<F>::T;
  F* A = (F*)a.A;
  const int lda = a.lda, k = a.k, W = a.W;
  const int cnt = *a.map_cnt;
  const int nleft = a.do_left ? k : 0, nright = a.c_end - a.c_begin;
  const int tiles_left = (nleft + 31) / 32;
  const int tiles_right = nright > 0 ? (nright + 31) / 32 : 0;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  constexpr int NW = 256 / 32;
  constexpr int ldx = 33;

  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int ldL = trsm_ldl(W, (int)sizeof(F));
  T* X = (T*)smem_raw;                       // W x ldx
  F* L = (F*)(X + (size_t)W * ldx);          // W x ldL (only when right tiles exist)
  size_t off = sizeof(T) * (size_t)W * ldx + sizeof(F) * (size_t)W * ldL;
  off = (off + 15) & ~(size_t)15;
  F* E = (F*)(smem_raw + off);               // (cnt - W) x 32 displaced rows
  int* val = (int*)(E + (size_t)W * 32);     // sources of the slots [2W]
  int* pos = val + 2 * W;                    // positions of the slots W .. cnt-1 (slot s < W is row s)
  __shared__ int s_nf;
  if (tid == 0) s_nf = 0;
  for (int s = tid; s < cnt; s += blockDim.x) {
    val[s] = a.map_val[s];
    if (s >= W) pos[s - W] = a.map_pos[s];
  }
  bool need_L = false;
  for (int t = blockIdx.x; t < tiles_left + tiles_right; t += gridDim.x)
    if (t >= tiles_left) need_L = true;
  constexpr int E16 = 16 / (int)sizeof(F);  // values per 16-byte load
  constexpr int LPR = 32 / E16;             // lanes per 32-column row segment
  if (need_L) {
    if (k % E16 == 0 && W % E16 == 0) {
      // eight 16-byte loads in flight per thread (rows of L in shared memory
      // are not 16-byte aligned: stored value by value)
      const int per = W / E16, tot = W * per;
      for (int i0 = tid; i0 < tot; i0 += 8 * 256) {
        uint4 u[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) {
          const int i = i0 + q * 256;
          if (i < tot) u[q] = *reinterpret_cast<const uint4*>(A + (size_t)(k + i / per) * lda + k + (i % per) * E16);
        }
#pragma unroll
        for (int q = 0; q < 8; ++q) {
          const int i = i0 + q * 256;
          if (i < tot) {
            F e[E16];
            memcpy(e, &u[q], 16);
#pragma unroll
            for (int c = 0; c < E16; ++c) L[(i / per) * ldL + (i % per) * E16 + c] = e[c];
          }
        }
      }
    } else {
      for (int i = warp; i < W; i += NW)
        for (int c = lane; c < W; c += 32) L[i * ldL + c] = A[(size_t)(k + i) * lda + k + c];
    }
  }
  __syncthreads();

  for (int t = blockIdx.x; t < tiles_left + tiles_right; t += gridDim.x) {
    const bool right = t >= tiles_left;
    const int c0 = right ? a.c_begin + (t - tiles_left) * 32 : t * 32;
    const int cend = right ? a.c_end : k;
    const int c = c0 + lane;
    // whole tiles at aligned columns move in 16-byte pieces, LPR lanes per
    // row and eight rows' loads in flight; ragged ones value by value
    const bool vec = c0 % E16 == 0 && c0 + 32 <= cend;
    const int vr = tid / LPR, vc = (tid % LPR) * E16;  // row and first column of a 16-byte piece
    constexpr int VR = 256 / LPR;                      // rows per pass of the block
    if (vec) {
      for (int s0 = vr; s0 < cnt; s0 += 8 * VR) {
        uint4 u[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) {
          const int s = s0 + q * VR;
          if (s < cnt) u[q] = *reinterpret_cast<const uint4*>(A + (size_t)(k + val[s]) * lda + c0 + vc);
        }
#pragma unroll
        for (int q = 0; q < 8; ++q) {
          const int s = s0 + q * VR;
          if (s >= cnt) continue;
          if (s < W) {
            F e[E16];
            memcpy(e, &u[q], 16);
#pragma unroll
            for (int v = 0; v < E16; ++v) X[s * ldx + vc + v] = (T)to_f(e[v]);
          } else {
            memcpy(E + (s - W) * 32 + vc, &u[q], 16);
          }
        }
      }
    } else {
      for (int s = warp; s < cnt; s += NW) {
        F v{};
        if (c < cend) v = A[(size_t)(k + val[s]) * lda + c];
        if (s < W) X[s * ldx + lane] = (T)to_f(v);
        else E[(s - W) * 32 + lane] = v;
      }
    }
    __syncthreads();
    if (vec) {
      for (int s = W + vr; s < cnt; s += VR) {
        uint4 u;
        memcpy(&u, E + (s - W) * 32 + vc, 16);
        *reinterpret_cast<uint4*>(A + (size_t)(k + pos[s - W]) * lda + c0 + vc) = u;
      }
    } else if (c < cend) {
      for (int s = W + warp; s < cnt; s += NW) A[(size_t)(k + pos[s - W]) * lda + c] = E[(s - W) * 32 + lane];
    }
    if (right) {
      for (int b0 = 0; b0 < W; b0 += 32) {
        const int bw = min(32, W - b0);
        // the block's own rows: columns 4 warp .. 4 warp + 3, row b0 + lane
        {
          T lr[32], x[4];
          const int i = min(b0 + lane, W - 1);
#pragma unroll
          for (int mm = 0; mm < 32; ++mm) lr[mm] = mm < bw ? (T)to_f(L[i * ldL + b0 + mm]) : (T)0;
#pragma unroll
          for (int q = 0; q < 4; ++q) x[q] = X[i * ldx + 4 * warp + q];
#pragma unroll
          for (int mm = 0; mm < 31; ++mm) {
            if (mm + 1 < bw) {
#pragma unroll
              for (int q = 0; q < 4; ++q) {
                const T xm = __shfl_sync(0xffffffffu, x[q], mm);
                if (lane > mm) x[q] = sub_rn(x[q], mul_rn(lr[mm], xm));
              }
            }
          }
          if (lane < bw) {
#pragma unroll
            for (int q = 0; q < 4; ++q) X[i * ldx + 4 * warp + q] = x[q];
          }
        }
        __syncthreads();
        // the rows below: four rows per warp and pass, one column per lane
        for (int r0 = b0 + 32 + warp * 4; r0 < W; r0 += 4 * NW) {
          T x[4];
          const F* lp[4];
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            const int r = min(r0 + q, W - 1);  // rows past W repeat the last one and are not stored
            x[q] = X[r * ldx + lane];
            lp[q] = L + r * ldL + b0;
          }
#pragma unroll 8
          for (int mm = 0; mm < 32; ++mm) {
            const T xm = X[(b0 + mm) * ldx + lane];
#pragma unroll
            for (int q = 0; q < 4; ++q) x[q] = sub_rn(x[q], mul_rn((T)to_f(lp[q][mm]), xm));
          }
#pragma unroll
          for (int q = 0; q < 4; ++q)
            if (r0 + q < W) X[(r0 + q) * ldx + lane] = x[q];
        }
        __syncthreads();
      }
    }
    int nf = 0;
    if (vec) {
      for (int s = vr; s < W; s += VR) {
        F e[E16];
#pragma unroll
        for (int v = 0; v < E16; ++v) {
          e[v] = store_rn<F>(X[s * ldx + vc + v]);
          if (right && !isfinite(to_f(e[v]))) nf = 1;
        }
        uint4 u;
        memcpy(&u, e, 16);
        *reinterpret_cast<uint4*>(A + (size_t)(k + s) * lda + c0 + vc) = u;
      }
    } else if (c < cend) {
      for (int s = warp; s < W; s += NW) {
        const F v = store_rn<F>(X[s * ldx + lane]);
        A[(size_t)(k + s) * lda + c] = v;
        if (right && !isfinite(to_f(v))) nf = 1;
      }
    }
    if (right && a.Ut != nullptr) {
      F* Ut = (F*)a.Ut;
      if (W % E16 == 0 && a.ldut % E16 == 0) {
        // 16 bytes (E16 rows of one column) per thread, neighbouring lanes on
        // neighbouring columns of X (no bank conflicts)
        for (int i = tid; i < 32 * (W / E16); i += 256) {
          const int cc = i % 32, s = (i / 32) * E16;
          if (c0 + cc >= cend) continue;
          F e[E16];
#pragma unroll
          for (int v = 0; v < E16; ++v) e[v] = store_rn<F>(X[(s + v) * ldx + cc]);
          uint4 u;
          memcpy(&u, e, 16);
          *reinterpret_cast<uint4*>(Ut + (size_t)(c0 + cc - k - W) * a.ldut + s) = u;
        }
      } else {
        for (int cc = warp; cc < 32; cc += NW)
          if (c0 + cc < cend)
            for (int s = lane; s < W; s += 32)
              Ut[(size_t)(c0 + cc - k - W) * a.ldut + s] = store_rn<F>(X[s * ldx + cc]);
      }
    }
    if (nf) s_nf = 1;
    __syncthreads();
  }
  if (tid == 0 && s_nf) atomicExch(a.nonfinite, 1);
}

// ------------------------------------------------------- SIMT update

// A22 <- A22 - L21 U12 for fp32 / fp64 factors: per element one ascending
// fused multiply-add chain from zero, then one rounded difference.  Tiles of
// BM x BN elements per block of 256 threads, BM/16 x BN/16 per thread (as
// two halves BM/2 and BN/2 apart, so that a warp's 16-byte shared-memory
// reads fall in different banks); the next BK slice is loaded into registers
// while the current one is used, and shared memory holds two slices, so a
// slice costs one block barrier.
template <typename T, int BM, int BN>
__global__ void __launch_bounds__(256, BM * BN > 64 * 64 ? 2 : sizeof(T) == 8 ? 3 : 4) lu_update_simt(UpdateArgs a) {
  constexpr int BK = 16;
  constexpr int E = 16 / (int)sizeof(T);       // values per 16-byte load
  constexpr int TM = BM / 16, TN = BN / 16;    // elements per thread
  constexpr int VM = TM < E ? TM : E, VN = TN < E ? TN : E;  // consecutive rows / columns of a thread
  constexpr int HM = TM / VM, HN = TN / VN;    // groups of them
  constexpr int LA = BM * BK / 256, LB = BK * BN / 256;  // values loaded per thread and slice
  static_assert(LA % E == 0 && LB % E == 0, "whole 16-byte loads");
  T* A = (T*)a.A;
  const int lda = a.lda, k = a.k, W = a.W;
  const int r0 = k + W, M = a.n - r0;
  const int c0 = a.c_begin, NC = a.c_end - a.c_begin;
  __shared__ __align__(16) T As[2][BK][BM + E];
  __shared__ __align__(16) T Bs[2][BK][BN];
  const int tid = threadIdx.x;
  const int tm = blockIdx.y * BM, tn = blockIdx.x * BN;
  const int ty = tid / 16, tx = tid % 16;
  // 16-byte loads need aligned columns (rows start on 64-element boundaries)
  const bool vecA = (k % E) == 0, vecB = (c0 % E) == 0;
  // C is read at the end: bring its lines to L2 meanwhile
  {
    constexpr int kLine = 128 / (int)sizeof(T);
    for (int l = tid; l < BM * (BN / kLine); l += 256) {
      const int i = tm + l / (BN / kLine), j = tn + l % (BN / kLine) * kLine;
      if (i < M && j < NC)
        asm volatile("prefetch.global.L2 [%0];" ::"l"(A + (size_t)(r0 + i) * lda + c0 + j));
    }
  }
  // fp32: two neighbouring columns per accumulator (one instruction for the
  // two fused multiply-adds, each rounded as usual)
  constexpr bool kPair = std::is_same<T, float>::value;
  using Acc = typename std::conditional<kPair, unsigned long long, T>::type;
  constexpr int NA = kPair ? TN / 2 : TN;
  Acc acc2[TM][NA];
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < NA; ++j) acc2[i][j] = 0;
  // slice loads: L21 values kq = E (idx % (BK / E)) .. of row idx / (BK / E);
  // U12 columns E (idx % (BN / E)) .. of row idx / (BN / E)
  T ra[LA], rb[LB];
  auto load = [&](int kc) {
#pragma unroll
    for (int v = 0; v < LA / E; ++v) {
      const int idx = tid + v * 256, i = tm + idx / (BK / E), kq = kc + (idx % (BK / E)) * E;
      const T* p = A + (size_t)(r0 + i) * lda + k + kq;
      if (i < M && kq + E <= W && vecA) {
        const uint4 u = *reinterpret_cast<const uint4*>(p);
        memcpy(&ra[v * E], &u, 16);
      } else {
#pragma unroll
        for (int e = 0; e < E; ++e) ra[v * E + e] = (i < M && kq + e < W) ? p[e] : (T)0;
      }
    }
#pragma unroll
    for (int v = 0; v < LB / E; ++v) {
      const int idx = tid + v * 256, kq = kc + idx / (BN / E), j = tn + (idx % (BN / E)) * E;
      const T* p = A + (size_t)(k + kq) * lda + c0 + j;
      if (kq < W && j + E <= NC && vecB) {
        const uint4 u = *reinterpret_cast<const uint4*>(p);
        memcpy(&rb[v * E], &u, 16);
      } else {
#pragma unroll
        for (int e = 0; e < E; ++e) rb[v * E + e] = (kq < W && j + e < NC) ? p[e] : (T)0;
      }
    }
  };
  auto put = [&](int buf) {
#pragma unroll
    for (int v = 0; v < LA / E; ++v) {
      const int idx = tid + v * 256;
#pragma unroll
      for (int e = 0; e < E; ++e) As[buf][(idx % (BK / E)) * E + e][idx / (BK / E)] = ra[v * E + e];
    }
#pragma unroll
    for (int v = 0; v < LB / E; ++v) {
      const int idx = tid + v * 256;
      uint4 u;
      memcpy(&u, &rb[v * E], 16);
      *reinterpret_cast<uint4*>(&Bs[buf][idx / (BN / E)][(idx % (BN / E)) * E]) = u;
    }
  };
  auto step = [&](int buf, int kq) {
    T av[TM];
    Acc bv[NA];
#pragma unroll
    for (int h = 0; h < HM; ++h)
#pragma unroll
      for (int i = 0; i < VM; ++i) av[h * VM + i] = As[buf][kq][h * (BM / HM) + ty * VM + i];
    constexpr int NV = NA / HN;
#pragma unroll
    for (int h = 0; h < HN; ++h)
      memcpy(&bv[h * NV], __builtin_assume_aligned(&Bs[buf][kq][h * (BN / HN) + tx * VN], VN * sizeof(T)), VN * sizeof(T));
#pragma unroll
    for (int i = 0; i < TM; ++i) {
      if constexpr (kPair) {
        unsigned long long a2;
        asm("mov.b64 %0, {%1, %1};" : "=l"(a2) : "f"(av[i]));
#pragma unroll
        for (int j = 0; j < NA; ++j)
          asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(acc2[i][j]) : "l"(a2), "l"(bv[j]));
      } else {
#pragma unroll
        for (int j = 0; j < NA; ++j) acc2[i][j] = fma_rn(av[i], bv[j], acc2[i][j]);
      }
    }
  };
  load(0);
  put(0);
  __syncthreads();
  int buf = 0;
  for (int kc = 0; kc < W; kc += BK, buf ^= 1) {
    const bool more = kc + BK < W;
    if (more) load(kc + BK);
    if (W - kc >= BK) {
#pragma unroll
      for (int kq = 0; kq < BK; ++kq) step(buf, kq);
    } else {
      for (int kq = 0; kq < W - kc; ++kq) step(buf, kq);
    }
    if (more) put(buf ^ 1);  // last read one slice ago, before the previous barrier
    __syncthreads();
  }
  const bool vecC = vecB && VN == E;
  T acc[TM][TN];
  memcpy(acc, acc2, sizeof(acc));
#pragma unroll
  for (int i = 0; i < TM; ++i) {
    const int row = tm + (i / VM) * (BM / HM) + ty * VM + i % VM;
    if (row >= M) continue;
#pragma unroll
    for (int h = 0; h < HN; ++h) {
      const int col = tn + h * (BN / HN) + tx * VN;
      T* p = A + (size_t)(r0 + row) * lda + c0 + col;
      if (vecC && col + VN <= NC) {
        uint4 u = *reinterpret_cast<const uint4*>(p);
        T c[E];
        memcpy(c, &u, 16);
#pragma unroll
        for (int j = 0; j < E; ++j) c[j] = sub_rn(c[j], acc[i][h * VN + (j < VN ? j : 0)]);
        memcpy(&u, c, 16);
        *reinterpret_cast<uint4*>(p) = u;
      } else {
#pragma unroll
        for (int j = 0; j < VN; ++j)
          if (col + j < NC) p[j] = sub_rn(p[j], acc[i][h * VN + j]);
      }
    }
  }
}

// ------------------------------------------------------------ launchers

size_t panel_smem_bytes(int fmt, int R_cap, int nb, int W) {
  const size_t ts = fmt == MSIR_FP64 ? 8 : 4;
  const int NBM = fmt == MSIR_FP64 ? 16 : 32;
  const size_t ldu = ((size_t)W + 7) / 8 * 8;
  const size_t NW = 512 / 32;  // the panel's most warps
  return 2 * 16 * kPanelCandBytes + ts * (2 * NW * NBM + NBM * NBM + NBM * ldu + (size_t)R_cap * (nb + 1)) +
         (size_t)W * sizeof(int) + 4 * NBM * sizeof(int);
}

size_t swap_trsm_smem_bytes(int fmt, int W) {
  const size_t ts = fmt == MSIR_FP64 ? 8 : 4;
  const size_t fs = fmt == MSIR_FP64 ? 8 : fmt == MSIR_FP32 ? 4 : 2;
  size_t off = ts * (size_t)W * 33 + fs * (size_t)W * trsm_ldl(W, (int)fs);
  off = (off + 15) & ~(size_t)15;
  return off + fs * (size_t)W * 32 + 3 * (size_t)W * sizeof(int);
}

cudaError_t launch_panel_f16(const PanelArgs& a, int C, cudaStream_t st);
cudaError_t launch_panel_bf16(const PanelArgs& a, int C, cudaStream_t st);
cudaError_t launch_panel_f32(const PanelArgs& a, int C, cudaStream_t st);
cudaError_t launch_panel_f64(const PanelArgs& a, int C, cudaStream_t st);

cudaError_t launch_panel(int fmt, const PanelArgs& a, int C, cudaStream_t st) {
  switch (fmt) {
    case MSIR_FP16: return launch_panel_f16(a, C, st);
    case MSIR_BF16: return launch_panel_bf16(a, C, st);
    case MSIR_FP32: return launch_panel_f32(a, C, st);
    case MSIR_FP64: return launch_panel_f64(a, C, st);
  }
  return cudaErrorInvalidValue;
}

template <typename F>
static cudaError_t launch_swap_trsm_t(const SwapTrsmArgs& a, int grid, cudaStream_t st) {
  size_t smem = swap_trsm_smem_bytes(Fmt<F>::code, a.W);
  cudaError_t e = cudaFuncSetAttribute(lu_outer_swap_trsm<F>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  lu_outer_swap_trsm<F><<<grid, 256, smem, st>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_swap_trsm(int fmt, const SwapTrsmArgs& a, int grid, cudaStream_t st) {
  switch (fmt) {
    case MSIR_FP16: return launch_swap_trsm_t<__half>(a, grid, st);
    case MSIR_BF16: return launch_swap_trsm_t<__nv_bfloat16>(a, grid, st);
    case MSIR_FP32: return launch_swap_trsm_t<float>(a, grid, st);
    case MSIR_FP64: return launch_swap_trsm_t<double>(a, grid, st);
  }
  return cudaErrorInvalidValue;
}

// fp32: 128 x 128 tiles (64 multiply-adds per four 16-byte shared-memory
// loads) when there are enough of them for the SMs, else 64 x 64; fp64: 64 x
// 64 (the narrow fp64 pipe bounds it, not the loads).
template <typename T, int BM, int BN>
static cudaError_t launch_simt_t(const UpdateArgs& a, int M, int NC, cudaStream_t st) {
  lu_update_simt<T, BM, BN><<<dim3((NC + BN - 1) / BN, (M + BM - 1) / BM), 256, 0, st>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_update_simt(int fmt, const UpdateArgs& a, cudaStream_t st) {
  const int M = a.n - a.k - a.W, NC = a.c_end - a.c_begin;
  if (M <= 0 || NC <= 0) return cudaSuccess;
  if (fmt == MSIR_FP64) return launch_simt_t<double, 64, 64>(a, M, NC, st);
  if (fmt != MSIR_FP32) return cudaErrorInvalidValue;
  if ((long long)((M + 127) / 128) * ((NC + 127) / 128) >= 128) return launch_simt_t<float, 128, 128>(a, M, NC, st);
  return launch_simt_t<float, 64, 64>(a, M, NC, st);
}

}  // namespace msir
