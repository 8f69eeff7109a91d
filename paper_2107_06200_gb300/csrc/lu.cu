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
//                       panel in registers; pivot candidates and their rows
//                       are pushed to every CTA of the cluster through
//                       distributed shared memory, so each column costs one
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

template <typename F>
__global__ void __launch_bounds__(256) lu_outer_swap_trsm(SwapTrsmArgs a) {
  using T = typename Fmt<F>::T;
  F* A = (F*)a.A;
  const int lda = a.lda, k = a.k, W = a.W;
  const int cnt = *a.map_cnt;
  const int nleft = a.do_left ? k : 0, nright = a.c_end - a.c_begin;
  const int tiles_left = (nleft + 31) / 32;
  const int tiles_right = nright > 0 ? (nright + 31) / 32 : 0;
  const int tid = threadIdx.x;

  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int ldL = W + (sizeof(F) == 2 ? 2 : 1);  // padded: rows of L fall in different banks
  T* X = (T*)smem_raw;                       // W x 32
  F* L = (F*)(X + (size_t)W * 32);           // W x ldL (only when right tiles exist)
  F* E = L + (size_t)W * ldL;                // (cnt - W) x 32 displaced rows
  size_t off = sizeof(T) * (size_t)W * 32 + sizeof(F) * ((size_t)W * ldL + (size_t)W * 32);
  off = (off + 15) & ~(size_t)15;
  int* pos = (int*)(smem_raw + off);
  int* val = pos + 2 * W;
  __shared__ int s_nf;
  if (tid == 0) s_nf = 0;
  for (int s = tid; s < cnt; s += blockDim.x) { pos[s] = a.map_pos[s]; val[s] = a.map_val[s]; }
  bool need_L = false;
  for (int t = blockIdx.x; t < tiles_left + tiles_right; t += gridDim.x)
    if (t >= tiles_left) need_L = true;
  if (need_L) {
    for (int idx = tid; idx < W * W; idx += blockDim.x) {
      const int i = idx / W, c = idx % W;
      L[i * ldL + c] = A[(size_t)(k + i) * lda + k + c];
    }
  }
  __syncthreads();

  for (int t = blockIdx.x; t < tiles_left + tiles_right; t += gridDim.x) {
    const bool right = t >= tiles_left;
    const int c0 = right ? a.c_begin + (t - tiles_left) * 32 : t * 32;
    const int cend = right ? a.c_end : k;
    // gather sources
    for (int idx = tid; idx < cnt * 32; idx += blockDim.x) {
      const int s = idx / 32, cc = idx % 32, c = c0 + cc;
      if (c < cend) {
        F v = A[(size_t)(k + val[s]) * lda + c];
        if (s < W) X[s * 32 + cc] = (T)to_f(v);
        else E[(s - W) * 32 + cc] = v;
      }
    }
    __syncthreads();
    for (int idx = tid; idx < (cnt - W) * 32; idx += blockDim.x) {
      const int s = W + idx / 32, cc = idx % 32, c = c0 + cc;
      if (c < cend) A[(size_t)(k + pos[s]) * lda + c] = E[(s - W) * 32 + cc];
    }
    if (right) {
      for (int mm = 0; mm < W - 1; ++mm) {
        const int rows = W - 1 - mm;
        for (int idx = tid; idx < rows * 32; idx += blockDim.x) {
          const int i = mm + 1 + idx / 32, cc = idx % 32;
          X[i * 32 + cc] = sub_rn(X[i * 32 + cc], mul_rn((T)to_f(L[i * ldL + mm]), X[mm * 32 + cc]));
        }
        __syncthreads();
      }
    }
    int nf = 0;
    for (int idx = tid; idx < W * 32; idx += blockDim.x) {
      const int s = idx / 32, cc = idx % 32, c = c0 + cc;
      if (c < cend) {
        F v = store_rn<F>(X[s * 32 + cc]);
        A[(size_t)(k + s) * lda + c] = v;
        if (right && !isfinite(to_f(v))) nf = 1;
      }
    }
    if (right && a.Ut != nullptr) {
      F* Ut = (F*)a.Ut;
      for (int idx = tid; idx < W * 32; idx += blockDim.x) {
        const int cc = idx / W, s = idx % W, c = c0 + cc;
        if (c < cend) Ut[(size_t)(c - k - W) * a.ldut + s] = store_rn<F>(X[s * 32 + cc]);
      }
    }
    if (nf) s_nf = 1;
    __syncthreads();
  }
  if (s_nf) atomicExch(a.nonfinite, 1);
}

// ------------------------------------------------------- SIMT update

template <typename F>
__global__ void __launch_bounds__(256) lu_update_simt(UpdateArgs a) {
  using T = typename Fmt<F>::T;
  F* A = (F*)a.A;
  const int lda = a.lda, k = a.k, W = a.W;
  const int r0 = k + W, M = a.n - r0;
  const int c0 = a.c_begin, NC = a.c_end - a.c_begin;
  constexpr int BM = 64, BN = 64, BK = 16;
  __shared__ T As[BK][BM + 1];
  __shared__ T Bs[BK][BN];
  const int tid = threadIdx.x;
  const int tm = blockIdx.y * BM, tn = blockIdx.x * BN;
  const int ty = tid / 16, tx = tid % 16;
  T acc[4][4];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = 0;
  for (int kc = 0; kc < W; kc += BK) {
    for (int idx = tid; idx < BM * BK; idx += 256) {
      const int i = idx / BK, kq = idx % BK;
      const int row = tm + i, kk = kc + kq;
      As[kq][i] = (row < M && kk < W) ? (T)to_f(A[(size_t)(r0 + row) * lda + k + kk]) : (T)0;
    }
    for (int idx = tid; idx < BK * BN; idx += 256) {
      const int kq = idx / BN, j = idx % BN;
      const int col = tn + j, kk = kc + kq;
      Bs[kq][j] = (col < NC && kk < W) ? (T)to_f(A[(size_t)(k + kk) * lda + c0 + col]) : (T)0;
    }
    __syncthreads();
#pragma unroll
    for (int kq = 0; kq < BK; ++kq) {
      T av[4], bv[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) av[i] = As[kq][ty * 4 + i];
#pragma unroll
      for (int j = 0; j < 4; ++j) bv[j] = Bs[kq][tx * 4 + j];
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = fma_rn(av[i], bv[j], acc[i][j]);
    }
    __syncthreads();
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int row = tm + ty * 4 + i;
    if (row >= M) continue;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int col = tn + tx * 4 + j;
      if (col >= NC) continue;
      F* p = A + (size_t)(r0 + row) * lda + c0 + col;
      *p = store_rn<F>(sub_rn((T)to_f(*p), acc[i][j]));
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
  const size_t ldL = W + (fs == 2 ? 2 : 1);
  size_t off = ts * (size_t)W * 32 + fs * ((size_t)W * ldL + (size_t)W * 32);
  off = (off + 15) & ~(size_t)15;
  return off + 4 * (size_t)W * sizeof(int);
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

cudaError_t launch_update_simt(int fmt, const UpdateArgs& a, cudaStream_t st) {
  const int M = a.n - a.k - a.W, NC = a.c_end - a.c_begin;
  if (M <= 0 || NC <= 0) return cudaSuccess;
  dim3 grid((NC + 63) / 64, (M + 63) / 64);
  switch (fmt) {
    case MSIR_FP16: lu_update_simt<__half><<<grid, 256, 0, st>>>(a); break;
    case MSIR_BF16: lu_update_simt<__nv_bfloat16><<<grid, 256, 0, st>>>(a); break;
    case MSIR_FP32: lu_update_simt<float><<<grid, 256, 0, st>>>(a); break;
    case MSIR_FP64: lu_update_simt<double><<<grid, 256, 0, st>>>(a); break;
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

}  // namespace msir
