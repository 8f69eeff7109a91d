// Persistent refinement kernel: the loop of Algorithm 4 after the LU.
//
// One cooperative launch runs SIR, SGMRES-IR and GMRES-IR steps, the
// stopping criteria of Sec. 2.1.1 and the stage switches, entirely on the
// device; it returns to the host only when the run has converged, has
// nothing left to try, or needs the factorisation redone in a finer u_f
// (the host then relaunches it in phase PH_ESCALATED).
//
// Work distribution: rows are grouped in blocks of kBlk = 64; CTA c owns
// blocks c, c+G, c+2G, ...  Residual and operator rows are produced in the
// pivoted order i -> perm[i], so the forward substitution of a block needs
// only rows its own CTA computed.  Triangular solves are wavefronts: a CTA
// accumulates the off-diagonal products of its block as soon as the blocks
// it depends on publish their values (epoch-tagged 64-bit words), then
// applies the inverse of its diagonal block and publishes.  The inverses
// and the scaled blocks are built here when a solve in their precision first
// needs them.
// Grid barriers are used only where a full vector is needed (matrix-vector
// products) or a global reduction (norms, Gram-Schmidt coefficients).  The
// stage controller is replicated in every CTA: all CTAs compute the same
// decisions from the same reduced values, so control flow stays uniform.
// All waits are bounded (MSIR_ERR_TIMEOUT).
#pragma once

#include "common.cuh"
#include <type_traits>

#include "inv_impl.cuh"
#include "refine.h"

namespace msir {

// ----------------------------------------------------------- helpers

struct Cx {
  int G, cta, tid, lane, warp, n, nblk;
  int team_k;  // RefineArgs::team_k
  unsigned epoch;
  unsigned nbar;             // arrivals that complete the latest grid barrier
  int redbuf;
  unsigned long long* t_ns;  // per-phase timers (CTA 0, thread 0), shared memory
  unsigned char* tsm;        // shared scratch of the substitutions (kTrsvSmem bytes)
  unsigned char* ssm;        // shared staging of the scaled-block construction (kScaledSmem)
  unsigned mready;           // RefState::mready of this launch (uniform)
  int C;                     // CTAs per cluster (1: no clusters)
  unsigned long long* inbox; // [kMaxCluster][kBlk][kLLWords] words written by cluster peers
};

// Barrier of the solve's grid (a block barrier when one block is the grid:
// nothing else reads its data, and data written during the kernel is never
// read through the non-coherent path).
static __device__ __forceinline__ bool grid_barrier(Cx& cx, const RefineArgs& a) {
  if (cx.G == 1) {
    __syncthreads();
    return true;
  }
  cx.nbar += cx.G;
  return grid_barrier_for(a.bar, a.err, cx.nbar, kWaitTimeoutNs);
}

// Phase timer: CTA 0 / thread 0 accumulates %globaltimer deltas.
struct PhaseTimer {
  Cx& cx;
  int ph;
  unsigned long long t0;
  __device__ PhaseTimer(Cx& c, int p) : cx(c), ph(p), t0(0) {
    if (cx.cta == 0 && cx.tid == 0) t0 = gtimer();
  }
  __device__ ~PhaseTimer() {
    if (cx.cta == 0 && cx.tid == 0) cx.t_ns[ph] += gtimer() - t0;
  }
};

static __device__ __forceinline__ double urnd(double v, int u) {
  return u == MSIR_FP32 ? (double)__double2float_rn(v) : v;
}
static __device__ __forceinline__ double umul(double a, double b, int u) {
  return u == MSIR_FP32 ? (double)__fmul_rn((float)a, (float)b) : __dmul_rn(a, b);
}
static __device__ __forceinline__ double uadd(double a, double b, int u) {
  return u == MSIR_FP32 ? (double)__fadd_rn((float)a, (float)b) : __dadd_rn(a, b);
}
static __device__ __forceinline__ double usub(double a, double b, int u) {
  return u == MSIR_FP32 ? (double)__fsub_rn((float)a, (float)b) : __dsub_rn(a, b);
}
static __device__ __forceinline__ double udiv(double a, double b, int u) {
  return u == MSIR_FP32 ? (double)__fdiv_rn((float)a, (float)b) : __ddiv_rn(a, b);
}
static __device__ __forceinline__ double usqrt(double a, int u) {
  return u == MSIR_FP32 ? (double)__fsqrt_rn((float)a) : __dsqrt_rn(a);
}
static __device__ __forceinline__ int square_of(int u) { return u == MSIR_FP32 ? MSIR_FP64 : MSIR_DD; }
static __device__ __forceinline__ double unit_roundoff(int f) {
  switch (f) {
    case MSIR_BF16: return 0x1p-8;
    case MSIR_FP16: return 0x1p-11;
    case MSIR_FP32: return 0x1p-24;
    case MSIR_FP64: return 0x1p-53;
    default: return 0x1p-106;
  }
}

// 16-byte asynchronous copy global -> shared (L2 only) with zero fill past
// `bytes` (0..16); groups of them are committed and waited for per thread.
__device__ __forceinline__ void cp_async16(void* sdst, const void* gsrc, int bytes) {
  const unsigned sa = (unsigned)__cvta_generic_to_shared(sdst);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(sa), "l"(gsrc), "r"(bytes) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// Accumulators of the row products: fp32 compensated (Dot2), fp64, and
// fp64 compensated (twice the working precision, result as dd).
template <int OP> struct RowAcc;
template <> struct RowAcc<MSIR_FP32> {
  using R = float;
  ff_t a{0.0f, 0.0f};
  __device__ __forceinline__ void add(float x, float y) { a = ff_fma(x, y, a); }
  __device__ __forceinline__ void merge(const RowAcc& o) { a = ff_merge(a, o.a); }
  __device__ __forceinline__ RowAcc peer(int m) const { return RowAcc{ff_shfl_xor(a, m)}; }
  __device__ __forceinline__ R fin() const { return ff_fin(a); }
};
template <> struct RowAcc<MSIR_FP64> {
  using R = double;
  double a = 0.0;
  __device__ __forceinline__ void add(double x, double y) { a = __fma_rn(x, y, a); }
  __device__ __forceinline__ void merge(const RowAcc& o) { a = __dadd_rn(a, o.a); }
  __device__ __forceinline__ RowAcc peer(int m) const { return RowAcc{__shfl_xor_sync(0xffffffffu, a, m)}; }
  __device__ __forceinline__ R fin() const { return a; }
};
template <> struct RowAcc<MSIR_DD> {
  using R = dd_t;
  double s = 0.0, c = 0.0;
  __device__ __forceinline__ void add(double x, double y) {
    const dd_t p = two_prod(x, y);
    const dd_t t = two_sum_ord(s, p.hi);
    s = t.hi;
    c = __dadd_rn(c, __dadd_rn(t.lo, p.lo));
  }
  __device__ __forceinline__ void merge(const RowAcc& o) {
    const dd_t v = dd_add(fast_two_sum(s, c), fast_two_sum(o.s, o.c));
    s = v.hi;
    c = v.lo;
  }
  __device__ __forceinline__ RowAcc peer(int m) const {
    return RowAcc{__shfl_xor_sync(0xffffffffu, s, m), __shfl_xor_sync(0xffffffffu, c, m)};
  }
  __device__ __forceinline__ R fin() const { return fast_two_sum(s, c); }
};

// Products of rows perm[i] of A with x in arithmetic OP, NR consecutive rows
// per warp; epi(i, perm[i], a . x) runs on one lane per row.
//
// The rows' values and x's reach each lane through a ring of asynchronous
// copies in the shared scratch (16 bytes per row and step, up to 4 steps
// deep; a lane reads only what it copied itself: no barriers), so a CTA
// keeps up to 100 KB of loads in flight whatever its registers hold.  NR is
// fixed at compile time and rows past the matrix repeat the last one: with a
// test per row the rows' sums ran one after another (n = 2000 fp64: 43 us
// instead of 11).  Each row has two sums (even and odd columns), because
// the chain of one is longer than a step's loads, and each warp starts at
// columns of its own; fp64 sums of fp32 rows with an fp64 vector have one,
// from the first column on (kAscending).  What bounds it: HBM for
// fp32 sums (n = 8192: 94 -> 60 us, 4.5 TB/s), the fp64 pipe (2 multiply-adds
// per clock and SM) for fp64 ones on fp32 data, where values are widened by
// integer instructions (steps with a subnormal, infinite or NaN operand on
// any lane take the hardware conversion).
template <typename A0, typename X, int OP, int NR, typename Epi>
__device__ __forceinline__ void gemv_rows_n(Cx& cx, const RefineArgs& a, const X* x, Epi& epi) {
  constexpr int VC = 16 / (int)sizeof(A0);               // columns per lane and step
  constexpr int XS = (VC * (int)sizeof(X) + 15) / 16;    // 16-byte pieces of x per lane and step
  constexpr int STEP = 32 * VC, UNIT = (NR + XS) * kRefThreads;
  static_assert(VC * sizeof(X) >= 16, "a lane's x fills whole pieces");
  static_assert(2 * UNIT * 16 <= kPhaseSmem, "the scratch holds two steps");
  using Acc = RowAcc<OP>;
  // fp64 sums on fp32 rows with an fp64 vector (the residual): one sum per
  // lane, columns ascending, the columns past the last multiple of 4 one per
  // lane at the end.  A residual is what its sums leave after cancellation,
  // so their order shows in it (1e-9 of it); with several rows per warp it
  // costs nothing on the fp64 pipe, which bounds this product.
  constexpr bool kAscending = OP == MSIR_FP64 && sizeof(A0) == 4 && sizeof(X) == 8;
  constexpr int kOdd = kAscending ? 0 : 1;
  const int nv = kAscending ? cx.n & ~3 : cx.n;  // columns of the steps
  const A0* A = (const A0*)a.A;
  const int n = cx.n, lane = cx.lane, nwarps = cx.G * (kRefThreads / 32), gw = cx.cta * (kRefThreads / 32) + cx.warp;
  const int depth = min(4, a.scratch / (UNIT * 16));     // 2, 3 or 4
  uint4* ring = (uint4*)cx.tsm + cx.tid;
  const int nsteps = (n + STEP - 1) / STEP;
  for (int i0 = gw * NR; i0 < n; i0 += nwarps * NR) {
    const A0* row[NR];
    Acc acc[NR][2];
#pragma unroll
    for (int r = 0; r < NR; ++r) row[r] = A + (size_t)a.perm[min(i0 + r, n - 1)] * a.lda;
    // each warp starts at columns of its own and wraps around: in step, the
    // warps would all read the same few lines of x at once, and the L2 slices
    // that hold them would serve one after another
    int ist = kAscending ? 0 : (int)((long long)gw * nsteps / nwarps), islot = 0;
    auto issue = [&](int st) {
      if (st < nsteps) {
        const int col = ist * STEP + lane * VC;
        ist = ist + 1 == nsteps ? 0 : ist + 1;
        const int valid = min(VC, max(0, nv - col)), c = valid > 0 ? col : 0;  // zeros past nv
        uint4* dst = ring + islot * UNIT;
#pragma unroll
        for (int r = 0; r < NR; ++r) cp_async16(dst + r * kRefThreads, row[r] + c, valid * (int)sizeof(A0));
#pragma unroll
        for (int q = 0; q < XS; ++q) {
          constexpr int XC = 16 / (int)sizeof(X);
          const int xc = col + q * XC, xv = min(XC, max(0, nv - xc));
          cp_async16(dst + (NR + q) * kRefThreads, x + (xv > 0 ? xc : 0), xv * (int)sizeof(X));
        }
      }
      islot = islot + 1 == depth ? 0 : islot + 1;
      cp_async_commit();
    };
    for (int st = 0; st < depth - 1; ++st) issue(st);
    int slot = 0;
    for (int st = 0; st < nsteps; ++st) {
      issue(st + depth - 1);
      if (depth == 4) cp_async_wait<3>();
      else if (depth == 3) cp_async_wait<2>();
      else cp_async_wait<1>();
      const uint4* src = ring + slot * UNIT;
      slot = slot + 1 == depth ? 0 : slot + 1;
      X xv[VC];
#pragma unroll
      for (int q = 0; q < XS; ++q) {
        const uint4 u = src[(NR + q) * kRefThreads];
        memcpy((char*)xv + 16 * q, &u, 16);
      }
      A0 av[NR][VC];
#pragma unroll
      for (int r = 0; r < NR; ++r) {
        const uint4 u = src[r * kRefThreads];
        memcpy(av[r], &u, 16);
      }
      if constexpr (OP != MSIR_FP32 && sizeof(A0) == 4) {
        bool sp = false;
        double xd[VC];
#pragma unroll
        for (int q = 0; q < VC; ++q) {
          if constexpr (sizeof(X) == 4) {
            sp |= widen_special(xv[q]);
            xd[q] = widen_normal(xv[q]);
          } else {
            xd[q] = xv[q];
          }
        }
#pragma unroll
        for (int r = 0; r < NR; ++r)
#pragma unroll
          for (int q = 0; q < VC; ++q) sp |= widen_special(av[r][q]);
        if (__any_sync(0xffffffffu, sp)) {
#pragma unroll
          for (int q = 0; q < VC; ++q)
#pragma unroll
            for (int r = 0; r < NR; ++r) acc[r][q & kOdd].add((double)av[r][q], (double)xv[q]);
        } else {
#pragma unroll
          for (int q = 0; q < VC; ++q)
#pragma unroll
            for (int r = 0; r < NR; ++r) acc[r][q & kOdd].add(widen_normal(av[r][q]), xd[q]);
        }
      } else {
#pragma unroll
        for (int q = 0; q < VC; ++q)
#pragma unroll
          for (int r = 0; r < NR; ++r) acc[r][q & kOdd].add(av[r][q], xv[q]);
      }
    }
    if constexpr (kAscending) {
      if (nv + lane < n) {
#pragma unroll
        for (int r = 0; r < NR; ++r) acc[r][0].add((double)row[r][nv + lane], (double)__ldcg(x + nv + lane));
      }
      __syncwarp();
    }
    // (Double-double sums are merged as renormalised pairs, 26 operations:
    // mean error 0.114 x 2^-106 sum |a x| at n = 2048, 0.220 at 8192.  As
    // terms of the row's sum, five operations, 0.151 at n = 2048; they took
    // 1.22 instead of 1.29 ms at n = 8192.)
#pragma unroll
    for (int r = 0; r < NR; ++r)
      if (kOdd) acc[r][0].merge(acc[r][1]);
#pragma unroll
    for (int m = 16; m > 0; m >>= 1)
#pragma unroll
      for (int r = 0; r < NR; ++r) acc[r][0].merge(acc[r][0].peer(m));
    Acc mine = acc[0][0];
#pragma unroll
    for (int r = 1; r < NR; ++r)
      if (lane == r) mine = acc[r][0];
    if (lane < NR && i0 + lane < n) epi(i0 + lane, a.perm[i0 + lane], mine.fin());
  }
  cp_async_wait<0>();  // (empty groups: every copy has been waited for)
}

// All rows: the fewest rows per warp (of 1, 2, 4, 7, 8) that take one round.
template <typename A0, typename X, int OP, typename Epi>
__device__ __forceinline__ void gemv_rows(Cx& cx, const RefineArgs& a, const X* x, Epi epi) {
  const int nwarps = cx.G * (kRefThreads / 32);
  const int rpw = (cx.n + nwarps - 1) / nwarps;
  if (rpw <= 1) gemv_rows_n<A0, X, OP, 1>(cx, a, x, epi);
  else if (rpw <= 2) gemv_rows_n<A0, X, OP, 2>(cx, a, x, epi);
  else if (rpw <= 4) gemv_rows_n<A0, X, OP, 4>(cx, a, x, epi);
  else if (rpw <= 7) gemv_rows_n<A0, X, OP, 7>(cx, a, x, epi);
  else gemv_rows_n<A0, X, OP, 8>(cx, a, x, epi);
}

// Reduce NV per-CTA values (each already reduced within the CTA and held by
// thread 0) across the grid.  op[i]: 0 = sum, 1 = NaN-propagating max.
template <int NV>
__device__ bool grid_reduce(Cx& cx, const RefineArgs& a, double (&v)[NV], const int (&op)[NV]) {
  PhaseTimer pt(cx, 5);
  __shared__ double s_res[kRedW];
  double* buf = a.red + (size_t)cx.redbuf * cx.G * kRedW;
  cx.redbuf ^= 1;
  if (cx.tid == 0)
    for (int i = 0; i < NV; ++i) buf[cx.cta * kRedW + i] = v[i];
  if (!grid_barrier(cx, a)) return false;
  if (cx.warp == 0) {
    for (int i = 0; i < NV; ++i) {
      double acc = op[i] ? 0.0 : 0.0;
      for (int c = cx.lane; c < cx.G; c += 32) {
        double q = __ldcg(buf + c * kRedW + i);
        acc = op[i] ? nanmax(acc, q) : __dadd_rn(acc, q);
      }
      acc = op[i] ? warp_nanmax_d(acc) : warp_sum_d(acc);
      if (cx.lane == 0) s_res[i] = acc;
    }
  }
  __syncthreads();
  for (int i = 0; i < NV; ++i) v[i] = s_res[i];
  __syncthreads();
  return true;
}

// CTA-level reduction of one value per thread (thread 0 gets the result).
static __device__ double cta_reduce(double v, int op, int tid) {
  __shared__ double s_w[kRefThreads / 32];
  v = op ? warp_nanmax_d(v) : warp_sum_d(v);
  if ((tid & 31) == 0) s_w[tid >> 5] = v;
  __syncthreads();
  double r = 0.0;
  if (tid == 0) {
    r = s_w[0];
    for (int i = 1; i < kRefThreads / 32; ++i) r = op ? nanmax(r, s_w[i]) : __dadd_rn(r, s_w[i]);
  }
  __syncthreads();
  return r;
}

// ----------------------------------------------------- triangular solves
//
// Block substitution with inverted diagonal blocks.  Block b of the forward
// solve computes z_b = c_b - sum_{j<b} L_bj y_j, then y_b = inv(L_bb) z_b
// rounded to the storage format; the backward solve runs the same way from
// the last block up with U.  The inverses (build_inverses) are in the
// arithmetic format of the solve.
//
// Thread (r, seg) of the CTA owning block b handles row r and the 16
// columns seg*16 .. seg*16+15 of every 64x64 tile of that row block.  As
// the blocks it depends on become available, the CTA accumulates their
// tiles (tile loads and payload loads issued one dependency ahead), so when
// the last one arrives only that tile, a 4-lane reduction, the 64x64
// product with the inverse and another 4-lane reduction remain on the
// critical path.
//
// Hand-off between CTAs: each solved value is published as 64-bit words
// carrying 32 payload bits and the 32-bit epoch of the solve.  A 64-bit
// aligned store or load is single-copy atomic, so a consumer that sees the
// current epoch in a word also sees that word's payload: no flag, fence or
// second round trip is needed.  Epochs grow by one per triangular solve and
// the payload buffer is zeroed whenever the epoch counter restarts.

// N consecutive factor values of one row (N in {4, 8, 16}), widened.  The
// first value's column is a multiple of N and rows start on 64-element
// boundaries, so the N values are aligned to N * sizeof(F) bytes.
__device__ __forceinline__ float h16_to_f(unsigned short b, __half*) { return __half2float(__ushort_as_half(b)); }
__device__ __forceinline__ float h16_to_f(unsigned short b, __nv_bfloat16*) { return __uint_as_float((unsigned)b << 16); }

template <typename F, int N> struct SegLd;
template <int N> struct SegLd<float, N> {
  template <typename Lt>
  static __device__ __forceinline__ void ld(const float* p, Lt (&v)[N]) {
#pragma unroll
    for (int m = 0; m < N / 4; ++m) {
      const float4 f = __ldcg((const float4*)p + m);
      v[4 * m] = (Lt)f.x; v[4 * m + 1] = (Lt)f.y; v[4 * m + 2] = (Lt)f.z; v[4 * m + 3] = (Lt)f.w;
    }
  }
};
template <int N> struct SegLd<double, N> {
  template <typename Lt>
  static __device__ __forceinline__ void ld(const double* p, Lt (&v)[N]) {
#pragma unroll
    for (int m = 0; m < N / 2; ++m) {
      const double2 f = __ldcg((const double2*)p + m);
      v[2 * m] = (Lt)f.x; v[2 * m + 1] = (Lt)f.y;
    }
  }
};
// 16-bit formats: each 32-bit word holds two values, the lower address in
// the low half
template <typename H, int N> struct SegLdH {
  template <typename Lt>
  static __device__ __forceinline__ void ld(const H* p, Lt (&v)[N]) {
    unsigned w[N / 2];
    if (N >= 8) {
#pragma unroll
      for (int m = 0; m < N / 8; ++m) {
        const uint4 u = __ldcg((const uint4*)p + m);
        w[4 * m] = u.x; w[4 * m + 1] = u.y; w[4 * m + 2] = u.z; w[4 * m + 3] = u.w;
      }
    } else {
      const uint2 u = __ldcg((const uint2*)p);
      w[0] = u.x; w[1] = u.y;
    }
#pragma unroll
    for (int k = 0; k < N / 2; ++k) {
      v[2 * k] = (Lt)h16_to_f((unsigned short)(w[k] & 0xffffu), (H*)nullptr);
      v[2 * k + 1] = (Lt)h16_to_f((unsigned short)(w[k] >> 16), (H*)nullptr);
    }
  }
};
template <int N> struct SegLd<__half, N> : SegLdH<__half, N> {};
template <int N> struct SegLd<__nv_bfloat16, N> : SegLdH<__nv_bfloat16, N> {};

// N consecutive factor values of one row, widened; zero outside the matrix.
template <typename F, typename Lt, int N>
__device__ __forceinline__ void load_seg(const F* LU, int ldf, int n, int row, int col, Lt (&v)[N]) {
  if (row < n && col + N <= n) {
    SegLd<F, N>::ld(LU + (size_t)row * ldf + col, v);
  } else {
#pragma unroll
    for (int k = 0; k < N; ++k)
      v[k] = (row < n && col + k < n) ? (Lt)to_f(LU[(size_t)row * ldf + col + k]) : (Lt)0;
  }
}

// Accumulator policies.  V: value type of the solve; A: running sum of
// products (fin() turns it into a V); L: factor element after widening;
// I: inverse element; kW: 32-bit payload words per value.  wsub(w, acc) is
// T(w - sum), the block's result before it is rounded to its storage format.
// Vectors live in double arrays (fp32 solves store floats in them, so that
// they never touch the scarce fp64 pipe; dd solves use a high and a low
// array).
// fp32 sums are compensated (ff_t, Dot2): their result is the accurately
// rounded fp32 value of the sum, which is the model of an fp32 sum that the
// solves follow (an accurate sum rounded once to the arithmetic precision),
// at a few fp32 instructions per term instead of fp64 work.
struct AccF {
  using V = float;
  using A = ff_t;
  using L = float;
  using I = float;
  static constexpr int kW = 1;
  static __device__ __forceinline__ V zero() { return 0.0f; }
  static __device__ __forceinline__ V load(const double* hi, const double*, int i) {
    return __ldcg((const float*)hi + i);
  }
  static __device__ __forceinline__ void save(double* hi, double*, int i, V v) { ((float*)hi)[i] = v; }
  static __device__ __forceinline__ void put(double* hi, double*, int i, double h, double) {
    ((float*)hi)[i] = (float)h;
  }
  static __device__ __forceinline__ double get(const double* hi, const double*, int i) {
    return (double)((const float*)hi)[i];
  }
  static __device__ __forceinline__ A azero() { return ff_t{0.0f, 0.0f}; }
  static __device__ __forceinline__ A merge(A a, A b) { return ff_merge(a, b); }
  static __device__ __forceinline__ A ax(A a, int m) { return ff_shfl_xor(a, m); }
  static __device__ __forceinline__ A fma(L l, V y, A acc) { return ff_fma(l, y, acc); }
  static __device__ __forceinline__ A ifma(I x, V z, A acc) { return ff_fma(x, z, acc); }
  static __device__ __forceinline__ V fin(A acc) { return ff_fin(acc); }
  static __device__ __forceinline__ V wsub(V w, A acc) { return ff_sub_from(w, acc); }
  static __device__ __forceinline__ V add(V a, V b) { return __fadd_rn(a, b); }
  static __device__ __forceinline__ V sub(V a, V b) { return __fsub_rn(a, b); }
  static __device__ __forceinline__ V store(V v, int fmt) { return round_f(v, fmt); }
  static __device__ __forceinline__ V sx(V v, int m) { return __shfl_xor_sync(0xffffffffu, v, m); }
  static __device__ __forceinline__ I inv(const RefineArgs& a, size_t o) { return __ldcg(a.inv32 + o); }
  // 16 consecutive scaled-block values of one row (zero outside the matrix)
  using Tm = float;
  template <int N>
  static __device__ __forceinline__ void tile(const RefineArgs& a, int n, int row, int col, Tm (&v)[N]) {
    load_seg<float, float, N>(a.M32, a.ldf, n, row, col, v);
  }
  static __device__ __forceinline__ const Tm* mat(const RefineArgs& a) { return a.M32; }
  static __device__ __forceinline__ A tfma(Tm m, V y, A acc) { return ff_fma(m, y, acc); }
  static __device__ __forceinline__ unsigned word(V v, int) { return __float_as_uint(v); }
  static __device__ __forceinline__ V unword(const unsigned* w) { return __uint_as_float(w[0]); }
};
struct AccD {
  using V = double;
  using A = double;
  using L = double;
  using I = double;
  static constexpr int kW = 2;
  static __device__ __forceinline__ V zero() { return 0.0; }
  static __device__ __forceinline__ V load(const double* hi, const double*, int i) { return __ldcg(hi + i); }
  static __device__ __forceinline__ void save(double* hi, double*, int i, V v) { hi[i] = v; }
  static __device__ __forceinline__ void put(double* hi, double*, int i, double h, double) { hi[i] = h; }
  static __device__ __forceinline__ double get(const double* hi, const double*, int i) { return hi[i]; }
  static __device__ __forceinline__ A azero() { return 0.0; }
  static __device__ __forceinline__ A merge(A a, A b) { return __dadd_rn(a, b); }
  static __device__ __forceinline__ A ax(A a, int m) { return __shfl_xor_sync(0xffffffffu, a, m); }
  static __device__ __forceinline__ A fma(L l, V y, A acc) { return __fma_rn(l, y, acc); }
  static __device__ __forceinline__ A ifma(I x, V z, A acc) { return __fma_rn(x, z, acc); }
  static __device__ __forceinline__ V fin(A acc) { return acc; }
  static __device__ __forceinline__ V wsub(V w, A acc) { return __dsub_rn(w, acc); }
  static __device__ __forceinline__ V add(V a, V b) { return __dadd_rn(a, b); }
  static __device__ __forceinline__ V sub(V a, V b) { return __dsub_rn(a, b); }
  static __device__ __forceinline__ V store(V v, int) { return v; }
  static __device__ __forceinline__ V sx(V v, int m) { return __shfl_xor_sync(0xffffffffu, v, m); }
  static __device__ __forceinline__ I inv(const RefineArgs& a, size_t o) { return __ldcg(a.inv_hi + o); }
  using Tm = double;
  template <int N>
  static __device__ __forceinline__ void tile(const RefineArgs& a, int n, int row, int col, Tm (&v)[N]) {
    load_seg<double, double, N>(a.M64, a.ldf, n, row, col, v);
  }
  static __device__ __forceinline__ const Tm* mat(const RefineArgs& a) { return a.M64; }
  static __device__ __forceinline__ A tfma(Tm m, V y, A acc) { return __fma_rn(m, y, acc); }
  static __device__ __forceinline__ unsigned word(V v, int k) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(v);
    return k == 0 ? (unsigned)b : (unsigned)(b >> 32);
  }
  static __device__ __forceinline__ V unword(const unsigned* w) {
    return __longlong_as_double((long long)(((unsigned long long)w[1] << 32) | w[0]));
  }
};
// Double-double sums of products are accumulated with compensation: each
// product is split exactly (TwoProduct) and its low-order parts kept apart,
// the running high word is updated by TwoSum and the rounding errors are
// summed in a second word (the scheme of Ogita, Rump and Oishi's Dot2,
// extended by the low words of the dd operands).  About 11 fp64 operations
// per term instead of 26 for a dd multiply and an accurate dd add, with an
// error of order n u^2 times the sum of |terms|, as for sums in dd.
struct DDAcc {
  double s, c;
};
struct AccDD {
  using V = dd_t;
  using A = DDAcc;
  using L = double;
  using I = dd_t;
  static constexpr int kW = 4;
  static __device__ __forceinline__ V zero() { return dd_t{0.0, 0.0}; }
  static __device__ __forceinline__ V load(const double* hi, const double* lo, int i) {
    return dd_t{__ldcg(hi + i), __ldcg(lo + i)};
  }
  static __device__ __forceinline__ void save(double* hi, double* lo, int i, V v) { hi[i] = v.hi; lo[i] = v.lo; }
  static __device__ __forceinline__ void put(double* hi, double* lo, int i, double h, double l) {
    hi[i] = h;
    lo[i] = l;
  }
  static __device__ __forceinline__ double get(const double* hi, const double* lo, int i) {
    return __dadd_rn(hi[i], lo[i]);
  }
  static __device__ __forceinline__ A azero() { return DDAcc{0.0, 0.0}; }
  // two partial sums: TwoSum of the running words, errors added (exact
  // error-free step, so every lane of a butterfly gets the same result)
  static __device__ __forceinline__ A merge(A a, A b) {
    const dd_t t = two_sum(a.s, b.s);
    return DDAcc{t.hi, __dadd_rn(__dadd_rn(a.c, b.c), t.lo)};
  }
  static __device__ __forceinline__ A ax(A a, int m) {
    return DDAcc{__shfl_xor_sync(0xffffffffu, a.s, m), __shfl_xor_sync(0xffffffffu, a.c, m)};
  }
  static __device__ __forceinline__ A fma(L l, V y, A acc) {
    const dd_t p = two_prod(l, y.hi);
    const double pl = __fma_rn(l, y.lo, p.lo);
    const dd_t t = two_sum_ord(acc.s, p.hi);
    return DDAcc{t.hi, __dadd_rn(acc.c, __dadd_rn(t.lo, pl))};
  }
  static __device__ __forceinline__ A ifma(I x, V z, A acc) {
    const dd_t p = two_prod(x.hi, z.hi);
    const double pl = __fma_rn(x.hi, z.lo, __fma_rn(x.lo, z.hi, p.lo));
    const dd_t t = two_sum_ord(acc.s, p.hi);
    return DDAcc{t.hi, __dadd_rn(acc.c, __dadd_rn(t.lo, pl))};
  }
  static __device__ __forceinline__ V fin(A acc) { return two_sum(acc.s, acc.c); }
  static __device__ __forceinline__ V wsub(V w, A acc) { return dd_sub(w, fin(acc)); }
  static __device__ __forceinline__ V add(V a, V b) { return dd_add(a, b); }
  static __device__ __forceinline__ V sub(V a, V b) { return dd_sub(a, b); }
  static __device__ __forceinline__ V store(V v, int) { return v; }
  static __device__ __forceinline__ V sx(V v, int m) { return dd_shfl_xor(v, m); }
  static __device__ __forceinline__ I inv(const RefineArgs& a, size_t o) {
    return dd_t{__ldcg(a.inv_hi + o), __ldcg(a.inv_lo + o)};
  }
  using Tm = dd_t;
  template <int N>
  static __device__ __forceinline__ void tile(const RefineArgs& a, int n, int row, int col, Tm (&v)[N]) {
    double h[N], l[N];
    load_seg<double, double, N>(a.Mdh, a.ldf, n, row, col, h);
    load_seg<double, double, N>(a.Mdl, a.ldf, n, row, col, l);
#pragma unroll
    for (int k = 0; k < N; ++k) v[k] = dd_t{h[k], l[k]};
  }
  static __device__ __forceinline__ A tfma(Tm m, V y, A acc) { return ifma(m, y, acc); }
  static __device__ __forceinline__ unsigned word(V v, int k) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(k < 2 ? v.hi : v.lo);
    return (k & 1) ? (unsigned)(b >> 32) : (unsigned)b;
  }
  static __device__ __forceinline__ V unword(const unsigned* w) {
    return dd_t{__longlong_as_double((long long)(((unsigned long long)w[1] << 32) | w[0])),
                __longlong_as_double((long long)(((unsigned long long)w[3] << 32) | w[2]))};
  }
};

static_assert(kRefThreads == 4 * kBlk, "substitution thread layout");

__device__ __forceinline__ unsigned long long ld_relaxed_u64(const unsigned long long* p) {
  unsigned long long v;
  asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void st_relaxed_u64(unsigned long long* p, unsigned long long v) {
  asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}

// Distributed shared memory: the address of `p` (this CTA's shared memory)
// in cluster peer `rank`, a relaxed store there, and a relaxed load of this
// CTA's own copy that observes such stores.
__device__ __forceinline__ unsigned peer_addr(const void* p, unsigned rank) {
  const unsigned a = (unsigned)__cvta_generic_to_shared(p);
  unsigned r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
  return r;
}
__device__ __forceinline__ void st_peer_u64(unsigned addr, unsigned long long v) {
  asm volatile("st.relaxed.cluster.shared::cluster.u64 [%0], %1;" ::"r"(addr), "l"(v) : "memory");
}
__device__ __forceinline__ unsigned long long ld_inbox_u64(const unsigned long long* p) {
  unsigned long long v;
  const unsigned a = (unsigned)__cvta_generic_to_shared(p);
  asm volatile("ld.relaxed.cluster.shared::cta.u64 %0, [%1];" : "=l"(v) : "r"(a) : "memory");
  return v;
}
// Cluster-wide barrier of all threads (release / acquire at cluster scope).
__device__ __forceinline__ void cluster_sync_all() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// Tag of an inbox word: the solve's epoch and the block's round (block /
// number of teams), bit 31 clear so that it never equals the all-ones fill
// of a fresh inbox.
__device__ __forceinline__ unsigned inbox_tag(unsigned epoch, int round) {
  return ((epoch << 8) | ((unsigned)round & 0xffu)) & 0x7fffffffu;
}

// Payload words of one block held by one lane: values lane and lane + 32.
template <int W>
struct LLRaw {
  unsigned long long w[2][W];
};

template <int W>
__device__ __forceinline__ void ll_issue(const unsigned long long* blk, int lane, LLRaw<W>& r) {
#pragma unroll
  for (int m = 0; m < 2; ++m)
#pragma unroll
    for (int k = 0; k < W; ++k) r.w[m][k] = ld_relaxed_u64(blk + (size_t)(lane + 32 * m) * W + k);
}

template <int W>
__device__ __forceinline__ bool ll_ready(const LLRaw<W>& r, unsigned epoch) {
  bool ok = true;
#pragma unroll
  for (int m = 0; m < 2; ++m)
#pragma unroll
    for (int k = 0; k < W; ++k) ok &= (unsigned)(r.w[m][k] >> 32) == epoch;
  return __all_sync(0xffffffffu, ok);
}

// Complete the payload of block `blk` whose loads were issued into r: poll
// until every word carries `epoch`, then stage the 64 values for the warp.
// Bounded like every device wait (MSIR_ERR_TIMEOUT, or another block's
// error).
template <typename ACC>
__device__ __forceinline__ bool ll_complete(const unsigned long long* blk, unsigned epoch, int lane,
                                            LLRaw<ACC::kW>& r, typename ACC::V* stage, int* err,
                                            int where) {
  constexpr int W = ACC::kW;
  unsigned long long t0 = 0;
  unsigned spins = 0;
  while (!ll_ready<W>(r, epoch)) {
    if ((++spins & 255u) == 0u) {
      int bad = 0;
      if (lane == 0) {
        if (t0 == 0) t0 = gtimer();
        if (ld_volatile_i32(err) != 0) bad = 1;
        else if (gtimer() - t0 > kWaitTimeoutNs) bad = 2;
      }
      bad = __shfl_sync(0xffffffffu, bad, 0);
      if (bad == 2) {
        // diagnostics: the first word still missing and the epoch it holds
        int idx = -1;
        unsigned tag = 0;
#pragma unroll
        for (int m = 0; m < 2; ++m)
#pragma unroll
          for (int k = 0; k < W; ++k)
            if (idx < 0 && (unsigned)(r.w[m][k] >> 32) != epoch) {
              idx = (lane + 32 * m) * W + k;
              tag = (unsigned)(r.w[m][k] >> 32);
            }
        const unsigned mk = __ballot_sync(0xffffffffu, idx >= 0);
        const int src = mk ? __ffs(mk) - 1 : 0;
        idx = __shfl_sync(0xffffffffu, idx, src);
        tag = __shfl_sync(0xffffffffu, tag, src);
        if (lane == 0) record_timeout(err, 2, where, (int)epoch, (idx << 20) | (int)(tag & 0xfffffu));
      }
      if (bad) return false;
    }
    ll_issue<W>(blk, lane, r);
  }
  __syncwarp();  // the previous block's staged values have been consumed
#pragma unroll
  for (int m = 0; m < 2; ++m) {
    unsigned p[W];
#pragma unroll
    for (int k = 0; k < W; ++k) p[k] = (unsigned)r.w[m][k];
    stage[lane + 32 * m] = ACC::unword(p);
  }
  __syncwarp();
  return true;
}

// ll_complete for a block that a cluster peer writes into this CTA's inbox
// slot: poll shared memory (no L2 round trip) until every word carries
// `tag`, then stage the values.  Bounded like every device wait.
template <typename ACC>
__device__ __forceinline__ bool ib_complete(const unsigned long long* slot, unsigned tag, int lane,
                                            typename ACC::V* stage, int* err, int where) {
  constexpr int W = ACC::kW;
  LLRaw<W> r;
  unsigned long long t0 = 0;
  unsigned spins = 0;
  while (true) {
#pragma unroll
    for (int m = 0; m < 2; ++m)
#pragma unroll
      for (int k = 0; k < W; ++k) r.w[m][k] = ld_inbox_u64(slot + (size_t)(lane + 32 * m) * W + k);
    if (ll_ready<W>(r, tag)) break;
    if ((++spins & 1023u) == 0u) {
      int bad = 0;
      if (lane == 0) {
        if (t0 == 0) t0 = gtimer();
        if (ld_volatile_i32(err) != 0) bad = 1;
        else if (gtimer() - t0 > kWaitTimeoutNs) bad = 2;
      }
      bad = __shfl_sync(0xffffffffu, bad, 0);
      if (bad == 2 && lane == 0) record_timeout(err, 2, where, (int)tag, -1);
      if (bad) return false;
    }
  }
  __syncwarp();  // the previous block's staged values have been consumed
#pragma unroll
  for (int m = 0; m < 2; ++m) {
    unsigned p[W];
#pragma unroll
    for (int k = 0; k < W; ++k) p[k] = (unsigned)r.w[m][k];
    stage[lane + 32 * m] = ACC::unword(p);
  }
  __syncwarp();
  return true;
}

// The factor storage type F of the refinement code is a template parameter
// of the single-system kernels (one instantiation per u_f); FAny stands for
// "the format in RefineArgs::f_fmt", read at run time, so that the batched
// engine, whose systems change u_f as they escalate, needs one
// instantiation.  Only the scaled-block construction reads the factors.
struct FAny {};
template <typename F>
__device__ __forceinline__ int factor_fmt(const RefineArgs&) {
  return Fmt<F>::code;
}
template <>
__device__ __forceinline__ int factor_fmt<FAny>(const RefineArgs& a) {
  return a.f_fmt;
}
template <typename F>
__device__ __forceinline__ double factor_at(const RefineArgs& a, size_t i) {
  return (double)to_f(((const F*)a.LU)[i]);
}
template <>
__device__ __forceinline__ double factor_at<FAny>(const RefineArgs& a, size_t i) {
  switch (a.f_fmt) {
    case MSIR_FP16: return (double)to_f(((const __half*)a.LU)[i]);
    case MSIR_BF16: return (double)to_f(((const __nv_bfloat16*)a.LU)[i]);
    case MSIR_FP32: return (double)((const float*)a.LU)[i];
    default: return ((const double*)a.LU)[i];
  }
}

static_assert(kInvScratch == (int)kInvSmem && kInvThreads == kRefThreads, "inverse scratch");

// Index of row r (of the n rows padded to whole superblocks) of triangle tri
// (0 L, 1 U) in the inverses of the diagonal superblocks, [2][npad][kSuper].
__device__ __forceinline__ size_t wide_row(const RefineArgs& a, int tri, int r) {
  return ((size_t)tri * a.npad + r) * kSuper;
}

// Inverses of the diagonal blocks of L and U by all CTAs of the grid, once
// per factorisation: as fp32 pairs (dd = false; inv32, inv32l) or in
// double-double (inv_hi, inv_lo, and for fp64 factors inv32, inv32l too);
// `wide`: the fp32 pairs go into the superblocks' array.
//
// The fp32 pairs of a block are formed in pair arithmetic if its diagonal is
// far from fp32's range ends and |X||B||X| is at most kInvCond times X
// (inv_cond_below): their error of 2^-46 times that is then below 2^-32, so
// that the inverse's fp32 rounding is the exact inverse's but for near ties.
// (LU factors of randsvd and normal matrices, plain and with rows or columns
// graded by 10^+-4: at most 1.4e3.  Solves with such inverses and scaled blocks
// against double-double ones, n = 1024 .. 7237: 1.000 times the error of
// those formed in double-double and fp64.)  Other blocks are formed in
// double-double and marked inv_hard.  Where double-double inverses are there
// already (kept factors), they are rounded to pairs instead.  The caller puts
// a grid barrier behind it; nothing here waits.
constexpr float kInvCond = 0x1p14f;
template <typename F>
__device__ __noinline__ void build_inverses(Cx& cx, const RefineArgs& a, bool dd, bool wide) {
  float* smf = (float*)cx.tsm;
  double* smd = (double*)cx.tsm;
  const bool want32 = !dd || factor_fmt<F>(a) == MSIR_FP64;
  const bool have = !dd && (cx.mready & RDY_INV);
  for (int q = cx.cta; q < 2 * cx.nblk; q += cx.G) {
    const int b = q % cx.nblk;
    const bool lower = q < cx.nblk;
    const size_t f0 = (size_t)b * kBlk * a.ldf + (size_t)b * kBlk;
    const size_t base = ((size_t)(lower ? 0 : 1) * cx.nblk + b) * kBlk * kBlk;
    const int nr = min(kBlk, cx.n - b * kBlk);
    auto get = [&](int i, int k) { return factor_at<F>(a, f0 + (size_t)i * a.ldf + k); };
    bool pair64 = dd;
    __syncthreads();  // the scratch is no longer read
    if (!dd) {
      inv_load<float>(smf, cx.n, b, lower, get);
      const float d = cx.tid < kBlk ? fabsf(smf[cx.tid * kXld + cx.tid]) : 1.0f;
      bool hard = __syncthreads_or(!(d >= 0x1p-60f && d <= 0x1p60f)) != 0;
      if (have) {
        for (int e = cx.tid; e < kBlk * kBlk; e += kRefThreads) {
          const double h = __ldcg(a.inv_hi + base + e), l = __ldcg(a.inv_lo + base + e);
          const float r = dd_to_f32(h, l);
          const int x = kIB * kXld + e / kBlk * kXld + e % kBlk;
          smf[x] = r;
          smf[x + kIB * kXld] = isfinite(r) ? (float)((h - (double)r) + l) : 0.0f;
        }
        __syncthreads();
      } else if (!hard) {
        inv_triangle<ArFF>(lower, smf);
      }
      hard = hard || !inv_cond_below(smf, kInvCond);
      if (cx.tid == 0) a.inv_hard[q] = hard;
      pair64 = hard && !have;
      __syncthreads();
    }
    if (pair64) {
      inv_load<double>(smd, cx.n, b, lower, get);
      inv_triangle<ArDD>(lower, smd);
    }
    // for wide solves the blocks go on the diagonals of the superblocks
    const size_t wbase = wide ? wide_row(a, lower ? 0 : 1, b * kBlk) + (b * kBlk) % kSuper : 0;
    const bool w32 = wide && !dd;
    float* o32h = w32 ? a.D32h + wbase : a.inv32 + base;
    float* o32l = w32 ? a.D32l + wbase : a.inv32l + base;
    const int ld32 = w32 ? kSuper : kBlk;
    for (int e = cx.tid; e < kBlk * kBlk; e += kRefThreads) {
      const int i = e / kBlk, k = e % kBlk, x = kIB * kXld + i * kXld + k;
      const bool in = i < nr && k < nr;
      if (pair64) {
        const double h = in ? smd[x] : 0.0, l = in ? smd[x + kIB * kXld] : 0.0;
        a.inv_hi[base + e] = h;
        a.inv_lo[base + e] = l;
        if (want32) {
          const float r = dd_to_f32(h, l);
          o32h[(size_t)i * ld32 + k] = r;
          o32l[(size_t)i * ld32 + k] = isfinite(r) ? (float)((h - (double)r) + l) : 0.0f;
        }
      } else {
        o32h[(size_t)i * ld32 + k] = in ? smf[x] : 0.0f;
        o32l[(size_t)i * ld32 + k] = in ? smf[x + kIB * kXld] : 0.0f;
      }
    }
  }
}

// Scaled off-diagonal blocks M_bj = D_b^{-1} F_bj (j != b; L below the
// diagonal blocks, U above), formed by all CTAs of the grid once per
// factorisation and precision, the first time a solve needs them: one 64x64
// tile per step.
//
// fp32 (bf16 / fp16 / fp32 factors): the inverse as an fp32 pair times the
// factor's values (exact in fp32), compensated sums, rounded once to fp32;
// its error before that rounding is about 2^-45 of the sum of magnitudes,
// and no fp64 instruction is issued (GB300's fp64 pipe runs 2 multiply-adds
// per clock and SM against 128 in fp32, and about 11 fp32 instructions do a
// term).  The inverse is staged transposed, so that a thread's 4 x 4 elements
// take three 16-byte loads per inner step; terms outside the triangle of the
// inverse are zero and skipped (a warp has 8 rows, warps w and w + 4 of one
// scheduler have long and short sums).  Measured (n = 8192): 7.2 -> 1.0 ms
// against fp64 sums.  Rows of blocks marked inv_hard take those: the fp64
// inverse, fp64 sums in the order of k, rounded once.
template <typename F>
__device__ __noinline__ bool build_scaled32(Cx& cx, const RefineArgs& a) {
  float* Xh = (float*)cx.ssm;  // [k][i], kBlk x kSc32Ld
  float* Xl = Xh + kBlk * kSc32Ld;
  float* Fb = Xl + kBlk * kSc32Ld;  // [k][c]
  const int n = cx.n, nb = cx.nblk, ld = a.ldf;
  const int wr = cx.warp < 4 ? cx.warp : 11 - cx.warp;
  const int i0 = wr * 8 + (cx.lane >> 4) * 4, c0 = (cx.lane & 15) * 4;
  for (int t = cx.cta; t < nb * nb; t += cx.G) {
    const int b = t / nb, j = t % nb;
    if (b == j) continue;
    const bool lower = j < b;
    const size_t ib = ((size_t)(lower ? 0 : 1) * nb + b) * kBlk * kBlk;
    const int r0 = b * kBlk, q0 = j * kBlk;
    __syncthreads();  // the previous staging is no longer read
    if (__ldcg(a.inv_hard + (lower ? 0 : nb) + b)) {
      for (int e = cx.tid; e < kBlk * kBlk; e += kRefThreads) {
        const int i = e / kBlk, row = r0 + i, col = q0 + e % kBlk;
        if (row >= n || col >= n) continue;
        double s = 0.0;
        const int k0 = lower ? 0 : i, k1 = lower ? i + 1 : min(kBlk, n - r0);
        for (int k = k0; k < k1; ++k)
          s = __fma_rn(__ldcg(a.inv_hi + ib + (size_t)i * kBlk + k), factor_at<F>(a, (size_t)(r0 + k) * ld + col), s);
        a.M32[(size_t)row * ld + col] = __double2float_rn(s);
      }
      continue;
    }
    for (int e = cx.tid; e < kBlk * kBlk; e += kRefThreads) {
      const int i = e / kBlk, k = e % kBlk;
      Xh[k * kSc32Ld + i] = __ldcg(a.inv32 + ib + e);
      Xl[k * kSc32Ld + i] = __ldcg(a.inv32l + ib + e);
      Fb[i * kSc32Ld + k] = (r0 + i < n && q0 + k < n) ? (float)factor_at<F>(a, (size_t)(r0 + i) * ld + q0 + k) : 0.0f;
    }
    __syncthreads();
    ff_t acc[4][4];
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
      for (int q = 0; q < 4; ++q) acc[r][q] = ff_t{0.0f, 0.0f};
    const int k0 = lower ? 0 : wr * 8, k1 = lower ? wr * 8 + 8 : kBlk;
    for (int k = k0; k < k1; ++k) {
      const float4 xh = *(const float4*)(Xh + k * kSc32Ld + i0);
      const float4 xl = *(const float4*)(Xl + k * kSc32Ld + i0);
      const float4 f = *(const float4*)(Fb + k * kSc32Ld + c0);
      const float h4[4] = {xh.x, xh.y, xh.z, xh.w}, l4[4] = {xl.x, xl.y, xl.z, xl.w}, f4[4] = {f.x, f.y, f.z, f.w};
#pragma unroll
      for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int q = 0; q < 4; ++q) acc[r][q] = ArFF::term(f4[q], ArFF::V{h4[r], l4[r]}, acc[r][q]);
    }
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const int row = r0 + i0 + r, col = q0 + c0;
      if (row >= n) continue;
      float* dst = a.M32 + (size_t)row * ld + col;
      if (col + 4 <= n) {
        *(float4*)dst = make_float4(ff_fin(acc[r][0]), ff_fin(acc[r][1]), ff_fin(acc[r][2]), ff_fin(acc[r][3]));
      } else {
#pragma unroll
        for (int q = 0; q < 4; ++q)
          if (col + q < n) dst[q] = ff_fin(acc[r][q]);
      }
    }
  }
  return grid_barrier(cx, a);
}

// fp64 and dd (and fp32 with fp64 factors): the inverse of the diagonal block
// and the factor block are staged in shared memory (half the inner dimension
// at a time); thread (i, g) forms row i, columns 16g .. 16g+15 of the
// product, 64 terms each.  fp64: fp64 inverse, fp64 sums (with fp64 factors
// rounded to fp32 for M32 too); dd: dd inverse, sums compensated as in the
// substitutions (Dot2 with the inverse's low word).
template <typename F>
__device__ __noinline__ bool build_scaled(Cx& cx, const RefineArgs& a, bool dd) {
  // staging of half the inner dimension at a time: inverse columns k0..k0+31
  // (high, low words) and factor rows k0..k0+31; the sums keep k order
  constexpr int KH = kBlk / 2;
  double* Xh = (double*)cx.ssm;       // 64 x (KH + 1)
  double* Xl = Xh + kBlk * (KH + 1);  // 64 x (KH + 1)
  double* Fb = Xl + kBlk * (KH + 1);  // KH x kScLd
  const bool with32 = factor_fmt<F>(a) == MSIR_FP64;
  const int n = cx.n, nb = cx.nblk, ld = a.ldf;
  const int i = cx.tid >> 2, cg = cx.tid & 3;
  for (int t = cx.cta; t < nb * nb; t += cx.G) {
    const int b = t / nb, j = t % nb;
    if (b == j) continue;
    const bool lower = j < b;
    const size_t ib = ((size_t)(lower ? 0 : 1) * nb + b) * kBlk * kBlk;
    const int r0 = b * kBlk, c0 = j * kBlk;
    const int row = r0 + i;
    double sh[16], sc[16];
#pragma unroll
    for (int q = 0; q < 16; ++q) sh[q] = sc[q] = 0.0;
    for (int k0 = 0; k0 < kBlk; k0 += KH) {
      __syncthreads();  // the previous staging is no longer read
      for (int e = cx.tid; e < kBlk * KH; e += kRefThreads) {
        const int rr = e / KH, kk = e % KH;
        Xh[rr * (KH + 1) + kk] = __ldcg(a.inv_hi + ib + (size_t)rr * kBlk + k0 + kk);
        if (dd) Xl[rr * (KH + 1) + kk] = __ldcg(a.inv_lo + ib + (size_t)rr * kBlk + k0 + kk);
      }
      for (int e = cx.tid; e < KH * kBlk; e += kRefThreads) {
        const int kk = e / kBlk, cc = e % kBlk;
        const int frow = r0 + k0 + kk, col = c0 + cc;
        Fb[kk * kScLd + cc] = (frow < n && col < n) ? factor_at<F>(a, (size_t)frow * ld + col) : 0.0;
      }
      __syncthreads();
      if (!dd) {
        for (int kk = 0; kk < KH; ++kk) {
          const double x = Xh[i * (KH + 1) + kk];
#pragma unroll
          for (int q = 0; q < 16; ++q) sh[q] = __fma_rn(x, Fb[kk * kScLd + cg * 16 + q], sh[q]);
        }
      } else {
        for (int kk = 0; kk < KH; ++kk) {
          const double xh = Xh[i * (KH + 1) + kk], xl = Xl[i * (KH + 1) + kk];
#pragma unroll
          for (int q = 0; q < 16; ++q) {
            const double f = Fb[kk * kScLd + cg * 16 + q];
            const dd_t p = two_prod(xh, f);
            const double pl = __fma_rn(xl, f, p.lo);
            const dd_t u = two_sum_ord(sh[q], p.hi);
            sh[q] = u.hi;
            sc[q] = __dadd_rn(sc[q], __dadd_rn(u.lo, pl));
          }
        }
      }
    }
    if (row < n) {
#pragma unroll
      for (int q = 0; q < 16; ++q) {
        const int col = c0 + cg * 16 + q;
        if (col >= n) continue;
        if (!dd) {
          a.M64[(size_t)row * ld + col] = sh[q];
          if (with32) a.M32[(size_t)row * ld + col] = __double2float_rn(sh[q]);
        } else {
          const dd_t v = two_sum(sh[q], sc[q]);
          a.Mdh[(size_t)row * ld + col] = v.hi;
          a.Mdl[(size_t)row * ld + col] = v.lo;
        }
      }
    }
  }
  return grid_barrier(cx, a);
}

// Depth of the ring of scaled-block tiles that fp32 / fp64 substitutions
// stream through shared memory (the scaled-block staging area, idle during
// the solves); a member's tile is R x 64 values.
constexpr int kTileRing = 3;

// One triangular solve (LOWER: L y = c, unit diagonal; else U z = y) over
// all blocks of this CTA's team, with the block rows scaled beforehand:
// y_b = w_b - sum_j M_bj y_j, w_b = inv(D_b) c_b (the backward solve the
// same with U).
//
// Teams: K CTAs (K in {1, 2, 4, 8}) share each 64-row block, member m
// taking rows m*64/K .. (m+1)*64/K - 1; teams own blocks t, t + T, t + 2T,
// ... (T = floor(G / K) teams; CTAs beyond K*T idle).  Each row is handled
// by TPR adjacent threads with 64/TPR columns of every tile each (TPR = 4,
// or 8 and 16 for K = 4 and 8 so that at least 4 warps work); the other
// warps only take part in the barriers.  Members need no exchange: each has all it
// needs for its rows (w from all of c_b, the tiles' rows, the published y).
// w_b is formed before the block's dependencies arrive, so the dependency
// chain carries one tile product and a 4-lane sum per block.  The backward
// solve takes y_b from the forward solve's published words (epoch - 1),
// because its rows may have been solved by other members.
//
// Not inlined: its register-heavy loop then does not raise the pressure of
// the rest of the kernel (the call costs a few register saves per solve).
template <typename F, typename ACC, bool LOWER, int K>
__device__ __noinline__ bool trsv_team(Cx& cx, const RefineArgs& a, int store_fmt, unsigned epoch) {
  using V = typename ACC::V;
  using I = typename ACC::I;
  using Tm = typename ACC::Tm;
  constexpr int W = ACC::kW;
  constexpr int R = kBlk / K;               // rows per member
  // threads per row: 4, or more so that a member keeps at least 4 warps
  // busy (one per SM sub-partition; each has its own fp64 unit)
  constexpr int TPR = R * 4 >= 128 ? 4 : 128 / R;
  constexpr int NC = kBlk / TPR;            // columns per thread and tile
  constexpr int NACT = R * TPR;             // working threads (whole warps)
  static_assert(NACT % 32 == 0 && NACT <= kRefThreads && NC >= 4, "team shape");
  V* s_stage = (V*)cx.tsm;                  // per warp: 64 staged values
  const int n = cx.n;
  const bool act = cx.tid < NACT;
  const int r = act ? cx.tid / TPR : 0, seg = cx.tid % TPR;
  V* stage = s_stage + cx.warp * kBlk;
  const int tri = LOWER ? 0 : 1;
  const double* in_hi = a.c_hi;  // forward solve input (backward: published y)
  const double* in_lo = a.c_lo;
  double* out_hi = LOWER ? a.y_hi : a.z_hi;
  double* out_lo = LOWER ? a.y_lo : a.z_lo;
  // hand-off words: [direction][block][64][W] (direction 0 forward, 1 backward)
  const size_t llblk = (size_t)kBlk * kLLWords;
  unsigned long long* ll_y = a.ll + (size_t)tri * cx.nblk * llblk;
  const unsigned long long* ll_fwd = a.ll;
  const int T = cx.G / K;
  const int team = cx.cta / K, member = cx.cta % K;
  const int nmine = team < T && team < cx.nblk ? (cx.nblk - 1 - team) / T + 1 : 0;
  // Clusters (cx.C > 1, K | C): the C / K teams of a cluster own
  // consecutive blocks of each round, and a team takes the blocks of the
  // teams before it in its cluster (forward; after it, backward) from its
  // inbox, where their owners write them through distributed shared memory,
  // instead of from the L2 hand-off words.  Every block is also published to
  // L2 for the other clusters.
  const bool clus = cx.C > 1 && K <= cx.C;
  const int TPC = clus ? cx.C / K : 1;  // teams per cluster
  const int tpos = team % TPC;          // this team's position in its cluster
  for (int q = 0; q < nmine; ++q) {
    const int b = LOWER ? team + q * T : team + (nmine - 1 - q) * T;
    const int r0 = b * kBlk;
    const int nr = min(kBlk, n - r0);
    const int rr = member * R + r;  // row within the block
    const int row = r0 + rr;
    const unsigned itag = inbox_tag(epoch, b / T);
    // dependencies taken from the inbox: forward b - tpos .. b - 1, backward
    // b + 1 .. b + TPC - 1 - tpos (the same round, this cluster)
    const int ib_lo = LOWER ? b - tpos : b + 1;
    const int ib_hi = LOWER ? b - 1 : b + (TPC - 1 - tpos);
    auto from_inbox = [&](int j) { return clus && j >= ib_lo && j <= ib_hi; };
    auto inbox_slot = [&](int j) {  // the source team's position
      return cx.inbox + (size_t)(tpos + (j - b)) * kBlk * W;
    };
    unsigned long long* ts = a.tsv ? a.tsv + ((LOWER ? 0 : 1) * (size_t)cx.nblk + b) * 4 : nullptr;
    if (ts && cx.tid == 0 && member == 0) ts[0] = gtimer();
    bool ok = true;  // a failed wait ends the warp's work; the CTA leaves together below
    // w_r = (row rr of inv(D_b)) c_b
    typename ACC::A wa = ACC::azero();
    if (act) {
      const V* cs;
      if (LOWER) {
        V cv[NC];
#pragma unroll
        for (int k = 0; k < NC; ++k) {
          const int kk = seg * NC + k;
          cv[k] = kk < nr ? ACC::load(in_hi, in_lo, r0 + kk) : ACC::zero();
        }
        const size_t inv_row = (((size_t)tri * cx.nblk + b) * kBlk + rr) * kBlk + seg * NC;
#pragma unroll
        for (int k = 0; k < NC; ++k) wa = ACC::ifma(ACC::inv(a, inv_row + k), cv[k], wa);
      } else {
        LLRaw<W> py;
        ll_issue<W>(ll_fwd + (size_t)b * llblk, cx.lane, py);
        ok = ll_complete<ACC>(ll_fwd + (size_t)b * llblk, epoch - 1, cx.lane, py, stage, a.err,
                              (tri << 24) | (1 << 23) | (b << 12) | b);
        cs = stage + seg * NC;
        const size_t inv_row = (((size_t)tri * cx.nblk + b) * kBlk + rr) * kBlk + seg * NC;
        if (ok) {
#pragma unroll
          for (int k = 0; k < NC; ++k) wa = ACC::ifma(ACC::inv(a, inv_row + k), cs[k], wa);
        }
      }
#pragma unroll
      for (int m = 1; m < TPR; m <<= 1) wa = ACC::merge(wa, ACC::ax(wa, m));
    }
    const V wr = ACC::fin(wa);
    // dependencies in the order they become available
    const int ndep = LOWER ? b : cx.nblk - 1 - b;
    // two interleaved partial sums (even and odd columns), merged at the
    // end: the tile product on the dependency chain is half as deep
    typename ACC::A acc = ACC::azero(), acc2 = ACC::azero();
    // fp32/fp64 tiles of at most a sixth of the staging area stream through a
    // ring in shared memory; wider ones (fp64 without teams) and dd tiles
    // are loaded into registers
    constexpr bool kRing = W <= 2 && (size_t)R * kBlk * sizeof(Tm) * kTileRing <= (size_t)kScaledSmem;
    if (ok && ndep > 0 && act) {
      if constexpr (kRing) {
        // fp32/fp64: the tiles stream through a ring in shared memory,
        // kTileRing - 1 dependencies ahead (asynchronous copies; each thread
        // copies and later reads only its own chunks, so no barrier), and the
        // hand-off words are loaded one dependency ahead
        constexpr int EPC = 16 / (int)sizeof(Tm);  // values per 16-byte chunk
        constexpr int NCH = NC / EPC;              // chunks per thread and tile
        Tm* ring = (Tm*)cx.ssm;                    // [kTileRing][NCH][NACT][EPC]
        const Tm* Mat = ACC::mat(a);
        auto issue = [&](int t) {
          if (t < ndep) {
            const int jt = LOWER ? t : cx.nblk - 1 - t;
            Tm* slot = ring + (size_t)(t % kTileRing) * NCH * NACT * EPC;
#pragma unroll
            for (int c = 0; c < NCH; ++c) {
              const int col = jt * kBlk + seg * NC + c * EPC;
              const int valid = row < n ? max(0, min(EPC, n - col)) : 0;
              const Tm* src = Mat + (valid > 0 ? (size_t)row * a.ldf + col : 0);
              cp_async16(slot + ((size_t)c * NACT + cx.tid) * EPC, src, valid * (int)sizeof(Tm));
            }
          }
          cp_async_commit();
        };
#pragma unroll
        for (int t = 0; t < kTileRing - 1; ++t) issue(t);
        LLRaw<W> pc, pn;
        int jb = LOWER ? 0 : cx.nblk - 1;
        if (!from_inbox(jb)) ll_issue<W>(ll_y + (size_t)jb * llblk, cx.lane, pc);
        for (int t = 0; t < ndep; ++t) {
          const int jn = LOWER ? jb + 1 : jb - 1;
          const bool more = t + 1 < ndep;
          issue(t + kTileRing - 1);
          if (more && !from_inbox(jn)) ll_issue<W>(ll_y + (size_t)jn * llblk, cx.lane, pn);
          cp_async_wait<kTileRing - 1>();  // this thread's copies of tile t are done
          Tm tc[NC];
          const Tm* slot = ring + (size_t)(t % kTileRing) * NCH * NACT * EPC;
#pragma unroll
          for (int c = 0; c < NCH; ++c)
#pragma unroll
            for (int e = 0; e < EPC; ++e) tc[c * EPC + e] = slot[((size_t)c * NACT + cx.tid) * EPC + e];
          const int where = (tri << 24) | (b << 12) | jb;
          if (!(from_inbox(jb) ? ib_complete<ACC>(inbox_slot(jb), itag, cx.lane, stage, a.err, where | (1 << 22))
                               : ll_complete<ACC>(ll_y + (size_t)jb * llblk, epoch, cx.lane, pc, stage, a.err, where))) {
            ok = false;
            break;
          }
          if (ts && !more && cx.tid == 0 && member == 0) ts[3] = gtimer();
          const V* ys = stage + seg * NC;
#pragma unroll
          for (int k = 0; k < NC; k += 2) {
            acc = ACC::tfma(tc[k], ys[k], acc);
            acc2 = ACC::tfma(tc[k + 1], ys[k + 1], acc2);
          }
          if (!more) break;
          pc = pn;
          jb = jn;
        }
        cp_async_wait<0>();  // no copy outlives the solve (the ring is reused)
      } else {
        // fp64 without teams: tile and payload loads one dependency ahead
        // (double buffer); dd: the next tile is loaded after the current
        // one is used (its products, not the loads, bound the dd solve)
        constexpr bool kDouble = W <= 2;
        Tm tc[NC], tn[kDouble ? NC : 1];
        LLRaw<W> pc, pn;
        int jb = LOWER ? 0 : cx.nblk - 1;
        ACC::template tile<NC>(a, n, row, jb * kBlk + seg * NC, tc);
        if (!from_inbox(jb)) ll_issue<W>(ll_y + (size_t)jb * llblk, cx.lane, pc);
        for (int t = 0; t < ndep; ++t) {
          const int jn = LOWER ? jb + 1 : jb - 1;
          const bool more = t + 1 < ndep;
          if (kDouble && more) {
            ACC::template tile<NC>(a, n, row, jn * kBlk + seg * NC, *(Tm(*)[NC])tn);
            if (!from_inbox(jn)) ll_issue<W>(ll_y + (size_t)jn * llblk, cx.lane, pn);
          }
          const int where = (tri << 24) | (b << 12) | jb;
          if (!(from_inbox(jb) ? ib_complete<ACC>(inbox_slot(jb), itag, cx.lane, stage, a.err, where | (1 << 22))
                               : ll_complete<ACC>(ll_y + (size_t)jb * llblk, epoch, cx.lane, pc, stage, a.err, where))) {
            ok = false;
            break;
          }
          if (ts && !more && cx.tid == 0 && member == 0) ts[3] = gtimer();
          const V* ys = stage + seg * NC;
#pragma unroll
          for (int k = 0; k < NC; k += 2) {
            acc = ACC::tfma(tc[k], ys[k], acc);
            acc2 = ACC::tfma(tc[k + 1], ys[k + 1], acc2);
          }
          if (!more) break;
          if (kDouble) {
#pragma unroll
            for (int k = 0; k < NC; ++k) tc[k] = tn[kDouble ? k : 0];
            pc = pn;
          } else {
            ACC::template tile<NC>(a, n, row, jn * kBlk + seg * NC, tc);
            if (!from_inbox(jn)) ll_issue<W>(ll_y + (size_t)jn * llblk, cx.lane, pc);
          }
          jb = jn;
        }
      }
    }
    acc = ACC::merge(acc, acc2);
    if (ts && cx.tid == 0 && member == 0) ts[1] = gtimer();
    if (act && ok) {
      // the TPR segments of the row: s_r, then y_r = S(T(w_r - s_r))
#pragma unroll
      for (int m = 1; m < TPR; m <<= 1) acc = ACC::merge(acc, ACC::ax(acc, m));
      V y = ACC::store(ACC::wsub(wr, acc), store_fmt);
      if (rr >= nr) y = ACC::zero();
      // publish: segment k writes payload word k of the row (rows past n as 0)
      if (seg < W)
        st_relaxed_u64(ll_y + (size_t)b * llblk + (size_t)rr * W + seg,
                       ((unsigned long long)epoch << 32) | ACC::word(y, seg));
      if (clus) {
        // and into the inboxes of the cluster's teams that take this block
        // next (their K members each): word k of the row for target CTA c,
        // spread over the row's TPR threads
        const int nteams = LOWER ? min(TPC - 1 - tpos, cx.nblk - 1 - b) : tpos;
        const unsigned long long* dst = cx.inbox + ((size_t)tpos * kBlk + rr) * W;
        for (int e = seg; e < nteams * K * W; e += TPR) {
          const int ci = e / W, k = e % W;
          const int cpos = LOWER ? tpos + 1 + ci / K : tpos - 1 - ci / K;
          st_peer_u64(peer_addr(dst + k, (unsigned)(cpos * K + ci % K)),
                      ((unsigned long long)itag << 32) | ACC::word(y, k));
        }
      }
      if (seg == 0 && rr < nr) ACC::save(out_hi, out_lo, row, y);
    }
    if (ts && cx.tid == 0 && member == 0) ts[2] = gtimer();
    if (__syncthreads_or(!ok)) return false;  // staged values are reused by the next block
  }
  return true;
}

// Team size of a solve in arithmetic ACC: fp32 solves keep one CTA per
// block (their products are cheap; teams need two grid barriers per
// solve).  fp64 and dd solves split each block's rows over K CTAs, which
// shortens the tile product on the dependency chain K-fold (on GB300's
// narrow fp64 pipe it costs more than the hand-off): K = 8 when each team
// then owns at most two blocks, else 4 when each owns at most four, else 2.
// Measured (one GPU, fp64 solves at n = 8192, dd solves at n = 4096): K = 4
// beats K = 2 by 15-20 %; K = 8, whose teams then own 7 or 4 blocks,
// gains nothing more.
template <typename ACC>
__device__ __forceinline__ int team_size(const Cx& cx) {
  if (ACC::kW == 1) return 1;
  int k;
  if (cx.team_k > 0) {
    k = cx.team_k <= cx.G ? cx.team_k : 1;
  } else {
    const int half = (cx.nblk + 1) / 2, quarter = (cx.nblk + 3) / 4;
    k = cx.G / 8 >= half ? 8 : (cx.G / 4 >= quarter ? 4 : (cx.G >= 2 ? 2 : 1));
  }
  return cx.C > 1 ? min(k, cx.C) : k;  // a team stays inside one cluster
}

// The same solve by a grid of one block (the batched engine) of at most
// kOneBlocks row blocks: the hand-offs are block barriers and y stays in
// shared memory, all w_b are formed first, and the tiles stream through one
// ring over all row blocks.  A row's four threads take alternate 16-byte
// pieces of it, so that the reads of y fall in different banks.  Bound by
// the fp64 pipe of its SM in fp64 solves (131k multiply-adds at n = 512: 32
// of 52 us).  n = 511, forward + backward, fp64: 197 us with a wait on
// published words and a tile fetched per dependency, 104 us so.
constexpr int kOneBlocks = 8;
template <typename ACC, bool LOWER>
__device__ __noinline__ bool trsv_one(Cx& cx, const RefineArgs& a, int store_fmt) {
  using V = typename ACC::V;
  using Tm = typename ACC::Tm;
  constexpr int EPC = 16 / (int)sizeof(Tm);      // values per 16-byte piece
  constexpr int NCH = kBlk / EPC / 4;            // pieces per thread and tile
  constexpr int kTile = kBlk * kBlk * (int)sizeof(Tm);
  constexpr int kFit = (kPhaseSmem - kTrsvSmem) / kTile, D = kFit < 6 ? kFit : 6;
  static_assert(D >= 2 && 2 * kOneBlocks * kBlk * sizeof(V) <= kTrsvSmem, "shared scratch");
  static_assert(NCH * kRefThreads * 16 == kTile, "four threads per row");
  V* ys = (V*)cx.tsm;                 // c (backward: y of the forward solve), then the solved values
  V* ws = ys + kOneBlocks * kBlk;
  uint4* ring = (uint4*)cx.ssm + cx.tid;
  const Tm* Mat = ACC::mat(a);
  const double* in_hi = LOWER ? a.c_hi : a.y_hi;
  const double* in_lo = LOWER ? a.c_lo : a.y_lo;
  double* out_hi = LOWER ? a.y_hi : a.z_hi;
  double* out_lo = LOWER ? a.y_lo : a.z_lo;
  const int n = cx.n, nblk = cx.nblk, rr = cx.tid >> 2, seg = cx.tid & 3, tri = LOWER ? 0 : 1;
  // row blocks in order q = 0, 1, ..; the q-th has q tiles
  int iq = 1, it = 0, islot = 0;
  auto issue = [&]() {
    if (iq < nblk) {
      const int row = (LOWER ? iq : nblk - 1 - iq) * kBlk + rr, c0 = (LOWER ? it : nblk - 1 - it) * kBlk;
#pragma unroll
      for (int c = 0; c < NCH; ++c) {
        const int col = c0 + (c * 4 + seg) * EPC;
        const int valid = row < n ? max(0, min(EPC, n - col)) : 0;
        cp_async16(ring + (islot * NCH + c) * kRefThreads, Mat + (valid > 0 ? (size_t)row * a.ldf + col : 0),
                   valid * (int)sizeof(Tm));
      }
      if (++it == iq) {
        it = 0;
        ++iq;
      }
    }
    islot = islot + 1 == D ? 0 : islot + 1;
    cp_async_commit();
  };
#pragma unroll
  for (int q = 0; q < D - 1; ++q) issue();
  __syncthreads();  // c (y) of every row
  for (int i = cx.tid; i < nblk * kBlk; i += kRefThreads) ys[i] = i < n ? ACC::load(in_hi, in_lo, i) : ACC::zero();
  __syncthreads();
#pragma unroll 2
  for (int b = 0; b < nblk; ++b) {
    typename ACC::A wa = ACC::azero(), wb = ACC::azero();
    const size_t inv_row = (((size_t)tri * nblk + b) * kBlk + rr) * kBlk + seg;
#pragma unroll
    for (int k = 0; k < 16; k += 2) {
      wa = ACC::ifma(ACC::inv(a, inv_row + k * 4), ys[b * kBlk + k * 4 + seg], wa);
      wb = ACC::ifma(ACC::inv(a, inv_row + k * 4 + 4), ys[b * kBlk + k * 4 + 4 + seg], wb);
    }
    wa = ACC::merge(wa, wb);
    wa = ACC::merge(wa, ACC::ax(wa, 1));
    wa = ACC::merge(wa, ACC::ax(wa, 2));
    if (seg == 0) ws[b * kBlk + rr] = ACC::fin(wa);
  }
  __syncthreads();
  int slot = 0;
  for (int q = 0; q < nblk; ++q) {
    const int b = LOWER ? q : nblk - 1 - q, row = b * kBlk + rr;
    typename ACC::A acc = ACC::azero(), acc2 = ACC::azero();
    for (int t = 0; t < q; ++t) {
      issue();
      cp_async_wait<D - 1>();
      const V* y = ys + (LOWER ? t : nblk - 1 - t) * kBlk + seg * EPC;
      const uint4* src = ring + slot * NCH * kRefThreads;
      slot = slot + 1 == D ? 0 : slot + 1;
#pragma unroll
      for (int c = 0; c < NCH; ++c) {
        const uint4 u = src[c * kRefThreads];
        Tm m[EPC];
        memcpy(m, &u, 16);
#pragma unroll
        for (int e = 0; e < EPC; e += 2) {
          acc = ACC::tfma(m[e], y[c * 4 * EPC + e], acc);
          acc2 = ACC::tfma(m[e + 1], y[c * 4 * EPC + e + 1], acc2);
        }
      }
    }
    acc = ACC::merge(acc, acc2);
    acc = ACC::merge(acc, ACC::ax(acc, 1));
    acc = ACC::merge(acc, ACC::ax(acc, 2));
    V y = ACC::store(ACC::wsub(ws[row], acc), store_fmt);
    if (row >= n) y = ACC::zero();
    if (seg == 0) {
      ys[row] = y;
      if (row < n) ACC::save(out_hi, out_lo, row, y);
    }
    __syncthreads();
  }
  cp_async_wait<0>();
  return true;
}

template <typename F, typename ACC, bool LOWER>
__device__ __forceinline__ bool trsv(Cx& cx, const RefineArgs& a, int store_fmt) {
  const unsigned epoch = ++cx.epoch;
  if constexpr (ACC::kW <= 2)
    if (cx.G == 1 && cx.nblk <= kOneBlocks) return trsv_one<ACC, LOWER>(cx, a, store_fmt);
  const int K = team_size<ACC>(cx);
  if (ACC::kW > 1 && K == 8) return trsv_team<F, ACC, LOWER, 8>(cx, a, store_fmt, epoch);
  if (ACC::kW > 1 && K == 4) return trsv_team<F, ACC, LOWER, 4>(cx, a, store_fmt, epoch);
  if (ACC::kW > 1 && K == 2) return trsv_team<F, ACC, LOWER, 2>(cx, a, store_fmt, epoch);
  return trsv_team<F, ACC, LOWER, 1>(cx, a, store_fmt, epoch);
}

// ------------------------------------------------ wide triangular solves
//
// For matrices of more than kWideMin rows the chain of 64-row blocks bounds
// the substitution above: n / 64 dependent hand-offs of about 1 us each, on
// few CTAs.  The wide solve takes superblocks of SB = kSuper rows:
//   z_s = c_s - sum_{j<s} F_sj y_j,   y_s = S(T(inv(F_ss) z_s))
// (backward: j > s, y for c), every CTA of the grid working on its share of
// each superblock's rows, with two hand-offs per superblock (z, then y)
// instead of SB / 64, and on the factors in their storage format instead of
// scaled blocks in the solve's precision.  Products with superblocks that
// are known early are formed while a hand-off is under way.
//
// Rounding: the inverse of a diagonal superblock and z are kept as pairs in
// fp32 solves (sums compensated), so the only fp32-sized error of a
// component is its final rounding.  fp64 solves use fp64 values: the inverse
// is the exact one rounded (wide_products), so that a solve's error stays
// within |X||T||y| 2^-53 as on the 64-row route (figures: see kWideMin64).
//
// Measured (forward + backward, alone on the GPU): n = 2000 94 -> 42 us
// (fp32), 112 -> 49 us (fp64); n = 8192 390 -> 200 us (fp32), 740 -> 350 us
// (fp64).  What bounds it now: two hand-offs of about 1 us per superblock
// (an L2 round trip alone is 0.4 us) and, at n = 8192, the compensated sums
// of the far products.
//
template <typename ACC> struct Wide;
template <> struct Wide<AccF> {
  using AR = ArFF;
  static constexpr int kZW = 2;  // hand-off words of a z value
  static __device__ __forceinline__ const float* inv_h(const RefineArgs& a) { return a.D32h; }
  static __device__ __forceinline__ const float* inv_l(const RefineArgs& a) { return a.D32l; }
  // z = c - acc as a pair
  static __device__ __forceinline__ ArFF::V zdiff(float c, ff_t acc) {
    float s, e;
    two_sum_f(c, -acc.s, s, e);
    e = __fsub_rn(e, acc.c);
    float h, l;
    two_sum_f(s, e, h, l);
    return ArFF::V{h, l};
  }
  static __device__ __forceinline__ ArFF::V zval(float c) { return ArFF::V{c, 0.0f}; }
  static __device__ __forceinline__ unsigned zword(ArFF::V z, int k) { return __float_as_uint(k ? z.l : z.h); }
  static __device__ __forceinline__ ArFF::V unzword(const unsigned* w) {
    return ArFF::V{__uint_as_float(w[0]), __uint_as_float(w[1])};
  }
};
// plain fp64 values in the pair interface (no low words)
struct ArD {
  using S = double;
  struct V { double h; };
  using Acc = double;
};
template <> struct Wide<AccD> {
  using AR = ArD;
  static constexpr int kZW = 2;
  static __device__ __forceinline__ const double* inv_h(const RefineArgs& a) { return a.D64; }
  static __device__ __forceinline__ const double* inv_l(const RefineArgs& a) { return a.D64; }
  static __device__ __forceinline__ ArD::V zdiff(double c, double acc) { return ArD::V{__dsub_rn(c, acc)}; }
  static __device__ __forceinline__ ArD::V zval(double c) { return ArD::V{c}; }
  static __device__ __forceinline__ unsigned zword(ArD::V z, int k) { return AccD::word(z.h, k); }
  static __device__ __forceinline__ ArD::V unzword(const unsigned* w) { return ArD::V{AccD::unword(w)}; }
};

// four consecutive values from 16-byte aligned shared memory
__device__ __forceinline__ void lds4(const float* p, float (&v)[4]) {
  const float4 f = *(const float4*)p;
  v[0] = f.x; v[1] = f.y; v[2] = f.z; v[3] = f.w;
}
__device__ __forceinline__ void lds4(const double* p, double (&v)[4]) {
  const double2 f = *(const double2*)p, g = *((const double2*)p + 1);
  v[0] = f.x; v[1] = f.y; v[2] = g.x; v[3] = g.y;
}

template <typename ACC, typename F>
__device__ __forceinline__ bool use_wide(const RefineArgs& a) {
  // (fp64 factors are not exact in the fp32 words of the inverses)
  if constexpr (std::is_same<F, FAny>::value || std::is_same<F, double>::value || ACC::kW == 4) return false;
  else return (a.wide & (ACC::kW == 1 ? 1 : 2)) != 0;
}

// Products of 64x64 tiles for the doubling of the superblock inverses: acc
// (4 x 4 per thread: rows 4 (tid / 16) .., columns 4 (tid % 16) ..) +=
// A B over 64 inner terms; A staged transposed ([k][i]), B as [k][j].  fp32
// pairs; A values or pairs (kPairA).
constexpr int kWtLd = kBlk + 4;
template <bool kPairA>
__device__ __forceinline__ void wide_tile_mma(const float* Ah, const float* Al, const float* Bh, const float* Bl,
                                              int i0, int j0, ff_t (&acc)[4][4]) {
#pragma unroll 2
  for (int k = 0; k < kBlk; ++k) {
    const float4 ah = *(const float4*)(Ah + k * kWtLd + i0);
    float4 al = make_float4(0.f, 0.f, 0.f, 0.f);
    if (kPairA) al = *(const float4*)(Al + k * kWtLd + i0);
    const float4 bh = *(const float4*)(Bh + k * kWtLd + j0), bl = *(const float4*)(Bl + k * kWtLd + j0);
    const float A4[4] = {ah.x, ah.y, ah.z, ah.w}, L4[4] = {al.x, al.y, al.z, al.w};
    const float H4[4] = {bh.x, bh.y, bh.z, bh.w}, M4[4] = {bl.x, bl.y, bl.z, bl.w};
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        if (kPairA) acc[i][j] = ArFF::term(ArFF::V{A4[i], L4[i]}, ArFF::V{H4[j], M4[j]}, acc[i][j]);
        else acc[i][j] = ArFF::term(A4[i], ArFF::V{H4[j], M4[j]}, acc[i][j]);
      }
  }
}

// Row sums of magnitudes and diagonals of the triangles within their
// superblocks (a warp per row; fp32 is enough for the test below).
template <typename F>
__device__ __forceinline__ void wide_rows(Cx& cx, const RefineArgs& a) {
  const int n = cx.n, nw = cx.G * (kRefThreads / 32);
  if (cx.cta == 0 && cx.tid == 0) a.wflag[0] = a.wflag[1] = 0;
  for (int q = cx.cta * (kRefThreads / 32) + cx.warp; q < 2 * n; q += nw) {
    const bool lower = q < n;
    const int r = lower ? q : q - n, s0 = r / kSuper * kSuper;
    const int c0 = lower ? s0 : r, c1 = lower ? r : min(s0 + kSuper, n);
    float s = 0.0f;
    for (int c = c0 + cx.lane; c < c1; c += 32) s += fabsf((float)factor_at<F>(a, (size_t)r * a.ldf + c));
    s = warp_sum_f(s);
    if (cx.lane == 0) {
      a.wrow[(size_t)(lower ? 0 : 1) * a.npad + r] = lower ? s + 1.0f : s;
      a.wrow[(size_t)(lower ? 2 : 3) * a.npad + r] = lower ? 1.0f : fabsf((float)factor_at<F>(a, (size_t)r * a.ldf + r));
    }
  }
}
// Whether the superblocks' inverses are safe in fp32 pairs (kWideRange,
// kWideCond), a warp per row: sets *wflag to 1 if the range is not, 2 if the
// condition may not be.  The products of a row i
// are X_ik T_kj with k between i and j, of the size of R_k / R_j where R are
// the rows' scales; out of range they overflow or vanish although X itself
// does not.
static __device__ __noinline__ void wide_check(Cx& cx, const RefineArgs& a) {
  const int n = cx.n, nw = cx.G * (kRefThreads / 32);
  for (int q = cx.cta * (kRefThreads / 32) + cx.warp; q < 2 * n; q += nw) {
    const bool lower = q < n;
    const int r = lower ? q : q - n, s0 = r / kSuper * kSuper, tri = lower ? 0 : 1;
    const float* sum = a.wrow + (size_t)tri * a.npad;
    const float* dia = a.wrow + (size_t)(2 + tri) * a.npad;
    const float* x = a.D32h + wide_row(a, tri, r) - s0;
    const int c0 = lower ? s0 : r, c1 = lower ? r + 1 : min(s0 + kSuper, n);
    float v = 0.0f, mx = 0.0f, mn = kWideRange;
    for (int c = c0 + cx.lane; c < c1; c += 32) {
      const float s = __ldcg(sum + c);
      v += fabsf(__ldcg(x + c)) * s;
      mx = fmaxf(mx, s);
      mn = fminf(mn, __ldcg(dia + c));
    }
    v = warp_sum_f(v);
#pragma unroll
    for (int m = 16; m > 0; m >>= 1) {
      mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, m));
      mn = fminf(mn, __shfl_xor_sync(0xffffffffu, mn, m));
    }
    const bool range = mx <= kWideRange && mn >= 1.0f / kWideRange && mx <= mn * kWideRange;
    if (cx.lane == 0 && !(range && v <= kWideCond)) atomicOr(a.wflag, range ? 2 : 1);
  }
}

// Running sum of fp32 products f (h + l) in three words: the first two take
// their terms by TwoSum, the third collects what those round off (Ogita,
// Rump and Oishi's K-fold summation, K = 3: about 2^-70 of the magnitudes).
struct ff3_t {
  float s0, s1, s2;
};
__device__ __forceinline__ void ff3_term(ff3_t& a, float f, float h, float l) {
  const float p = __fmul_rn(f, h), pe = __fmaf_rn(f, h, -p);
  const float q = __fmul_rn(f, l), qe = __fmaf_rn(f, l, -q);
  float t, u1, u2, u3;
  two_sum_f(a.s0, p, a.s0, t);
  two_sum_f(a.s1, t, a.s1, u1);
  two_sum_f(a.s1, pe, a.s1, u2);
  two_sum_f(a.s1, q, a.s1, u3);
  a.s2 = __fadd_rn(a.s2, __fadd_rn(__fadd_rn(u1, u2), __fadd_rn(u3, qe)));
}

// fp64 inverses of the diagonal superblocks from the fp32 pairs X by one
// Newton step, X (2 I - T X) = X + X R with the residual R = I - T X.  The
// factor's values are exact in fp32, so T X is summed on the fp32 pipe in
// three words; R is then known to some 2^-60 of its terms, and its own
// rounding to fp32 and the plain fp32 product X R are a correction's.  What
// is left is R^2 and the final rounding: the result is the inverse to about
// one fp64 rounding.  (Doubled up in plain fp64 instead, the inverses carry
// the superblock's Skeel condition number, some 1e4 for LU factors, times
// 2^-53, and a solve with random right-hand sides was up to 2.6 times, with
// graded rows 13 times, as inaccurate as the 64-row one.)
//
// R waits in M64, whose scaled blocks belong to the 64-row route (their bit
// is cleared).  R scaled by the row sums s of |T|, R_ij s_j / s_i, has to
// stay below kWideResid, so that R^2 (512 terms) is below 2^-54; otherwise
// RDY_NO64 is set and the solves keep the 64-row route.
//
// The same two products of tiles, with magnitudes instead (kCond), are
// |X|(|T||X|), whose columns' largest elements relative to those of X are to
// be at most kWideCond (wide_columns has left the latter in wrow).
//
// The tiles of a superblock with the most inner tiles come first.
template <typename F, bool kCond>
__device__ __noinline__ bool wide_products(Cx& cx, const RefineArgs& a) {
  constexpr int NT = kSuper / kBlk, NP = NT * (NT + 1) / 2;
  float* R = (float*)a.M64;
  float* As = (float*)cx.tsm;     // [k][i]
  float* Bs = As + kBlk * kWtLd;  // [k][j]
  float* Bl = Bs + kBlk * kWtLd;
  const int n = cx.n, ldf = a.ldf, NS = a.npad / kSuper;
  const int i0 = (cx.tid >> 4) * 4, j0 = (cx.tid & 15) * 4;
  cx.mready &= ~RDY_M64;
  for (int pass = 0; pass < 2; ++pass) {
    bool bad = false;
    for (int t = cx.cta; t < 2 * NS * NP; t += cx.G) {
      const int tri = t % 2, s0 = (t / 2) % NS * kSuper;
      // the q-th pair of tiles, distance NT - 1 first
      int q = t / (2 * NS), d = NT - 1;
      for (int cnt = 1; q >= cnt; ++cnt, --d) q -= cnt;
      const bool lower = tri == 0;
      const int ti = lower ? q + d : q, tj = lower ? q : q + d;
      const int r0 = s0 + ti * kBlk, c0 = s0 + tj * kBlk;  // first row and column of the tile
      if (max(r0, c0) >= n) continue;
      ff3_t acc[4][4];
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = ff3_t{0.0f, 0.0f, 0.0f};
      for (int kt = min(ti, tj); kt <= max(ti, tj); ++kt) {
        const int k0 = s0 + kt * kBlk;
        __syncthreads();  // the previous staging is no longer read
        for (int e = cx.tid; e < kBlk * kBlk; e += kRefThreads) {
          const int r = e / kBlk, c = e % kBlk;
          const int arow = r0 + r, acol = k0 + c, brow = k0 + r;
          float av = 0.0f, bh = 0.0f, bl = 0.0f;
          if (pass == 0) {
            if (arow < n && acol < n && (lower ? acol < arow : acol >= arow))
              av = (float)factor_at<F>(a, (size_t)arow * ldf + acol);
            else if (lower && acol == arow)
              av = 1.0f;
          } else if (arow < n) {
            av = __ldcg(a.D32h + wide_row(a, tri, arow) + kt * kBlk + c);
          }
          if (brow < n) {
            const size_t x = wide_row(a, tri, brow) + tj * kBlk + c;
            bh = pass == 0 ? __ldcg(a.D32h + x) : __ldcg(R + x);
            if (pass == 0) bl = __ldcg(a.D32l + x);
          }
          As[c * kWtLd + r] = kCond ? fabsf(av) : av;
          Bs[r * kWtLd + c] = kCond ? fabsf(bh) : bh;
          if (!kCond) Bl[r * kWtLd + c] = bl;
        }
        __syncthreads();
#pragma unroll 2
        for (int k = 0; k < kBlk; ++k) {
          const float4 f = *(const float4*)(As + k * kWtLd + i0);
          const float4 bh = *(const float4*)(Bs + k * kWtLd + j0);
          const float F4[4] = {f.x, f.y, f.z, f.w}, H4[4] = {bh.x, bh.y, bh.z, bh.w};
          if (pass == 0 && !kCond) {
            const float4 bl = *(const float4*)(Bl + k * kWtLd + j0);
            const float L4[4] = {bl.x, bl.y, bl.z, bl.w};
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
              for (int j = 0; j < 4; ++j) ff3_term(acc[i][j], F4[i], H4[j], L4[j]);
          } else {
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
              for (int j = 0; j < 4; ++j) acc[i][j].s0 = __fmaf_rn(F4[i], H4[j], acc[i][j].s0);
          }
        }
      }
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int row = r0 + i0 + i;
        if (row >= n) continue;
        const size_t x = wide_row(a, tri, row) + tj * kBlk + j0;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const int col = c0 + j0 + j;
          const ff3_t v = acc[i][j];
          if (kCond) {
            if (pass == 0) R[x + j] = v.s0;
            else if (col < n) bad |= !(v.s0 <= kWideCond * __ldcg(a.wrow + (size_t)(4 + tri) * a.npad + col));
          } else if (pass == 0) {
            float h, l;
            two_sum_f(__fsub_rn(v.s0, row == col ? 1.0f : 0.0f), v.s1, h, l);
            const float r = -__fadd_rn(h, __fadd_rn(l, v.s2));
            R[x + j] = r;
            if (col < n)
              bad |= !(fabsf(r) * __ldcg(a.wrow + (size_t)tri * a.npad + col) <=
                       kWideResid * __ldcg(a.wrow + (size_t)tri * a.npad + row));
          } else {
            a.D64[x + j] = __dadd_rn((double)__ldcg(a.D32h + x + j),
                                     __dadd_rn((double)__ldcg(a.D32l + x + j), (double)v.s0));
          }
        }
      }
    }
    if (bad) atomicOr(a.wflag + (kCond ? 0 : 1), 1);
    if (!grid_barrier(cx, a)) return false;
  }
  if (kCond) cx.mready |= __ldcg(a.wflag) & 1 ? RDY_NO32 : RDY_W32;
  else cx.mready |= __ldcg(a.wflag + 1) ? RDY_NO64 : RDY_W64;
  return true;
}

// Largest element of each column of the superblocks' inverses into wrow, a
// lane per column; behind a grid barrier.
static __device__ __noinline__ void wide_columns(Cx& cx, const RefineArgs& a) {
  const int n = cx.n, nc = (n + 31) / 32, nw = cx.G * (kRefThreads / 32);
  for (int q = cx.cta * (kRefThreads / 32) + cx.warp; q < 2 * nc; q += nw) {
    const int tri = q < nc ? 0 : 1, col = (q % nc) * 32 + cx.lane, s0 = col / kSuper * kSuper;
    if (col >= n) continue;
    const int r0 = tri == 0 ? col : s0, r1 = tri == 0 ? min(s0 + kSuper, n) : col + 1;
    float m = 0.0f;
    for (int r = r0; r < r1; ++r) m = fmaxf(m, fabsf(__ldcg(a.D32h + wide_row(a, tri, r) + (col - s0))));
    a.wrow[(size_t)(4 + tri) * a.npad + col] = m;
  }
}

// Inverses of the diagonal superblocks from those of the 64x64 blocks
// (build_inverses has put them on the diagonal), by doubling h = 64, 128, ..:
//   L: X21 = -X22 (L21 X11)     U: X12 = -X11 (U12 X22)
// as fp32 pairs, in 64x64 tiles over all CTAs.  The inner product T waits in
// the opposite off-diagonal block of the same arrays, which the inverse does
// not use (its readers stay inside the triangle).
template <typename F>
__device__ __noinline__ bool build_wide(Cx& cx, const RefineArgs& a) {
  float* D0 = a.D32h;
  float* D1 = a.D32l;
  float* As = (float*)cx.tsm;         // [k][i], high words
  float* Bs = As + kBlk * kWtLd;      // [k][j]
  float* Al = Bs + kBlk * kWtLd;      // low words
  float* Bl = Al + kBlk * kWtLd;
  constexpr int sb = kSuper;
  const int n = cx.n, ldf = a.ldf;
  const int i0 = (cx.tid >> 4) * 4, j0 = (cx.tid & 15) * 4;
  wide_rows<F>(cx, a);  // (read behind the barriers of the doubling)
  for (int h = kBlk; h < sb; h *= 2) {
    const int nt = h / kBlk, npair = (a.npad / 2) / h;
    for (int pass = 0; pass < 2; ++pass) {
      for (int t = cx.cta; t < 2 * npair * nt * nt; t += cx.G) {
        const int tj = t % nt, ti = (t / nt) % nt, pr = (t / (nt * nt)) % npair, tri = t / (nt * nt * npair);
        const bool lower = tri == 0;
        const int o = pr * 2 * h;
        if (o + h >= n) continue;  // no second half
        const int oc = o % sb;     // column of the pair inside its superblock
        // pass 0: T = F[fr..][fc..] X[xr..][xr..]; pass 1: X_off = -X T
        const int xr = lower ? o : o + h;       // the X of pass 0 (11 / 22)
        const int fr = lower ? o + h : o;       // rows of F, of T's target in pass 1 and of the other X
        const int xk0 = lower ? tj : 0, xk1 = lower ? nt : tj + 1;      // pass 0: inner tiles
        const int yk0 = lower ? 0 : ti, yk1 = lower ? ti + 1 : nt;      // pass 1
        const int tr = lower ? o : o + h, tc = lower ? oc + h : oc;     // where T waits
        const int k0 = pass ? yk0 : xk0, k1 = pass ? yk1 : xk1;
        ff_t acc[4][4];
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
          for (int j = 0; j < 4; ++j) acc[i][j] = ff_t{0.0f, 0.0f};
        for (int kt = k0; kt < k1; ++kt) {
          __syncthreads();  // the previous staging is no longer read
          for (int e = cx.tid; e < kBlk * kBlk; e += kRefThreads) {
            const int r = e / kBlk, c = e % kBlk;
            if (pass == 0) {
              const int frow = fr + ti * kBlk + r, fcol = xr + kt * kBlk + c;
              As[c * kWtLd + r] = (frow < n && fcol < n) ? (float)factor_at<F>(a, (size_t)frow * ldf + fcol) : 0.0f;
              const int xrow = xr + kt * kBlk + r;
              const size_t x = wide_row(a, tri, xrow) + (xr - o) + oc + tj * kBlk + c;
              Bs[r * kWtLd + c] = xrow < n ? __ldcg(D0 + x) : 0.0f;
              Bl[r * kWtLd + c] = xrow < n ? __ldcg(D1 + x) : 0.0f;
            } else {
              const int xrow = fr + ti * kBlk + r;
              const size_t x = wide_row(a, tri, xrow) + (fr - o) + oc + kt * kBlk + c;
              As[c * kWtLd + r] = xrow < n ? __ldcg(D0 + x) : 0.0f;
              Al[c * kWtLd + r] = xrow < n ? __ldcg(D1 + x) : 0.0f;
              const int trow = kt * kBlk + r;  // inner index of T
              const size_t y = wide_row(a, tri, tr + trow) + tc + tj * kBlk + c;
              const bool in = fr + trow < n;   // rows of T past the matrix were not formed
              Bs[r * kWtLd + c] = in ? __ldcg(D0 + y) : 0.0f;
              Bl[r * kWtLd + c] = in ? __ldcg(D1 + y) : 0.0f;
            }
          }
          __syncthreads();
          if (pass == 0) wide_tile_mma<false>(As, Al, Bs, Bl, i0, j0, acc);
          else wide_tile_mma<true>(As, Al, Bs, Bl, i0, j0, acc);
        }
        // T to its waiting place (row index: inner index of the second
        // product), X_off negated
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int r = ti * kBlk + i0 + i;
          if (fr + r >= n) continue;
          const size_t x = pass == 0 ? wide_row(a, tri, tr + r) + tc : wide_row(a, tri, fr + r) + (xr - o) + oc;
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            const size_t y = x + tj * kBlk + j0 + j;
            ArFF::V v = ArFF::fin(acc[i][j]);
            if (pass) v = ArFF::neg(v);
            D0[y] = v.h;
            D1[y] = v.l;
          }
        }
      }
      if (!grid_barrier(cx, a)) return false;
    }
  }
  wide_check(cx, a);
  if (!grid_barrier(cx, a)) return false;
  const int flag = __ldcg(a.wflag);
  if (flag == 2) {
    wide_columns(cx, a);
    return wide_products<F, true>(cx, a);
  }
  cx.mready |= flag ? RDY_NO32 : RDY_W32;
  return true;
}

// Wait until every word of `nval` values (W words each, at p) carries
// `epoch`, and hand each value to put(index, words): values tid, tid +
// kRefThreads, ... of this thread, loads of kIn values in flight.  Bounded
// like every device wait.
template <int W, typename Put>
__device__ __forceinline__ bool wide_collect(const unsigned long long* p, int nval, unsigned epoch, int tid, int* err,
                                             int where, Put put) {
  constexpr int kIn = 4;
  for (int v0 = tid; v0 < nval; v0 += kIn * kRefThreads) {
    unsigned long long w[kIn][W];
    unsigned todo = 0;
#pragma unroll
    for (int q = 0; q < kIn; ++q)
      if (v0 + q * kRefThreads < nval) todo |= 1u << q;
    unsigned long long t0 = 0;
    unsigned spins = 0;
    while (true) {
#pragma unroll
      for (int q = 0; q < kIn; ++q)
        if (todo >> q & 1u) {
#pragma unroll
          for (int k = 0; k < W; ++k) w[q][k] = ld_relaxed_u64(p + (size_t)(v0 + q * kRefThreads) * W + k);
        }
#pragma unroll
      for (int q = 0; q < kIn; ++q)
        if (todo >> q & 1u) {
          bool ok = true;
#pragma unroll
          for (int k = 0; k < W; ++k) ok &= (unsigned)(w[q][k] >> 32) == epoch;
          if (ok) {
            unsigned x[W];
#pragma unroll
            for (int k = 0; k < W; ++k) x[k] = (unsigned)w[q][k];
            put(v0 + q * kRefThreads, x);
            todo &= ~(1u << q);
          }
        }
      if (!todo) break;
      if ((++spins & 255u) == 0u) {
        if (t0 == 0) t0 = gtimer();
        if (ld_volatile_i32(err) != 0) return false;
        if (gtimer() - t0 > kWaitTimeoutNs) {
          record_timeout(err, 2, where, (int)epoch, v0);
          return false;
        }
      }
    }
  }
  return true;
}


// The factor values of one thread of a wide solve, in the order of their
// use: near(1), far(2), near(2), far(3), ...  A segment is one row's steps
// over consecutive columns: near(t) those of superblock t - 1, far(t + 1)
// those of superblocks 0 .. t - 1.  issue() copies the next step into the
// ring (an empty step once nothing is left, so that every step is one copy
// group), take() reads the oldest.
template <typename F, bool LOWER, int WPR>
struct WideStream {
  static constexpr int VC = 16 / (int)sizeof(F), STEP = 32 * VC * WPR, SPB = kSuper / STEP;
  const F* LU;
  const F* src;
  uint4* ring;
  int ldf, n, NS, rpc, npass, r_lo, wp, wrow, lane, tid;
  int t, far, ps, left, col, slot, cslot, depth;
  bool row;
  __device__ __forceinline__ int super(int i) const { return LOWER ? i : NS - 1 - i; }
  // row of pass p within superblock s, or -1
  __device__ __forceinline__ int my_row(int s, int p) const {
    const int rr = r_lo + p * (8 / WPR) + wrow;
    return rr < min(min(r_lo + rpc, kSuper), n - s * kSuper) ? rr : -1;
  }
  __device__ __forceinline__ void init(const F* LU_, int ldf_, int n_, int NS_, int rpc_, int npass_, int r_lo_, int wp_,
                                       int wrow_, int lane_, int tid_, uint4* ring_, int depth_) {
    LU = LU_; ldf = ldf_; n = n_; NS = NS_; rpc = rpc_; npass = npass_; r_lo = r_lo_; wp = wp_; wrow = wrow_;
    lane = lane_; tid = tid_; ring = ring_; depth = depth_;
    t = 0; far = 1; ps = npass - 1; left = 0; col = 0; slot = 0; cslot = 0;
    row = false;
    src = LU;
  }
  __device__ __forceinline__ void next_segment() {
    if (t < NS && ++ps >= npass) {
      ps = 0;
      if (!far && t + 1 < NS) {
        far = 1;
      } else {
        far = 0;
        ++t;
      }
    }
    left = 0x7fffffff;
    row = false;
    if (t < NS) {
      const int s = super(far ? t + 1 : t);
      const int rr = my_row(s, ps);
      row = rr >= 0;
      left = (far ? t : 1) * SPB;
      col = (far && LOWER ? 0 : super(t - 1)) * kSuper + (wp * 32 + lane) * VC;
      src = LU + (size_t)(s * kSuper + max(rr, 0)) * ldf;
    }
  }
  __device__ __forceinline__ void issue() {
    if (left == 0) next_segment();
    if (row) {
      const int valid = min(VC, max(0, n - col));  // columns past the matrix are zeros
      cp_async16(ring + slot * kRefThreads + tid, src + (valid > 0 ? col : 0), valid * (int)sizeof(F));
      col += STEP;
    }
    --left;
    slot = slot + 1 == depth ? 0 : slot + 1;
    cp_async_commit();
  }
  __device__ __forceinline__ void fill() {
    for (int i = 4; i < depth; ++i) issue();
  }
  __device__ __forceinline__ uint4 take() {
    const uint4 u = ring[cslot * kRefThreads + tid];
    cslot = cslot + 1 == depth ? 0 : cslot + 1;
    return u;
  }
};

// Interleaved sums of a thread: four in fp32 (the chain of a compensated sum
// is long), one in fp64 (the narrow pipe serves the CTA's warps in turn).
template <typename ACC> constexpr int kWideAcc = ACC::kW == 1 ? 4 : 1;
template <typename ACC>
__device__ __forceinline__ typename ACC::A wide_sum(const typename ACC::A (&acc)[4]) {
  return ACC::merge(ACC::merge(acc[0], acc[1]), ACC::merge(acc[2], acc[3]));
}
template <typename ACC>
__device__ __forceinline__ typename ACC::A wide_sum(const typename ACC::A (&acc)[1]) {
  return acc[0];
}

// The next U steps of a wide solve's stream, in the solve's precision.
template <typename ACC, int U, typename F, bool LOWER, int WPR>
__device__ __forceinline__ void wide_fetch(WideStream<F, LOWER, WPR>& q,
                                           typename ACC::L (&l)[U][WideStream<F, LOWER, WPR>::VC]) {
  using Lt = typename ACC::L;
  constexpr int VC = WideStream<F, LOWER, WPR>::VC;
  static_assert(U <= 4, "the ring holds depth copies");
#pragma unroll
  for (int h = 0; h < U; ++h) q.issue();
  // depth - 4 + U copies are under way or waiting; the U oldest are due
  if (q.depth == kRingDeep) cp_async_wait<kRingDeep - 4>();
  else cp_async_wait<kRingFlat - 4>();
  uint4 raw[U];
#pragma unroll
  for (int h = 0; h < U; ++h) raw[h] = q.take();
#pragma unroll
  for (int h = 0; h < U; ++h) {
    F f[VC];
    memcpy(f, &raw[h], 16);
    if constexpr (sizeof(Lt) == 8 && sizeof(F) < 8) {
      // widened by integer instructions (see gemv_rows_n)
      bool sp = false;
#pragma unroll
      for (int e = 0; e < VC; ++e) {
        const float v = (float)to_f(f[e]);
        sp |= widen_special(v);
        l[h][e] = widen_normal(v);
      }
      if (__any_sync(0xffffffffu, sp)) {
#pragma unroll
        for (int e = 0; e < VC; ++e) l[h][e] = (Lt)to_f(f[e]);
      }
    } else {
#pragma unroll
      for (int e = 0; e < VC; ++e) l[h][e] = (Lt)to_f(f[e]);
    }
  }
}
// Their products with the y at yp, yp + STEP, .., into interleaved sums.
template <typename ACC, int U, int VC, int STEP>
__device__ __forceinline__ void wide_apply(const typename ACC::L (&l)[U][VC], const typename ACC::V* yp,
                                           typename ACC::A (&acc)[kWideAcc<ACC>]) {
  using V = typename ACC::V;
#pragma unroll
  for (int h = 0; h < U; ++h) {
    V y[VC];
    if constexpr (VC >= 4) {
#pragma unroll
      for (int e = 0; e < VC; e += 4) {
        V y4[4];
        lds4(yp + h * STEP + e, y4);
#pragma unroll
        for (int i = 0; i < 4; ++i) y[e + i] = y4[i];
      }
    } else {
      y[0] = yp[h * STEP];
      y[1] = yp[h * STEP + 1];
    }
#pragma unroll
    for (int e = 0; e < VC; ++e) acc[e % kWideAcc<ACC>] = ACC::fma(l[h][e], y[e], acc[e % kWideAcc<ACC>]);
  }
}

// Sum over the 32 WPR threads that share a row, for the CTA's 8 / WPR rows at
// once.  fp32: the total is on lane 0 of the row's first warp.  fp64: an
// addition by a whole warp holds the SM's pipe for 16 cycles, so the partial
// sums go through shared memory and warp 0 adds them for all rows (4 WPR
// lanes per row), instead of five additions on every warp; the total of row
// r is on warp 0's lane 4 WPR r.  One block barrier (none for fp32 with one
// warp per row); the buffers of successive calls alternate.
template <typename ACC, int WPR>
__device__ __forceinline__ typename ACC::A wide_total(typename ACC::A acc, typename ACC::A* part, int& pbuf, int tid,
                                                      int lane, int warp) {
  using A = typename ACC::A;
  if constexpr (ACC::kW == 1) {
#pragma unroll
    for (int m = 16; m > 0; m >>= 1) acc = ACC::merge(acc, ACC::ax(acc, m));
    if constexpr (WPR > 1) {
      pbuf ^= 8;
      if (warp % WPR > 0 && lane == 0) part[pbuf + warp] = acc;
      __syncthreads();
      if (warp % WPR == 0) {
#pragma unroll
        for (int h = 1; h < WPR; ++h) acc = ACC::merge(acc, part[pbuf + warp + h]);
      }
    }
  } else {
    pbuf ^= kRefThreads;
    part[pbuf + tid] = acc;
    __syncthreads();
    if (warp == 0) {
      constexpr int LPR = 4 * WPR, PER = 32 * WPR / LPR;  // lanes per row, partial sums per lane
      const A* p = part + pbuf + (lane / LPR) * (32 * WPR) + lane % LPR;
      A s0 = p[0], s1 = p[LPR];
#pragma unroll
      for (int h = 2; h < PER; h += 2) {
        s0 = ACC::merge(s0, p[h * LPR]);
        s1 = ACC::merge(s1, p[(h + 1) * LPR]);
      }
      acc = ACC::merge(s0, s1);
#pragma unroll
      for (int m = LPR / 2; m > 0; m >>= 1) acc = ACC::merge(acc, ACC::ax(acc, m));
    }
  }
  return acc;
}

// One wide triangular solve (LOWER: L y = c; else U x = y).  WPR warps share
// a row (columns split between them); a CTA takes rpc consecutive rows of
// every superblock.  Not inlined (see trsv_team).
//
// Per superblock t (in the order of the solve):
//   y of superblock t - 1 arrives; its products (`near`) complete z, which is
//   handed on; while it travels, the products of superblock t + 1's rows with
//   superblocks 0 .. t - 1 (`far`) are formed and the inverse's rows are
//   loaded; z arrives, y = inv z is handed on.
// The factor's values reach each thread through a ring of asynchronous
// copies in shared memory in the order of their use, a.ring - 4 steps ahead
// across superblocks (16 bytes per thread and step; a thread reads only what
// it copied, so the ring needs no barrier): the loads run at memory speed
// whatever the hand-offs do.  Every CTA keeps all of y in shared memory.
template <typename F, typename ACC, bool LOWER, int WPR>
__device__ __noinline__ bool trsv_wide(Cx& cx, const RefineArgs& a, int store_fmt, unsigned epoch) {
  using WA = Wide<ACC>;
  using AR = typename WA::AR;
  using V = typename ACC::V;
  using Z = typename AR::V;
  using A = typename ACC::A;
  using S = typename AR::S;
  using Lt = typename ACC::L;
  constexpr int W = ACC::kW, ZW = WA::kZW;
  constexpr int RG = (kRefThreads / 32) / WPR;  // rows of a CTA at a time
  constexpr int SB = kSuper;
  constexpr int VC = 16 / (int)sizeof(F);       // factor values per thread and step
  constexpr int STEP = 32 * VC * WPR;           // columns of a row per step
  constexpr int SPB = SB / STEP;                // steps per superblock
  static_assert(SPB * STEP == SB, "whole steps");
  constexpr bool kPair = sizeof(Z) > sizeof(S);
  constexpr int kAcc = kWideAcc<ACC>;
  const int n = cx.n, NS = a.npad / SB;
  const int tri = LOWER ? 0 : 1;
  const int rpc = (SB + cx.G - 1) / cx.G;       // rows of each superblock per CTA
  const int npass = (rpc + RG - 1) / RG;
  V* ys = (V*)cx.tsm;                           // y, npad values
  S* zh = (S*)(ys + a.npad);                    // z of the superblock
  S* zl = zh + SB;                              // low words (fp32)
  A* part = (A*)(zl + SB);                      // partial sums of the rows' other warps [2][8] (fp64: of every thread [2][256])
  A* facc = part + (W == 1 ? 16 : 2 * kRefThreads);  // far sums of the next superblock's rows [npass][256]
  uint4* ring = (uint4*)(cx.tsm + a.ring_off);  // [a.ring][256]
  const size_t llblk = (size_t)kBlk * kLLWords;
  unsigned long long* wy = a.ll + (size_t)tri * cx.nblk * llblk;
  unsigned long long* wz = a.ll + (size_t)(2 + tri) * cx.nblk * llblk;
  const unsigned long long* wfwd = a.ll;
  const double* in_hi = LOWER ? a.c_hi : a.y_hi;
  double* out_hi = LOWER ? a.y_hi : a.z_hi;
  const F* LU = (const F*)a.LU;
  const S* Ih = WA::inv_h(a);
  const S* Il = WA::inv_l(a);
  const int wp = cx.warp % WPR, wrow = cx.warp / WPR;
  const int r_lo = cx.cta * rpc;
  auto super = [&](int t) { return LOWER ? t : NS - 1 - t; };
  // row of pass ps within superblock s, or -1
  auto my_row = [&](int s, int ps) {
    const int rr = r_lo + ps * RG + wrow;
    return rr < min(min(r_lo + rpc, SB), n - s * SB) ? rr : -1;
  };


  WideStream<F, LOWER, WPR> q;
  q.init(LU, a.ldf, n, NS, rpc, npass, r_lo, wp, wrow, cx.lane, cx.tid, ring, a.ring);
  int pbuf = 0;
  auto row_total = [&](A acc) -> A { return wide_total<ACC, WPR>(acc, part, pbuf, cx.tid, cx.lane, cx.warp); };
  // the lane that holds a row's total, and which of the pass's rows (see wide_total)
  const bool wr_lane = W == 1 ? (wp == 0 && cx.lane == 0) : (cx.warp == 0 && cx.lane % (32 / RG) == 0);
  const int wr_row = W == 1 ? wrow : cx.lane / (32 / RG);
  auto out_row = [&](int s, int ps) {  // the row this lane hands on, or -1
    const int rr = r_lo + ps * RG + wr_row;
    return wr_lane && rr < min(min(r_lo + rpc, SB), n - s * SB) ? rr : -1;
  };

  q.fill();
  for (int t = 0; t < NS; ++t) {
    const int s = super(t);
    const int R0 = s * SB, SBn = min(SB, n - R0);
    const int where = (tri << 24) | (1 << 23) | s;
    // z past the matrix meets zeros of the inverse (filled behind a barrier:
    // until then the previous superblock's z may still be read)
    auto fill_z = [&]() {
      for (int i = SBn + cx.tid; i < SB; i += kRefThreads) {
        zh[i] = (S)0;
        if constexpr (kPair) zl[i] = (S)0;
      }
    };
    if (t == 0) {
      fill_z();
      // z = c: the input of the whole superblock is already known to all
      // (forward: c is complete; backward: the forward solve's last words)
      bool ok = true;
      if (LOWER) {
        for (int i = cx.tid; i < SBn; i += kRefThreads) {
          const Z z = WA::zval(ACC::load(in_hi, nullptr, R0 + i));
          zh[i] = z.h;
          if constexpr (kPair) zl[i] = z.l;
        }
      } else {
        ok = wide_collect<W>(wfwd + (size_t)R0 * W, SBn, epoch - 1, cx.tid, a.err, where, [&](int i, const unsigned* w) {
          const Z z = WA::zval(ACC::unword(w));
          zh[i] = z.h;
          if constexpr (kPair) zl[i] = z.l;
        });
      }
      if (__syncthreads_or(!ok)) return false;
    } else {
      const int u = super(t - 1), N0 = u * SB, Nn = min(SB, n - N0);
      constexpr int PG = SPB < 4 ? SPB : 4;
      Lt ln[PG][VC];
      wide_fetch<ACC, PG>(q, ln);  // ahead of y
      const bool ok = wide_collect<W>(wy + (size_t)N0 * W, Nn, epoch, cx.tid, a.err, where,
                                      [&](int i, const unsigned* w) { ys[N0 + i] = ACC::unword(w); });
      for (int i = N0 + Nn + cx.tid; i < N0 + SB; i += kRefThreads) ys[i] = ACC::zero();
      if (__syncthreads_or(!ok)) return false;
      fill_z();
      for (int ps = 0; ps < npass; ++ps) {
        if (ps > 0) wide_fetch<ACC, PG>(q, ln);
        const int ro = out_row(s, ps);
        const V c_in = ro >= 0 ? ACC::load(in_hi, nullptr, R0 + ro) : ACC::zero();
        A ac[kAcc];
#pragma unroll
        for (int e = 0; e < kAcc; ++e) ac[e] = ACC::azero();
        if (t > 1) ac[0] = facc[ps * kRefThreads + cx.tid];
        const V* yp = ys + u * SB + (wp * 32 + cx.lane) * VC;
        wide_apply<ACC, PG, VC, STEP>(ln, yp, ac);
#pragma unroll
        for (int g = PG; g < SPB; g += PG) {
          wide_fetch<ACC, PG>(q, ln);
          wide_apply<ACC, PG, VC, STEP>(ln, yp + g * STEP, ac);
        }
        const A acc = row_total(wide_sum<ACC>(ac));
        if (ro >= 0) {
          const Z z = WA::zdiff(c_in, acc);
#pragma unroll
          for (int k = 0; k < ZW; ++k)
            st_relaxed_u64(wz + (size_t)(R0 + ro) * ZW + k, ((unsigned long long)epoch << 32) | WA::zword(z, k));
        }
      }
    }
    // the inverse's rows (this lane's columns, 4 at a time), ahead of z
    constexpr int kGrp = SB / (32 * 4 * WPR);   // groups of 4 columns per lane
    constexpr int kU = 4 * (int)sizeof(S) / 16; // 16-byte loads per group
    uint4 ih[kGrp][kU], il[kPair ? kGrp : 1][kU];
    auto load_inv = [&](int rr) {
      const size_t ir = wide_row(a, tri, R0 + max(rr, 0));
#pragma unroll
      for (int q = 0; q < kGrp; ++q) {
        const int c = (q * WPR + wp) * 128 + cx.lane * 4;
        const bool in = rr >= 0 && (LOWER ? c <= rr : c + 4 > rr);
#pragma unroll
        for (int m = 0; m < kU; ++m) {
          ih[q][m] = in ? __ldcg((const uint4*)(Ih + ir + c) + m) : make_uint4(0, 0, 0, 0);
          if constexpr (kPair) il[q][m] = in ? __ldcg((const uint4*)(Il + ir + c) + m) : make_uint4(0, 0, 0, 0);
        }
      }
    };
    load_inv(my_row(s, 0));
    if (t > 0 && t + 1 < NS) {
      for (int ps = 0; ps < npass; ++ps) {
        const bool have = my_row(super(t + 1), ps) >= 0;
        A ac[kAcc];
#pragma unroll
        for (int e = 0; e < kAcc; ++e) ac[e] = ACC::azero();
        const V* yp = ys + (LOWER ? 0 : super(t - 1) * SB) + (wp * 32 + cx.lane) * VC;
        int k = 0;
        // (U = 2 in fp64: more widened values would not fit in registers)
        constexpr int U = W == 1 ? 4 : 2;
        for (; k + U <= t * SPB; k += U, yp += U * STEP) {
          Lt l[U][VC];
          wide_fetch<ACC, U>(q, l);
          if (have) wide_apply<ACC, U, VC, STEP>(l, yp, ac);
        }
        for (; k < t * SPB; ++k, yp += STEP) {
          Lt l[1][VC];
          wide_fetch<ACC, 1>(q, l);
          if (have) wide_apply<ACC, 1, VC, STEP>(l, yp, ac);
        }
        facc[ps * kRefThreads + cx.tid] = wide_sum<ACC>(ac);
      }
    }
    if (t > 0) {
      const bool ok = wide_collect<ZW>(wz + (size_t)R0 * ZW, SBn, epoch, cx.tid, a.err, where | (1 << 22),
                                       [&](int i, const unsigned* w) {
                                         const Z z = WA::unzword(w);
                                         zh[i] = z.h;
                                         if constexpr (kPair) zl[i] = z.l;
                                       });
      if (__syncthreads_or(!ok)) return false;
    }
    // y_s = S(T(inv(F_ss) z_s))
    for (int ps = 0; ps < npass; ++ps) {
      const int rr = my_row(s, ps);
      if (ps > 0) load_inv(rr);
      A ac[kAcc];
#pragma unroll
      for (int e = 0; e < kAcc; ++e) ac[e] = ACC::azero();
#pragma unroll
      for (int q = 0; q < kGrp; ++q) {
        const int c = (q * WPR + wp) * 128 + cx.lane * 4;
        S xh[4], xl[4], h4[4], l4[4];
        memcpy(xh, ih[q], 4 * sizeof(S));
        if constexpr (kPair) memcpy(xl, il[q], 4 * sizeof(S));
        lds4(zh + c, h4);
        if constexpr (kPair) lds4(zl + c, l4);
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          // inside the triangle only (the rest of the array holds other data)
          const bool in = (LOWER ? c + e <= rr : c + e >= rr) && c + e < SBn;
          const S x = in ? xh[e] : (S)0;
          if constexpr (kPair) ac[e % kAcc] = ArFF::term(ArFF::V{x, in ? xl[e] : (S)0}, ArFF::V{h4[e], l4[e]}, ac[e % kAcc]);
          else ac[e % kAcc] = __fma_rn(x, h4[e], ac[e % kAcc]);
        }
      }
      const A acc = row_total(wide_sum<ACC>(ac));
      const int ro = out_row(s, ps);
      if (ro >= 0) {
        const V y = ACC::store(ACC::fin(acc), store_fmt);
#pragma unroll
        for (int k = 0; k < W; ++k)
          st_relaxed_u64(wy + (size_t)(R0 + ro) * W + k, ((unsigned long long)epoch << 32) | ACC::word(y, k));
        ACC::save(out_hi, nullptr, R0 + ro, y);
      }
    }
  }
  cp_async_wait<0>();  // no copy outlives the solve
  __syncthreads();     // the scratch is free for the next phase
  return true;
}

template <typename F, typename ACC, bool LOWER>
__device__ __forceinline__ bool trsv_wide_any(Cx& cx, const RefineArgs& a, int store_fmt) {
  const unsigned epoch = ++cx.epoch;
  // two warps per row while a CTA has at most four rows of a superblock
  if (kSuper <= 4 * cx.G) return trsv_wide<F, ACC, LOWER, 2>(cx, a, store_fmt, epoch);
  return trsv_wide<F, ACC, LOWER, 1>(cx, a, store_fmt, epoch);
}

// M^{-1} applied to the right-hand side already placed in c (permuted
// order, scaled by R, rounded to the storage format): forward then backward
// substitution.  Result in z (natural order, before the S*mu scaling).
// `synced`: c is complete grid-wide (a barrier lies behind it), and the
// caller puts a barrier before it reads z; otherwise c and z belong to the
// CTAs b mod G of the 64-row blocks.
template <typename F, typename ACC>
__device__ bool msolve(Cx& cx, const RefineArgs& a, int store_fmt, bool synced) {
  // (a solve that rounds its components to a 16-bit format hands each 64-row
  // block's rounded values on to the next: in superblocks the components of
  // one superblock would not see each other's rounding, which doubles the
  // error of the result)
  if (use_wide<ACC, F>(a) && (ACC::kW == 2 || store_fmt >= MSIR_FP32)) {
    if constexpr (!std::is_same<F, FAny>::value && !std::is_same<F, double>::value && ACC::kW <= 2) {
      constexpr bool k32 = ACC::kW == 1;
      const unsigned need = k32 ? RDY_W32 : RDY_W64;
      if (!(cx.mready & (RDY_W32 | RDY_NO32))) {
        build_inverses<F>(cx, a, false, true);
        if (!grid_barrier(cx, a) || !build_wide<F>(cx, a)) return false;
      }
      if (!k32 && (cx.mready & RDY_W32) && !(cx.mready & (RDY_W64 | RDY_NO64)))
        if (!wide_products<F, false>(cx, a)) return false;
      if (cx.mready & need) {
        if (!synced && !grid_barrier(cx, a)) return false;
        {
          PhaseTimer pt(cx, 1);
          if (!trsv_wide_any<F, ACC, true>(cx, a, store_fmt)) return false;
        }
        PhaseTimer pt(cx, 2);
        if (!trsv_wide_any<F, ACC, false>(cx, a, store_fmt)) return false;
        return synced || grid_barrier(cx, a);
      }
    }
  }
  // inverses and scaled blocks of the current factors in this precision, once
  const bool f64 = factor_fmt<F>(a) == MSIR_FP64;
  const unsigned need = ACC::kW == 4 ? RDY_MDD : (ACC::kW == 2 || f64) ? RDY_M64 : RDY_M32;
  if (!(cx.mready & need)) {
    if (need == RDY_M32) {
      build_inverses<F>(cx, a, false, false);
      if (!grid_barrier(cx, a) || !build_scaled32<F>(cx, a)) return false;
    } else {
      if (!(cx.mready & RDY_INV)) {
        build_inverses<F>(cx, a, true, false);
        if (!grid_barrier(cx, a)) return false;
      }
      if (!build_scaled<F>(cx, a, need == RDY_MDD)) return false;
      cx.mready |= RDY_INV;
    }
    cx.mready |= need;
  }
  // Rows of block b are prepared (c) and consumed (z) by CTA b mod G.  A
  // team of K > 1 CTAs spreads them over other CTAs, so c must be visible
  // grid-wide before the forward solve and z after the backward solve.
  const bool team = !synced && team_size<ACC>(cx) > 1;
  if (team && !grid_barrier(cx, a)) return false;
  {
    PhaseTimer pt(cx, 1);
    if (!trsv<F, ACC, true>(cx, a, store_fmt)) return false;
  }
  PhaseTimer pt(cx, 2);
  if (!trsv<F, ACC, false>(cx, a, store_fmt)) return false;
  return !team || grid_barrier(cx, a);
}

template <typename F>
__device__ bool msolve_arith(Cx& cx, const RefineArgs& a, int arith, int store_fmt, bool synced = false) {
  if (arith == MSIR_FP32) return msolve<F, AccF>(cx, a, store_fmt, synced);
  if (arith == MSIR_FP64) return msolve<F, AccD>(cx, a, store_fmt, synced);
  return msolve<F, AccDD>(cx, a, store_fmt, synced);
}

// right-hand side element of a substitution in precision `arith`
__device__ __forceinline__ void put_c(const RefineArgs& a, int arith, int i, double h, double l) {
  if (arith == MSIR_FP32) AccF::put(a.c_hi, a.c_lo, i, h, l);
  else if (arith == MSIR_FP64) AccD::put(a.c_hi, a.c_lo, i, h, l);
  else AccDD::put(a.c_hi, a.c_lo, i, h, l);
}
// solution element (z) of a substitution in precision `arith`, as a double
__device__ __forceinline__ double get_z(const RefineArgs& a, int arith, int i) {
  if (arith == MSIR_FP32) return AccF::get(a.z_hi, a.z_lo, i);
  if (arith == MSIR_FP64) return AccD::get(a.z_hi, a.z_lo, i);
  return AccDD::get(a.z_hi, a.z_lo, i);
}

// iterate over the rows of my blocks
#define FOR_MY_ROWS(cx, i)                                                          \
  for (int _b = (cx).cta; _b < (cx).nblk; _b += (cx).G)                               \
    for (int i = _b * kBlk + (cx).tid; i < min((_b + 1) * kBlk, (cx).n); i += kRefThreads)

// Squeezed factors of B = mu R A S (Sec. 2.1.2's cited scaling): A x = c is
// solved as B y = mu R c, x = S y; mu scales the right-hand side before it
// is rounded to the solve's storage format, which keeps it (and y) inside
// the bf16 / fp16 range when A's entries are far from 1.
static __device__ __forceinline__ double rscale(const RefineArgs& a, int row) {
  return a.Rsc ? a.Rsc[row] * a.mu : 1.0;
}
static __device__ __forceinline__ double cscale(const RefineArgs& a, int col) {
  return a.Ssc ? a.Ssc[col] : 1.0;
}

// ------------------------------------------------------------ residual

// r_p[i] = b[perm[i]] - A[perm[i]] x in ur; rows are spread over every warp
// of the grid (the fp64 work needs all SMs).  Returns (via grid reduction)
// s = ||r||_inf and ||x||_inf, and, with an exact solution given (MSIR_CONV_TRUE),
// ferr = ||x - x_ref||_inf / ||x_ref||_inf.  The caller has made x complete
// (barrier).
template <typename A0>
__device__ __noinline__ bool residual(Cx& cx, const RefineArgs& a, const double* x, int ur, double& s,
                         double& xnorm, double* ferr = nullptr) {
  PhaseTimer pt(cx, 0);
  double mr = 0.0, mx = 0.0;
  if (ur == MSIR_DD) {
    gemv_rows<A0, double, MSIR_DD>(cx, a, x, [&](int i, int ar, dd_t ax) {
      const dd_t r = dd_sub(dd_t{a.b[ar], 0.0}, ax);
      a.r_hi[i] = r.hi;
      a.r_lo[i] = r.lo;
      mr = nanmax(mr, fabs(r.hi));
    });
  } else {
    gemv_rows<A0, double, MSIR_FP64>(cx, a, x, [&](int i, int ar, double ax) {
      const double r = __dsub_rn(a.b[ar], ax);
      a.r_hi[i] = r;
      a.r_lo[i] = 0.0;
      mr = nanmax(mr, fabs(r));
    });
  }
  double mf = 0.0, mref = 0.0;
  for (int i = cx.cta * kRefThreads + cx.tid; i < cx.n; i += cx.G * kRefThreads) {
    const double xi = __ldcg(x + i);
    mx = nanmax(mx, fabs(xi));
    if (a.xref) {
      const double ri = __ldg(a.xref + i);
      mf = nanmax(mf, fabs(__dsub_rn(xi, ri)));
      mref = nanmax(mref, fabs(ri));
    }
  }
  mr = cta_reduce(mr, 1, cx.tid);
  mx = cta_reduce(mx, 1, cx.tid);
  if (a.xref) {
    mf = cta_reduce(mf, 1, cx.tid);
    mref = cta_reduce(mref, 1, cx.tid);
    double v[4] = {mr, mx, mf, mref};
    const int op[4] = {1, 1, 1, 1};
    if (!grid_reduce<4>(cx, a, v, op)) return false;
    s = v[0];
    xnorm = v[1];
    if (ferr) *ferr = v[3] > 0.0 ? v[2] / v[3] : v[2];
    return true;
  }
  double v[2] = {mr, mx};
  const int op[2] = {1, 1};
  if (!grid_reduce<2>(cx, a, v, op)) return false;
  s = v[0];
  xnorm = v[1];
  if (ferr) *ferr = 0.0;
  return true;
}

// fl_u(r_p[i] / s), division in u_r
static __device__ __forceinline__ double scaled_r(const RefineArgs& a, int i, double s, int ur, int u) {
  if (ur == MSIR_DD) {
    const dd_t q = dd_div_d(dd_t{__ldcg(a.r_hi + i), __ldcg(a.r_lo + i)}, s);
    return urnd(q.hi, u);
  }
  return urnd(__ddiv_rn(__ldcg(a.r_hi + i), s), u);
}

// --------------------------------------------------------------- GMRES

struct GmresOut {
  int k;
  bool nonfinite;
};

// Working-precision arithmetic for the GMRES vectors and the Givens /
// least-squares scalars (U = float for u = fp32, double for u = fp64).
template <typename U> struct UA;
template <> struct UA<float> {
  static __device__ __forceinline__ float mul(float a, float b) { return __fmul_rn(a, b); }
  static __device__ __forceinline__ float add(float a, float b) { return __fadd_rn(a, b); }
  static __device__ __forceinline__ float sub(float a, float b) { return __fsub_rn(a, b); }
  static __device__ __forceinline__ float div(float a, float b) { return __fdiv_rn(a, b); }
  static __device__ __forceinline__ float sqrt_(float a) { return __fsqrt_rn(a); }
  static __device__ __forceinline__ float fma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
  static __device__ __forceinline__ float wsum(float v) { return warp_sum_f(v); }
  static __device__ __forceinline__ float rnd(double v) { return __double2float_rn(v); }
};
template <> struct UA<double> {
  static __device__ __forceinline__ double mul(double a, double b) { return __dmul_rn(a, b); }
  static __device__ __forceinline__ double add(double a, double b) { return __dadd_rn(a, b); }
  static __device__ __forceinline__ double sub(double a, double b) { return __dsub_rn(a, b); }
  static __device__ __forceinline__ double div(double a, double b) { return __ddiv_rn(a, b); }
  static __device__ __forceinline__ double sqrt_(double a) { return __dsqrt_rn(a); }
  static __device__ __forceinline__ double fma(double a, double b, double c) { return __fma_rn(a, b, c); }
  static __device__ __forceinline__ double wsum(double v) { return warp_sum_d(v); }
  static __device__ __forceinline__ double rnd(double v) { return v; }
};

// Operator t = A v (rows perm[i]) in the operator precision, scaled by R,
// placed in c, rows over every warp of the grid, followed by a grid barrier.
// op = FP32: compensated fp32 sums (the accurately rounded fp32 value of
// each row's sum).
template <typename A0, typename U>
__device__ __noinline__ bool apply_A(Cx& cx, const RefineArgs& a, const U* v, int op) {
  PhaseTimer pt(cx, 4);
  // (an fp32 vector comes with an fp32 matrix: u >= u0)
  if constexpr (sizeof(A0) == 4 || sizeof(U) == 8) {
    if (op == MSIR_FP32) {
      if constexpr (sizeof(U) == 4)
        gemv_rows<A0, U, MSIR_FP32>(cx, a, v, [&](int i, int ar, float t) {
          ((float*)a.c_hi)[i] = __fmul_rn(t, (float)rscale(a, ar));
        });
    } else if (op == MSIR_DD) {
      if constexpr (sizeof(U) == 8)
        gemv_rows<A0, U, MSIR_DD>(cx, a, v, [&](int i, int ar, dd_t t) {
          const double R = rscale(a, ar);
          a.c_hi[i] = t.hi * R;
          a.c_lo[i] = t.lo * R;
        });
    } else {
      gemv_rows<A0, U, MSIR_FP64>(cx, a, v, [&](int i, int ar, double t) { a.c_hi[i] = t * rscale(a, ar); });
    }
  }
  return grid_barrier(cx, a);
}

// GMRES's vector work (Gram-Schmidt, norms, basis updates) uses a flat
// partition: CTA c owns the contiguous rows [c*chunk, (c+1)*chunk) with
// chunk = ceil(n / G), so every CTA shares it (the substitutions' block
// partition leaves all but n/64 CTAs without rows).  Grid barriers separate
// the phases that hand rows between the two partitions.
__device__ __forceinline__ void flat_rows(const Cx& cx, int& r0, int& r1) {
  const int chunk = (cx.n + cx.G - 1) / cx.G;
  r0 = min(cx.n, cx.cta * chunk);
  r1 = min(cx.n, r0 + chunk);
}

// out_i = fl_u(z_i * S_i * mu), flat rows (after the substitution's rows
// are visible grid-wide)
template <typename U>
__device__ bool finish_solve(Cx& cx, const RefineArgs& a, U* out, int arith) {
  if (!grid_barrier(cx, a)) return false;
  int r0, r1;
  flat_rows(cx, r0, r1);
  for (int i = r0 + cx.tid; i < r1; i += kRefThreads) out[i] = UA<U>::rnd(get_z(a, arith, i) * cscale(a, i));
  __syncthreads();
  return true;
}

// Two-stage grid reduction of the (k+1) Gram-Schmidt partial sums; the
// result (rounded to u) lands in s_h[0..k].
template <typename U>
__device__ bool cgs_reduce(Cx& cx, const RefineArgs& a, int kp1, U* s_h) {
  PhaseTimer pt(cx, 3);
  if (!grid_barrier(cx, a)) return false;
  if (cx.G == 1) {  // one block's partial sums are the sums
    for (int j = cx.tid; j < kp1; j += kRefThreads) s_h[j] = UA<U>::rnd(a.hred[j]);
    __syncthreads();
    return true;
  }
  for (int j = cx.cta * 8 + cx.warp; j < kp1; j += cx.G * 8) {
    double acc = 0.0;
    for (int c = cx.lane; c < cx.G; c += 32) acc = __dadd_rn(acc, __ldcg(a.hred + (size_t)c * (a.kcap + 1) + j));
    acc = warp_sum_d(acc);
    if (cx.lane == 0) a.hvec[j] = (double)UA<U>::rnd(acc);
  }
  if (!grid_barrier(cx, a)) return false;
  for (int j = cx.tid; j < kp1; j += kRefThreads) s_h[j] = (U)__ldcg(a.hvec + j);
  __syncthreads();
  return true;
}

// partial sums p_j = sum over my rows of V_j[i] * w[i], j = 0..k, then
// summed over the CTAs in fp64 and rounded to u (the oracle's reading of
// "inner products in u": an accurate sum rounded once).  u = fp64: fp64
// sums.  u = fp32: compensated fp32 sums (Dot2: every product's and
// addition's rounding error kept in a second word), passed on as the fp64
// value s + c; fp64 arithmetic on fp32 data spends most of its time
// widening operands on GB300's narrow fp64 pipe.
//
// The phase is bound by load latency, not bandwidth: each thread takes
// kVec consecutive basis vectors (one 16-byte load per row; the basis is
// row-major with ldv a multiple of 32) and loads kChunk rows ahead of the
// sums.  While there are few basis vectors, groups of gw threads (a power of
// two) take every 256 / gw-th row each, and their sums are added by
// shuffles and through shared memory.
template <typename U>
__device__ __noinline__ void cgs_partials(Cx& cx, const RefineArgs& a, const U* V, const U* w, int kp1) {
  PhaseTimer pt(cx, 3);
  constexpr int kVec = 16 / (int)sizeof(U);
  constexpr int kChunk = 12;
  constexpr bool kF = sizeof(U) == 4;
  using Vec = typename std::conditional<kF, float4, double2>::type;
  using Acc = typename std::conditional<kF, ff_t, double>::type;
  int r0, r1;
  flat_rows(cx, r0, r1);
  const int nq = (kp1 + kVec - 1) / kVec;
  int gw = 4;
  while (gw < nq && gw < kRefThreads) gw *= 2;
  const int ngrp = kRefThreads / gw;
  Acc* part = (Acc*)cx.tsm;  // [warp][column of the warp's groups]
  for (int jq = cx.tid & (gw - 1); jq < (nq + gw - 1) / gw * gw; jq += gw) {
    const int j0 = min(jq, nq - 1) * kVec;
    // columns j0 .. j0 + kVec - 1 (those past k are summed and not stored)
    Acc acc[kVec];
#pragma unroll
    for (int e = 0; e < kVec; ++e) {
      if constexpr (kF) acc[e] = ff_t{0.0f, 0.0f};
      else acc[e] = 0.0;
    }
    for (int i0 = r0 + cx.tid / gw; i0 < r1; i0 += kChunk * ngrp) {
      U vv[kChunk][kVec], wv[kChunk];
#pragma unroll
      for (int c = 0; c < kChunk; ++c) {
        const int i = min(i0 + c * ngrp, r1 - 1);
        const Vec t = __ldcg((const Vec*)(V + (size_t)i * a.ldv + j0));
        const U* tp = (const U*)&t;
#pragma unroll
        for (int e = 0; e < kVec; ++e) vv[c][e] = tp[e];
        wv[c] = __ldcg(w + i);
      }
#pragma unroll
      for (int c = 0; c < kChunk; ++c) {
        if (i0 + c * ngrp < r1) {
#pragma unroll
          for (int e = 0; e < kVec; ++e) {
            if constexpr (kF) acc[e] = ff_fma(vv[c][e], wv[c], acc[e]);
            else acc[e] = __fma_rn(vv[c][e], wv[c], acc[e]);
          }
        }
      }
    }
    auto add = [](Acc x, Acc y) {
      if constexpr (kF) return ff_merge(x, y);
      else return __dadd_rn(x, y);
    };
    for (int m = gw; m < 32; m *= 2) {
#pragma unroll
      for (int e = 0; e < kVec; ++e) {
        if constexpr (kF) acc[e] = ff_merge(acc[e], ff_shfl_xor(acc[e], m));
        else acc[e] = __dadd_rn(acc[e], __shfl_xor_sync(0xffffffffu, acc[e], m));
      }
    }
    if (ngrp > 1) {
#pragma unroll
      for (int e = 0; e < kVec; ++e) part[cx.tid * kVec + e] = acc[e];
      __syncthreads();
      // the threads of the first group (of each warp: of its first one) hold
      // the sums' columns; with gw < 32 a warp holds all of them
      const int hop = gw < 32 ? 32 : gw;
      if (cx.tid < gw) {
#pragma unroll
        for (int e = 0; e < kVec; ++e) {
          Acc s[kRefThreads / 32];
#pragma unroll
          for (int g = 0; g < kRefThreads / 32; ++g) {
            if constexpr (kF) s[g] = ff_t{0.0f, 0.0f};
            else s[g] = 0.0;
            if (g * hop < kRefThreads) s[g] = part[(cx.tid + g * hop) * kVec + e];
          }
          acc[e] = add(add(add(s[0], s[1]), add(s[2], s[3])), add(add(s[4], s[5]), add(s[6], s[7])));
        }
      }
    }
    if (cx.tid < gw && jq < nq) {
#pragma unroll
      for (int e = 0; e < kVec; ++e) {
        if (j0 + e >= kp1) break;
        double v;
        if constexpr (kF) v = __dadd_rn((double)acc[e].s, (double)acc[e].c);
        else v = acc[e];
        a.hred[(size_t)cx.cta * (a.kcap + 1) + j0 + e] = v;
      }
    }
  }
}

// sum_j V_j[i] c_j for the CTA's flat rows, handed to epi(i, pre(i), sum):
// gw lanes (a power of two, 32 from 128 columns on; fp64: 64) share a row,
// each summing groups of kVec consecutive columns by 16-byte loads, then a
// butterfly over them; a warp has kRows rows per group of lanes in flight,
// and what epi reads beside the sum (pre) is loaded with them.  The sum is a
// compensated pair (u = fp32: Dot2 in fp32, the pair's sum is the value;
// u = fp64: an fp64 sum in .s, .c = 0).
struct RowSum {
  double s, c;
};
template <typename U, int kRows, typename Pre, typename Epi>
__device__ __forceinline__ void basis_rows_n(const Cx& cx, const RefineArgs& a, const U* V, int kp1, const U* c,
                                             int gw, int r0, int r1, Pre pre, Epi epi) {
  constexpr int kVec = 16 / (int)sizeof(U);
  constexpr bool kF = sizeof(U) == 4;
  using Vec = typename std::conditional<kF, float4, double2>::type;
  const int l = cx.lane & (gw - 1), sub = cx.lane / gw, spw = 32 / gw;
  for (int i0 = r0 + cx.warp * kRows * spw; i0 < r1; i0 += (kRefThreads / 32) * kRows * spw) {
    ff_t af[kRows];
    double ad[kRows];
    U pv[kRows];
    size_t row[kRows];
#pragma unroll
    for (int q = 0; q < kRows; ++q) {
      const int i = min(i0 + q * spw + sub, r1 - 1);
      row[q] = (size_t)i * a.ldv;
      pv[q] = pre(i);
      af[q] = ff_t{0.0f, 0.0f};
      ad[q] = 0.0;
    }
    auto step = [&](int j0, bool full) {
      U vv[kRows][kVec], cj[kVec];
#pragma unroll
      for (int e = 0; e < kVec; ++e) cj[e] = full || j0 + e < kp1 ? c[j0 + e] : (U)0;
#pragma unroll
      for (int q = 0; q < kRows; ++q) {
        const Vec t = __ldcg((const Vec*)(V + row[q] + j0));
        const U* tp = (const U*)&t;
#pragma unroll
        for (int e = 0; e < kVec; ++e) vv[q][e] = full || j0 + e < kp1 ? tp[e] : (U)0;  // past k: anything
      }
#pragma unroll
      for (int q = 0; q < kRows; ++q)
#pragma unroll
        for (int e = 0; e < kVec; ++e) {
          if constexpr (kF) af[q] = ff_fma(vv[q][e], cj[e], af[q]);
          else ad[q] = __fma_rn(vv[q][e], cj[e], ad[q]);
        }
    };
    int j0 = l * kVec;
#pragma unroll 2
    for (; j0 + kVec <= kp1; j0 += gw * kVec) step(j0, true);
    if (j0 < kp1) step(j0, false);
    __syncwarp();
    for (int m = gw / 2; m > 0; m >>= 1) {
#pragma unroll
      for (int q = 0; q < kRows; ++q) {
        if constexpr (kF) af[q] = ff_merge(af[q], ff_shfl_xor(af[q], m));
        else ad[q] = __dadd_rn(ad[q], __shfl_xor_sync(0xffffffffu, ad[q], m));
      }
    }
#pragma unroll
    for (int q = 0; q < kRows; ++q) {
      const int i = i0 + q * spw + sub;
      if (l == (q & (gw - 1)) && i < r1)
        epi(i, pv[q], kF ? RowSum{(double)af[q].s, (double)af[q].c} : RowSum{ad[q], 0.0});
    }
  }
}
template <typename U, typename Pre, typename Epi>
__device__ __forceinline__ void basis_rows(const Cx& cx, const RefineArgs& a, const U* V, int kp1, const U* c, Pre pre,
                                           Epi epi) {
  constexpr int kVec = 16 / (int)sizeof(U);
  int r0, r1;
  flat_rows(cx, r0, r1);
  int gw = 4;
  while (gw < 32 && gw * kVec < kp1) gw *= 2;
  const int spw = 32 / gw;
  // rows per group of lanes that let all warps work
  const int per = (r1 - r0 + kRefThreads / 32 * spw - 1) / (kRefThreads / 32 * spw);
  if (per <= 2) basis_rows_n<U, 2>(cx, a, V, kp1, c, gw, r0, r1, pre, epi);
  else if (per <= 4) basis_rows_n<U, 4>(cx, a, V, kp1, c, gw, r0, r1, pre, epi);
  else basis_rows_n<U, 8>(cx, a, V, kp1, c, gw, r0, r1, pre, epi);
}

// w_i = fl_u(w_i - sum_j V_j[i] h_j) with the difference taken from the
// accurate sum (fp32: w - (s + c) by ff_sub_from); flat rows
template <typename U>
__device__ __noinline__ void cgs_update(Cx& cx, const RefineArgs& a, const U* V, U* w, int kp1, const U* s_h) {
  PhaseTimer pt(cx, 3);
  basis_rows<U>(cx, a, V, kp1, s_h, [&](int i) { return w[i]; }, [&](int i, U wi, RowSum acc) {
    if constexpr (sizeof(U) == 4)
      w[i] = ff_sub_from(wi, ff_t{(float)acc.s, (float)acc.c});
    else
      w[i] = UA<U>::rnd(__dsub_rn((double)wi, acc.s));
  });
  __syncthreads();
}

// d_i = fl_u(sum_j V_j[i] y_j) over the flat rows (the GMRES correction)
template <typename U>
__device__ __noinline__ void basis_combine(Cx& cx, const RefineArgs& a, const U* V, int kdone, const U* y) {
  basis_rows<U>(cx, a, V, kdone, y, [](int) { return (U)0; }, [&](int i, U, RowSum acc) {
    a.d[i] = sizeof(U) == 4 ? (double)ff_fin(ff_t{(float)acc.s, (float)acc.c}) : (double)UA<U>::rnd(acc.s);
  });
}

template <typename U>
__device__ bool grid_sum_sq(Cx& cx, const RefineArgs& a, const U* w, double& out) {
  double ss = 0.0;
  int r0, r1;
  flat_rows(cx, r0, r1);
  for (int i = r0 + cx.tid; i < r1; i += kRefThreads) {
    const double wv = (double)w[i];
    ss = __fma_rn(wv, wv, ss);
  }
  double v[1] = {cta_reduce(ss, 0, cx.tid)};
  const int opr[1] = {0};
  if (!grid_reduce<1>(cx, a, v, opr)) return false;
  out = v[0];
  return true;
}

// y of the rotated (triangular) Hessenberg system by one warp, into ys and
// a.yv: row i from the last up, y_i = (g_i - sum_j H_ij y_j) / H_ii with every
// product and difference rounded, j ascending.  The subtractions of a row
// are a chain; the products of 32 columns are formed by the lanes beside it,
// and the next 32 entries of H (row-major) are loaded ahead, across rows
// too.  (One thread that loads each entry when the chain reaches it took 50
// ms for 820 columns, a fifth of a GMRES cycle at n = 8192.)
template <typename U>
__device__ __noinline__ void hessenberg_solve(const RefineArgs& a, int kcap, int kdone, const U* g, U* ys, int lane) {
  using M = UA<U>;
  const int ld = kcap + 1;
  auto entry = [&](int i, int j) { return i >= 0 && j < kdone ? (U)__ldcg(a.H + (size_t)i * ld + j) : (U)0; };
  // the chunks of row i start at its diagonal: columns i + lane, i + 32 + lane, ..
  int i = kdone - 1, j0 = i;
  U h = entry(i, j0 + lane);
  U acc = (U)0, diag = (U)0;
  while (i >= 0) {
    const bool last = j0 + 32 >= kdone;
    const int ni = last ? i - 1 : i, nj = last ? i - 1 : j0 + 32;
    const U hn = entry(ni, nj + lane);
    int l0 = 0;
    if (j0 == i) {
      acc = g[i];
      diag = __shfl_sync(0xffffffffu, h, 0);
      l0 = 1;
    }
    const int cnt = min(32, kdone - j0);
    const U p = lane >= l0 && lane < cnt ? M::mul(h, ys[j0 + lane]) : (U)0;
    for (int l = l0; l < cnt; ++l) acc = M::sub(acc, __shfl_sync(0xffffffffu, p, l));
    if (last) {
      const U y = M::div(acc, diag);
      if (lane == 0) {
        ys[i] = y;
        a.yv[i] = (double)y;
      }
      __syncwarp();
    }
    h = hn;
    i = ni;
    j0 = nj;
  }
}

template <typename A0, typename F, typename U>
__device__ bool gmres(Cx& cx, const RefineArgs& a, double s, int ur, int u, int op, double tau,
                      unsigned char* gsm, GmresOut& out) {
  using M = UA<U>;
  __shared__ double s_bc[1];
  const int kcap = a.kcap;
  U* sm_cs = (U*)gsm;
  U* sm_sn = sm_cs + kcap + 1;
  U* sm_g = sm_sn + kcap + 1;   // kcap + 2
  U* s_h = sm_g + kcap + 2;     // 2 (kcap + 1)
  U* V = (U*)a.V;
  U* vk = (U*)a.vk;
  U* w = (U*)a.w;
  out.k = 0;
  out.nonfinite = false;
  // w0 = fl_u(M^{-1} r~) with the substitutions in op
  for (int b = cx.cta; b < cx.nblk; b += cx.G)
    for (int i = b * kBlk + cx.tid; i < min((b + 1) * kBlk, cx.n); i += kRefThreads)
      put_c(a, op, i, scaled_r(a, i, s, ur, u) * rscale(a, a.perm[i]), 0.0);
  __syncthreads();
  if (!msolve_arith<F>(cx, a, op, op)) return false;
  if (!finish_solve<U>(cx, a, w, op)) return false;
  double ss;
  if (!grid_sum_sq<U>(cx, a, w, ss)) return false;
  const U beta = M::sqrt_(M::rnd(ss));
  if (!isfinite((double)beta)) { out.nonfinite = true; return true; }
  int f0, f1;
  flat_rows(cx, f0, f1);
  if (beta == (U)0) {
    for (int i = f0 + cx.tid; i < f1; i += kRefThreads) a.d[i] = 0.0;
    return grid_barrier(cx, a);  // d is read by the block partition
  }
  for (int i = f0 + cx.tid; i < f1; i += kRefThreads) {
    const U v = M::div(w[i], beta);
    V[(size_t)i * a.ldv] = v;
    vk[i] = v;
  }
  if (cx.tid == 0) sm_g[0] = beta;
  __syncthreads();
  int kdone = 0;
  for (int k = 0; k < kcap; ++k) {
    // full V_k needed by the matrix-vector product
    if (!grid_barrier(cx, a)) return false;
    if (!apply_A<A0, U>(cx, a, vk, op)) return false;
    if (!msolve_arith<F>(cx, a, op, op, true)) return false;
    if (!finish_solve<U>(cx, a, w, op)) return false;
    // classical Gram-Schmidt, twice
    cgs_partials<U>(cx, a, V, w, k + 1);
    if (!cgs_reduce<U>(cx, a, k + 1, s_h)) return false;
    cgs_update<U>(cx, a, V, w, k + 1, s_h);
    for (int j = cx.tid; j <= k; j += kRefThreads) s_h[kcap + 1 + j] = s_h[j];
    __syncthreads();
    cgs_partials<U>(cx, a, V, w, k + 1);
    if (!cgs_reduce<U>(cx, a, k + 1, s_h)) return false;
    cgs_update<U>(cx, a, V, w, k + 1, s_h);
    for (int j = cx.tid; j <= k; j += kRefThreads) s_h[j] = M::add(s_h[kcap + 1 + j], s_h[j]);
    __syncthreads();
    double ww;
    if (!grid_sum_sq<U>(cx, a, w, ww)) return false;
    const U hk1 = M::sqrt_(M::rnd(ww));
    // Givens rotations (every CTA computes the same numbers)
    unsigned long long tg0 = (cx.cta == 0 && cx.tid == 0) ? gtimer() : 0;
    // The rotations are a chain from entry to entry, carry = -sn carry +
    // cs x, linear in the carry, so one warp scans it: each lane composes
    // the rotations of its piece (odd length: no bank conflicts) into
    // carry -> A carry + B, five shuffles give every piece its carry, and
    // the lanes apply their rotations.  |A| <= 1 and B is at most the norm of
    // the piece, so the rounding errors stay below those of the chain, whose
    // dependent fp64 pair took 180 ns a rotation (n = 2000 in single with
    // 435 iterations: 5.9 of 54 ms in the chain).
    if (cx.warp == 0) {
      const int len = ((k + 31) / 32) | 1;
      const int i0 = min(cx.lane * len, k), i1 = min(i0 + len, k);
      U sa = (U)1, sb = (U)0;
      for (int i = i0; i < i1; ++i) {
        const U sn = sm_sn[i];
        sb = fma(-sn, sb, M::mul(sm_cs[i], s_h[i + 1]));
        sa = M::mul(-sn, sa);
      }
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const U pa = __shfl_up_sync(0xffffffffu, sa, o), pb = __shfl_up_sync(0xffffffffu, sb, o);
        if (cx.lane >= o) {
          sb = fma(sa, pb, sb);
          sa = M::mul(sa, pa);
        }
      }
      const U h0 = s_h[0];
      const U end = fma(sa, h0, sb);
      U carry = __shfl_up_sync(0xffffffffu, end, 1);
      if (cx.lane == 0) carry = h0;
      const U last = s_h[i1];  // the next lane's first result takes its place
      __syncwarp();
      for (int i = i0; i < i1; ++i) {
        const U x0 = carry, cs = sm_cs[i], sn = sm_sn[i];
        const U x1 = i + 1 < i1 ? s_h[i + 1] : last;
        carry = fma(-sn, x0, M::mul(cs, x1));
        s_h[i] = fma(cs, x0, M::mul(sn, x1));
      }
      __syncwarp();
      if (cx.lane == 31) s_h[k] = carry;
    }
    __syncthreads();
    if (cx.tid == 0) {
      const U f = s_h[k], g = hk1;
      U c, sn, r;
      if (g == (U)0) {
        c = (U)1; sn = (U)0; r = f;
      } else {
        r = M::sqrt_(M::add(M::mul(f, f), M::mul(g, g)));
        c = M::div(f, r);
        sn = M::div(g, r);
      }
      sm_cs[k] = c;
      sm_sn[k] = sn;
      s_h[k] = r;
      const U gk = sm_g[k];
      sm_g[k] = M::mul(c, gk);
      sm_g[k + 1] = M::mul(-sn, gk);
      s_bc[0] = fabs((double)sm_g[k + 1]) / (double)beta;
    }
    __syncthreads();
    if (cx.cta == 0)
      for (int i = cx.tid; i <= k; i += kRefThreads) a.H[(size_t)i * (kcap + 1) + k] = (double)s_h[i];
    if (cx.cta == 0 && cx.tid == 0) cx.t_ns[6] += gtimer() - tg0;
    const double relres = s_bc[0];
    kdone = k + 1;
    if (hk1 != (U)0 && isfinite((double)hk1)) {
      for (int i = f0 + cx.tid; i < f1; i += kRefThreads) {
        const U v = M::div(w[i], hk1);
        V[(size_t)i * a.ldv + k + 1] = v;
        vk[i] = v;
      }
    }
    __syncthreads();
    if (!isfinite(relres) || relres <= tau || hk1 == (U)0) break;
  }
  // y from the rotated Hessenberg matrix (warp 0 of CTA 0), then d = fl_u(V y)
  __syncthreads();  // CTA 0's rows of H are written
  if (cx.cta == 0 && cx.warp == 0) hessenberg_solve<U>(a, kcap, kdone, sm_g, s_h, cx.lane);
  if (!grid_barrier(cx, a)) return false;
  for (int j = cx.tid; j < kdone; j += kRefThreads) s_h[j] = (U)__ldcg(a.yv + j);
  __syncthreads();
  basis_combine<U>(cx, a, V, kdone, s_h);
  out.k = kdone;
  return grid_barrier(cx, a);  // d is read by the block partition
}

// -------------------------------------------------------------- kernel

// (cta: the block's index in the solve's grid; block 0 writes the report)
static __device__ void rep_new_stage(const RefineArgs& a, RefState& S, int cta) {
  if (cta == 0 && threadIdx.x == 0 && S.nstages < MSIR_MAX_STAGES) {
    msir_stage& g = a.rep->stage[S.nstages];
    g.uf = S.uf;
    g.u = S.u;
    g.ur = S.ur;
    g.alg = S.alg;
    g.steps = 0;
    g.nonfinite = 0;
  }
  S.nstages++;
}

// Algorithm 4's stopping logic after one completed step (mirrors Sec. 2.1.1
// with the readings listed in the library documentation).  Thread 0 only.
// Returns 0 continue, 1 converged, 2 switch (reset = phi > phi_0).
static __device__ int ctl_step(RefState& S, const RefineArgs& a, double s, double dnorm, double xnorm,
                               double nbe, double ferr, int kg, int* reset) {
  const double delta = s * dnorm;
  const double z = xnorm > 0.0 ? delta / xnorm : __longlong_as_double(0x7ff0000000000000ll);
  const double v = isfinite(S.delta_prev) ? delta / S.delta_prev : 0.0;
  S.rho_max = fmax(S.rho_max, v);
  const double phi =
      S.rho_max < 1.0 ? z / (1.0 - S.rho_max) : __longlong_as_double(0x7ff0000000000000ll);
  S.phi = phi;
  if (!S.have_phi0) { S.phi0 = phi; S.have_phi0 = 1; }
  S.delta_prev = delta;
  const double gamma = a.gamma > 0.0 ? a.gamma : sqrt((double)a.n);
  const double uu0 = unit_roundoff(a.u0);
  const double thr = gamma * uu0;
  bool conv = phi >= 0.0 && phi <= thr;
  if (a.conv == MSIR_CONV_COMBINED) conv = conv && nbe <= 2.0 * uu0;
  if (a.conv == MSIR_CONV_TRUE) conv = ferr <= uu0 && nbe <= uu0;
  *reset = 0;
  if (conv) return 1;
  const bool trig = z <= unit_roundoff(S.u) || v >= a.rho_thresh || S.it >= a.i_max ||
                    (S.alg != MSIR_ALG_SIR && kg >= 0 && (double)kg >= a.kmax);
  if (trig) {
    *reset = phi > S.phi0 ? 1 : 0;
    return 2;
  }
  return 0;
}

// Algorithm 4 after the factorisation (the MSIR mode of the refinement
// kernel): x0, then SIR / SGMRES-IR / GMRES-IR steps with the stopping
// logic, until convergence, a stage that needs a finer u_f (S.phase =
// PH_NEED_ESC) or the end.  Run by every CTA of a cooperative launch, or by
// one CTA alone (cx.G = 1) in the batched engine.  S, s_act, s_reset and
// s_alg live in shared memory.  Returns false if a device wait failed.
template <typename A0, typename F>
__device__ __forceinline__ bool refine_msir(Cx& cx, const RefineArgs& a, RefState& S, unsigned char* gsm, int& s_act,
                            int& s_reset, int& s_alg) {
  bool ok = true;
  const int ff = factor_fmt<F>(a);
  const int arith_f = ff == MSIR_FP64 ? MSIR_FP64 : MSIR_FP32;
  double s = S.s, xnorm = 0.0, nbe = S.nbe;
  if (S.phase == PH_START) {
    if (a.normb == 0.0) {
      FOR_MY_ROWS(cx, i) { a.x[i] = 0.0; a.xbest[i] = 0.0; }
      if (cx.tid == 0) { S.cged = 1; S.status = MSIR_OK; S.phase = PH_DONE; S.nbe = 0.0; S.s = 0.0; }
      __syncthreads();
      return true;  // b = 0: x = 0, converged
    }
    // x0 = fl_u(fl_u(||b||) M_f^{-1} fl_u(b / ||b||)) with the u_f model
    for (int b = cx.cta; b < cx.nblk; b += cx.G)
      for (int i = b * kBlk + cx.tid; i < min((b + 1) * kBlk, cx.n); i += kRefThreads) {
        const int pr = a.perm[i];
        const double bt = urnd(__ddiv_rn(a.b[pr], a.normb), S.u);
        put_c(a, arith_f, i, round_to(bt * rscale(a, pr), S.uf), 0.0);
      }
    __syncthreads();
    ok = msolve_arith<F>(cx, a, arith_f, S.uf);
    if (!ok) return false;
    {
      const double nb_u = urnd(a.normb, S.u);
      double mx = 0.0;
      FOR_MY_ROWS(cx, i) {
        const double d0 = urnd(get_z(a, arith_f, i) * cscale(a, i), S.u);
        const double x0 = urnd(nb_u * d0, S.u);
        a.x0[i] = x0;
        mx = nanmax(mx, fabs(x0));
      }
      mx = cta_reduce(mx, 1, cx.tid);
      double v[1] = {mx};
      const int op[1] = {1};
      if (!(ok = grid_reduce<1>(cx, a, v, op))) return false;
      const bool bad = !isfinite(v[0]);
      FOR_MY_ROWS(cx, i) {
        if (bad) a.x0[i] = 0.0;
        a.x[i] = a.x0[i];
        a.xbest[i] = a.x0[i];
      }
    }
    if (!(ok = grid_barrier(cx, a))) return false;
    if (!(ok = residual<A0>(cx, a, a.x, S.ur, s, xnorm))) return false;
    nbe = s / (a.normA * xnorm + a.normb);
    if (cx.tid == 0) {
      S.best_nbe = nbe;
      S.alg = MSIR_ALG_SIR;
      S.it = 0;
      S.rho_max = 0.0;
      S.delta_prev = __longlong_as_double(0x7ff0000000000000ll);
      S.phase = PH_ESCALATED + 10;  // running
      rep_new_stage(a, S, cx.cta);
    }
    __syncthreads();
  } else if (S.phase == PH_ESCALATED) {
    if (!(ok = grid_barrier(cx, a))) return false;
    if (!(ok = residual<A0>(cx, a, a.x, S.ur, s, xnorm))) return false;
    nbe = s / (a.normA * xnorm + a.normb);
    if (cx.tid == 0) {
      if (nbe < S.best_nbe) S.best_nbe = nbe;
      S.alg = MSIR_ALG_SIR;
      S.it = 0;
      S.rho_max = 0.0;
      S.delta_prev = __longlong_as_double(0x7ff0000000000000ll);
      S.phase = PH_ESCALATED + 10;
      rep_new_stage(a, S, cx.cta);
    }
    __syncthreads();
    if (nbe <= S.best_nbe) FOR_MY_ROWS(cx, i) a.xbest[i] = a.x[i];
  }

  while (true) {
    if (s == 0.0) {
      if (cx.tid == 0) { S.cged = 1; S.status = MSIR_OK; }
      break;
    }
    if (!isfinite(s)) break;
    const int u = S.u, ur = S.ur;
    int kg = -1;
    bool nonfinite = false;
    if (S.alg == MSIR_ALG_SIR) {
      for (int b = cx.cta; b < cx.nblk; b += cx.G)
        for (int i = b * kBlk + cx.tid; i < min((b + 1) * kBlk, cx.n); i += kRefThreads) {
          const double rt = scaled_r(a, i, s, ur, u);
          put_c(a, arith_f, i, round_to(rt * rscale(a, a.perm[i]), S.uf), 0.0);
        }
      __syncthreads();
      if (!(ok = msolve_arith<F>(cx, a, arith_f, S.uf))) break;
      FOR_MY_ROWS(cx, i) a.d[i] = urnd(get_z(a, arith_f, i) * cscale(a, i), u);
      __syncthreads();
    } else {
      const int op = S.alg == MSIR_ALG_SGMRES ? u : square_of(u);
      const double tau = a.tau > 0.0 ? a.tau : (u == MSIR_FP32 ? 1e-6 : 1e-10);
      GmresOut go;
      if (u == MSIR_FP32) {
        if (!(ok = gmres<A0, F, float>(cx, a, s, ur, u, op, tau, gsm, go))) break;
      } else {
        if (!(ok = gmres<A0, F, double>(cx, a, s, ur, u, op, tau, gsm, go))) break;
      }
      kg = go.k;
      nonfinite = go.nonfinite;
    }
    // tentative update x_{i+1} = fl_u(x_i + fl_u(fl_u(s) d)) and the norms
    double md = 0.0, mx = 0.0;
    const double su = urnd(s, u);
    FOR_MY_ROWS(cx, i) {
      const double dv = nonfinite ? 0.0 : a.d[i];
      const double xv = a.x[i];
      a.xn[i] = urnd(xv + urnd(su * dv, u), u);
      md = nanmax(md, fabs(dv));
      mx = nanmax(mx, fabs(xv));
    }
    md = cta_reduce(md, 1, cx.tid);
    mx = cta_reduce(mx, 1, cx.tid);
    {
      double v[2] = {md, mx};
      const int op[2] = {1, 1};
      if (!(ok = grid_reduce<2>(cx, a, v, op))) break;
      md = v[0];
      mx = v[1];
    }
    if (nonfinite || !isfinite(md)) {
      // Inf/NaN correction: no update, the step is not counted, next stage
      if (cx.tid == 0) {
        if (cx.cta == 0 && S.nstages >= 1 && S.nstages <= MSIR_MAX_STAGES)
          a.rep->stage[S.nstages - 1].nonfinite = 1;
        if (S.alg == MSIR_ALG_GMRES) {
          S.phase = PH_NEED_ESC;
        } else {
          S.alg += 1;
          S.it = 0;
          S.rho_max = 0.0;
          S.delta_prev = __longlong_as_double(0x7ff0000000000000ll);
          rep_new_stage(a, S, cx.cta);
        }
      }
      __syncthreads();
      if (S.phase == PH_NEED_ESC) break;
      continue;
    }
    const double s_old = s, xnorm_old = mx;
    FOR_MY_ROWS(cx, i) a.x[i] = a.xn[i];
    if (!(ok = grid_barrier(cx, a))) break;
    double ferr = 0.0;
    if (!(ok = residual<A0>(cx, a, a.x, ur, s, xnorm, &ferr))) break;
    nbe = s / (a.normA * xnorm + a.normb);
    const bool better = nbe < S.best_nbe;
    // every thread has read S before thread 0 updates it (shared memory)
    __syncthreads();
    if (better) FOR_MY_ROWS(cx, i) a.xbest[i] = a.x[i];
    if (cx.tid == 0) {
      if (better) S.best_nbe = nbe;
      S.it += 1;
      S.total_steps += 1;
      if (kg >= 0) S.total_gmres += kg;
      if (cx.cta == 0 && S.nstages >= 1 && S.nstages <= MSIR_MAX_STAGES) {
        msir_stage& g = a.rep->stage[S.nstages - 1];
        if (kg >= 0 && g.steps < MSIR_MAX_STEPS) g.gmres_iters[g.steps] = kg;
        g.steps += 1;
      }
      int rs = 0;
      s_act = ctl_step(S, a, s_old, md, xnorm_old, nbe, ferr, kg, &rs);
      s_reset = rs;
      s_alg = S.alg;
      S.nbe = nbe;
    }
    __syncthreads();
    // decisions below use s_act/s_reset/s_alg: thread 0 changes S.alg
    // inside this branch while other warps may not have reached it yet
    if (s_act == 1) {
      if (cx.tid == 0) { S.cged = 1; S.status = MSIR_OK; }
      break;
    }
    if (s_act == 2) {
      const bool reset = s_reset != 0;
      if (reset) FOR_MY_ROWS(cx, i) a.x[i] = a.x0[i];
      if (s_alg == MSIR_ALG_GMRES) {
        if (cx.tid == 0) S.phase = PH_NEED_ESC;
        __syncthreads();
        break;
      }
      if (cx.tid == 0) {
        S.alg += 1;
        S.it = 0;
        S.rho_max = 0.0;
        S.delta_prev = __longlong_as_double(0x7ff0000000000000ll);
        rep_new_stage(a, S, cx.cta);
      }
      __syncthreads();
      if (reset) {
        if (!(ok = grid_barrier(cx, a))) break;
        if (!(ok = residual<A0>(cx, a, a.x, ur, s, xnorm))) break;
        nbe = s / (a.normA * xnorm + a.normb);
        const bool b2 = nbe < S.best_nbe;
        if (b2) FOR_MY_ROWS(cx, i) a.xbest[i] = a.x[i];
        __syncthreads();
        if (cx.tid == 0 && b2) S.best_nbe = nbe;
        __syncthreads();
      }
    }
  }
  if (cx.tid == 0) {
    S.s = s;
    S.nbe = nbe;
    if (S.phase != PH_NEED_ESC) S.phase = PH_DONE;
  }
  __syncthreads();
  if (ok && S.phase == PH_DONE && !S.cged) {
    // not converged: return the iterate of smallest nbe
    FOR_MY_ROWS(cx, i) a.x[i] = a.xbest[i];
    if (cx.tid == 0) { S.status = MSIR_NOT_CONVERGED; S.nbe = S.best_nbe; }
  }
  return ok;
}

template <typename A0, typename F>
// One CTA per SM.  (Two per SM, with 128 registers per thread, let
// concurrent systems share SMs, but measured slower: spinning and fp64 work
// of one system then slow the other's.)
__global__ void __launch_bounds__(kRefThreads, 1) refine_kernel(RefineArgs a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  unsigned char* gsm = smem_raw + a.gmres_off;  // GMRES scalars
  __shared__ RefState S;
  __shared__ int s_act, s_reset, s_alg;

  Cx cx;
  cx.tsm = smem_raw + kScratchOff;
  cx.ssm = cx.tsm + kTrsvSmem;
  cx.G = gridDim.x;
  cx.cta = blockIdx.x;
  cx.tid = threadIdx.x;
  cx.lane = threadIdx.x & 31;
  cx.warp = threadIdx.x >> 5;
  cx.n = a.n;
  cx.nblk = (a.n + kBlk - 1) / kBlk;
  cx.team_k = a.team_k;
  cx.redbuf = 0;
  cx.nbar = 0;
  cx.inbox = (unsigned long long*)smem_raw;
  cx.C = 1;
  if (a.cluster > 1) {
    // the inbox starts all ones (a tag no hand-off uses); peers write into
    // it only after every CTA of the cluster has filled its own
    for (int i = cx.tid; i < kInboxSmem / 8; i += kRefThreads) cx.inbox[i] = ~0ull;
    unsigned rank, nrank;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
    asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(nrank));
    // the block-to-team mapping assumes rank = block index mod cluster size
    if ((int)nrank == a.cluster && (int)rank == cx.cta % a.cluster && a.cluster <= kMaxCluster) cx.C = a.cluster;
    cluster_sync_all();
  }
  if (cx.tid == 0) S = *a.st;
  __syncthreads();
  cx.epoch = S.epoch;
  cx.mready = S.mready;
  cx.t_ns = S.t_ns;
  bool ok = true;
  if (a.mode == MODE_RESIDUAL) {
    double s = 0.0, xn = 0.0;
    ok = grid_barrier(cx, a) && residual<A0>(cx, a, a.x, a.ap_arith, s, xn);
    if (ok && cx.cta == 0 && cx.tid == 0) *a.res_s = s;
  } else if (a.mode == MODE_PREP) {
    build_inverses<F>(cx, a, true, false);
  } else if (a.mode == MODE_APPLY) {
    for (int b = cx.cta; b < cx.nblk; b += cx.G)
      for (int i = b * kBlk + cx.tid; i < min((b + 1) * kBlk, cx.n); i += kRefThreads) {
        const int pr = a.perm[i];
        const double v = a.ap_in[pr] * rscale(a, pr);
        put_c(a, a.ap_arith, i, a.ap_arith == MSIR_DD ? v : round_to(v, a.ap_store), 0.0);
      }
    __syncthreads();
    ok = msolve_arith<F>(cx, a, a.ap_arith, a.ap_store);
    if (ok) FOR_MY_ROWS(cx, i) a.ap_out[i] = get_z(a, a.ap_arith, i) * cscale(a, i);
  } else {
    ok = refine_msir<A0, F>(cx, a, S, gsm, s_act, s_reset, s_alg);
  }
  __syncthreads();
  if (!ok && cx.tid == 0) { S.phase = PH_ERROR; S.status = MSIR_ERR_TIMEOUT; }
  if (cx.tid == 0) {
    S.epoch = cx.epoch;
    S.mready = cx.mready;
  }
  __syncthreads();
  if (cx.cta == 0 && cx.tid == 0) *a.st = S;
  // no CTA leaves while a cluster peer may still write into its inbox (every
  // wait before this point is bounded, so every peer arrives)
  if (a.cluster > 1) cluster_sync_all();
}

// Entry point of one instantiation (defined in refine_<a>_<f>.cu).
template <typename A0, typename F> void* refine_entry();

}  // namespace msir
