// Arguments and state of the persistent refinement kernel (refine.cu).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/msir.h"

namespace msir {

constexpr int kRefThreads = 256;  // 8 warps
constexpr int kBlk = 64;          // rows per block of the row distribution / TRSV
constexpr int kMaxKcap = 2048;    // GMRES iteration cap supported
// 64-bit payload words per value of the substitution hand-off buffer (4:
// enough for a double-double value).  The buffer holds, per direction
// (forward, backward), the solved values and the team-exchanged z of every
// block: 2 * 2 * ceil(n/kBlk) * kBlk * kLLWords words.
constexpr int kLLWords = 4;
// Shared scratch of the substitutions: 8 warps x 64 staged values plus the
// 64 values of z, for the widest value type (double-double, 16 bytes).
constexpr int kTrsvSmem = (kRefThreads / 32 + 1) * kBlk * 16;
// Shared staging of the scaled-block construction.  fp64 / dd: half the
// inner dimension of one tile at a time (inverse high and low words, 64 x 33
// doubles each; factor rows, 32 x 65 doubles).  fp32: the whole tile
// (inverse high and low words transposed and factor rows, 64 x 68 floats).
constexpr int kScLd = kBlk + 1;
constexpr int kSc32Ld = kBlk + 4;
constexpr int kScaledSmem64 = (2 * kBlk * (kBlk / 2 + 1) + (kBlk / 2) * kScLd) * 8;
constexpr int kScaledSmem32 = 3 * kBlk * kSc32Ld * 4;
constexpr int kScaledSmem = kScaledSmem64 > kScaledSmem32 ? kScaledSmem64 : kScaledSmem32;
// Shared scratch of one phase at a time: the substitutions (staged values
// and the tile ring in the staging area), the scaled-block construction, or
// the inverse of one diagonal block (inv_impl.cuh).
constexpr int kInvScratch = 8 * (3 * kBlk * (kBlk + 1) + 2 * (kBlk / 2) * (kBlk / 2 + 1) + 2 * kBlk);
constexpr int kPhaseSmem = kTrsvSmem + kScaledSmem > kInvScratch ? kTrsvSmem + kScaledSmem : kInvScratch;
// Thread-block clusters of the refinement launch: at most kMaxCluster CTAs.
// Each CTA keeps an inbox in shared memory where the CTAs of its cluster
// that solve the blocks just before it (forward) or after it (backward)
// write their solved values: one slot of kBlk values of kLLWords words per
// team position in the cluster.
constexpr int kMaxCluster = 8;
constexpr int kInboxSmem = kMaxCluster * kBlk * kLLWords * 8;

// Dynamic shared memory of the refinement: the inbox (it keeps its contents
// between phases), the scratch, the GMRES scalars.
constexpr int kScratchOff = kInboxSmem;
constexpr int kGmresOff = kInboxSmem + kPhaseSmem;  // (without wide solves)

// What a workspace holds for the current factors (RefState::mready).
enum ReadyBits : unsigned {
  RDY_M32 = 1u,  // inv32 and the fp32 scaled blocks
  RDY_MDD = 2u,  // double-double scaled blocks
  RDY_M64 = 4u,  // fp64 scaled blocks
  RDY_INV = 8u,  // inv_hi, inv_lo
  RDY_W32 = 16u, // fp32-pair inverses of the diagonal superblocks
  RDY_W64 = 32u, // fp64 ones
  RDY_NO32 = 64u, // fp32 pairs do not hold these superblocks' inverses: 64-row solves
  RDY_NO64 = 128u // nor the fp64 ones made from them
};

// Wide solves (refine_impl.cuh): rows of a superblock, and the smallest
// matrices that take them.  fp32: from two superblocks on (n = 1024 .. 2000:
// 20-40 us for a pair of solves against 45-95).  fp64: from 1792 rows on
// (n = 2000: 49 us against 112; below, the superblocks' construction, 1 ms,
// takes the solves of a short run to earn).  Errors against double-double
// solves, mean over n = 1300 .. 7237 and kappa = 1e2 .. 1e8, relative to the
// 64-row solves': fp32 0.08 (right-hand sides A x) and 0.09 (random ones),
// fp64 0.14 and 0.27.
constexpr int kSuper = 512;
constexpr int kWideMin = 1024;
constexpr int kWideMin64 = 1792;
// Smallest matrix whose factors' fp64 applies are wide: below, the first
// apply of a handle would pay more for the superblocks (n = 2000: 1.1 ms)
// than for the scaled blocks (0.7 ms); n = 5000: 2.7 and 3.7 ms.
constexpr int kWideApply64 = 3072;
// A superblock's inverse is formed in fp32 pairs (2^-46 an operation) only if
// its row sums and diagonal lie within 2^+-60 of 1 and of each other, so that
// no product or error term of the doubling leaves fp32's range, and its
// condition is at most kWideCond: the pair's error is some 2^-46 |X||T||X|.
// As for the 64-row blocks that is bounded by Skeel's condition number
// max_i (|X||T|e)_i, and where this is above the limit (columns of very
// different scale) formed and compared with X column by column.  (LU factors
// of randsvd, normal and other dense matrices, plain and with rows or columns
// graded by 10^+-4: at most 4.7e4 by either.)
// kWideResid: the largest scaled residual of a pair that one Newton step
// takes to fp64 (wide_products).
constexpr float kWideRange = 0x1p60f, kWideCond = 0x1p17f, kWideResid = 0x1p-32f;
constexpr int kRingDeep = 16, kRingFlat = 8;  // steps of the ring of factor values
// Shared memory of a wide solve in values of `vbytes` on a grid of G CTAs:
// y of every row, z of a superblock (high and low words), partial sums; then
// the ring of factor values (16 bytes per thread and step).
constexpr size_t wide_ring_off(int npad, int G, int vbytes) {
  const size_t rows = (size_t)(kSuper + G - 1) / G, passes = (rows + 3) / 4;  // at least 4 rows of a CTA at a time
  return ((size_t)npad * vbytes + 2 * (size_t)kSuper * vbytes + (2 + passes) * kRefThreads * 8 + 127) / 128 * 128;
}
constexpr size_t wide_smem(int npad, int G, int vbytes, int ring) {
  return wide_ring_off(npad, G, vbytes) + (size_t)ring * kRefThreads * 16;
}

// MODE_PREP: the double-double inverses of the diagonal blocks alone (a
// factorisation that is handed out); no CTA waits for another
enum RefMode { MODE_SOLVE = 0, MODE_APPLY = 1, MODE_RESIDUAL = 2, MODE_PREP = 3 };
enum RefPhase {
  PH_START = 0,      // compute x0, then refine
  PH_ESCALATED = 1,  // factors replaced by a finer u_f: recompute r, start SIR
  PH_DONE = 2,
  PH_NEED_ESC = 3,   // GMRES-IR stage ended without convergence: host refactors
  PH_ERROR = 4
};

// Controller state of Algorithm 4 kept on the device between launches.
struct RefState {
  int phase;
  int alg, it;
  int uf, u, ur;
  int cged, status;
  int have_phi0;
  unsigned epoch;     // substitution epoch (one per triangular solve)
  unsigned mready;    // ReadyBits of the current factors
  int nstages;
  int total_steps, total_gmres;
  double rho_max, delta_prev, phi0, phi;
  double s, nbe, best_nbe;
  // device time (ns) spent by CTA 0 per phase: 0 residual, 1 forward
  // substitution, 2 backward substitution, 3 Gram-Schmidt, 4 operator
  // matrix-vector product, 5 update/norm reductions, 6 Givens/least squares
  unsigned long long t_ns[8];
};

struct RefineArgs {
  int mode;
  int n;
  int a_fmt;               // storage of A_u: MSIR_FP32 or MSIR_FP64
  const void* A;           // A_u, row-major
  int lda;
  const double* b;         // b_u (values in u0)
  const void* LU;          // packed factors in u_f storage, row-major
  int ldf;
  int f_fmt;               // storage format of LU (MSIR_BF16 .. MSIR_FP64)
  const int* perm;         // (P A)[i] = A[perm[i]]
  const double* Rsc;       // squeezing row scalings (nullptr: none)
  const double* Ssc;       // column scalings
  double mu;
  double normA, normb;
  double* x;               // current iterate (values in u)
  double* xn;              // next iterate
  double* x0;
  double* xbest;
  double* r_hi;            // residual, permuted order: r_p[i] = r[perm[i]]
  double* r_lo;
  double* c_hi;            // TRSV right-hand side / work (permuted order)
  double* c_lo;
  double* y_hi;            // forward-substitution result
  double* y_lo;
  double* z_hi;            // backward-substitution result (natural order)
  double* z_lo;
  double* d;               // correction
  double* w;               // GMRES work vector
  double* V;               // Krylov basis in u, row-major: entry j of row i at
  int ldv;                 //   V + i*ldv (ldv >= kcap + 1)
  double* vk;              // the newest basis vector, contiguous (operator input)
  double* H;               // rotated Hessenberg, row-major, leading dimension kcap + 1
  double* yv;              // GMRES least-squares solution (kcap)
  double* red;             // reduction scratch: 2 * gridDim.x * kRedW
  double* hred;            // CGS partial sums: gridDim.x * (kcap+1)
  double* hvec;            // reduced CGS coefficients (kcap+1)
  unsigned long long* ll;  // substitution hand-off words (see kLLWords)
  // inverses of the diagonal blocks of L and U, [2][ceil(n/kBlk)][kBlk][kBlk],
  // zero outside the n - 64 b rows and columns of a ragged last block: a pair
  // of fp32 (inv32 is its fp32 rounding) and a double-double (inv_hi is its
  // fp64 rounding); built in the kernel when first needed
  float* inv32;
  float* inv32l;
  double* inv_hi;
  double* inv_lo;
  int* inv_hard;           // [2][ceil(n/kBlk)]: block kept out of the fp32 pairs' sums
  // scaled off-diagonal blocks D_b^{-1} F_bj (j != b) of L (j < b) and U
  // (j > b), row-major with leading dimension ldf, built in the kernel when a
  // solve in that precision first needs them (RefState::mready)
  float* M32;
  double* M64;
  double* Mdh;
  double* Mdl;
  // wide solves: n rounded up to whole superblocks, which precisions take
  // them (bit 0 fp32, bit 1 fp64), steps of the ring of factor values
  // (kRingDeep or kRingFlat) and its offset in the scratch, the inverses of the diagonal
  // superblocks of L and U, [2][npad][kSuper] (fp32 pairs, fp64)
  int npad, wide, ring, ring_off;
  int gmres_off;           // offset of the GMRES scalars in shared memory, and
  int scratch;             // bytes of the scratch before them (set by the launcher)
  float* D32h;
  float* D32l;
  double* D64;
  // of the triangles within their superblocks, [2][npad] each: the rows' sums
  // of magnitudes, the diagonal's magnitudes, the largest one of each column
  // of the inverse (wide_columns); what build_wide and wide_products found
  // (0: safe)
  float* wrow;
  int* wflag;
  unsigned* bar;           // grid barrier counter (zeroed before launch)
  int* err;
  RefState* st;
  msir_report* rep;        // device copy of the report
  // parameters of Algorithm 4
  int i_max;
  double rho_thresh;
  double kmax;
  int kcap;
  int team_k;              // substitution team size for fp64/dd (0: the rule in team_size)
  double tau;              // <= 0: by u
  double gamma;
  int conv;
  const double* xref;      // MSIR_CONV_TRUE: exact solution (natural order), else nullptr
  int allow_escalation;
  int u0;
  // MODE_APPLY: arith / store formats and input/output (natural order)
  int ap_arith, ap_store;
  const double* ap_in;
  double* ap_out;
  // MODE_RESIDUAL: output s
  double* res_s;
  // optional wavefront timestamps of the last substitution pair (ns):
  // [direction][block][start, off-diagonal done, published, last dependency seen]
  unsigned long long* tsv;
  // CTAs per thread-block cluster of this launch (1: no clusters); the
  // substitutions hand solved blocks to the CTAs of their cluster through
  // distributed shared memory
  int cluster;
};

constexpr int kRedW = 4;

cudaError_t launch_refine(int a_fmt, int f_fmt, const RefineArgs& a, int grid, cudaStream_t st);
int refine_max_grid(int a_fmt, int f_fmt, int kcap);
// Largest cooperative grid of `cluster`-CTA clusters that fits on the
// device for every u_f instantiation with A_u in a_fmt (0 if none).
int refine_max_cluster_grid(int a_fmt, int kcap, int cluster);
// Dynamic shared memory of a launch: the inbox, the scratch of the phase that
// needs most (`phase` bytes for the wide solves), the GMRES scalars.
size_t refine_smem_bytes(int kcap, size_t phase = 0);

}  // namespace msir
