// Launch wrappers of the device kernels (kernels.cu).
#pragma once

#include <cuda_runtime.h>

#include "internal.h"

namespace psi {

// Programmatic dependent launch.  The level loops are chains of kernels of a few
// microseconds; a kernel launched with launch_dep may start while its predecessor in
// the stream still runs, reads what no kernel writes (its task, the supernode's
// metadata) and waits in after_previous() for the predecessor's end.  Every kernel
// launched so calls after_previous() in all its threads before anything else in
// memory, so that a kernel's end implies the end of all before it; the next one
// may start only after that wait, so at most one kernel per stream waits resident.
// One exception: merged_update takes its ticket before the wait.  A level's ticket is
// touched by its own launch alone, and the memset that clears it precedes the chain's
// first kernel, which starts in the ordinary way and so after the memset.
__device__ __forceinline__ void after_previous() {
#ifdef __CUDA_ARCH__
  cudaGridDependencySynchronize();
  cudaTriggerProgrammaticLaunchCompletion();
#endif
}

//
// Only grids of at most kDepCtas CTAs, the latency-bound ones: CTAs placed while the
// predecessor still holds the SMs land where slots are free, several on one SM
// beside empty ones, and a launch that is bound by the FP64 pipe then ends later
// than after an ordinary start (no limit: 20^3 adjoint step 10.9 -> 14.0 ms; 64
// against none: 31 x 31 grid 648 -> 590 us, 200 x 147 grid 1,911 -> 1,857, 24^3
// log det step 6,685 -> 6,558, adjoint step 10,934 -> 10,778; 152 is within 2%
// of 64 either way).
constexpr int64_t kDepCtas = 64;

// dep = false: an ordinary launch (the first of a stream's chain, or after a wait
// on another stream's event).
template <class... P, class... A>
cudaError_t launch_dep(void (*kernel)(P...), dim3 grid, unsigned block, size_t smem, cudaStream_t st, bool dep, A... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(block);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at = {};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &at;
  cfg.numAttrs = dep && (int64_t)grid.x * grid.y * grid.z <= kDepCtas ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}

// Per-batch-member sizes (elements of the scalar) of every batched array.
struct Sizes {
  int64_t panel;  // L and X panels
  int64_t lhat;   // normalised factor Lhat
  int64_t linv;   // diagonal-block inverses
  int64_t n;      // pivots
  int64_t part;   // step-3 partial products
  int64_t ypart;  // step-2 partial products
  int batch;
};

enum class Kern {
  Trsm, NormM, Lhat, Gemm1, Gemm2, DiagFinal, Gemm1Reduce,
  FactorDiagBK, CopyBackBK   // Bunch-Kaufman pivoted factor
};

// Everything a kernel may need; device pointers typed by dtype inside.
struct KArgs {
  int dtype;  // PSELINV_F64 / PSELINV_C128
  int maxw;   // widest supernode (shared-memory size of the diagonal kernels)
  const SnMeta* meta;
  const ColDesc* desc;
  const int32_t* relidx;
  void* L;
  void* D;
  void* Linv;
  void* Lhat;
  void* X;
  void* part;
  void* ypart;
  int* status;
  // split step 2: per-output-tile counters (batch x tctr_total, zero between
  // launches); set: the last slice CTA of a tile sums the slices in slice
  // order and writes X_{C,K} (no separate reduction); nullptr: partials only.
  // Step 3: set where the CTA of a supernode's last tile runs the finish
  int* tctr;
  int64_t tctr_n;  // counters per batch member
  Sizes sz;
  // non-symmetric handles (nullptr / 0 for symmetric ones)
  void* U;     // U panels: U'_{j,i} at panel position (i, j)
  void* Uinv;  // (U'_KK^T)^{-1}, linv layout
  void* XU;    // XU panels: X_{j,i} at panel position (i, j); step 2 reads X_{C,C} above the
               // diagonal from here, step 3 finish writes X_KK^T here
  // Bunch-Kaufman pivoted factor (nullptr when not pivoted), batch x n each:
  const int32_t* piv;  // supernode-local original column at each pivot position
  const int8_t* ptype; // 0 = 1x1 pivot, 1 / 2 = first / second column of a 2x2 pivot
  const void* E;       // D_{k+1,k} of a 2x2 pivot, at its first column
  // pole sum accumulated in the step-3 finish (pselinv_selinv_pole_sum):
  // weights w_b (batch), Gamma = sum_b w_b X_b (one panel array), counters
  // (nsn x kFinishCtas, zero between launches); nullptr otherwise
  const void* gw;
  void* gam;
  int* gctr;
  // pivoted factor: W_{C,K} = L_{C,K} D_K (see FArgs); nullptr elsewhere
  void* W;
};

// The factorisation's kernels.  Symmetric factors have one side; non-symmetric
// ones two: side 0 the lower triangle (L panels, (L_KK)^{-1}), side 1 the
// transposed upper one (U panels, (U'_KK^T)^{-1}).
struct FArgs {
  const SnMeta* meta;
  const ColDesc* desc;
  const int32_t* relidx;
  void* L[2];     // L, U panels
  void* Linv[2];  // inverses of the diagonal blocks' unit triangles
  // W_{C,K} = L_{C,K} D_K (side 1: U'_{K,C}^T D_K; pivoted: D_K's 1 x 1 and
  // 2 x 2 blocks, columns in pivot order), the panel solve's product before the
  // D^{-1} scaling, kept for the panel and Schur updates, in the panel layout
  // of this array (the X and XU panels, free during the factorisation)
  void* W[2];
  void* D;
  int* status;
  Sizes sz;
  int sides;
};
enum class FKern { Panel, Update, VInv, Schur };
// Status words set when a wait of a merged launch ran out: the factorisation's until
// the next factorisation, the adjoint's until pselinv_sync_status has reported it.
constexpr int kFactorTimeoutWord = 5, kAdjointTimeoutWord = 6;
// One merged launch (merged_update.cuh): the level's ticket, and for the
// level's first group on the tiles per group and the finished tiles per (group,
// copy), copy = side and batch member.
struct MergedArgs {
  int* ticket;
  int* abort;        // set when a wait ran out: the factorisation's status word, or the adjoint's flag
  const int32_t* gcnt;
  int* done;
  int ntile;         // tiles of one copy
  long long spin_ns; // bound of every wait
};

// CTAs of the per-level step-3 finish per supernode (blockIdx.z of k_diag_final).
constexpr int kFinishCtas = 32;

// Original local column of pivot position k of the supernode starting at f.
__device__ __forceinline__ int pcol(const KArgs& a, int b, int f, int k) {
  return a.piv ? a.piv[(int64_t)b * a.sz.n + f + k] : k;
}

cudaError_t setup_kernels();
cudaError_t launch_scatter_values(int dtype, const void* vals, const int64_t* vmap, int64_t nnz, void* L,
                                  const Sizes& sz, cudaStream_t st);
// Non-symmetric values: lower (A_ij) to the L panels, upper (A_ji) to the U
// panels, swapped where flip[q] (the ordering transposed entry q).
cudaError_t launch_scatter_values_lu(int dtype, const void* lower, const void* upper, const int64_t* vmap,
                                     const uint8_t* flip, int64_t nnz, void* L, void* U, const Sizes& sz,
                                     cudaStream_t st);
// Non-symmetric gather: X_ij (upper = 0) or X_ji (upper = 1) at stored entry q.
cudaError_t launch_gather_values_lu(int dtype, const void* XL, const void* XU, const int64_t* vmap,
                                    const uint8_t* flip, int64_t nnz, int upper, void* out, const Sizes& sz,
                                    cudaStream_t st);
// diagmask == nullptr: plain gather; else off-diagonal entries doubled.  invalid: a
// device flag; where it is set the output is NaN and *report becomes 1.
cudaError_t launch_gather_values(int dtype, const void* X, const int64_t* vmap, const uint8_t* diagmask, int64_t nnz,
                                 void* out, const Sizes& sz, cudaStream_t st, const int* invalid = nullptr,
                                 int* report = nullptr);
// Tile kernels (Trsm, NormM, Lhat, Gemm1, Gemm2) over n tasks of one tile
// width variant (BN = 8 << var).
cudaError_t launch_tiles(Kern k, int var, const KArgs& a, const Task* tasks, int64_t n, cudaStream_t st,
                         bool dep = true);
// Per-supernode kernels (DiagFinal, Gemm1Reduce, FactorDiagBK, CopyBackBK) over
// the nsn supernodes listed in sns.  threads: block size of FactorDiagBK (at
// most 512).
cudaError_t launch_per_sn(Kern k, const KArgs& a, const int32_t* sns, int nsn, cudaStream_t st, int threads = 256,
                          bool dep = true);
// Blocked factorisation: the diagonal block p of the listed supernodes (all wider
// than p blocks), and its tile lists (var: tile variant of the Schur groups).
// w: the widest such block.
cudaError_t launch_fdiag(int dtype, const FArgs& f, const int32_t* sns, int nsn, int p, int w, cudaStream_t st,
                         bool dep = true);
cudaError_t launch_schur_merged(int dtype, const FArgs& f, const MergedArgs& q, const Task* t, cudaStream_t st, bool dep);
// Inverses of the 32 x 32 diagonal blocks of L_KK of the listed supernodes (the widest wmax).
cudaError_t launch_vdiag(int dtype, const FArgs& f, const int32_t* sns, int nsn, int wmax, cudaStream_t st);
cudaError_t launch_ftiles(FKern k, int var, int dtype, const FArgs& f, const Task* t, int64_t n, cudaStream_t st,
                          bool dep = true);
// CTAs per batch member; work: batch x 2 x logdet_parts(n) doubles.
constexpr int logdet_parts(int64_t n) { return n <= 256 ? 1 : n >= 128 * 256 ? 128 : (int)((n + 255) / 256); }
cudaError_t launch_logdet(int dtype, const void* D, int64_t n, double* work, double* out, int batch, cudaStream_t st,
                          const int8_t* ptype = nullptr, const void* E = nullptr);
cudaError_t launch_pole_sum(int dtype, const void* X, int64_t panel_total, int batch, const void* w, void* out,
                            cudaStream_t st);
cudaError_t launch_trace_sum(int dtype, const void* X, int64_t panel_total, const int64_t* vmap,
                             const uint8_t* diagmask, const void* vals, int64_t nnz, int batch, void* out,
                             cudaStream_t st);

// ---- step 2 with FP64 arithmetic emulated on the bf16 tensor cores (emulate.cu) ----
// Real symmetric positive definite X only: |X_pq| <= sqrt(X_pp X_qq), so with
// e_p = ceil(log2 sqrt(X_pp)) every entry of Xt = 2^-(e_p + e_q) X has |Xt| < 1.
// Each entry of Xt (and of B' = diag(2^e_C) Lhat over a per-column exponent)
// is cut once into 7 signed 8-bit slices held as bf16; step 2 forms the 28
// slice products of weight >= 2^-48 with exact FP32 sums over 32-row chunks
// folded into 64-bit integers.
struct EmArgs {
  void* xs;              // [batch][panel_total] uint4: 7 bf16 slices of Xt per X panel entry
  void* ls;              // [batch][lhat_total] uint4: 7 bf16 slices of B' per Lhat entry
  int32_t* sig;          // [batch][n] e_p of every column (written when its level finishes)
  int32_t* lexp;         // [batch][n] column exponent F of B' (|B'_{:,j}| < 2^F), per global column
  int32_t* gexp;         // [batch][n] column exponent G of X'' = diag(2^-e_C) X_{C,K} (step 3)
  const int32_t* crow;   // [sum r] global row of C[i] of supernode K at desc offset of K
  int64_t n;
};
// Emulation status word: kEmRange after an X diagonal <= 0 / not finite or a
// scaled entry outside its slice range (X not positive definite).
constexpr int kEmStatusWord = 4;
constexpr int kEmRange = 1;
// After steps 2-3 of a level: e_p of the level's columns and the slices of
// its X panels.  Before step 2 of a level: F and the slices of its B'.
cudaError_t launch_em_split_x(const KArgs& a, const EmArgs& e, const int32_t* sns, int nsn, cudaStream_t st);
// max_r: the largest |C| among the supernodes (sizes the shared memory).
cudaError_t launch_em_split_lhat(const KArgs& a, const EmArgs& e, const int32_t* sns, int nsn, int max_r,
                                 cudaStream_t st);
// After step 2 of a level (step 3 emulated): G and the slices of X'' for its
// supernodes, written over the slice array at the rows of C of their panels.
cudaError_t launch_em_split_xck(const KArgs& a, const EmArgs& e, const int32_t* sns, int nsn, int max_r,
                                cudaStream_t st);
// Step-3 partial products (the Gemm2 task list of tile variant var) on the slices.
cudaError_t launch_em_gemm2(int var, const KArgs& a, const EmArgs& e, const Task* tasks, int64_t n, cudaStream_t st);
// Dynamic shared-memory limits of the step-2 kernels (called by setup_kernels).
cudaError_t setup_em_kernels();
// Step-2 tiles (the Gemm1 task list of tile variant var) on the slices:
// 64 x 8 / 64 x 16 tiles on mma.sync (var 0, 1).
cudaError_t launch_em_gemm1(int var, const KArgs& a, const EmArgs& e, const Task* tasks, int64_t n,
                            cudaStream_t st);

// ---- persistent per-level schedule (persistent.cu) ----
struct PArgs {
  const Task* g1;       // step-2 task array (t_gemm1)
  const Task* g2;       // step-3 task array (t_gemm2)
  int* c1;              // [batch][nsn] finished step-2 tiles
  int* c2;              // [batch][nsn] finished step-3 tiles
  int* cr;              // [batch][nsn] finished slice reductions
  int* cf;              // [batch][nsn] finished step-3 finish parts (X of the supernode final at kFinishParts)
  int* lvl;             // [nlevels] finished finish parts of a level, all batch members
  const int32_t* n1;    // [nsn] step-2 tiles per supernode
  const int32_t* n2;    // [nsn] step-3 tiles per supernode
  const int32_t* snlevel;   // [nsn] level (0 = roots)
  const int32_t* snparent;  // [nsn] supernodal parent, -1 = root
  const int32_t* level_ptr; // [nlevels + 1] supernodes per level (prefix sums)
  int* head;            // dequeue counter
  int nsn;
  int64_t yslot, pslot; // elements of one level slot of the step-2 / step-3 partial buffers
  long long spin_ns;    // bound of every wait
};
// Slots of the partial-product ring: a level starts its step 2 only once the
// level kRing above it has finished, so at most kRing levels hold partials.
constexpr int kRing = 4;
cudaError_t launch_persistent(const KArgs& a, const PArgs& p, const PTask* list, int64_t ntask, int grid,
                              cudaStream_t st);
cudaError_t persistent_grid(int dtype, int* grid);

// ---- adjoint (adjoint.cu) ----
struct AdjArgs {
  KArgs k;
  const void* G;  // seed, X panel layout
  int g_kind;     // PSELINV_G_SYMMETRIC / PSELINV_G_PANEL
  void* Xb;       // adjoint of X panels; later adjoint of the updated factor panels
  void* Lb;       // adjoint of L (panel layout)
  void* Db;       // adjoint of D
  void* Zb;       // s x s per supernode (linv layout): Zbar, then Vbar, then P
  void* W1;       // s x s per supernode scratch
  void* Yb;       // r x s per supernode (lhat layout): Ybar, then T1
  void* Hb;       // r x s per supernode: Lhat-bar
};
enum class AdjKern { Ybar, Lhbar, LbarOff, T1, Q, Vpart, Rpart, Syr2k, Dr1, Dr3, Dr4, Df2, Df3, Df4 };
enum class AdjSn { Seed, Ev, Zbar, Dr2, Df1, Df5 };
cudaError_t launch_adj_tiles(AdjKern k, int var, const AdjArgs& a, const Task* tasks, int64_t n, cudaStream_t st,
                             bool dep = true);
cudaError_t launch_adj_merged(const AdjArgs& a, const MergedArgs& q, const Task* t, cudaStream_t st);
// wmax: the widest supernode of the launch (64 at most where every supernode takes part).
cudaError_t launch_adj_per_sn(AdjSn k, const AdjArgs& a, const int32_t* sns, int nsn, int wmax, cudaStream_t st,
                              bool dep = true);

}  // namespace psi
