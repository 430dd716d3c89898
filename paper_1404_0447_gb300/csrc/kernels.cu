// Device kernels of the supernodal LDL^T and the selected inversion,
// templated on the scalar (double, or complex symmetric Cplx) and on the
// output tile width BN of the tile GEMMs.
//
// Storage (per batch member, offsets in SnMeta, elements of the scalar):
// L and X panels are (s + r) x s column-major blocks with ld = s + r whose
// rows are the supernode's own columns followed by R(K) = C; Lhat_{C,K} is
// r x s with ld = r; (L_KK)^{-1} is s x s with ld = s; D holds the pivots.
#include <cuda_runtime.h>

#include <algorithm>

#include "block_inverse.cuh"
#include "internal.h"
#include "kernels.h"
#include "merged_update.cuh"
#include "selinv_steps.cuh"
#include "tile_gemm.cuh"

namespace psi {

// packed lower-triangular index, column-major: (i, j), i >= j, order s
__device__ __forceinline__ int pk(int i, int j, int s) { return j * s - (j * (j - 1)) / 2 + (i - j); }

// Status words 0-1 hold one 64-bit key (column << 2 | kind), kind 1 = zero
// pivot, 2 = non-finite: the minimum is the first bad column and, within
// it, a zero pivot before its consequences.
__device__ void report_pivot(int* status, int col, bool zero) {
  atomicMin(reinterpret_cast<unsigned long long*>(status),
            ((unsigned long long)(unsigned)col << 2) | (zero ? 1ull : 2ull));
}

// Whether u / d may be taken as u (1 / d) (one division a column, a product of 60
// cycles instead of a division of 574 per entry): 1 / d is a normal number.
// Elsewhere (|d| < 2^-1021 or >= 2^1022) the product would lose bits or overflow where
// the quotient is an ordinary number, and the kernels divide, outside the code that
// ordinary pivots run: a test and a division in the pivot loop of k_fdiag cost 0.8 to
// 1.3% of a 24^3 log det step and a 24^3 non-symmetric pass, this form 0 and 0.5%.
// Complex: division squares |d|, which leaves its own range first.
__device__ __forceinline__ bool by_reciprocal(double d) {
  return ((unsigned)__double2hiint(d) >> 20 & 0x7ffu) - 2u < 2043u;
}
__device__ __forceinline__ bool by_reciprocal(Cplx) { return true; }
// A zero in the place of the reciprocal (a normal number has no zero high word).
__device__ __forceinline__ bool no_reciprocal(double rd) { return __double2hiint(rd) == 0; }
__device__ __forceinline__ bool no_reciprocal(Cplx) { return false; }

// --------------------------------------------------------------------------
// value scatter / selected-entry gather (HBM-bound, index driven)
// --------------------------------------------------------------------------

template <class T>
__global__ void k_scatter_values(const T* __restrict__ vals, const int64_t* __restrict__ vmap, int64_t nnz,
                                 T* __restrict__ L, int64_t panel_total) {
  const int b = blockIdx.y;
  const T* v = vals + (int64_t)b * nnz;
  T* Lb = L + (int64_t)b * panel_total;
  for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < nnz; q += (int64_t)gridDim.x * blockDim.x)
    Lb[vmap[q]] = v[q];
}

// Non-symmetric values: entry q's pair (A_ij, A_ji) goes to the L and U
// panels at its position, or to the U and L panels where the ordering
// transposed it.
template <class T>
__global__ void k_scatter_values_lu(const T* __restrict__ lo, const T* __restrict__ up,
                                    const int64_t* __restrict__ vmap, const uint8_t* __restrict__ flip,
                                    int64_t nnz, T* __restrict__ L, T* __restrict__ U, int64_t panel_total) {
  const int b = blockIdx.y;
  const T* vl = lo + (int64_t)b * nnz;
  const T* vu = up + (int64_t)b * nnz;
  T* Lb = L + (int64_t)b * panel_total;
  T* Ub = U + (int64_t)b * panel_total;
  for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < nnz; q += (int64_t)gridDim.x * blockDim.x) {
    const int64_t p = vmap[q];
    const bool f = flip[q] != 0;
    Lb[p] = f ? vu[q] : vl[q];
    Ub[p] = f ? vl[q] : vu[q];
  }
}

// Non-symmetric gather: X_ij (upper = 0) or X_ji (upper = 1) for the stored
// entry q at (i, j), from the XL or XU panel depending on the flip.
template <class T>
__global__ void k_gather_values_lu(const T* __restrict__ XL, const T* __restrict__ XU, int64_t panel_total,
                                   const int64_t* __restrict__ vmap, const uint8_t* __restrict__ flip, int64_t nnz,
                                   int upper, T* __restrict__ out) {
  const int b = blockIdx.y;
  const T* Xl = XL + (int64_t)b * panel_total;
  const T* Xu = XU + (int64_t)b * panel_total;
  T* o = out + (int64_t)b * nnz;
  for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < nnz; q += (int64_t)gridDim.x * blockDim.x)
    o[q] = ((flip[q] != 0) != (upper != 0)) ? Xu[vmap[q]] : Xl[vmap[q]];
}

// out[q] = X at the panel position of stored entry q; with a diagonal mask,
// off-diagonal entries are doubled (gradient with respect to a stored value
// that stands for both A_ij and A_ji).  NaN throughout where *invalid is set, which
// *report then says.
template <class T>
__global__ void k_gather_values(const T* __restrict__ X, int64_t panel_total, const int64_t* __restrict__ vmap,
                                const uint8_t* __restrict__ diagmask, int64_t nnz, T* __restrict__ out,
                                const int* __restrict__ invalid, int* report) {
  const int b = blockIdx.y;
  const T* Xb = X + (int64_t)b * panel_total;
  T* o = out + (int64_t)b * nnz;
  const bool bad = invalid && *invalid;
  if (bad && threadIdx.x == 0) *report = 1;
  for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < nnz; q += (int64_t)gridDim.x * blockDim.x) {
    const T v = bad ? Sc<T>::nan() : Xb[vmap[q]];
    o[q] = (diagmask && !diagmask[q]) ? 2.0 * v : v;
  }
}

// --------------------------------------------------------------------------
// diagonal blocks
// --------------------------------------------------------------------------

// Blocked factorisation of the panel of supernode K, 32 columns at a time: for
// block p, k_fdiag (diagonal block), k_fpanel (the rows below it) and k_fupdate
// (the remaining columns of the panel).  One SM's FP64 pipe takes 97 us for the
// s^3 / 3 flops of a 128-wide block and as long again for its inverse, so the
// work is spread over the GPU and only the 32 x 32 blocks stay on one SM;
// (L_KK)^{-1} off the diagonal blocks waits until after the last level
// (k_vinv), where all supernodes run at once.  Against one CTA per supernode
// factoring and inverting the whole block in shared memory: see k_fdiag.
constexpr int kFdUpdate = 192;  // threads holding a 32 x 32 triangle, beside the pivot warp: 6 warps fill the FP64 pipe
constexpr int kFdEntries = (kFB * (kFB + 1) / 2 + kFdUpdate - 1) / kFdUpdate;  // lower entries per thread
// ... and a narrower one (levels of thousands of small supernodes): 64 threads for
// w <= 8 (36 entries), 96 for w <= 16 (136), 128 for w <= 24 (300)
inline int fd_update(int w) { return w <= 8 ? 64 : w <= 16 ? 96 : w <= 24 ? 128 : kFdUpdate; }

// Value of lane src, to all lanes of the warp.
__device__ __forceinline__ double shfl(double v, int src) { return __shfl_sync(0xffffffffu, v, src); }
__device__ __forceinline__ Cplx shfl(Cplx v, int src) { return {shfl(v.re, src), shfl(v.im, src)}; }

// Block p of the supernodes in sns (width above 32 p): LDL^T of the w x w
// diagonal block (w <= 32) and the inverse V of its unit lower triangle, by
// in-place elimination on [A | I]: at column j, row i > j becomes row i - l_i
// row j, and the freed slot (i, j) takes V's -l_i.
// SIDES 2, non-symmetric block A = L D U': the lower triangle (panel L, V to
// linv) and the transposed upper one (panel U, V = (U'^T)^{-1} to uinv) are
// eliminated side by side, each with its own l and the other's unscaled column
// u; the pivots are those of the lower triangle, and on symmetric input both
// sides do the arithmetic of SIDES 1.
// Bound: the chain of w pivots.  Warp 0 runs that chain one column ahead of the
// others: in phase j it updates column j + 1 (lane = row), takes 1 / d (364
// cycles) and scales (60), while the other warps apply column j to the entries
// right of column j + 1 and to V (up to three entries per thread, in
// registers).  They exchange l and u of column j, column j + 1 before its last
// update and V's row j through shared memory, double buffered, one barrier per
// column.  Out: L (unit diagonal implied, d on the diagonal) to the panel, d to
// D, V to linv (zeros above the diagonal).
template <class T, int SIDES>
__global__ void __launch_bounds__(32 + SIDES * kFdUpdate) k_fdiag(FArgs f, const int32_t* __restrict__ sns, int p) {
  __shared__ __align__(16) double raw[SIDES * 2 * 4 * kFB * Sc<T>::P];
  // per side, of parity j & 1: l and u of column j, column j before the update by column j - 1, V's row j
  constexpr int SD = 8 * kFB;
  T* sh = reinterpret_cast<T*>(raw);
  const int b = blockIdx.y;
  const SnMeta m = f.meta[sns[blockIdx.x]];
  after_previous();
  const int s = m.s, ld = m.s + m.r, c0 = p * kFB, w = min(kFB, s - c0);
  const int64_t po = b * f.sz.panel + m.panel + c0 + (int64_t)c0 * ld, vo = b * f.sz.linv + m.linv + c0 + (int64_t)c0 * s;
  if (threadIdx.x < 32) {
    const int i = threadIdx.x;
    T* d = (T*)f.D + b * f.sz.n + m.f + c0;
    T c[SIDES];
#pragma unroll
    for (int e = 0; e < SIDES; ++e) c[e] = i < w ? ((T*)f.L[e] + po)[i] : Sc<T>::zero();  // column 0
    T dl = c[0];  // lane j: d_j, once column j is final
    auto column = [&](int j, T dj, bool prod) {
      const T rd = Sc<T>::one() / dj;
      const int o = (j & 1) * kFB;
      T l[SIDES], u[SIDES];
#pragma unroll
      for (int e = 0; e < SIDES; ++e) {
        l[e] = prod ? c[e] * rd : c[e] / dj;
        sh[e * SD + o + i] = l[e];  // rows above j are not read
        sh[e * SD + 2 * kFB + o + i] = c[e];
        u[e] = shfl(c[e], j + 1);
      }
      __syncthreads();
#pragma unroll
      for (int e = 0; e < SIDES; ++e) {
        // rows above j + 1 and from w: never used
        c[e] = sh[e * SD + 4 * kFB + (kFB - o) + i] - l[e] * u[SIDES - 1 - e];
        if (i > j && i < w) ((T*)f.L[e] + po)[i + (int64_t)j * ld] = l[e];
      }
      if (i == j + 1) dl = c[0];
    };
    int j = 0;
    for (; j + 1 < w; ++j) {
      const T dj = shfl(c[0], j);
      if constexpr (Sc<T>::P == 1)
        if (__any_sync(0xffffffffu, !by_reciprocal(dj))) break;  // a vote: no divergent code in the chain
      column(j, dj, true);
    }
    if constexpr (Sc<T>::P == 1)
      for (; j + 1 < w; ++j) {  // from the first pivot out of range on
        const T dj = shfl(c[0], j);
        column(j, dj, by_reciprocal(dj));
      }
    // off the chain: a test of d_j inside the loop would hold this warp for the
    // FP64 compares of every column
    if (i < w) {
      if (Sc<T>::bad(dl)) report_pivot(f.status, m.f + c0 + i, Sc<T>::is_zero(dl));
      d[i] = dl;
      ((T*)f.L[0] + po)[i + (int64_t)i * ld] = dl;
#pragma unroll
      for (int e = 0; e < SIDES; ++e) ((T*)f.Linv[e] + vo)[i + (int64_t)i * s] = Sc<T>::one();
    }
    return;
  }
  const int nu = (blockDim.x - 32) / SIDES;  // threads per side
  const int side = SIDES == 1 ? 0 : (threadIdx.x - 32) / nu;
  const int t = threadIdx.x - 32 - side * nu;
  const T* P = (const T*)f.L[side] + po;
  T* V = (T*)f.Linv[side] + vo;
  T *sl = sh + side * SD, *spre = sl + 4 * kFB, *sv = sl + 6 * kFB;
  const T* su = sh + (SIDES - 1 - side) * SD + 2 * kFB;
  const int ne = w * (w + 1) / 2;
  T x[kFdEntries];
  int ri[kFdEntries], ck[kFdEntries];
#pragma unroll
  for (int q = 0; q < kFdEntries; ++q) {
    const int e = t + q * nu;
    ri[q] = ck[q] = 0;  // no entry: never live
    x[q] = Sc<T>::zero();
    if (e < ne) {
      tri_entry(e, ri[q], ck[q]);
      if (ck[q] > 0) x[q] = P[ri[q] + (int64_t)ck[q] * ld];  // column 0 is the pivot warp's
      if (ck[q] == 1) spre[kFB + ri[q]] = x[q];
    }
  }
  for (int j = 0; j + 1 < w; ++j) {
    __syncthreads();
    const int o = (j & 1) * kFB;
    // all operands first, then the products of the three entries back to back: with
    // a branch per kind of entry they ran one after the other and the phase took
    // 924 cycles instead of 655 (34.2k -> 24.5k cycles for 32 columns)
    T a[kFdEntries], v[kFdEntries];
#pragma unroll
    for (int q = 0; q < kFdEntries; ++q) {
      a[q] = sl[o + ri[q]];
      v[q] = (ck[q] > j ? su : sv)[o + ck[q]];  // k > j: u_k; k < j: V_jk
    }
#pragma unroll
    for (int q = 0; q < kFdEntries; ++q) {
      const int i = ri[q], k = ck[q];
      if (i > j && k != j + 1)  // column j + 1 is the pivot warp's
        x[q] = (k == j ? Sc<T>::zero() : x[q]) - a[q] * (k == j ? Sc<T>::one() : v[q]);
    }
#pragma unroll
    for (int q = 0; q < kFdEntries; ++q) {
      const int i = ri[q], k = ck[q];
      if (k == j + 2 && i >= k) spre[o + i] = x[q];    // parity of column j + 2
      if (i == j + 1 && k <= j) sv[kFB - o + k] = x[q];  // V's row j + 1
    }
  }
#pragma unroll
  for (int q = 0; q < kFdEntries; ++q) {
    const int i = ri[q], k = ck[q];
    if (i <= k) continue;
    V[i + (int64_t)k * s] = x[q];
    V[k + (int64_t)i * s] = Sc<T>::zero();
  }
}

// Blocked factorisation, 16 (32, 64) rows from m0 of the panel below the diagonal block
// p (task c): W = A V_pp^T = L D, kept in the X panels (same layout) as the
// first operand of the panel and Schur updates, and L = W D^{-1} in place.
// Warp j takes the block's columns 8 j .. 8 j + 7 (k < 8 j + 8: V_pp^T is upper
// triangular) of 16 rows; blocks of at most 8 or 16 columns put the free warps on
// further rows (fpanel_rows).  The CTA's rows are its own, so after one barrier L
// replaces A.
// Operand fragments go straight from global memory to registers, all loads in
// flight at once.  Bound: the FP64 pipe (40 m8n8k4 MMAs of 145 cycles) where a
// level has many rows; near the root, latency: 64 x 8 tiles staged in shared
// memory took 8.7 us however few there were, a warp per 8 rows and 32 columns 9.5.
// blockIdx.z = 1: the U side of a non-symmetric factor, U'_{K,C}^T = A_{K,C}^T
// L_KK^{-T} D^{-1}, as L_{C,K} = A_{C,K} U'_KK^{-1} D^{-1} uses (U'_KK^T)^{-1}.
template <class T>
__global__ void __launch_bounds__(kFB * 4) k_fpanel(FArgs f, const Task* __restrict__ tasks) {
  constexpr int RF = 2;
  const Task tk = tasks[blockIdx.x];
  const int b = blockIdx.y, side = blockIdx.z;
  const SnMeta m = f.meta[tk.sn];
  after_previous();
  const int s = m.s, ld = s + m.r, c0 = tk.c * kFB, w = min(kFB, s - c0);
  const int lane = threadIdx.x & 31, g = lane >> 2, q = lane & 3, warp = threadIdx.x >> 5;
  const int nw = 64 / fpanel_rows(w);  // warps side by side
  const int j = warp % nw, m0 = tk.m0 + warp / nw * 16;
  T* A = (T*)f.L[side] + b * f.sz.panel + m.panel + (int64_t)c0 * ld;
  T* Wp = (T*)f.W[side] + b * f.sz.panel + m.panel + (int64_t)c0 * ld;
  const T* Vi = (const T*)f.Linv[f.sides - 1 - side] + b * f.sz.linv + m.linv + c0 + (int64_t)c0 * s;
  T a[RF][kFB / 4], bf[kFB / 4], dc[2], rd[2];
#pragma unroll
  for (int u = 0; u < kFB / 4; ++u) {
    const int k = 4 * u + q, n = 8 * j + g;
    const bool on = u < 2 * j + 2 && k < w;
    bf[u] = on && n < w ? Vi[n + (int64_t)k * s] : Sc<T>::zero();
#pragma unroll
    for (int h = 0; h < RF; ++h) {
      const int row = m0 + 8 * h + g;
      a[h][u] = on && row < ld ? A[row + (int64_t)k * ld] : Sc<T>::zero();
    }
  }
#pragma unroll
  for (int e = 0; e < 2; ++e) {
    const int col = 8 * j + 2 * q + e;
    dc[e] = col < w ? ((const T*)f.D + b * f.sz.n + m.f + c0)[col] : Sc<T>::one();
    rd[e] = Sc<T>::one() / dc[e];
  }
  double acc[RF][Sc<T>::P][2] = {};
#pragma unroll
  for (int h = 0; h < RF; ++h) {
    if (j == 0) frag_mma<T, 2>(acc[h], a[h], bf);
    if (j == 1) frag_mma<T, 4>(acc[h], a[h], bf);
    if (j == 2) frag_mma<T, 6>(acc[h], a[h], bf);
    if (j == 3) frag_mma<T, 8>(acc[h], a[h], bf);
  }
  __syncthreads();  // every warp has read its rows' entries
#pragma unroll
  for (int h = 0; h < RF; ++h)
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      const int row = m0 + 8 * h + g, col = 8 * j + 2 * q + e;
      if (row >= ld || col >= w) continue;
      const T v = frag_value<T>(acc[h], e);
      Wp[row + (int64_t)col * ld] = v;
      A[row + (int64_t)col * ld] = v * rd[e];
    }
  if (by_reciprocal(dc[0]) && by_reciprocal(dc[1])) return;
#pragma unroll
  for (int h = 0; h < RF; ++h)  // behind the stores of every ordinary pivot
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      const int row = m0 + 8 * h + g, col = 8 * j + 2 * q + e;
      if (row < ld && col < w && !by_reciprocal(dc[e])) A[row + (int64_t)col * ld] = frag_value<T>(acc[h], e) / dc[e];
    }
}

// Blocked factorisation, the columns right of block p (task c) of the panel:
// A_ij -= sum_k W_ik L_jk over the block's 32 columns k, rows i >= j of the
// whole panel (i > j on the U side), each entry by one thread; one warp per
// 8 x 8 fragment of a 16 x 8 tile, operands straight to registers (see k_fpanel).
// Bound: latency near the root, 8 us a step (staged 64 x 8 tiles 8.5).
constexpr int kFUpdateThreads = 4 * kFUpdateRows;
template <class T>
__global__ void __launch_bounds__(kFUpdateThreads) k_fupdate(FArgs f, const Task* __restrict__ tasks) {
  const Task tk = tasks[blockIdx.x];
  const int b = blockIdx.y, side = blockIdx.z;
  const SnMeta m = f.meta[tk.sn];
  after_previous();
  const int s = m.s, ld = s + m.r, c0 = tk.c * kFB;
  const int lane = threadIdx.x & 31, g = lane >> 2, q = lane & 3;
  const int64_t po = b * f.sz.panel + m.panel;
  T* P = (T*)f.L[side] + po;
  const T* L2 = (const T*)f.L[f.sides - 1 - side] + po + (int64_t)c0 * ld;
  const T* Wp = (const T*)f.W[side] + po + (int64_t)c0 * ld;
  const int r0 = tk.m0 + 8 * (threadIdx.x >> 5);
  if (r0 >= ld) return;
  T a[kFB / 4], bf[kFB / 4];
#pragma unroll
  for (int u = 0; u < kFB / 4; ++u) {
    const int64_t k = (int64_t)(4 * u + q) * ld;
    a[u] = r0 + g < ld ? Wp[r0 + g + k] : Sc<T>::zero();
    bf[u] = tk.n0 + g < s ? L2[tk.n0 + g + k] : Sc<T>::zero();
  }
  double acc[Sc<T>::P][2] = {};
  frag_mma<T, kFB / 4>(acc, a, bf);
#pragma unroll
  for (int e = 0; e < 2; ++e) {
    const int row = r0 + g, col = tk.n0 + 2 * q + e;
    if (row < ld && col < s && row >= col + side) P[row + (int64_t)col * ld] -= frag_value<T>(acc, e);
  }
}

// (L_KK)^{-1} off its 32 x 32 diagonal blocks, all supernodes wider than 32 of the
// task list at once (pivot-free: after the last level): one strip of 8 columns
// (task n0) per CTA; blockIdx.z = side.  Bound: the chain of a strip's blocks, 54 us
// for all supernodes of a 33 x 29 x 27 grid (inside the level loop, with the block on
// one SM, (L_KK)^{-1} was most of the 345 us of a 128-wide block).
template <class T>
__global__ void __launch_bounds__(TG_THREADS) k_vinv(FArgs f, const Task* __restrict__ tasks) {
  __shared__ VsSmem<T> sm;
  const Task tk = tasks[blockIdx.x];
  const SnMeta m = f.meta[tk.sn];
  after_previous();
  inverse_strip<T>((const T*)f.L[blockIdx.z] + blockIdx.y * f.sz.panel + m.panel, m.s + m.r,
                   (T*)f.Linv[blockIdx.z] + blockIdx.y * f.sz.linv + m.linv, m.s, tk.n0, sm);
}

// Inverses of the 32 x 32 diagonal blocks of L_KK (pivoted factorisation; the
// pivot-free one forms them in k_fdiag): blockIdx.z = block of the supernode.
template <class T>
__global__ void __launch_bounds__(kVdThreads) k_vdiag(FArgs f, const int32_t* __restrict__ sns) {
  __shared__ __align__(16) unsigned char raw[sizeof(VdSmem<T>)];
  const SnMeta m = f.meta[sns[blockIdx.x]];
  after_previous();
  const int c0 = blockIdx.z * kFB, ld = m.s + m.r;
  if (c0 >= m.s) return;
  diag_inverse<T>((const T*)f.L[0] + blockIdx.y * f.sz.panel + m.panel + c0 + (int64_t)c0 * ld, ld,
                  (T*)f.Linv[0] + blockIdx.y * f.sz.linv + m.linv + c0 + (int64_t)c0 * m.s, m.s, min(kFB, m.s - c0),
                  *reinterpret_cast<VdSmem<T>*>(raw));
}

// |re| + |im|: the magnitude Bunch-Kaufman compares (plain |x| for real)
__device__ __forceinline__ double bk_abs(double x) { return fabs(x); }
__device__ __forceinline__ double bk_abs(Cplx x) { return fabs(x.re) + fabs(x.im); }

// bk_abs as an ordered key: magnitudes compare like their bit patterns, in integer
// instructions (an FP64 compare waits 55 cycles for the one pipe); 0 for a NaN.
constexpr unsigned long long kBkInf = 0x7ff0000000000000ull;
__device__ __forceinline__ unsigned long long bk_key(double mag) {
  const unsigned long long u = (unsigned long long)__double_as_longlong(mag);
  return u > kBkInf ? 0ull : u + 1ull;
}

// Largest key over warp lanes and its index (the first on ties), to all lanes:
// three 32-bit warp reductions.  Key 0 is no candidate; none where all are.
__device__ __forceinline__ void warp_argmax(unsigned long long& key, int& idx, int none) {
  const unsigned hi = (unsigned)(key >> 32), lo = (unsigned)key;
  const unsigned mh = __reduce_max_sync(0xffffffffu, hi);
  const unsigned ml = __reduce_max_sync(0xffffffffu, hi == mh ? lo : 0u);
  const bool top = key && hi == mh && lo == ml;
  idx = (int)__reduce_min_sync(0xffffffffu, top ? (unsigned)idx : (unsigned)none);
  key = ((unsigned long long)mh << 32) | ml;
}

// Factorisation with Bunch-Kaufman pivoting restricted to the supernode's
// diagonal block (Bunch and Kaufman 1977, the lower form of LAPACK's
// xSYTF2), one CTA per supernode of the level, the block packed in shared
// memory.  For pivot position k of the reduced block: a = |T_kk|, colmax =
// max_{i>k} |T_ik| at imax; a >= alpha colmax -> 1x1; else with rowmax the
// largest off-diagonal magnitude of row/column imax: a rowmax >= alpha
// colmax^2 -> 1x1; |T_imax,imax| >= alpha rowmax -> 1x1 after swapping k
// and imax; else 2x2 on (k, k+1) after swapping k+1 and imax.  Swaps are
// symmetric interchanges of the whole block, including the computed L rows.
// Out: L_KK (pivot order, zero beside 2x2 blocks) and D to the panel's
// diagonal block, D, E (2x2 off-diagonals), pivot types, the local pivot
// order piv.  (L_KK)^{-1} is k_vdiag's and k_vinv's.
// A reduced column that is entirely zero, a singular 2x2 block or a non-finite
// value is reported in the status words.
// Bound: per column the search and the reciprocal of the pivot (one warp), three
// barriers, and the trailing update on this SM's FP64 pipe (s^3 / 6 FMAs, 100 us
// of a 128-wide real block), one FMA per entry: L_i u_j with the unscaled column u
// kept beside L (L_i L_j d took three FP64 operations, 300 of the 440-530 us of
// such a block).  Searching column k + 1 beside the update was slower (350
// against 300 us): the update's FMAs keep the one warp waiting for the pipe.
template <class T>
__global__ void __launch_bounds__(512) k_factor_diag_bk(const SnMeta* __restrict__ meta,
                                                        const int32_t* __restrict__ sns, T* __restrict__ L,
                                                        T* __restrict__ D, T* __restrict__ E,
                                                        int8_t* __restrict__ ptype, int32_t* __restrict__ piv,
                                                        Sizes sz, int* status) {
  extern __shared__ __align__(16) unsigned char shraw[];
  T* Tp = reinterpret_cast<T*>(shraw);
  const int k0 = sns[blockIdx.x];
  const int b = blockIdx.y;
  const SnMeta m = meta[k0];
  after_previous();
  const int s = m.s, ld = m.s + m.r;
  T* l1 = Tp + s * (s + 1) / 2;  // 1x1 step: the unscaled column; 2x2 step: the new L columns
  T* l2 = l1 + s;                // 1x1 step: the new L column
  int* perm = reinterpret_cast<int*>(l2 + s);
  __shared__ int sh_kp, sh_kstep, sh_bad, sh_row;  // sh_row: column of the row search still to do, or -1
  __shared__ __align__(16) double rraw[Sc<T>::P];
  T* rpiv = reinterpret_cast<T*>(rraw);  // 1 / pivot of a 1 x 1 step; 0: divide by the pivot
  __shared__ double sh_colmax;
  T* P = L + b * sz.panel + m.panel;
  const int nt = blockDim.x, t = threadIdx.x;
  const double alpha = (1.0 + sqrt(17.0)) / 8.0;
  for (int e = t; e < s * s; e += nt) {
    const int i = e % s, j = e / s;
    if (i >= j) Tp[pk(i, j, s)] = P[i + (int64_t)j * ld];
  }
  for (int q = t; q < s; q += nt) perm[q] = q;
  if (t == 0) sh_bad = 0;
  __syncthreads();
  T* dd = D + b * sz.n + m.f;
  T* ee = E + b * sz.n + m.f;
  int8_t* ty = ptype + b * sz.n + m.f;
  // warp 0, column c final: the decision for pivot position c, up to the row search
  auto search = [&](int c) {
    const T acc = Tp[pk(c, c, s)];
    const T r0 = Sc<T>::one() / acc;  // the reciprocal pivot of a 1 x 1 step without interchange
    const int cc = pk(c, c, s) - c;
    unsigned long long ck = 0;
    int ci = s;
#pragma unroll
    for (int h = 0; h < kMaxWidth / 32; ++h) {
      const int i = c + 1 + t + 32 * h;
      const unsigned long long key = i < s ? bk_key(bk_abs(Tp[cc + i])) : 0ull;
      if (key > ck) {
        ck = key;
        ci = i;
      }
    }
    warp_argmax(ck, ci, s);
    if (t == 0) {
      const unsigned long long ak = bk_key(bk_abs(acc));
      const double colmax = ck ? __longlong_as_double((long long)(ck - 1)) : 0.0;
      sh_kp = c;
      sh_kstep = 1;
      sh_row = -1;
      *rpiv = by_reciprocal(acc) ? r0 : Sc<T>::zero();
      if (ak == 0 || ak > kBkInf || ck > kBkInf) {  // NaN or infinite
        sh_bad = 2;
      } else if (ak == 1 && ck <= 1) {
        sh_bad = 1;
      } else if (ak < bk_key(alpha * colmax)) {
        sh_row = ci;
        sh_colmax = colmax;
      }
    }
  };
  int k = 0;
  while (k < s) {
    if (t < 32) search(k);
    __syncthreads();
    if (sh_bad) break;
    if (sh_row >= 0) {
      if (t < 32) {
        const int imax = sh_row;
        unsigned long long rk = 0;
        int ri = s;
        for (int j = k + t; j < s; j += 32)
          if (j != imax) {
            const unsigned long long key = bk_key(bk_abs(j < imax ? Tp[pk(imax, j, s)] : Tp[pk(j, imax, s)]));
            if (key > rk) {
              rk = key;
              ri = j;
            }
          }
        warp_argmax(rk, ri, s);
        if (t == 0) {
          const double rowmax = rk ? __longlong_as_double((long long)(rk - 1)) : 0.0, colmax = sh_colmax;
          const double absakk = bk_abs(Tp[pk(k, k, s)]);
          if (!(absakk * rowmax >= alpha * colmax * colmax)) {
            sh_kp = imax;
            const T d = Tp[pk(imax, imax, s)];
            if (bk_abs(d) >= alpha * rowmax)
              *rpiv = by_reciprocal(d) ? Sc<T>::one() / d : Sc<T>::zero();
            else
              sh_kstep = 2;
          }
        }
      }
      __syncthreads();
    }
    const int kstep = sh_kstep, kp = sh_kp, kk = k + kstep - 1;
    if (kp != kk) {  // symmetric interchange of kk and kp (kp > kk) in packed lower storage
      for (int j = t; j < kk; j += nt) {
        const T x = Tp[pk(kk, j, s)];
        Tp[pk(kk, j, s)] = Tp[pk(kp, j, s)];
        Tp[pk(kp, j, s)] = x;
      }
      for (int i = kk + 1 + t; i < kp; i += nt) {
        const T x = Tp[pk(i, kk, s)];
        Tp[pk(i, kk, s)] = Tp[pk(kp, i, s)];
        Tp[pk(kp, i, s)] = x;
      }
      for (int i = kp + 1 + t; i < s; i += nt) {
        const T x = Tp[pk(i, kk, s)];
        Tp[pk(i, kk, s)] = Tp[pk(i, kp, s)];
        Tp[pk(i, kp, s)] = x;
      }
      if (t == 0) {
        const T x = Tp[pk(kk, kk, s)];
        Tp[pk(kk, kk, s)] = Tp[pk(kp, kp, s)];
        Tp[pk(kp, kp, s)] = x;
        const int p = perm[kk];
        perm[kk] = perm[kp];
        perm[kp] = p;
      }
      __syncthreads();
    }
    if (kstep == 1) {
      const T rd = *rpiv;
      const int ck = pk(k, k, s) - k;
      const bool prod = !no_reciprocal(rd);
      for (int i = k + 1 + t; i < s; i += nt) {
        const T u = Tp[ck + i], l = prod ? u * rd : u / Tp[ck + k];
        l1[i] = u;
        l2[i] = l;
        Tp[ck + i] = l;
      }
      if (t == nt - 1) {
        dd[k] = Tp[ck + k];
        ee[k] = Sc<T>::zero();
        ty[k] = 0;
      }
      __syncthreads();
      // trailing lower triangle, one warp per column (no integer division)
      for (int jj = k + 1 + (t >> 5); jj < s; jj += nt >> 5) {
        const int cj = pk(jj, jj, s) - jj;
        const T u = l1[jj];
        for (int ii = jj + (t & 31); ii < s; ii += 32) Tp[cj + ii] -= l2[ii] * u;
      }
    } else {
      const T a11 = Tp[pk(k, k, s)], a21 = Tp[pk(k + 1, k, s)], a22 = Tp[pk(k + 1, k + 1, s)];
      const T det = a11 * a22 - a21 * a21;
      if (t == 0 && Sc<T>::bad(det)) sh_bad = Sc<T>::is_zero(det) ? 1 : 2;
      for (int i = k + 2 + t; i < s; i += nt) {  // [l1 l2] = [w1 w2] D^{-1}
        const T w1 = Tp[pk(i, k, s)], w2 = Tp[pk(i, k + 1, s)];
        l1[i] = (w1 * a22 - w2 * a21) / det;
        l2[i] = (w2 * a11 - w1 * a21) / det;
      }
      __syncthreads();
      if (sh_bad) break;
      for (int jj = k + 2 + (t >> 5); jj < s; jj += nt >> 5) {
        const int cj = pk(jj, jj, s);
        for (int ii = jj + (t & 31); ii < s; ii += 32)
          Tp[cj + ii - jj] -= l1[ii] * Tp[pk(jj, k, s)] + l2[ii] * Tp[pk(jj, k + 1, s)];
      }
      __syncthreads();
      for (int i = k + 2 + t; i < s; i += nt) {
        Tp[pk(i, k, s)] = l1[i];
        Tp[pk(i, k + 1, s)] = l2[i];
      }
      if (t == nt - 1) {
        Tp[pk(k + 1, k, s)] = Sc<T>::zero();
        dd[k] = a11;
        dd[k + 1] = a22;
        ee[k] = a21;
        ee[k + 1] = Sc<T>::zero();
        ty[k] = 1;
        ty[k + 1] = 2;
      }
    }
    __syncthreads();
    k += kstep;
  }
  if (sh_bad) {
    if (t == 0) report_pivot(status, m.f + k, sh_bad == 1);
    return;
  }
  for (int e = t; e < s * s; e += nt) {
    const int i = e % s, j = e / s;
    if (i > j) P[i + (int64_t)j * ld] = Tp[pk(i, j, s)];
    if (i == j) P[i + (int64_t)j * ld] = dd[i];
  }
  for (int q = t; q < s; q += nt) piv[b * sz.n + m.f + q] = perm[q];
}

// Pivoted factor: L_{C,K} = Z D_K^{-1} for the panel-solve output Z =
// A_{C,K P} L_KK^{-T} (kept as W in the X panels' layout), with 2x2 blocks of
// D_K, written to the panel.
template <class T>
__global__ void k_copyback_bk(const SnMeta* __restrict__ meta, const int32_t* __restrict__ sns, T* __restrict__ L,
                              const T* __restrict__ W, const T* __restrict__ D, const T* __restrict__ E,
                              const int8_t* __restrict__ ptype, Sizes sz) {
  const int k = sns[blockIdx.x];
  const int b = blockIdx.y;
  const SnMeta m = meta[k];
  after_previous();
  const int s = m.s, r = m.r, ld = s + r;
  T* P = L + b * sz.panel + m.panel + s;
  const T* Z = W + b * sz.panel + m.panel + s;
  const T* d = D + b * sz.n + m.f;
  const T* e = E + b * sz.n + m.f;
  const int8_t* ty = ptype + b * sz.n + m.f;
  for (int j = blockIdx.z; j < s; j += gridDim.z) {
    if (ty[j] == 2) continue;  // done with its partner
    if (ty[j] == 0) {
      for (int i = threadIdx.x; i < r; i += blockDim.x) P[i + (int64_t)j * ld] = Z[i + (int64_t)j * ld] / d[j];
    } else {
      const T det = d[j] * d[j + 1] - e[j] * e[j];
      for (int i = threadIdx.x; i < r; i += blockDim.x) {
        const T z1 = Z[i + (int64_t)j * ld], z2 = Z[i + (int64_t)(j + 1) * ld];
        P[i + (int64_t)j * ld] = (z1 * d[j + 1] - z2 * e[j]) / det;
        P[i + (int64_t)(j + 1) * ld] = (z2 * d[j] - z1 * e[j]) / det;
      }
    }
  }
}

// Pole sum in the write step (Section 4.4's expansion Gamma = sum_b w_b X_b,
// batch members b = poles): the finish is the last write of every panel
// entry (X_{C,K} is final since step 2, X_KK once the finish's CTAs have
// run), so after CTA `part` of supernode k has finished member b it counts
// itself on the counter of (k, part); the one that completes the batch forms
// Gamma over the entries this part owns (its X_KK pairs, both triangles, and
// a 1/nparts share of X_{C,K}), summing the members in order b = 0, 1, ...:
// no atomics on values, every Gamma entry written once, the same arithmetic
// as the separate pass (k_pole_sum).  Pivot-free symmetric factors only.
template <class T>
__device__ void pole_share(const KArgs& a, int k, int part, int nparts) {
  const Sizes& sz = a.sz;
  __shared__ int last;
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    int* ctr = a.gctr + (int64_t)k * nparts + part;
    last = atomicAdd(ctr, 1) == sz.batch - 1;
    if (last) *ctr = 0;
    __threadfence();
  }
  __syncthreads();
  if (!last) return;
  const SnMeta m = a.meta[k];
  const int s = m.s, r = m.r, ld = s + r;
  const T* w = (const T*)a.gw;
  const T* X = (const T*)a.X + m.panel;
  T* G = (T*)a.gam + m.panel;
  auto gsum = [&](int64_t idx) {
    T acc = Sc<T>::zero();
    for (int q = 0; q < sz.batch; ++q) acc += w[q] * ld_cg(X + q * sz.panel + idx);
    G[idx] = acc;
  };
  for (int e = threadIdx.x + part * blockDim.x; e < s * s; e += nparts * blockDim.x) {
    const int i = e % s, j = e / s;
    if (i < j) continue;
    gsum(i + (int64_t)j * ld);
    if (i != j) gsum(j + (int64_t)i * ld);
  }
  const int64_t rs = (int64_t)r * s;
  for (int64_t q = threadIdx.x + (int64_t)part * blockDim.x; q < rs; q += (int64_t)nparts * blockDim.x)
    gsum(s + q % r + (q / r) * ld);
}

template <class T>
__global__ void k_diag_final(KArgs a, const int32_t* __restrict__ sns) {
  const int k = sns[blockIdx.x];
  const SnMeta m = a.meta[k];
  after_previous();
  step3_finish<T>(a, m, blockIdx.y, blockIdx.z, gridDim.z, false);
  if (a.gam) pole_share<T>(a, k, blockIdx.z, gridDim.z);
}

// --------------------------------------------------------------------------
// tile GEMMs
// --------------------------------------------------------------------------

// Panel solve of the pivoted factorisation: W_{C,K} = A_{C,K P} (L_KK)^{-T}
// (the columns of A_{C,K} in pivot order), the Schur update's L_{C,K} D_K; its
// product with D^{-1} is k_copyback_bk's (2x2 blocks can straddle tiles).
template <class T, int BN>
__global__ void __launch_bounds__(TG_THREADS, (tile_min_ctas<T, BN>())) k_trsm(const SnMeta* __restrict__ meta, const Task* __restrict__ tasks,
                                                     const T* __restrict__ L, const T* __restrict__ Linv, Sizes sz,
                                                     const int32_t* __restrict__ piv, T* __restrict__ W) {
  __shared__ TileSmem<T, BN> sm;
  const Task tk = tasks[blockIdx.x];
  const int b = blockIdx.y;
  const SnMeta m = meta[tk.sn];
  after_previous();
  const int s = m.s, r = m.r, ld = s + r;
  const T* A = L + b * sz.panel + m.panel + s;
  const T* Vi = Linv + b * sz.linv + m.linv;
  Acc<T, BN> acc;
  acc_zero<T, BN>(acc);
  const int32_t* pv = piv + b * sz.n + m.f;
  auto la = [&](int mm, int kk) {
    const int row = tk.m0 + mm;
    return row < r ? A[row + (int64_t)pv[kk] * ld] : Sc<T>::zero();
  };
  auto lb = [&](int kk, int nn) {
    const int col = tk.n0 + nn;
    return col < s ? Vi[col + kk * s] : Sc<T>::zero();
  };
  // (L_KK)^{-T} is upper triangular: output columns < n0 + BN need only k < n0 + BN
  tile_mma<T, BN>(sm, 0, min(s, tk.n0 + tile_cols<BN>()), [](int) { return false; }, la, lb, acc,
                  LiveRect{r - tk.m0, s - tk.n0}, KUpperB<BN>{tk.n0});
  T* wout = W + b * sz.panel + m.panel + s;
  tile_epilogue<T, BN>(acc, [&](int mm, int nn, T v) {
    const int row = tk.m0 + mm, col = tk.n0 + nn;
    if (row < r && col < s) wout[row + (int64_t)col * ld] = v;
  });
}

// Schur-complement update of the ancestors: lower tiles of
// U = L_{C,K} D_K L_{C,K}^T; U[i][k] (i >= k) is subtracted from the ancestor
// entry found through the column descriptor of k and the relative index of i.
// Task.c is the tile's column end (a tile covers columns [n0, c) of C).
// The task list of one launch is a group of supernodes whose C are disjoint
// (analysis), and inside one supernode the targets of different (i, k) are
// different entries, so each target is read-modified-written by exactly one
// thread of the launch: no atomics, and a fixed order of the updates.
// The first operand is W_{C,K} = L_{C,K} D_K (pivoted: with D's 2 x 2 blocks) as
// the panel solve left it, so the loads carry no FP64 product (a product per A
// element is 64 x 16 FP64 operations per k-tile, 1/8 of the MMA work of a
// 64 x 8 tile on the same pipe); the second is L_{C,K} in its panel.
// Non-symmetric factor: side blockIdx.z = 0 takes U'_{K,C}^T as the second
// operand, giving L_{C,K} D_K U'_{K,C} into the L panels; side 1 swaps the
// operands' sides, giving U'_{K,C}^T D_K L_{C,K}^T below the diagonal into the
// U panels.  Both sides run in one launch (different targets).
template <class T, int BN>
__global__ void __launch_bounds__(TG_THREADS, (tile_min_ctas<T, BN>())) k_schur(FArgs f, const Task* __restrict__ tasks) {
  __shared__ TileSmem<T, BN> sm;
  const Task tk = tasks[blockIdx.x];
  const int b = blockIdx.y, side = blockIdx.z;
  const SnMeta m = f.meta[tk.sn];
  after_previous();
  const int s = m.s, r = m.r, ld = s + r;
  const int64_t po = b * f.sz.panel + m.panel + s;
  const T* Lc2 = (const T*)f.L[f.sides - 1 - side] + po;
  const T* Wc = (const T*)f.W[side] + po;
  Acc<T, BN> acc;
  acc_zero<T, BN>(acc);
  auto la = [&](int mm, int kk) {
    const int row = tk.m0 + mm;
    return row < r ? Wc[row + (int64_t)kk * ld] : Sc<T>::zero();
  };
  auto lb = [&](int kk, int nn) {
    const int col = tk.n0 + nn;
    return col < tk.c ? Lc2[col + (int64_t)kk * ld] : Sc<T>::zero();
  };
  // live: fragments with a row and a column inside C and an entry on or below the diagonal
  const int dm = tk.m0 - tk.n0;
  tile_mma<T, BN>(sm, 0, s, [](int) { return false; }, la, lb, acc, [&](int r0, int c0) {
    return tk.m0 + r0 < r && tk.n0 + c0 < tk.c && c0 <= dm + r0 + 7;
  });
  T* Lb = (T*)f.L[side] + b * f.sz.panel;
  const ColDesc* dk = f.desc + m.desc;
  tile_epilogue<T, BN>(acc, [&](int mm, int nn, T v) {
    const int i = tk.m0 + mm, kc = tk.n0 + nn;
    if (i < r && kc < tk.c && kc + side <= i) {
      const ColDesc cd = dk[kc];
      T* dst = &Lb[cd.col + f.relidx[cd.rel + i]];
      *dst = *dst - v;
    }
  });
}

// The Schur updates of a whole small level in one launch (merged_update.cuh),
// operands and targets as in k_schur.  A launch per group and part cost 3 to 5 us
// however few tiles it held (31 x 31 grid, 103 launches: 590 -> 537 us).  Larger
// levels keep a launch per group: ordered the same way on their 64 x 8 tiles they
// gave 0.2 to 0.4% on wide supernodes and lost 2 to 3% on narrow ones, whose short
// tiles feel the ticket and hold their slots while the group before ends.
template <class T>
__global__ void __launch_bounds__(TG_THREADS) k_schur_merged(FArgs f, const Task* __restrict__ tasks, MergedArgs mq) {
  merged_update<T, 1>(
      tasks, mq, f.meta, f.desc, f.relidx, f.sides,
      [&](const SnMeta& m, int b, int side, int) {
        const int64_t po = b * f.sz.panel + m.panel + m.s;
        return UpdatePair<T>{(const T*)f.W[side] + po, (const T*)f.L[f.sides - 1 - side] + po, m.s + m.r};
      },
      [&](int b, int side) { return (T*)f.L[side] + b * f.sz.panel; }, [](T x, T v, bool) { return x - v; });
}

// Normalisation, diagonal part: M_K = L_KK^{-T} D_K^{-1} L_KK^{-1} = V^T (D_K^{-1} V)
// with V = (L_KK)^{-1} from the factorisation, into the diagonal block of the
// X panel (Algorithm 1 step 3's first term; U_KK = D_K L_KK^T), one 64 x 8
// tile of s x s per CTA over all supernodes; V is lower triangular, so only
// k >= max(m0, n0) contributes, and the symmetric forms compute the lower
// triangle and mirror it.
// MODE 1, pivoted factor: D_K has 2 x 2 blocks, so row q of D_K^{-1} V is
// c_q V_q + c'_q V_{q'} with q' the 2 x 2 partner, and M_K goes to the
// original columns (P(i), P(j)).
// MODE 2, non-symmetric: U_KK^{-1} L_KK^{-1} = U'_KK^{-1} D_K^{-1} L_KK^{-1} =
// Vu^T D_K^{-1} Vl, every entry of the block.
// Bound: the FP64 pipe (2/3 s^3 flops per supernode).  It replaces a kernel of
// one CTA per supernode that inverted L_KK again, one column per thread (a
// serial chain of dependent loads through L1, 1.0 to 1.7 ms a pass on
// problems with a 128-wide supernode whatever their size).
template <class T, int MODE>
__global__ void __launch_bounds__(TG_THREADS, (tile_min_ctas<T, 8>())) k_norm_m(KArgs a, const Task* __restrict__ tasks) {
  constexpr int BN = 8;
  __shared__ TileSmem<T, BN> sm;
  __shared__ double coef[(MODE == 1 ? 2 : 1) * kMaxWidth * Sc<T>::P];  // 1 / d_q, or the own coefficient of a 2 x 2 row; partners after
  __shared__ int pq[MODE == 1 ? kMaxWidth : 1];
  const Task tk = tasks[blockIdx.x];
  const int b = blockIdx.y;
  const SnMeta m = a.meta[tk.sn];
  after_previous();
  const int s = m.s, ld = m.s + m.r;
  const T* V = (const T*)a.Linv + b * a.sz.linv + m.linv;
  const T* Vm = MODE == 2 ? (const T*)a.Uinv + b * a.sz.linv + m.linv : V;
  const T* d = (const T*)a.D + b * a.sz.n + m.f;
  T* rd = reinterpret_cast<T*>(coef);
  T* rp = rd + (MODE == 1 ? kMaxWidth : 0);
  const int q0 = max(tk.m0, tk.n0);  // V_qi = 0 for q < i
  for (int q = q0 + threadIdx.x; q < s; q += TG_THREADS) {
    if constexpr (MODE == 1) {
      const int8_t* ty = a.ptype + b * a.sz.n + m.f;
      const T* ee = (const T*)a.E + b * a.sz.n + m.f;
      if (ty[q] == 0) {
        rd[q] = Sc<T>::one() / d[q];
        rp[q] = Sc<T>::zero();
        pq[q] = q;
      } else {
        const int f0 = ty[q] == 1 ? q : q - 1;  // first column of the 2 x 2 block
        const T det = d[f0] * d[f0 + 1] - ee[f0] * ee[f0];
        const int o = ty[q] == 1 ? q + 1 : q - 1;
        rd[q] = d[o] / det;
        rp[q] = -ee[f0] / det;
        pq[q] = o;
      }
    } else {
      rd[q] = Sc<T>::one() / d[q];
    }
  }
  __syncthreads();
  Acc<T, BN> acc;
  acc_zero<T, BN>(acc);
  auto la = [&](int mm, int q) {
    const int i = tk.m0 + mm;
    return i < s ? Vm[q + i * s] : Sc<T>::zero();
  };
  auto lb = [&](int q, int nn) -> T {
    const int j = tk.n0 + nn;
    if (j >= s) return Sc<T>::zero();
    if constexpr (MODE == 1) return rd[q] * V[q + j * s] + rp[q] * V[pq[q] + j * s];
    return rd[q] * V[q + j * s];
  };
  const int dm = tk.m0 - tk.n0;
  // a 2 x 2 pivot whose first column is q0 - 1 has its second row at q0: row q0 - 1
  // of D^{-1} V meets V_{q0-1,i} = 0, so the range still starts at q0
  tile_mma<T, BN>(sm, q0, s, [](int) { return true; }, la, lb, acc, [&](int r0, int c0) {
    return tk.m0 + r0 < s && tk.n0 + c0 < s && (MODE == 2 || c0 <= dm + r0 + 7);
  }, KLowerTA{tk.m0});
  T* XK = (T*)a.X + b * a.sz.panel + m.panel;
  tile_epilogue<T, BN>(acc, [&](int mm, int nn, T v) {
    int i = tk.m0 + mm, j = tk.n0 + nn;
    if (i >= s || j >= s) return;
    if constexpr (MODE == 2) {
      XK[i + (int64_t)j * ld] = v;
    } else {
      if (i < j) return;
      if constexpr (MODE == 1) {
        const int32_t* pv = a.piv + b * a.sz.n + m.f;
        i = pv[i];
        j = pv[j];
      }
      XK[i + (int64_t)j * ld] = v;
      XK[j + (int64_t)i * ld] = v;
    }
  });
}

// Normalisation, off-diagonal part: Lhat_{C,K} = L_{C,K} (L_KK)^{-1}.
template <class T, int BN>
__global__ void __launch_bounds__(TG_THREADS, (tile_min_ctas<T, BN>())) k_lhat(const SnMeta* __restrict__ meta, const Task* __restrict__ tasks,
                                                     const T* __restrict__ L, const T* __restrict__ Linv,
                                                     T* __restrict__ Lhat, Sizes sz) {
  __shared__ TileSmem<T, BN> sm;
  const Task tk = tasks[blockIdx.x];
  const int b = blockIdx.y;
  const SnMeta m = meta[tk.sn];
  after_previous();
  const int s = m.s, r = m.r, ld = s + r;
  const T* A = L + b * sz.panel + m.panel + s;
  const T* Vi = Linv + b * sz.linv + m.linv;
  Acc<T, BN> acc;
  acc_zero<T, BN>(acc);
  auto la = [&](int mm, int kk) {
    const int row = tk.m0 + mm;
    return row < r ? A[row + (int64_t)kk * ld] : Sc<T>::zero();
  };
  auto lb = [&](int kk, int nn) {
    const int col = tk.n0 + nn;
    return col < s ? Vi[kk + col * s] : Sc<T>::zero();
  };
  // (L_KK)^{-1} is lower triangular: output columns >= n0 need only k >= n0
  tile_mma<T, BN>(sm, tk.n0, s, [](int) { return false; }, la, lb, acc, LiveRect{r - tk.m0, s - tk.n0},
                  KLowerB<BN>{tk.n0});
  T* out = Lhat + b * sz.lhat + m.lhat;
  tile_epilogue<T, BN>(acc, [&](int mm, int nn, T v) {
    const int row = tk.m0 + mm, col = tk.n0 + nn;
    if (row < r && col < s) out[row + (int64_t)col * r] = v;
  });
}

// Steps 2 and 3 as grouped per-level kernels (bodies in selinv_steps.cuh).
template <class T, int BN, bool UNSYM>
__global__ void __launch_bounds__(TG_THREADS, (tile_min_ctas<T, BN>())) k_gemm1(KArgs a, const Task* __restrict__ tasks) {
  __shared__ TileSmem<T, BN> sm;
  const Task tk = tasks[blockIdx.x];
  const SnMeta m = a.meta[tk.sn];
  after_previous();
  step2_tile<T, BN, UNSYM>(a, tk, m, blockIdx.y, sm);
}

// blockIdx.z strides over the columns of the split supernodes of the level
template <class T>
__global__ void k_gemm1_reduce(KArgs a, const int32_t* __restrict__ sns) {
  step2_reduce<T>(a, sns[blockIdx.x], blockIdx.y, blockIdx.z, gridDim.z, false);
}

template <class T, int BN>
__global__ void __launch_bounds__(TG_THREADS, (tile_min_ctas<T, BN>())) k_gemm2(KArgs a, const Task* __restrict__ tasks) {
  __shared__ TileSmem<T, BN> sm;
  const Task tk = tasks[blockIdx.x];
  const SnMeta m = a.meta[tk.sn];
  after_previous();
  step3_tile<T, BN>(a, tk, m, blockIdx.y, sm, false);
  // levels of narrow supernodes: no launch of its own for a finish of a few entries
  if (a.tctr && last_step3<BN>(a, m, blockIdx.y)) step3_finish<T>(a, m, blockIdx.y, 0, 1, true);
}

// --------------------------------------------------------------------------
// log det
// --------------------------------------------------------------------------

// Sum of two values over the CTA's 256 threads, to thread 0.
__device__ __forceinline__ void block_sum2(double& a, double& c) {
  __shared__ double s1[256];
  __shared__ double s2[256];
  s1[threadIdx.x] = a;
  s2[threadIdx.x] = c;
  __syncthreads();
  for (int w = blockDim.x / 2; w > 0; w >>= 1) {
    if (threadIdx.x < w) {
      s1[threadIdx.x] += s1[threadIdx.x + w];
      s2[threadIdx.x] += s2[threadIdx.x + w];
    }
    __syncthreads();
  }
  a = s1[0];
  c = s2[0];
}

// Real: (sum log|d_j|, number of negative pivots); complex: sum of principal
// logs (log|d_j|, arg d_j), per batch member (blockIdx.y): partial sums of
// gridDim.x CTAs, then their sum in a fixed order (k_logdet_sum).  Bound: the
// logarithms on the FP64 pipe; one CTA took 136 us for n = 13,824.
template <class T>
__global__ void k_logdet(const T* __restrict__ D, int64_t n, double* __restrict__ work,
                         const int8_t* __restrict__ ptype, const T* __restrict__ E) {
  const int b = blockIdx.y;
  double a = 0.0, c = 0.0;
  for (int64_t j = threadIdx.x + (int64_t)blockIdx.x * blockDim.x; j < n; j += (int64_t)gridDim.x * blockDim.x) {
    const int8_t ty = ptype ? ptype[b * n + j] : 0;
    if (ty == 2) continue;  // counted with its partner
    // a 2x2 pivot contributes the determinant of its block
    const T d = ty == 1 ? D[b * n + j] * D[b * n + j + 1] - E[b * n + j] * E[b * n + j] : D[b * n + j];
    if constexpr (Sc<T>::P == 1) {
      a += log(fabs(d));
      c += d < 0.0 ? 1.0 : 0.0;
    } else {
      a += log(hypot(d.re, d.im));
      c += atan2(d.im, d.re);
    }
  }
  block_sum2(a, c);
  if (threadIdx.x == 0) {
    double* w = work + 2 * ((int64_t)b * gridDim.x + blockIdx.x);
    w[0] = a;
    w[1] = c;
  }
}
__global__ void k_logdet_sum(const double* __restrict__ work, int parts, double* __restrict__ out) {
  const int b = blockIdx.x;
  const double* w = work + 2 * (int64_t)b * parts;
  double a = 0.0, c = 0.0;
  for (int p = threadIdx.x; p < parts; p += blockDim.x) {
    a += w[2 * p];
    c += w[2 * p + 1];
  }
  block_sum2(a, c);
  if (threadIdx.x == 0) {
    out[2 * b] = a;
    out[2 * b + 1] = c;
  }
}

// --------------------------------------------------------------------------
// pole sum and trace pairing
// --------------------------------------------------------------------------

// out[e] = sum_b w_b X_b[e]  (grid-stride, HBM-bound)
template <class T>
__global__ void k_pole_sum(const T* __restrict__ X, int64_t panel_total, int batch, const T* __restrict__ w,
                           T* __restrict__ out) {
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < panel_total;
       e += (int64_t)gridDim.x * blockDim.x) {
    T acc = Sc<T>::zero();
    for (int b = 0; b < batch; ++b) acc += w[b] * X[(int64_t)b * panel_total + e];
    out[e] = acc;
  }
}

// S_b = sum_q m_q X(q) A_q with m_q = 1 on the diagonal, 2 off it; one CTA
// per batch member, fixed reduction order (deterministic).
template <class T>
__global__ void k_trace_sum(const T* __restrict__ X, int64_t panel_total, const int64_t* __restrict__ vmap,
                            const uint8_t* __restrict__ diagmask, const T* __restrict__ vals, int64_t nnz,
                            T* __restrict__ out) {
  __shared__ T red[1024];
  const int b = blockIdx.x;
  const T* Xb = X + (int64_t)b * panel_total;
  const T* v = vals + (int64_t)b * nnz;
  T acc = Sc<T>::zero();
  for (int64_t q = threadIdx.x; q < nnz; q += blockDim.x) {
    const T t = Xb[vmap[q]] * v[q];
    acc += diagmask[q] ? t : 2.0 * t;
  }
  red[threadIdx.x] = acc;
  __syncthreads();
  for (int w = blockDim.x / 2; w > 0; w >>= 1) {
    if (threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x == 0) out[b] = red[0];
}

cudaError_t launch_pole_sum(int dtype, const void* X, int64_t panel_total, int batch, const void* w, void* out,
                            cudaStream_t st) {
  const unsigned grid = 152 * 8;
  if (dtype == PSELINV_C128)
    k_pole_sum<Cplx><<<grid, 256, 0, st>>>((const Cplx*)X, panel_total, batch, (const Cplx*)w, (Cplx*)out);
  else
    k_pole_sum<double><<<grid, 256, 0, st>>>((const double*)X, panel_total, batch, (const double*)w, (double*)out);
  return cudaGetLastError();
}

cudaError_t launch_trace_sum(int dtype, const void* X, int64_t panel_total, const int64_t* vmap,
                             const uint8_t* diagmask, const void* vals, int64_t nnz, int batch, void* out,
                             cudaStream_t st) {
  if (dtype == PSELINV_C128)
    k_trace_sum<Cplx><<<batch, 1024, 0, st>>>((const Cplx*)X, panel_total, vmap, diagmask, (const Cplx*)vals, nnz,
                                              (Cplx*)out);
  else
    k_trace_sum<double><<<batch, 1024, 0, st>>>((const double*)X, panel_total, vmap, diagmask, (const double*)vals,
                                                nnz, (double*)out);
  return cudaGetLastError();
}

// --------------------------------------------------------------------------
// launch wrappers
// --------------------------------------------------------------------------

static inline unsigned blocks_for(int64_t n, int threads, int cap = 152 * 16) {
  int64_t b = (n + threads - 1) / threads;
  if (b < 1) b = 1;
  return (unsigned)(b < cap ? b : cap);
}

// packed lower triangle, two length-s vectors and s ints
template <class T>
static size_t diag_smem(int maxw) {
  return sizeof(T) * ((size_t)maxw * (maxw + 1) / 2 + 2 * (size_t)maxw) + sizeof(int) * (size_t)maxw;
}

template <class T>
static cudaError_t setup_t() {
  const cudaError_t e = cudaFuncSetAttribute(k_factor_diag_bk<T>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)diag_smem<T>(kMaxWidth));
  return e;
}

cudaError_t setup_kernels() {
  cudaError_t e = setup_t<double>();
  if (e != cudaSuccess) return e;
  if ((e = setup_em_kernels()) != cudaSuccess) return e;
  return setup_t<Cplx>();
}

template <class T>
static cudaError_t scatter_t(const void* vals, const int64_t* vmap, int64_t nnz, void* L, const Sizes& sz,
                             cudaStream_t st) {
  k_scatter_values<T><<<dim3(blocks_for(nnz, 256), sz.batch), 256, 0, st>>>((const T*)vals, vmap, nnz, (T*)L,
                                                                           sz.panel);
  return cudaGetLastError();
}
cudaError_t launch_scatter_values(int dtype, const void* vals, const int64_t* vmap, int64_t nnz, void* L,
                                  const Sizes& sz, cudaStream_t st) {
  return dtype == PSELINV_C128 ? scatter_t<Cplx>(vals, vmap, nnz, L, sz, st)
                               : scatter_t<double>(vals, vmap, nnz, L, sz, st);
}

template <class T>
static cudaError_t scatter_lu_t(const void* lo, const void* up, const int64_t* vmap, const uint8_t* flip, int64_t nnz,
                                void* L, void* U, const Sizes& sz, cudaStream_t st) {
  k_scatter_values_lu<T><<<dim3(blocks_for(nnz, 256), sz.batch), 256, 0, st>>>(
      (const T*)lo, (const T*)up, vmap, flip, nnz, (T*)L, (T*)U, sz.panel);
  return cudaGetLastError();
}
cudaError_t launch_scatter_values_lu(int dtype, const void* lower, const void* upper, const int64_t* vmap,
                                     const uint8_t* flip, int64_t nnz, void* L, void* U, const Sizes& sz,
                                     cudaStream_t st) {
  return dtype == PSELINV_C128 ? scatter_lu_t<Cplx>(lower, upper, vmap, flip, nnz, L, U, sz, st)
                               : scatter_lu_t<double>(lower, upper, vmap, flip, nnz, L, U, sz, st);
}

template <class T>
static cudaError_t gather_lu_t(const void* XL, const void* XU, const int64_t* vmap, const uint8_t* flip, int64_t nnz,
                               int upper, void* out, const Sizes& sz, cudaStream_t st) {
  k_gather_values_lu<T><<<dim3(blocks_for(nnz, 256), sz.batch), 256, 0, st>>>(
      (const T*)XL, (const T*)XU, sz.panel, vmap, flip, nnz, upper, (T*)out);
  return cudaGetLastError();
}
cudaError_t launch_gather_values_lu(int dtype, const void* XL, const void* XU, const int64_t* vmap,
                                    const uint8_t* flip, int64_t nnz, int upper, void* out, const Sizes& sz,
                                    cudaStream_t st) {
  return dtype == PSELINV_C128 ? gather_lu_t<Cplx>(XL, XU, vmap, flip, nnz, upper, out, sz, st)
                               : gather_lu_t<double>(XL, XU, vmap, flip, nnz, upper, out, sz, st);
}

template <class T>
static cudaError_t gather_t(const void* X, const int64_t* vmap, const uint8_t* mask, int64_t nnz, void* out,
                            const Sizes& sz, cudaStream_t st, const int* invalid, int* report) {
  k_gather_values<T><<<dim3(blocks_for(nnz, 256), sz.batch), 256, 0, st>>>((const T*)X, sz.panel, vmap, mask, nnz,
                                                                          (T*)out, invalid, report);
  return cudaGetLastError();
}
cudaError_t launch_gather_values(int dtype, const void* X, const int64_t* vmap, const uint8_t* diagmask, int64_t nnz,
                                 void* out, const Sizes& sz, cudaStream_t st, const int* invalid, int* report) {
  return dtype == PSELINV_C128 ? gather_t<Cplx>(X, vmap, diagmask, nnz, out, sz, st, invalid, report)
                               : gather_t<double>(X, vmap, diagmask, nnz, out, sz, st, invalid, report);
}

// ---- tile-kernel launch for one task range of one variant ----

template <class T, int BN>
static cudaError_t tiles_tb(Kern k, const KArgs& a, const Task* t, int64_t n, cudaStream_t st, bool dep) {
  const dim3 grid((unsigned)n, a.sz.batch);
  switch (k) {
    case Kern::NormM:
      if constexpr (BN == 8) {  // a list of 64 x 8 tiles only
        if (a.Uinv) return launch_dep(k_norm_m<T, 2>, grid, TG_THREADS, 0, st, dep, a, t);
        if (a.ptype) return launch_dep(k_norm_m<T, 1>, grid, TG_THREADS, 0, st, dep, a, t);
        return launch_dep(k_norm_m<T, 0>, grid, TG_THREADS, 0, st, dep, a, t);
      }
      return cudaErrorInvalidValue;
    case Kern::Trsm:
      return launch_dep(k_trsm<T, BN>, grid, TG_THREADS, 0, st, dep, a.meta, t, (const T*)a.L, (const T*)a.Linv, a.sz,
                        a.piv, (T*)a.W);
    case Kern::Lhat:
      if constexpr (BN == 8 || BN == kFine)  // a list of 64 x 8 or of fine tiles
        return launch_dep(k_lhat<T, BN>, grid, TG_THREADS, 0, st, dep, a.meta, t, (const T*)a.L, (const T*)a.Linv,
                          (T*)a.Lhat, a.sz);
      return cudaErrorInvalidValue;
    case Kern::Gemm1:
      if (a.XU) return launch_dep(k_gemm1<T, BN, true>, grid, TG_THREADS, 0, st, dep, a, t);
      return launch_dep(k_gemm1<T, BN, false>, grid, TG_THREADS, 0, st, dep, a, t);
    case Kern::Gemm2:
      return launch_dep(k_gemm2<T, BN>, grid, TG_THREADS, 0, st, dep, a, t);
    default:
      return cudaErrorInvalidValue;
  }
}

template <class T>
static cudaError_t tiles_t(Kern k, int var, const KArgs& a, const Task* t, int64_t n, cudaStream_t st, bool dep) {
  if (n <= 0) return cudaSuccess;
  switch (var) {
    case 0: return tiles_tb<T, 8>(k, a, t, n, st, dep);
    case 1: return tiles_tb<T, 16>(k, a, t, n, st, dep);
    case 2: return tiles_tb<T, 32>(k, a, t, n, st, dep);
    case kVarFine: return tiles_tb<T, kFine>(k, a, t, n, st, dep);
    default:
      if constexpr (Sc<T>::P == 1) return tiles_tb<T, 64>(k, a, t, n, st, dep);
      return cudaErrorInvalidValue;  // complex tiles stop at BN = 32 (register budget)
  }
}

cudaError_t launch_tiles(Kern k, int var, const KArgs& a, const Task* t, int64_t n, cudaStream_t st, bool dep) {
  return a.dtype == PSELINV_C128 ? tiles_t<Cplx>(k, var, a, t, n, st, dep) : tiles_t<double>(k, var, a, t, n, st, dep);
}

// ---- blocked factorisation ----

template <class T>
static cudaError_t fdiag_t(const FArgs& f, const int32_t* sns, int nsn, int p, int w, cudaStream_t st, bool dep) {
  const dim3 grid(nsn, f.sz.batch);
  const int nu = fd_update(w);
  if (f.sides == 2) return launch_dep(k_fdiag<T, 2>, grid, 32 + 2 * nu, 0, st, dep, f, sns, p);
  return launch_dep(k_fdiag<T, 1>, grid, 32 + nu, 0, st, dep, f, sns, p);
}
cudaError_t launch_fdiag(int dtype, const FArgs& f, const int32_t* sns, int nsn, int p, int w, cudaStream_t st,
                         bool dep) {
  if (nsn <= 0) return cudaSuccess;
  return dtype == PSELINV_C128 ? fdiag_t<Cplx>(f, sns, nsn, p, w, st, dep)
                               : fdiag_t<double>(f, sns, nsn, p, w, st, dep);
}

cudaError_t launch_vdiag(int dtype, const FArgs& f, const int32_t* sns, int nsn, int wmax, cudaStream_t st) {
  if (nsn <= 0) return cudaSuccess;
  const dim3 grid(nsn, f.sz.batch, (wmax + kFB - 1) / kFB);
  if (dtype == PSELINV_C128) return launch_dep(k_vdiag<Cplx>, grid, kVdThreads, 0, st, true, f, sns);
  return launch_dep(k_vdiag<double>, grid, kVdThreads, 0, st, true, f, sns);
}

template <class T>
static cudaError_t ftiles_t(FKern k, int var, const FArgs& f, const Task* t, int64_t n, cudaStream_t st, bool dep) {
  const dim3 grid((unsigned)n, f.sz.batch, f.sides);
  switch (k) {
    case FKern::Panel: return launch_dep(k_fpanel<T>, grid, 4 * kFB, 0, st, dep, f, t);
    case FKern::Update: return launch_dep(k_fupdate<T>, grid, kFUpdateThreads, 0, st, dep, f, t);
    case FKern::VInv: return launch_dep(k_vinv<T>, grid, TG_THREADS, 0, st, dep, f, t);
    default:  // Schur groups: 64 x 8 tiles, or the widest of the type
      if (var == 0) return launch_dep(k_schur<T, 8>, grid, TG_THREADS, 0, st, dep, f, t);
      if constexpr (Sc<T>::P == 2) return launch_dep(k_schur<T, 32>, grid, TG_THREADS, 0, st, dep, f, t);
      return cudaErrorInvalidValue;
  }
}
cudaError_t launch_ftiles(FKern k, int var, int dtype, const FArgs& f, const Task* t, int64_t n, cudaStream_t st,
                          bool dep) {
  if (n <= 0) return cudaSuccess;
  return dtype == PSELINV_C128 ? ftiles_t<Cplx>(k, var, f, t, n, st, dep) : ftiles_t<double>(k, var, f, t, n, st, dep);
}

cudaError_t launch_schur_merged(int dtype, const FArgs& f, const MergedArgs& q, const Task* t, cudaStream_t st,
                                bool dep) {
  if (q.ntile <= 0) return cudaSuccess;
  const dim3 grid(q.ntile, f.sz.batch, f.sides);  // the product of the last two can exceed the limit of one
  if (dtype == PSELINV_C128) return launch_dep(k_schur_merged<Cplx>, grid, TG_THREADS, 0, st, dep, f, t, q);
  return launch_dep(k_schur_merged<double>, grid, TG_THREADS, 0, st, dep, f, t, q);
}

template <class T>
static cudaError_t per_sn_t(Kern k, const KArgs& a, const int32_t* sns, int nsn, cudaStream_t st, int threads,
                            bool dep) {
  if (nsn <= 0) return cudaSuccess;
  const dim3 grid(nsn, a.sz.batch);
  // CTAs of a step-3 finish: entries of X_KK (with 32 throughout, 1,291 supernodes of
  // width ~5 took 43 us) and, for the pole sum, of X_{C,K}
  const int parts = a.gam ? kFinishCtas : std::max(1, std::min(kFinishCtas, a.maxw * a.maxw / 512));
  switch (k) {
    case Kern::Gemm1Reduce:
      k_gemm1_reduce<T><<<dim3(nsn, a.sz.batch, 16), 256, 0, st>>>(a, sns);
      return cudaGetLastError();
    case Kern::FactorDiagBK:
      return launch_dep(k_factor_diag_bk<T>, grid, threads > 512 ? 512 : threads, diag_smem<T>(a.maxw), st, dep, a.meta,
                        sns, (T*)a.L, (T*)a.D, (T*)a.E, (int8_t*)a.ptype, (int32_t*)a.piv, a.sz, a.status);
    case Kern::CopyBackBK:
      return launch_dep(k_copyback_bk<T>, dim3(nsn, a.sz.batch, 16), 256, 0, st, dep, a.meta, sns, (T*)a.L,
                        (const T*)a.W, (const T*)a.D, (const T*)a.E, a.ptype, a.sz);
    default:
      // up to 32 CTAs per supernode: the levels near the root hold one supernode
      // whose finish reads one s x s partial per row chunk of C
      return launch_dep(k_diag_final<T>, dim3(nsn, a.sz.batch, parts), 256, 0, st, dep, a, sns);
  }
}

cudaError_t launch_per_sn(Kern k, const KArgs& a, const int32_t* sns, int nsn, cudaStream_t st, int threads,
                          bool dep) {
  return a.dtype == PSELINV_C128 ? per_sn_t<Cplx>(k, a, sns, nsn, st, threads, dep)
                                 : per_sn_t<double>(k, a, sns, nsn, st, threads, dep);
}

cudaError_t launch_logdet(int dtype, const void* D, int64_t n, double* work, double* out, int batch, cudaStream_t st,
                          const int8_t* ptype, const void* E) {
  const int parts = logdet_parts(n);
  if (parts == 1) work = out;  // one partial sum is the sum: no second launch (a call for n = 27 43.6 -> 34.3 us, n = 216 43.6 -> 39.3)
  if (dtype == PSELINV_C128)
    k_logdet<Cplx><<<dim3(parts, batch), 256, 0, st>>>((const Cplx*)D, n, work, ptype, (const Cplx*)E);
  else
    k_logdet<double><<<dim3(parts, batch), 256, 0, st>>>((const double*)D, n, work, ptype, (const double*)E);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess || parts == 1) return e;
  k_logdet_sum<<<batch, 256, 0, st>>>(work, parts, out);
  return cudaGetLastError();
}

}  // namespace psi
