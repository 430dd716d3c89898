// The updates of the ancestors by a whole level in one launch: the tiles of all its
// Schur groups, 16 x 8, in group order (factorisation: k_schur_merged; adjoint:
// k_syr2k_merged).  Targets of different groups overlap, so a tile's
// read-modify-write waits until the groups before its own have finished (same
// order per target as a launch per group, so the same bits); the products do not
// wait.  CTAs take their tile by a ticket: the holder of a tile only waits on
// tiles with lower tickets, which running CTAs hold, and those of the lowest
// group wait on nothing, so the waits end whatever else is resident; each is
// bounded in time all the same (bounded_wait.cuh).
// Warp w computes the k range [w kq, (w + 1) kq) of the tile from fragments loaded
// straight to registers; the four partial sums are added in warp order.
// Bound: latency (loads, at most 16 MMAs a warp and product, the group order).
#pragma once

#include "bounded_wait.cuh"
#include "kernels.h"
#include "selinv_steps.cuh"
#include "tile_gemm.cuh"

namespace psi {

// One product of the update: A (rows of C x s) B^T (columns of C x s), both
// column-major.
template <class T>
struct UpdatePair {
  const T* a;
  const T* b;
  int64_t ld;
};

// pairs(m, b, side, p): operands of product p < NP.  target(b, side): the panels
// updated.  apply(x, v, diag): the new value of a target x given the products' sum.
template <class T, int NP, class PAIRS, class TARGET, class APPLY>
__device__ __forceinline__ void merged_update(const Task* __restrict__ tasks, const MergedArgs& mq,
                                              const SnMeta* __restrict__ meta, const ColDesc* __restrict__ desc,
                                              const int32_t* __restrict__ relidx, int sides, const PAIRS& pairs,
                                              const TARGET& target, const APPLY& apply) {
  constexpr int P = Sc<T>::P, RF = kMergedRows / 8, LDP = kMergedRows + 1, KW = 32;
  __shared__ double part[4][P][8][LDP];
  __shared__ int sh_ticket;
  if (threadIdx.x == 0) sh_ticket = atomicAdd(mq.ticket, 1);  // zeroed before the chain's first kernel
  __syncthreads();
  const int ticket = sh_ticket, copies = gridDim.y * gridDim.z, copy = ticket % copies;
  const Task tk = tasks[ticket / copies];
  const int side = copy % sides, b = copy / sides;
  const int grp = tk.c >> kMergedShift, cend = tk.c & ((1 << kMergedShift) - 1);
  const SnMeta m = meta[tk.sn];
  const int s = m.s, r = m.r;
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5, g = lane >> 2, q = lane & 3;
  // this thread's entry of the tile and its target
  const int ei = tk.m0 + t % kMergedRows, ec = tk.n0 + t / kMergedRows;
  const bool live = ei < r && ec < cend && ec + side <= ei;
  T* dst = nullptr;
  if (live) {
    const ColDesc cd = desc[m.desc + ec];
    dst = target(b, side) + cd.col + relidx[cd.rel + ei];
  }
  const int need = grp > 0 ? mq.gcnt[grp - 1] : 0;
  after_previous();
  double acc[RF][P][2] = {};
  const int kq = (s + 15) / 16 * 4, k0 = warp * kq, k1 = min(s, k0 + kq);  // at most KW
  if (k0 < k1) {
#pragma unroll
    for (int p = 0; p < NP; ++p) {
      const UpdatePair<T> pr = pairs(m, b, side, p);
      T fa[RF][KW / 4], fb[KW / 4];
#pragma unroll
      for (int u = 0; u < KW / 4; ++u) {
        const int k = k0 + 4 * u + q;
        const bool on = k < k1;
        fb[u] = on && tk.n0 + g < cend ? pr.b[tk.n0 + g + k * pr.ld] : Sc<T>::zero();
#pragma unroll
        for (int h = 0; h < RF; ++h) {
          const int row = tk.m0 + 8 * h + g;
          fa[h][u] = on && row < r ? pr.a[row + k * pr.ld] : Sc<T>::zero();
        }
      }
#pragma unroll
      for (int h = 0; h < RF; ++h) {
        if (tk.m0 + 8 * h >= r) continue;
#pragma unroll
        for (int u = 0; u < KW / 4; ++u)
          if (k0 + 4 * u < k1) frag_mma<T, 1>(acc[h], fa[h] + u, fb + u);
      }
    }
  }
#pragma unroll
  for (int h = 0; h < RF; ++h)
#pragma unroll
    for (int p = 0; p < P; ++p)
#pragma unroll
      for (int e = 0; e < 2; ++e) part[warp][p][2 * q + e][8 * h + g] = acc[h][p][e];
  __syncthreads();
  double v[P];
#pragma unroll
  for (int p = 0; p < P; ++p) {
    v[p] = part[0][p][t / kMergedRows][t % kMergedRows];
#pragma unroll
    for (int w = 1; w < 4; ++w) v[p] += part[w][p][t / kMergedRows][t % kMergedRows];
  }
  if (grp > 0 && !cta_wait(mq.done + (int64_t)(grp - 1) * copies + copy, need, mq.spin_ns, mq.abort, 20)) return;
  if (live) {
    if constexpr (P == 1)
      *dst = apply(ld_cg(dst), v[0], ei == ec);
    else
      *dst = apply(ld_cg(dst), T{v[0], v[1]}, ei == ec);
  }
  cta_signal(mq.done + (int64_t)grp * copies + copy);
}

}  // namespace psi
