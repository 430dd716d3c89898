// Inverse V of a unit lower triangle of order s <= 128 in blocks of kFactorBlock:
// the diagonal blocks first, then strips of 8 columns, each strip independent
// of the others.  Shared by the factorisation (kernels.cu) and the
// allocation-free block inverse (static_scratch.cu).
//
// One CTA inverting a whole 128-wide triangle is held to one SM's FP64 pipe
// (s^3 / 3 flops, 97 us) and, column per thread, to a chain of dependent
// loads (above 400 us); strips put 16 CTAs of at most 20 us on a block.
#pragma once

#include "internal.h"
#include "tile_gemm.cuh"

namespace psi {

constexpr int kFB = kFactorBlock;

// Row and column of entry e of a lower triangle stored row by row.
__device__ __forceinline__ void tri_entry(int e, int& i, int& k) {
  i = (int)((sqrtf(8.0f * (float)e + 1.0f) - 1.0f) * 0.5f);
  while ((i + 1) * (i + 2) / 2 <= e) ++i;
  while (i * (i + 1) / 2 > e) --i;
  k = e - i * (i + 1) / 2;
}

constexpr int kVdThreads = 192;  // 6 warps fill the FP64 pipe; three strictly lower entries per thread
template <class T>
struct VdSmem {
  T l[kFB][kFB + 1];
  T v[2][kFB];  // V's row j, by parity
};

// V = A^{-1} for the unit lower triangle of order w <= 32 at A (ld; its diagonal
// and upper part are not read), the whole w x w block of V written.  Row by
// row: V_ik -= A_ij V_jk for k < j < i, one barrier per column j.
template <class T>
__device__ void diag_inverse(const T* A, int64_t ld, T* V, int64_t vld, int w, VdSmem<T>& sm) {
  constexpr int E = (kFB * (kFB - 1) / 2 + kVdThreads - 1) / kVdThreads;
  const int t = threadIdx.x, ne = w * (w - 1) / 2;
  for (int e = t; e < w * w; e += kVdThreads) {
    const int i = e % w, k = e / w;
    if (i > k) sm.l[i][k] = A[i + (int64_t)k * ld];
    if (i <= k) V[i + (int64_t)k * vld] = i == k ? Sc<T>::one() : Sc<T>::zero();
  }
  T x[E];
  int ri[E], ck[E];
#pragma unroll
  for (int q = 0; q < E; ++q) {
    const int e = t + q * kVdThreads;
    ri[q] = ck[q] = 0;  // no entry: never live
    x[q] = Sc<T>::zero();
    if (e < ne) {
      tri_entry(e, ri[q], ck[q]);
      ++ri[q];  // strictly lower: row i holds columns 0 .. i - 1
    }
  }
  for (int j = 0; j + 1 < w; ++j) {
    __syncthreads();
    const T* vr = sm.v[j & 1];
#pragma unroll
    for (int q = 0; q < E; ++q) {
      const int i = ri[q], k = ck[q];
      if (i > j && k <= j) {
        const T l = sm.l[i][j];
        x[q] = k == j ? -l : x[q] - l * vr[k];
        if (i == j + 1) sm.v[~j & 1][k] = x[q];
      }
    }
  }
#pragma unroll
  for (int q = 0; q < E; ++q)
    if (ri[q] > 0) V[ri[q] + (int64_t)ck[q] * vld] = x[q];
}

template <class T>
struct VsSmem {
  static constexpr int LDX = 12;  // 4 (mod 16) doubles
  double x[Sc<T>::P][kMaxWidth][LDX];
  double s[Sc<T>::P][kFB][LDX];
};

// Columns n0 .. n0+7 of V = A^{-1} (unit lower triangle of order s, ld; V s x s,
// its diagonal blocks filled): with j the block of the columns, X_j = V_jj and,
// for i = j+1, j+2, ...: X_i = -V_ii sum_{k=j}^{i-1} A_ik X_k.  Four warps; warp
// w holds rows 8w .. 8w+7 of the 32-row block on m8n8k4 MMAs, its operand
// fragments straight from global memory (eight 64-byte row runs per k-block,
// loaded before the products), X in shared memory.  Blocks above the diagonal
// are written as zeros.
template <class T>
__device__ void inverse_strip(const T* A, int64_t ld, T* V, int s, int n0, VsSmem<T>& sm) {
  constexpr int P = Sc<T>::P;
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5, g = lane >> 2, q = lane & 3;
  const int j0 = n0 / kFB * kFB, j1 = min(s, j0 + kFB), n1 = min(s, n0 + 8);
  for (int e = t; e < j0 * 8; e += TG_THREADS) {
    const int col = n0 + e / j0;
    if (col < n1) V[e % j0 + (int64_t)col * s] = Sc<T>::zero();
  }
  for (int e = t; e < kFB * 8; e += TG_THREADS) {
    const int row = j0 + e % kFB, col = n0 + e / kFB;
    const T v = row < j1 && col < n1 ? V[row + (int64_t)col * s] : Sc<T>::zero();
#pragma unroll
    for (int pl = 0; pl < P; ++pl) sm.x[pl][row][e / kFB] = Sc<T>::plane(v, pl);
  }
  __syncthreads();
  // acc += (row `row` of M, columns k0 .. k0 + 31 before klim) (the 32 rows of x
  // at xr0), k-steps u0 .. u1 - 1 of 4 (the others meet zeros of a triangle)
  auto product = [&](const T* M, int64_t mld, int row, int k0, int klim, const double* x, int64_t plane, int u0, int u1,
                     double (&acc)[P][2]) {
    T fa[kFB / 4], fb[kFB / 4];
#pragma unroll
    for (int u = 0; u < kFB / 4; ++u) {
      if (u < u0 || u >= u1) continue;
      const int kk = k0 + 4 * u + q;
      fa[u] = row < s && kk < klim ? M[row + (int64_t)kk * mld] : Sc<T>::zero();
      const double* xb = x + (4 * u + q) * VsSmem<T>::LDX + g;
      if constexpr (P == 1)
        fb[u] = xb[0];
      else
        fb[u] = T{xb[0], xb[plane]};
    }
#pragma unroll
    for (int u = 0; u < kFB / 4; ++u)
      if (u >= u0 && u < u1) frag_mma<T, 1>(acc, fa + u, fb + u);
  };
  constexpr int64_t XP = (int64_t)kMaxWidth * VsSmem<T>::LDX, SP = (int64_t)kFB * VsSmem<T>::LDX;
  const int ustrip = (n0 - j0) / 4;  // X_j is zero above the strip's own rows
  for (int i0 = j1; i0 < s; i0 += kFB) {
    const int row = i0 + 8 * warp + g;
    const bool live = i0 + 8 * warp < s;  // the last block may hold fewer rows than four fragments
    double acc[P][2] = {};
    if (live)
      for (int k0 = j0; k0 < i0; k0 += kFB)
        product(A, ld, row, k0, s, &sm.x[0][k0][0], XP, k0 == j0 ? ustrip : 0, kFB / 4, acc);
#pragma unroll
    for (int pl = 0; pl < P; ++pl)
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        sm.s[pl][8 * warp + g][2 * q + e] = acc[pl][e];
        acc[pl][e] = 0.0;
      }
    __syncthreads();
    // V_ii is lower triangular: rows 8 w .. 8 w + 7 need k < 8 w + 8
    if (live) product(V, s, row, i0, min(s, i0 + kFB), &sm.s[0][0][0], SP, 0, 2 * warp + 2, acc);
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      const int col = n0 + 2 * q + e;
#pragma unroll
      for (int pl = 0; pl < P; ++pl) sm.x[pl][i0 + 8 * warp + g][2 * q + e] = -acc[pl][e];
      if (row < s && col < n1) V[row + (int64_t)col * s] = -frag_value<T>(acc, e);
    }
    __syncthreads();
  }
}

}  // namespace psi
