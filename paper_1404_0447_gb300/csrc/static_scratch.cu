// Allocation-free entry point: inverses of a batch of small dense blocks
// from their LDL^T factors, with the intermediate L^{-1} blocks kept in a
// fixed device array that belongs to this library instead of memory from
// cudaMalloc.
//
// Why: cudaMalloc can stall and cudaFree synchronises the whole device, and
// some callers may not call either -- code running inside another
// framework's memory pool or under a fixed memory budget, real-time loops
// that must never block on the allocator.  This entry point allocates
// nothing: the caller passes inputs and outputs, and the only scratch is
// g_block_scratch below (16 MiB, held by every GPU that loads the library
// until the process exits).
#include <cuda_runtime.h>

#include <mutex>
#include <string>

#include "block_inverse.cuh"
#include "internal.h"
#include "tile_gemm.cuh"

namespace psi {
void set_global_error(const std::string& msg);  // capi.cu
}

namespace {

constexpr int64_t kScratchDoubles = int64_t(1) << 21;  // 16 MiB of doubles
constexpr int kMaxDevices = 64;

// The shared scratch: L^{-1} of every block of the current call, s x s
// column-major, block-major.  Every call overwrites what it uses.
__device__ __align__(256) double g_block_scratch[kScratchDoubles];

// Phase 1: the 32 x 32 diagonal blocks of V = L^{-1} (entries on and above the
// diagonal of L are not read); CTA (block of the batch, block of V).
__global__ void __launch_bounds__(psi::kVdThreads) k_static_vdiag(int s, const double* __restrict__ L,
                                                                  double* __restrict__ scratch) {
  __shared__ psi::VdSmem<double> sm;
  const int c0 = blockIdx.y * psi::kFB;
  const int64_t at = (int64_t)blockIdx.x * s * s + c0 + (int64_t)c0 * s;
  psi::diag_inverse<double>(L + at, s, scratch + at, s, min(psi::kFB, s - c0), sm);
}

// Phase 2: the rest of V in strips of 8 columns (blockIdx.y); every entry of V's
// s x s block is written by phases 1 and 2 (zeros above the diagonal), so nothing
// from an earlier call survives into this one.
__global__ void __launch_bounds__(psi::TG_THREADS) k_static_vinv(int s, const double* __restrict__ L,
                                                                 double* __restrict__ scratch) {
  __shared__ psi::VsSmem<double> sm;
  const int64_t at = (int64_t)blockIdx.x * s * s;
  psi::inverse_strip<double>(L + at, s, scratch + at, s, blockIdx.y * 8, sm);
}

// Phase 3, one CTA per 64 x 8 tile on or below the diagonal of a block: M =
// V^T (D^{-1} V) on the FP64 pipe, which bounds it, from row k = max(m0, n0) of V
// on (V is lower triangular), mirrored above the diagonal.
__global__ void __launch_bounds__(psi::TG_THREADS, (psi::tile_min_ctas<double, 8>()))
    k_static_m(int s, const double* __restrict__ scratch, const double* __restrict__ d, double* __restrict__ M) {
  constexpr int BN = 8;
  __shared__ psi::TileSmem<double, BN> sm;
  __shared__ double rd[psi::kMaxWidth];
  const int b = blockIdx.x, n0 = blockIdx.y * BN, m0 = n0 + blockIdx.z * psi::TG_BM;
  if (m0 >= s) return;
  const double* V = scratch + (int64_t)b * s * s;
  const double* db = d + (int64_t)b * s;
  for (int q = m0 + threadIdx.x; q < s; q += psi::TG_THREADS) rd[q] = 1.0 / db[q];
  __syncthreads();
  psi::Acc<double, BN> acc;
  psi::acc_zero<double, BN>(acc);
  auto la = [&](int mm, int q) { const int i = m0 + mm; return i < s ? V[q + i * s] : 0.0; };
  auto lb = [&](int q, int nn) { const int j = n0 + nn; return j < s ? rd[q] * V[q + j * s] : 0.0; };
  const int dm = m0 - n0;
  psi::tile_mma<double, BN>(sm, m0, s, [](int) { return true; }, la, lb, acc, [&](int r0, int c0) {
    return m0 + r0 < s && n0 + c0 < s && c0 <= dm + r0 + 7;
  }, psi::KLowerTA{m0});
  double* Mb = M + (int64_t)b * s * s;
  psi::tile_epilogue<double, BN>(acc, [&](int mm, int nn, double v) {
    const int i = m0 + mm, j = n0 + nn;
    if (i >= s || j >= s || i < j) return;
    Mb[i + j * s] = v;
    Mb[j + i * s] = v;
  });
}

std::mutex g_mu;
double* g_scratch_ptr[kMaxDevices] = {};

// Once per device, with that device current: the device address of the
// scratch array (the host-side symbol is only a stand-in).
cudaError_t setup_device(int dev, double** out) {
  std::lock_guard<std::mutex> lock(g_mu);
  if (!g_scratch_ptr[dev]) {
    void* p = nullptr;
    cudaError_t e = cudaGetSymbolAddress(&p, g_block_scratch);
    if (e != cudaSuccess) return e;
    g_scratch_ptr[dev] = (double*)p;
  }
  *out = g_scratch_ptr[dev];
  return cudaSuccess;
}

int fail(int code, const std::string& msg) {
  psi::set_global_error(msg);
  return code;
}

}  // namespace

extern "C" int pselinv_block_inverse_static(int32_t s, int32_t count, const double* d_L, const double* d_d,
                                            double* d_M, void* stream) {
  if (s < 1 || s > psi::kMaxWidth) return fail(PSELINV_ERR_ARG, "block order s must be 1..128");
  if (count < 1) return fail(PSELINV_ERR_ARG, "count must be >= 1");
  if ((int64_t)count * s * s > kScratchDoubles)
    return fail(PSELINV_ERR_ARG, "count * s * s exceeds the static scratch (2^21 doubles = 16 MiB): " +
                                     std::to_string((int64_t)count * s * s) + " requested");
  if (!d_L || !d_d || !d_M) return fail(PSELINV_ERR_ARG, "NULL pointer");
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess || dev < 0 || dev >= kMaxDevices)
    return fail(PSELINV_ERR_CUDA, std::string("cudaGetDevice: ") + cudaGetErrorString(e));
  double* scratch = nullptr;
  e = setup_device(dev, &scratch);
  if (e != cudaSuccess) return fail(PSELINV_ERR_CUDA, std::string("static scratch set-up: ") + cudaGetErrorString(e));
  cudaStream_t st = (cudaStream_t)stream;
  // one CTA for the whole inverse of a block, a column per thread, took 1,000 of
  // the 1,097 us of 192 blocks of order 100
  const int strips = (s + 7) / 8;
  k_static_vdiag<<<dim3(count, (s + psi::kFB - 1) / psi::kFB), psi::kVdThreads, 0, st>>>(s, d_L, scratch);
  if (s > psi::kFB) k_static_vinv<<<dim3(count, strips), psi::TG_THREADS, 0, st>>>(s, d_L, scratch);
  k_static_m<<<dim3(count, strips, (s + psi::TG_BM - 1) / psi::TG_BM), psi::TG_THREADS, 0, st>>>(s, scratch, d_d, d_M);
  e = cudaGetLastError();
  if (e != cudaSuccess) return fail(PSELINV_ERR_CUDA, std::string("launch: ") + cudaGetErrorString(e));
  return PSELINV_OK;
}
