// Generic per-cell chemistry kernels for sm_103a: plain (one pass, one cell per
// thread) and queue (persistent CTAs, substep-granular refill from a device work
// queue), compiled for 2, 3 and 9 species and for both integrators (RODAS3 and
// ROS2); the body is in chem_kernel_body.cuh.
#include <cuda_runtime.h>

#include <mutex>

#include "chem_kernel_body.cuh"

namespace rde {

namespace {

template <int K, bool QUEUE, int METHOD>
__global__ void __launch_bounds__(kThreads, 1) chem_advance_kernel(const LaunchArgs a) {
  advance_body<K, QUEUE, GenericRhs, METHOD>(a);
}

template <int K>
size_t smem_bytes(int mech_bytes, int n_blocks) {
  return (size_t)mech_bytes + Slots<K>::bytes(kThreads) + (n_blocks > 0 ? sizeof(long long) * (n_blocks + 1) : 0);
}

template <int K, bool QUEUE, int METHOD>
cudaError_t set_smem(size_t smax) {
  return raise_shared_limit(reinterpret_cast<const void*>(chem_advance_kernel<K, QUEUE, METHOD>), smax);
}

template <int K>
cudaError_t prepare_k(int mech_bytes, int* fit) {
  const size_t smax = smem_bytes<K>(mech_bytes, kMaxBlocks);
  cudaError_t e = set_smem<K, true, kMethodRodas3>(smax);
  if (e == cudaSuccess) e = set_smem<K, false, kMethodRodas3>(smax);
  if (e == cudaSuccess) e = set_smem<K, true, kMethodRos2>(smax);
  if (e == cudaSuccess) e = set_smem<K, false, kMethodRos2>(smax);
  if (e == cudaSuccess) e = set_smem<K, true, kMethodExtrap>(smax);
  // one resident CTA per SM for every instance (launch bounds and shared memory);
  // the fit of the RODAS3 queue kernel sizes the persistent grid of both methods
  if (e == cudaSuccess)
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(fit, chem_advance_kernel<K, true, kMethodRodas3>, kThreads,
                                                      smax);
  if (e == cudaSuccess && *fit < 1) e = cudaErrorInvalidConfiguration;
  return e;
}

template <int K, bool QUEUE, int METHOD>
cudaError_t launch_one(const LaunchArgs& a, cudaStream_t stream) {
  const size_t smem = smem_bytes<K>(a.mech_bytes, a.blocks ? a.n_blocks : 0);
  const long long blocks_needed = (a.n_total + kThreads - 1) / kThreads;
  long long grid = blocks_needed;
  if (QUEUE) {
    const int fit = a.fit > 0 ? a.fit : 1;
    const int per_sm = a.ctas_per_sm > 0 ? min(a.ctas_per_sm, fit) : fit;
    grid = min(blocks_needed, (long long)a.num_sms * per_sm);
  }
  if (grid < 1) grid = 1;
  chem_advance_kernel<K, QUEUE, METHOD><<<(unsigned)grid, kThreads, smem, stream>>>(a);
  return cudaGetLastError();
}

template <int K>
cudaError_t launch_k(const LaunchArgs& a, cudaStream_t stream) {
  const bool plain = a.schedule == RDE_SCHED_PLAIN;
  if (a.opt.method == RDE_METHOD_ROS2)
    return plain ? launch_one<K, false, kMethodRos2>(a, stream) : launch_one<K, true, kMethodRos2>(a, stream);
  if (a.opt.method == RDE_METHOD_EXTRAP)   // queue schedule only: the Jacobian scratch is per resident lane
    return plain ? cudaErrorInvalidValue : launch_one<K, true, kMethodExtrap>(a, stream);
  return plain ? launch_one<K, false, kMethodRodas3>(a, stream) : launch_one<K, true, kMethodRodas3>(a, stream);
}

}  // namespace

bool kernel_supports(int K) { return K == 2 || K == 3 || K == 9; }

int kernel_threads() { return kThreads; }

size_t kernel_shared_bytes(int K, int mech_bytes) {
  switch (K) {
    case 2: return smem_bytes<2>(mech_bytes, 0);
    case 3: return smem_bytes<3>(mech_bytes, 0);
    case 9: return smem_bytes<9>(mech_bytes, 0);
    default: return 0;
  }
}

cudaError_t raise_shared_limit(const void* kernel, size_t bytes) {
  static std::mutex mu;   // the limit is read and written as one step
  std::lock_guard<std::mutex> lk(mu);
  cudaFuncAttributes at;
  const cudaError_t e = cudaFuncGetAttributes(&at, kernel);
  if (e != cudaSuccess || bytes <= (size_t)at.maxDynamicSharedSizeBytes) return e;
  return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}

cudaError_t prepare_advance(int K, int mech_bytes, int* fit) {
  switch (K) {
    case 2: return prepare_k<2>(mech_bytes, fit);
    case 3: return prepare_k<3>(mech_bytes, fit);
    case 9: return prepare_k<9>(mech_bytes, fit);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t launch_advance(const LaunchArgs& a, cudaStream_t stream) {
  if (a.blocks && a.n_blocks > kMaxBlocks) return cudaErrorInvalidValue;
  switch (a.K) {
    case 2: return launch_k<2>(a, stream);
    case 3: return launch_k<3>(a, stream);
    case 9: return launch_k<9>(a, stream);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace rde

// ---- queue order by predicted cost ----
// A cell takes 50 to 1,000 attempts, and a call ends when its last cell does: a lane that
// takes a long cell late keeps its SM sub-partition busy on its own.  The queue therefore
// hands the cells out by predicted cost, longest first (as the paper weights its ranks by
// cost, Section 3.3.1): a counting sort into kOrderBins bins, a quarter octave each, of
//   dt / h_hint    where the caller carries a step size (the attempts a step needs), else
//   T^2 p          (rank correlation with the attempts 0.92 on the RDE-like field and 0.81
//                  on uniform cells; T alone 0.84 and 0.72).
// Two passes over T and p (or h_hint), a few microseconds for 100,000 cells; with the first
// cells spread over the CTAs (advance_body) 60,001 field cells took 159 ms instead of 212,
// 120,000 194 ms instead of 299.  The order
// within a bin varies from run to run; a cell's result does not depend on the order.
namespace rde {
namespace {
constexpr int kOrderThreads = 256;
constexpr int kOrderChunk = 2048;   // cells per CTA of either pass

__device__ __forceinline__ int cost_bin(const LaunchArgs& a, const long long* offs, long long n_total, long long g) {
  LaneCell c{};
  if (!locate(a, offs, n_total, g, c)) return 0;
  float x;
  int base;
  const double hint = c.h_hint ? c.h_hint[c.i] : 0.0;
  if (hint > 0.0) {
    x = (float)(a.dt / hint);
    base = 127;             // bin 0: a hint of dt or more
  } else {
    const double T = c.T[c.i];
    x = (float)(T * T * c.p[c.i]);
    base = 127 + 24;        // bins from 2^24 K^2 Pa to 2^56
  }
  const int b = (int)(__float_as_uint(x) >> 21) - 4 * base;
  // infinity goes first, NaN and what is not positive last
  return x > 0.0f ? max(0, min(kOrderBins - 1, b)) : 0;
}

__device__ __forceinline__ long long block_offsets(const LaunchArgs& a, long long* offs) {
  if (a.blocks && threadIdx.x == 0) {
    long long acc = 0;
    for (int b = 0; b < a.n_blocks; ++b) {
      offs[b] = acc;
      const long long nb = (long long)a.blocks[b].n;
      acc += nb > 0 ? nb : 0;
    }
    offs[a.n_blocks] = acc;
  }
  __syncthreads();
  return a.blocks ? min(a.n_total, offs[a.n_blocks]) : a.n_total;
}

__global__ void __launch_bounds__(kOrderThreads) order_count_kernel(const LaunchArgs a, unsigned* counts) {
  extern __shared__ __align__(16) unsigned char smem[];
  unsigned* mine = reinterpret_cast<unsigned*>(smem);
  long long* offs = reinterpret_cast<long long*>(smem + sizeof(unsigned) * kOrderBins);
  for (int b = threadIdx.x; b < kOrderBins; b += kOrderThreads) mine[b] = 0;
  const long long n = block_offsets(a, offs);   // its barrier covers the zeros above
  const long long first = (long long)blockIdx.x * kOrderChunk, last = min(n, first + kOrderChunk);
  for (long long g = first + threadIdx.x; g < last; g += kOrderThreads) atomicAdd(&mine[cost_bin(a, offs, n, g)], 1u);
  __syncthreads();
  for (int b = threadIdx.x; b < kOrderBins; b += kOrderThreads)
    if (mine[b]) atomicAdd(&counts[b], mine[b]);
}

__global__ void __launch_bounds__(kOrderThreads) order_place_kernel(const LaunchArgs a, const unsigned* counts,
                                                                    unsigned* cursors, long long* order) {
  extern __shared__ __align__(16) unsigned char smem[];
  unsigned* mine = reinterpret_cast<unsigned*>(smem);       // this CTA's cells per bin
  unsigned* base = mine + kOrderBins;                       // where they go
  unsigned* used = base + kOrderBins;
  long long* offs = reinterpret_cast<long long*>(smem + 3 * sizeof(unsigned) * kOrderBins);
  for (int b = threadIdx.x; b < kOrderBins; b += kOrderThreads) mine[b] = used[b] = 0;
  const long long n = block_offsets(a, offs);
  const long long first = (long long)blockIdx.x * kOrderChunk, last = min(n, first + kOrderChunk);
  int bin[kOrderChunk / kOrderThreads];
#pragma unroll
  for (int q = 0; q < kOrderChunk / kOrderThreads; ++q) {
    const long long g = first + threadIdx.x + (long long)q * kOrderThreads;
    bin[q] = g < last ? cost_bin(a, offs, n, g) : -1;
    if (bin[q] >= 0) atomicAdd(&mine[bin[q]], 1u);
  }
  __syncthreads();
  for (int b = threadIdx.x; b < kOrderBins; b += kOrderThreads) {
    unsigned before = 0;   // cells of costlier bins
    for (int c = b + 1; c < kOrderBins; ++c) before += counts[c];
    base[b] = mine[b] ? before + atomicAdd(&cursors[b], mine[b]) : 0;
  }
  __syncthreads();
#pragma unroll
  for (int q = 0; q < kOrderChunk / kOrderThreads; ++q) {
    if (bin[q] < 0) continue;
    const long long at = (long long)base[bin[q]] + atomicAdd(&used[bin[q]], 1u);
    // T is read twice and must not change in between; an index is never written out of range
    if (at < n) order[at] = first + threadIdx.x + (long long)q * kOrderThreads;
  }
}
}  // namespace

cudaError_t launch_order(const LaunchArgs& args, unsigned* counts, long long* order, cudaStream_t stream) {
  LaunchArgs a = args;
  a.order = nullptr;
  const unsigned grid = (unsigned)((a.n_total + kOrderChunk - 1) / kOrderChunk);
  const size_t offs = a.blocks ? sizeof(long long) * (a.n_blocks + 1) : 0;
  order_count_kernel<<<grid, kOrderThreads, sizeof(unsigned) * kOrderBins + offs, stream>>>(a, counts);
  order_place_kernel<<<grid, kOrderThreads, 3 * sizeof(unsigned) * kOrderBins + offs, stream>>>(
      a, counts, counts + kOrderBins, order);
  return cudaGetLastError();
}
}  // namespace rde

// ---- test hook: the library's exp / log / reciprocal on device arrays ----
namespace rde {
namespace {
__global__ void selftest_math_kernel(int fn, long long n, const double* x, double* y, const double* tabs) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  y[i] = fn == 0   ? exp_tab(x[i], reinterpret_cast<const unsigned long long*>(tabs))
         : fn == 1 ? log_tab(x[i], tabs + kExpTabSize)
                   : recip(x[i]);
}
}  // namespace

cudaError_t launch_selftest_math(int fn, long long n, const double* x, double* y, const double* tabs,
                                 cudaStream_t stream) {
  if (n <= 0) return cudaSuccess;
  selftest_math_kernel<<<(unsigned)((n + 255) / 256), 256, 0, stream>>>(fn, n, x, y, tabs);
  return cudaGetLastError();
}
}  // namespace rde
