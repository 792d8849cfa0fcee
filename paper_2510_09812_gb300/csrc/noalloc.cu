// Allocation-free volume average.
//
// Some callers cannot allocate device memory: code that runs inside another framework's fixed
// memory pool (where a cudaMalloc outside the pool would break its budget or fragment it),
// real-time loops and host callbacks where cudaMalloc's implicit device synchronisation is not
// acceptable, and plug-ins that only receive pointers.  gspm_volume_avg_noalloc serves them: the
// caller passes the field, the quadrature weights and the output on the device; the reduction's
// scratch (one partial per block plus an arrival counter) lives in a file-scope __device__ array
// of fixed size that every GPU loading this library holds until the process exits.
//
// The host never dereferences the array's name (in host code it is only a stand-in symbol); the
// device address is looked up once per device with cudaGetSymbolAddress, with that device
// current, on the first call made on that device.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>
#include <mutex>

#include "gspm.h"

namespace gspm {
void set_error(const char* fmt, ...);
}

namespace {

constexpr int kThreads = 256;
constexpr int kComp = 16;                        // partial slots per block (ncomp <= 9 used)
constexpr int kMaxBlocks = GSPM_NOALLOC_MAX_BLOCKS;
constexpr int kScratch = kMaxBlocks * kComp + 32;  // partials, then the counter slot

// Reduction scratch shared by every call on this device: kMaxBlocks x 16 doubles of block
// partials followed by the arrival counter (first 4 bytes of the next 256-byte run).
static __device__ __align__(256) double g_noalloc_scratch[kScratch];

constexpr int kMaxGrid = 608;       // 4 x 152 SMs
constexpr int64_t kOneBlock = 4096;  // values (rows x components) summed by a single block
static_assert(kMaxGrid <= kMaxBlocks, "one scratch slot per block");

constexpr int kMaxDevices = 64;
std::mutex g_mu;
double* g_addr[kMaxDevices] = {};

// Block sum per component of the per-thread values v (thread t holds component t % nc; threads
// t >= active hold none), valid in threads c < nc: eight partial sums per component in a fixed
// order, then their sum.
__device__ __forceinline__ double block_sum(double v, int nc, int active, double* sm) {
  const int t = threadIdx.x;
  __syncthreads();
  sm[t] = v;
  __syncthreads();
  double s = 0.0;
  if (t < 8 * nc)
    for (int k = t; k < active; k += 8 * nc) s += sm[k];
  __syncthreads();
  if (t < 8 * nc) sm[t] = s;
  __syncthreads();
  s = 0.0;
  if (t < nc)
    for (int j = 0; j < 8; ++j) s += sm[t + j * nc];
  return s;
}

// out[c] = sum_i w_i f[i*nc + c].  The field is read as the flat array it is: the largest multiple
// of nc up to the block size takes part, so a thread keeps one component and one accumulator, and
// a warp's loads are 256 contiguous bytes (a thread per row reads every 32-byte sector nc times).
// kDeep loads of the field and of the weights are in flight per thread.  The FP64 pipe bounds it
// (two FMAs per SM and clock: 30 us for 3M rows of six, against 25 us for the bytes), so the
// reduction trees must stay small against the rows: four blocks per SM and no more.  At 2,963,088
// rows of six: 136.1 us before (thread per row, 2048 blocks, nine warp trees each), 47.2 us now
// (3.5 TB/s; rows of one 133 -> 18 us, of nine 134 -> 66 us).  One block needs neither counter nor
// scratch and writes `out` itself: 300 rows of three 18.7 -> 4.2 us, against 8.3 us for several
// blocks and the counter's clear.
constexpr int kDeep = 8;
__global__ void __launch_bounds__(kThreads)
k_wsum_noalloc(int64_t n, int nc, const double* __restrict__ f, const double* __restrict__ w,
               double* __restrict__ out, double* scratch) {
  __shared__ double sm[kThreads];
  __shared__ int last;
  const int rows = kThreads / nc, active = rows * nc, t = threadIdx.x;
  const int64_t step = (int64_t)gridDim.x * rows;
  double v = 0.0;
  if (t < active) {
    int64_t i = (int64_t)blockIdx.x * rows + t / nc;
    const int c = t % nc;
    for (; i < n; i += kDeep * step) {
      double a[kDeep], b[kDeep];
#pragma unroll
      for (int u = 0; u < kDeep; ++u) {
        const int64_t k = i + u * step;
        const bool ok = k < n;
        a[u] = ok ? __ldcs(f + k * nc + c) : 0.0;
        b[u] = ok ? __ldg(w + k) : 0.0;
      }
#pragma unroll
      for (int u = 0; u < kDeep; ++u) v += b[u] * a[u];
    }
  }
  double x = block_sum(v, nc, active, sm);
  if (gridDim.x == 1) {
    if (t < nc) out[t] = x;
    return;
  }
  unsigned* counter = reinterpret_cast<unsigned*>(scratch + (int64_t)kMaxBlocks * kComp);
  if (t < nc) {
    scratch[(int64_t)blockIdx.x * kComp + t] = x;
    __threadfence();
  }
  __syncthreads();
  if (t == 0) last = (atomicAdd(counter, 1u) == gridDim.x - 1);
  __syncthreads();
  if (!last) return;
  __threadfence();
  // the last block to arrive sums the block partials in block order
  v = 0.0;
  if (t < active)
    for (int b = t / nc; b < (int)gridDim.x; b += kDeep * rows) {
      double a[kDeep];
#pragma unroll
      for (int u = 0; u < kDeep; ++u)
        a[u] = b + u * rows < (int)gridDim.x
                   ? __ldcg(scratch + (int64_t)(b + u * rows) * kComp + t % nc) : 0.0;
#pragma unroll
      for (int u = 0; u < kDeep; ++u) v += a[u];
    }
  x = block_sum(v, nc, active, sm);
  if (t < nc) out[t] = x;
  if (t == 0) *counter = 0u;
}

// Device address of the scratch for the current device, looked up once per device.
int scratch_address(double** out) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) {
    gspm::set_error("volume_avg_noalloc: cudaGetDevice: %s", cudaGetErrorString(e));
    return GSPM_ECUDA;
  }
  if (dev < 0 || dev >= kMaxDevices) {
    gspm::set_error("volume_avg_noalloc: device ordinal %d above %d", dev, kMaxDevices - 1);
    return GSPM_EINVAL;
  }
  std::lock_guard<std::mutex> lock(g_mu);
  if (!g_addr[dev]) {
    void* p = nullptr;
    e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
    if (e != cudaSuccess || !p) {
      gspm::set_error("volume_avg_noalloc: cudaGetSymbolAddress: %s", cudaGetErrorString(e));
      return GSPM_ECUDA;
    }
    g_addr[dev] = static_cast<double*>(p);
  }
  *out = g_addr[dev];
  return GSPM_OK;
}

}  // namespace

extern "C" int gspm_volume_avg_noalloc(const double* field, const double* weights, int64_t n,
                                       int ncomp, double* out, void* stream) {
  if (!field || !weights || !out) {
    gspm::set_error("volume_avg_noalloc: null pointer");
    return GSPM_EINVAL;
  }
  if (n <= 0) {
    gspm::set_error("volume_avg_noalloc: n must be positive (got %lld)", (long long)n);
    return GSPM_EINVAL;
  }
  if (ncomp < 1 || ncomp > GSPM_NOALLOC_MAX_COMP) {
    gspm::set_error("volume_avg_noalloc: ncomp %d outside 1..%d (the fixed scratch holds at most "
                    "%d components per block)", ncomp, GSPM_NOALLOC_MAX_COMP,
                    GSPM_NOALLOC_MAX_COMP);
    return GSPM_EINVAL;
  }
  double* scratch = nullptr;
  int st = scratch_address(&scratch);
  if (st != GSPM_OK) return st;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  cudaError_t e = cudaSuccess;
  // up to kOneBlock values one block does it all; beyond, a block per round of kDeep loads, at most
  // four per SM (GB300: 152 SMs)
  const int64_t rows = kThreads / ncomp;
  int64_t blocks = 1;
  if (n * ncomp > kOneBlock) {
    blocks = std::min<int64_t>((n + kDeep * rows - 1) / (kDeep * rows), kMaxGrid);
    // the arrival counter must start at zero (a previous call resets it; clear it regardless)
    e = cudaMemsetAsync(scratch + (int64_t)kMaxBlocks * kComp, 0, sizeof(unsigned), s);
    if (e != cudaSuccess) {
      gspm::set_error("volume_avg_noalloc: cudaMemsetAsync: %s", cudaGetErrorString(e));
      return GSPM_ECUDA;
    }
  }
  k_wsum_noalloc<<<(int)blocks, kThreads, 0, s>>>(n, ncomp, field, weights, out, scratch);
  e = cudaGetLastError();
  if (e != cudaSuccess) {
    gspm::set_error("volume_avg_noalloc: launch: %s", cudaGetErrorString(e));
    return GSPM_ECUDA;
  }
  return GSPM_OK;
}
