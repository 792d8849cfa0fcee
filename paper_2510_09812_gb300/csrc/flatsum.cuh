// Weighted sums of a nodal field read as a flat array: sum_i w_i f[i * nc + c] per component.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>

namespace gspm {

constexpr int kSumThreads = 256;
constexpr int kSumComp = 16;             // partial slots per block (at most 9 used)
constexpr int kSumDeep = 8;
constexpr int kSumGrid = 608;            // 4 x 152 SMs
constexpr int64_t kSumOneBlock = 4096;   // values (rows x components) summed by a single block

// Blocks for n rows of nc: up to kSumOneBlock values one block does it all; beyond, a block per round
// of kSumDeep loads, at most four per SM.
__host__ __device__ inline int sum_blocks(int64_t n, int nc) {
  if (n * nc <= kSumOneBlock) return 1;
  const int64_t per = (int64_t)kSumDeep * (kSumThreads / nc), b = (n + per - 1) / per;
  return (int)(b < kSumGrid ? b : kSumGrid);
}

namespace {

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

// out[c] = sum_i w_i f[i*nc + c], by the blocks blockIdx.x < nblocks.  The field is read as the flat
// array it is: the largest multiple of nc up to the block size takes part, so a thread keeps one
// component and one accumulator, and a warp's loads are 256 contiguous bytes (a thread per row reads
// every 32-byte sector nc times).  kSumDeep loads of the field and of the weights are in flight per
// thread.  The FP64 pipe bounds it (two FMAs per SM and clock: 28 us for 3M rows of six, against 25 us
// for the bytes), so the reduction trees must stay small against the rows: four blocks per SM and no
// more.  At 2,963,088 rows of six: 136.1 us before (thread per row, 2048 blocks, nine warp trees each),
// 47.2 us now with the counter's clear, a launch of its own (3.5 TB/s; rows of one 133 -> 18 us, of nine
// 134 -> 66 us).  One block needs neither counter nor scratch and writes `out` itself: 300 rows of three
// 18.7 -> 4.2 us, against 8.3 us for several blocks and the counter's clear.
__device__ __forceinline__ void flat_sum(int nblocks, int64_t n, int nc, const double* __restrict__ f,
                                         const double* __restrict__ w, double* out,
                                         double* partials, unsigned* counter) {
  __shared__ double sm[kSumThreads];
  __shared__ int last;
  const int rows = kSumThreads / nc, active = rows * nc, t = threadIdx.x;
  const int64_t step = (int64_t)nblocks * rows;
  double v = 0.0;
  if (t < active) {
    int64_t i = (int64_t)blockIdx.x * rows + t / nc;
    const int c = t % nc;
    for (; i < n; i += kSumDeep * step) {
      double a[kSumDeep], b[kSumDeep];
#pragma unroll
      for (int u = 0; u < kSumDeep; ++u) {
        const int64_t k = i + u * step;
        const bool ok = k < n;
        a[u] = ok ? __ldcs(f + k * nc + c) : 0.0;
        b[u] = ok ? __ldg(w + k) : 0.0;
      }
#pragma unroll
      for (int u = 0; u < kSumDeep; ++u) v += b[u] * a[u];
    }
  }
  double x = block_sum(v, nc, active, sm);
  if (nblocks == 1) {
    if (t < nc) out[t] = x;
    return;
  }
  if (t < nc) {
    partials[(int64_t)blockIdx.x * kSumComp + t] = x;
    __threadfence();
  }
  __syncthreads();
  if (t == 0) last = (atomicAdd(counter, 1u) == (unsigned)nblocks - 1u);
  __syncthreads();
  if (!last) return;
  __threadfence();
  // the last block to arrive sums the block partials in block order
  v = 0.0;
  if (t < active)
    for (int b = t / nc; b < nblocks; b += kSumDeep * rows) {
      double a[kSumDeep];
#pragma unroll
      for (int u = 0; u < kSumDeep; ++u)
        a[u] = b + u * rows < nblocks
                   ? __ldcg(partials + (int64_t)(b + u * rows) * kSumComp + t % nc) : 0.0;
#pragma unroll
      for (int u = 0; u < kSumDeep; ++u) v += a[u];
    }
  x = block_sum(v, nc, active, sm);
  if (t < nc) out[t] = x;
  if (t == 0) *counter = 0u;
}

}  // namespace

}  // namespace gspm
