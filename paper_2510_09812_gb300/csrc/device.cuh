// Device helpers shared by the kernel files: SELL-32 row products, compensated and double-float
// sums, deterministic per-segment reductions.
#pragma once

#include <cuda_runtime.h>

#include <type_traits>

#include "kernels.cuh"

namespace gspm {

namespace {

constexpr unsigned kFull = 0xffffffffu;

// Compensated summation (Kahan): s + c carries the running sum with the low-order part lost by
// each add kept in c (subtracted at the end: total = s - c)
template <typename T>
__device__ __forceinline__ void kahan_add(T& s, T& c, T x) {
  const T y = x - c;
  const T t = s + y;
  c = (t - s) - y;
  s = t;
}

__device__ __forceinline__ int64_t gtid() { return (int64_t)blockIdx.x * blockDim.x + threadIdx.x; }
__device__ __forceinline__ int64_t gstride() { return (int64_t)gridDim.x * blockDim.x; }

// Programmatic dependent launch (the CG loop kernels): a kernel launched with
// launch_pdl first waits until the previous kernel of the stream has completed and its memory
// is visible, then lets the next kernel be scheduled (its blocks wait the same way), so
// launch latency overlaps the running kernel.  Outside such a launch both are no-ops.
__device__ __forceinline__ void pdl_enter() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// Double-float addition (h, l) += (bh, bl): Knuth's TwoSum of the high parts, the low parts
// added to its error term, renormalised (the _rn intrinsics keep the compiler from contracting
// or reassociating the steps)
__device__ __forceinline__ void df_add(float& h, float& l, float bh, float bl) {
  const float s = __fadd_rn(h, bh);
  const float z = __fsub_rn(s, h);
  float e = __fadd_rn(__fsub_rn(h, __fsub_rn(s, z)), __fsub_rn(bh, z));
  e = __fadd_rn(e, __fadd_rn(l, bl));
  h = __fadd_rn(s, e);
  l = __fsub_rn(e, __fsub_rn(h, s));
}

// a double-float value; the three operations that the sums over lanes need, for each type
struct DF {
  float h, l;
};
__device__ __forceinline__ DF lane_xor(DF v, int o) {
  return DF{__shfl_xor_sync(kFull, v.h, o), __shfl_xor_sync(kFull, v.l, o)};
}
template <typename V>
__device__ __forceinline__ V lane_xor(V v, int o) {
  return __shfl_xor_sync(kFull, v, o);
}
__device__ __forceinline__ DF plus(DF a, DF b) {
  df_add(a.h, a.l, b.h, b.l);
  return a;
}
template <typename V>
__device__ __forceinline__ V plus(V a, V b) {
  return a + b;
}
__device__ __forceinline__ double as_double(DF v) { return (double)v.h + (double)v.l; }
__device__ __forceinline__ double as_double(double v) { return v; }

__host__ __device__ constexpr int pow2_up(int n) { return n <= 1 ? 1 : 2 * pow2_up((n + 1) / 2); }

// Sums of M values (a power of two) over each group of LANES lanes.  While several values are
// left, a pair of lanes splits them: each keeps half of them and adds the other lane's, so M
// values take M - 1 + log2(LANES / M) additions where M separate trees take M log2(LANES).  The
// result is value (lane % LANES) / (LANES / M), the same bits in every lane that has it: those of a
// tree per value with halving distances.
template <int M, int LANES, typename V>
__device__ __forceinline__ V lane_sums(V (&v)[M]) {
  const int lane = threadIdx.x & 31;
  int o = LANES / 2;
#pragma unroll
  for (int w = M / 2; w >= 1; w >>= 1) {
    const bool up = lane & o;
#pragma unroll
    for (int i = 0; i < w; ++i) {
      const V send = up ? v[i] : v[i + w];
      v[i] = plus(up ? v[i + w] : v[i], lane_xor(send, o));
    }
    o >>= 1;
  }
#pragma unroll
  for (int r = LANES / M; r > 1; r >>= 1) v[0] = plus(v[0], lane_xor(v[0], r / 2));
  return v[0];
}

// The same with doubling distances (the bits of a tree per value that starts with neighbours): the
// result is value lane % M with its bits in reverse order.
template <int M, int LANES, typename V>
__device__ __forceinline__ V lane_sums_up(V (&v)[M]) {
  const int lane = threadIdx.x & 31;
  int o = 1;
#pragma unroll
  for (int w = M / 2; w >= 1; w >>= 1) {
    const bool up = lane & o;
#pragma unroll
    for (int i = 0; i < w; ++i) {
      const V send = up ? v[i] : v[i + w];
      v[i] = plus(up ? v[i + w] : v[i], lane_xor(send, o));
    }
    o <<= 1;
  }
#pragma unroll
  for (; o < LANES; o <<= 1) v[0] = plus(v[0], lane_xor(v[0], o));
  return v[0];
}
// lane % M with its bits in reverse order
template <int M>
__device__ __forceinline__ int lane_value_up(int lane) {
  int k = 0;
#pragma unroll
  for (int w = M / 2, o = 1; w >= 1; w >>= 1, o <<= 1) k += lane & o ? w : 0;
  return k;
}

// The last item of `seg` to arrive (its block partials, a row of pow2_up(NC) values, already in
// red.partial) sums the segment's item partials in a fixed order and returns true (totals in
// res[0..NC), valid in every thread of that block).  The partials of a segment are one run that
// the whole block loads in order, every load independent of the others; thread t sums value
// t % pow2_up(NC).  FP64 additions bound this tail (2 per clock and SM): one per partial value,
// the trees over lanes only as deep as a value has lanes.  Against one strided pass, one tree of 32
// lanes and one of the block per value: 16 meshes of 65,536 nodes in a batch 41.6 -> 39.2 ms, two
// steps of 2,963,088 nodes 217.4 -> 211.9 ms.
template <int NC>
__device__ __forceinline__ bool seg_arrive(int item, int seg, const DSeg& G, const ItemList& IL,
                                           const Red& red, double* res) {
  constexpr int M = pow2_up(NC), NW = kBlock / 32;
  __shared__ double sm[NW][M];
  __shared__ int am_last;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (threadIdx.x == 0) {
    __threadfence();
    const unsigned t = atomicAdd(G.counter + seg, 1u);
    am_last = (t == (unsigned)IL.seg_nitems[seg] - 1u);
  }
  __syncthreads();
  if (!am_last) return false;
  __threadfence();
  const double* p = red.partial + (int64_t)IL.seg_item0[seg] * M;
  const int ne = IL.seg_nitems[seg] * M;
  double a[4] = {0.0, 0.0, 0.0, 0.0};
  int e = threadIdx.x;
  for (; e + 3 * kBlock < ne; e += 4 * kBlock) {
    double x[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) x[u] = __ldcg(p + e + u * kBlock);
#pragma unroll
    for (int u = 0; u < 4; ++u) a[u] += x[u];
  }
  for (; e < ne; e += kBlock) a[0] += __ldcg(p + e);
  double acc = (a[0] + a[1]) + (a[2] + a[3]);
#pragma unroll
  for (int o = M; o < 32; o <<= 1) acc += __shfl_xor_sync(kFull, acc, o);
  if (lane < M) sm[warp][lane] = acc;
  __syncthreads();
  if (threadIdx.x < NC) {
    double x[NW];
#pragma unroll
    for (int w = 0; w < NW; ++w) x[w] = sm[w][threadIdx.x];
#pragma unroll
    for (int h = NW / 2; h >= 1; h >>= 1)
#pragma unroll
      for (int w = 0; w < h; ++w) x[w] += x[w + h];
    res[threadIdx.x] = x[0];
  }
  if (threadIdx.x == 0) G.counter[seg] = 0u;
  __syncthreads();
  return true;
}

// Block reduction of NC values (v: padded with zeros to a power of two) into the item's partials,
// then seg_arrive.  Blocks of kBlock threads.
template <int NC, typename V>
__device__ __forceinline__ bool seg_reduce_of(V (&v)[pow2_up(NC)], int item, int seg, const DSeg& G,
                                              const ItemList& IL, const Red& red, double* res) {
  constexpr int M = pow2_up(NC), NW = kBlock / 32, R = 32 / M;
  __shared__ V sm[M][NW];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const V s = lane_sums<M, 32>(v);
  if (lane % R == 0) sm[lane / R][warp] = s;
  __syncthreads();
  if (warp == 0) {
    // NW lanes per value, 32 / NW values at a time
#pragma unroll
    for (int c0 = 0; c0 < NC; c0 += 32 / NW) {
      const int c = c0 + lane / NW;
      V x = sm[c < M ? c : 0][lane % NW];
#pragma unroll
      for (int o = NW / 2; o >= 1; o >>= 1) x = plus(x, lane_xor(x, o));
      if (lane % NW == 0 && c < M) red.partial[(int64_t)item * M + c] = as_double(x);
    }
    __syncwarp();
  }
  return seg_arrive<NC>(item, seg, G, IL, red, res);
}

// Sum over a warp's lanes, distances halving; the result is lane 0's
__device__ __forceinline__ double warp_sum(double x) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) x += __shfl_down_sync(kFull, x, o);
  return x;
}

// The reduction of FP64 contexts: one tree of 32 lanes and one of the warps per value, then the item
// partials strided over the block's threads and the same trees.  A CG solve in FP64 that stops at a
// loose tolerance magnifies the rounding of its sums (1e-16) to 1e-9 .. 1e-8 of the solution, so this
// order of additions is part of what such a context returns and does not follow the faster one above.
template <int NC>
__device__ __forceinline__ bool seg_reduce_fixed(double (&v)[NC], int item, int seg, const DSeg& G,
                                                 const ItemList& IL, const Red& red, double* res) {
  __shared__ double sm[NC][32];
  __shared__ int am_last;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
#pragma unroll
  for (int c = 0; c < NC; ++c) {
    const double x = warp_sum(v[c]);
    if (lane == 0) sm[c][warp] = x;
  }
  __syncthreads();
  if (warp == 0) {
#pragma unroll
    for (int c = 0; c < NC; ++c) {
      const double x = warp_sum(lane < nw ? sm[c][lane] : 0.0);
      if (lane == 0) red.partial[(int64_t)item * kRedComp + c] = x;
    }
  }
  if (threadIdx.x == 0) {
    __threadfence();
    const unsigned t = atomicAdd(G.counter + seg, 1u);
    am_last = (t == (unsigned)IL.seg_nitems[seg] - 1u);
  }
  __syncthreads();
  if (!am_last) return false;
  __threadfence();
  const int i0 = IL.seg_item0[seg], ni = IL.seg_nitems[seg];
#pragma unroll
  for (int c = 0; c < NC; ++c) {
    double acc = 0.0;
    for (int b = threadIdx.x; b < ni; b += blockDim.x)
      acc += __ldcg(red.partial + (int64_t)(i0 + b) * kRedComp + c);
    acc = warp_sum(acc);
    if (lane == 0) sm[c][warp] = acc;
  }
  __syncthreads();
  if (warp == 0) {
#pragma unroll
    for (int c = 0; c < NC; ++c) {
      const double x = warp_sum(lane < nw ? sm[c][lane] : 0.0);
      if (lane == 0) res[c] = x;
    }
  }
  if (threadIdx.x == 0) G.counter[seg] = 0u;
  __syncthreads();
  return true;
}

// FP64 values in a context of working precision T
template <typename T, int NC>
__device__ __forceinline__ bool seg_reduce(double (&v)[NC], int item, int seg, const DSeg& G,
                                           const ItemList& IL, const Red& red, double* res) {
  if constexpr (std::is_same<T, double>::value) {
    return seg_reduce_fixed<NC>(v, item, seg, G, IL, red, res);
  } else {
    double x[pow2_up(NC)];
#pragma unroll
    for (int c = 0; c < pow2_up(NC); ++c) x[c] = c < NC ? v[c < NC ? c : 0] : 0.0;
    return seg_reduce_of<NC>(x, item, seg, G, IL, red, res);
  }
}

// seg_reduce of per-thread values given as unevaluated sums hi + lo in T.  T = float: the warp
// and block trees run in double-float arithmetic (FP32 operations, about 44 significant bits;
// an FP64 instruction costs ~64 FP32 ones on this part and the FP64 trees dominated the short
// CG vector kernels), one FP64 conversion per block and value.  T = double: seg_reduce.
template <typename T, int NC>
__device__ __forceinline__ bool seg_reduce_hl(const T (&hi)[NC], const T (&lo)[NC], int item,
                                              int seg, const DSeg& G, const ItemList& IL,
                                              const Red& red, double* res) {
  if constexpr (std::is_same<T, double>::value) {
    double v[NC];
#pragma unroll
    for (int c = 0; c < NC; ++c) v[c] = hi[c] + lo[c];
    return seg_reduce<T, NC>(v, item, seg, G, IL, red, res);
  } else {
    DF x[pow2_up(NC)];
#pragma unroll
    for (int c = 0; c < pow2_up(NC); ++c)
      x[c] = c < NC ? DF{hi[c < NC ? c : 0], lo[c < NC ? c : 0]} : DF{0.f, 0.f};
    return seg_reduce_of<NC>(x, item, seg, G, IL, red, res);
  }
}

// The difference forms sum_j A_ij (x_j - x_i) of the zero-row-sum operators (K^ms, K^mech, F^ms,
// G) are used in FP32, where they keep smooth fields from cancelling; in FP64 the plain products
// are accurate enough and each extra subtraction costs FP64 issue slots.
template <typename T>
constexpr int kDiff = std::is_same<T, float>::value ? 1 : 0;

__device__ __forceinline__ bool row_valid(const DSeg& G, int seg, int64_t row) {
  return row - G.seg_row0[seg] < G.seg_nrow[seg];
}

// y_r(row) = sum_k A(row, k) x_r(col(row, k)) for one row of a scalar SELL matrix, neighbours
// k = k0, k0 + kstep, ...  diff != 0 (an operator whose rows sum to zero: K^ms, K^mech): formed as
// sum_k A(row, k) (x_r(col) - x_r(row)), equal in exact arithmetic; a smooth x then does not
// cancel in the sum, and the FP32 rounding of the values cannot make the operator act on the
// constants (its rows' rounded sums no longer enter).
template <typename V, typename X, typename Acc, int NR, int VAR = 0>
__device__ __forceinline__ void sell_scalar_row(const DSell& A, const V* __restrict__ val,
                                                int64_t s, int lane, const X* __restrict__ x,
                                                int64_t ld, const int (&skip)[NR],
                                                Acc (&acc)[NR], int k0 = 0, int kstep = 1,
                                                int diff = 0) {
  const int64_t base = A.sptr[s];
  const int len = A.slen[s];
  const int32_t* cp = A.col + base + lane;
  const V* vp = val + base + lane;
  const int64_t row = s * 32 + lane;
  X xi[NR];
#pragma unroll
  for (int r = 0; r < NR; ++r) {
    acc[r] = Acc(0);
    xi[r] = diff && row < A.n ? x[r * ld + row] : X(0);
  }
  if (VAR == 1 || VAR == 3) {
    // eight neighbours per round: their columns and values first, then the gathers, then the
    // FMAs (more loads in flight per thread).  Past the row's end the round re-reads entry kb
    // (kb < len), so every load is unconditional and inside the slice, with weight 0.
    for (int kb = k0; kb < len; kb += 8 * kstep) {
      int j[8];
      V w[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const int k = kb + u * kstep;
        const int kc = k < len ? k : kb;
        j[u] = __ldcs(cp + (int64_t)kc * 32);
        const V wv = __ldcs(vp + (int64_t)kc * 32);
        w[u] = k < len ? wv : V(0);
      }
#pragma unroll
      for (int r = 0; r < NR; ++r)
        if (!skip[r]) {
          X g[8];
#pragma unroll
          for (int u = 0; u < 8; ++u) g[u] = __ldg(x + r * ld + j[u]) - xi[r];
#pragma unroll
          for (int u = 0; u < 8; ++u) acc[r] += (Acc)w[u] * (Acc)g[u];
        }
    }
    return;
  }
#pragma unroll 4
  for (int k = k0; k < len; k += kstep) {
    const int j = __ldcs(cp + (int64_t)k * 32);
    const Acc a = (Acc)__ldcs(vp + (int64_t)k * 32);
#pragma unroll
    for (int r = 0; r < NR; ++r)
      if (!skip[r]) acc[r] += a * (Acc)(__ldg(x + r * ld + j) - xi[r]);
  }
}

// Values of a stored 3x3 block: B = 9 row-major, B = 6 the upper triangle (00, 01, 02, 11, 12, 22)
// of a symmetric block.  blk(a, b) is the position of A_ab.  Every block of K^mech is symmetric on
// a periodic mesh with one stiffness: integrating d_c phi_i d_d phi_j by parts twice swaps c and d,
// and the quadrature is exact for that difference.  The product is bound by its value stream, so
// storing 6 of 9 values takes 28 instead of 40 bytes per FP32 entry (column index included):
// 289 -> 217 us per FP32 launch at 2,963,088 nodes (1.317 GB, 6.06 TB/s), 58 -> 46 us at 524,288.
template <int B>
__device__ __forceinline__ constexpr int blk(int a, int b) {
  return B == 9 ? 3 * a + b : (a <= b ? 3 * a - a * (a - 1) / 2 + b - a : 3 * b - b * (b - 1) / 2 + a - b);
}

// 3x3-block row: y(row, a) = sum_k sum_b A(row, k)_ab x(col, b); x, y arrays of [n][3].
// diff != 0: sum_k A(row, k) (x(col) - x(row)), as in sell_scalar_row.
template <int B, typename V, typename X, typename Acc, int VAR>
__device__ __forceinline__ void sell_block_row(const DSell& A, const V* __restrict__ val,
                                               int64_t s, int lane, const X* __restrict__ x,
                                               Acc (&acc)[3], int k0 = 0, int kstep = 1,
                                               int diff = 0) {
  const int64_t base = A.sptr[s];
  const int len = A.slen[s];
  const int32_t* cp = A.col + base + lane;
  const V* vp = val + base * B + lane;
  const int64_t row = s * 32 + lane;
  const bool own = diff && row < A.n;
  const X xi0 = own ? x[3 * row] : X(0), xi1 = own ? x[3 * row + 1] : X(0),
          xi2 = own ? x[3 * row + 2] : X(0);
  acc[0] = acc[1] = acc[2] = Acc(0);
  if (VAR == 1 || VAR == 3) {
    // five neighbours per round: all loads first, then the FMAs; past the row's end entry kb
    // is re-read with weight 0 (unconditional loads, all inside the slice)
    for (int kb = k0; kb < len; kb += 5 * kstep) {
      int j[5];  // 32-bit: five fewer registers than 64-bit indices in this unrolled round
      V w[5][B];
#pragma unroll
      for (int u = 0; u < 5; ++u) {
        const int k = kb + u * kstep;
        const bool ok = k < len;
        const int kc = ok ? k : kb;
        j[u] = __ldcs(cp + (int64_t)kc * 32);
        const V* bp = vp + (int64_t)kc * (32 * B);
#pragma unroll
        for (int e = 0; e < B; ++e) {
          const V wv = __ldcs(bp + e * 32);
          w[u][e] = ok ? wv : V(0);
        }
      }
#pragma unroll
      for (int u = 0; u < 5; ++u) {
        const X* xj = x + 3 * (int64_t)j[u];
        const Acc x0 = (Acc)(__ldg(xj) - xi0), x1 = (Acc)(__ldg(xj + 1) - xi1),
                  x2 = (Acc)(__ldg(xj + 2) - xi2);
#pragma unroll
        for (int a = 0; a < 3; ++a)
          acc[a] += (Acc)w[u][blk<B>(a, 0)] * x0 + (Acc)w[u][blk<B>(a, 1)] * x1 +
                    (Acc)w[u][blk<B>(a, 2)] * x2;
      }
    }
  } else {
#pragma unroll 2
    for (int k = k0; k < len; k += kstep) {
      const int64_t j = __ldcs(cp + (int64_t)k * 32);
      const V* bp = vp + (int64_t)k * (32 * B);
      const Acc x0 = (Acc)(__ldg(x + 3 * j) - xi0), x1 = (Acc)(__ldg(x + 3 * j + 1) - xi1),
                x2 = (Acc)(__ldg(x + 3 * j + 2) - xi2);
      V w[B];
#pragma unroll
      for (int e = 0; e < B; ++e) w[e] = __ldcs(bp + e * 32);
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        acc[a] += (Acc)w[blk<B>(a, 0)] * x0;
        acc[a] += (Acc)w[blk<B>(a, 1)] * x1;
        acc[a] += (Acc)w[blk<B>(a, 2)] * x2;
      }
    }
  }
}

// Compensated dot product in FP32 (Ogita, Rump and Oishi, "Accurate sum and dot product", SIAM
// J. Sci. Comput. 26 (2005), Algorithm Dot2): each product is split exactly into p + e with an
// FMA, the running sum kept exactly as s plus the accumulated errors c by Knuth's TwoSum, so
// s + c is as accurate as the dot product computed in twice the working precision.  The CG
// initial residuals b - A x (which cancel heavily with a warm start) use it instead of FP64
// arithmetic, whose rate on this part is 1/64 of FP32's.
struct Dot2 {
  float s = 0.f, c = 0.f;
  // the _rn intrinsics keep the compiler from contracting or reassociating these steps
  __device__ __forceinline__ void add(float a, float b) {
    const float p = __fmul_rn(a, b);
    const float e = fmaf(a, b, -p);
    const float t = __fadd_rn(s, p);
    const float z = __fsub_rn(t, s);
    const float d = __fadd_rn(__fsub_rn(s, __fsub_rn(t, z)), __fsub_rn(p, z));
    c = __fadd_rn(c, __fadd_rn(d, e));
    s = t;
  }
  __device__ __forceinline__ double value() const { return (double)s + (double)c; }
};

// sell_scalar_row / sell_block_row with Dot2 accumulators (FP32 operands)
template <int NR>
__device__ __forceinline__ void sell_scalar_row_dot2(const DSell& A, const float* __restrict__ val,
                                                     int64_t s, int lane,
                                                     const float* __restrict__ x, int64_t ld,
                                                     Dot2 (&acc)[NR], int diff = 0) {
  const int64_t base = A.sptr[s];
  const int len = A.slen[s];
  const int32_t* cp = A.col + base + lane;
  const float* vp = val + base + lane;
  const int64_t row = s * 32 + lane;
  float xi[NR];
#pragma unroll
  for (int r = 0; r < NR; ++r) xi[r] = diff && row < A.n ? x[r * ld + row] : 0.f;
#pragma unroll 4
  for (int k = 0; k < len; ++k) {
    const int j = __ldcs(cp + (int64_t)k * 32);
    const float a = __ldcs(vp + (int64_t)k * 32);
#pragma unroll
    for (int r = 0; r < NR; ++r) acc[r].add(a, __fsub_rn(__ldg(x + r * ld + j), xi[r]));
  }
}
template <int B>
__device__ __forceinline__ void sell_block_row_dot2(const DSell& A, const float* __restrict__ val,
                                                    int64_t s, int lane,
                                                    const float* __restrict__ x,
                                                    Dot2 (&acc)[3], int diff = 0) {
  const int64_t base = A.sptr[s];
  const int len = A.slen[s];
  const int32_t* cp = A.col + base + lane;
  const float* vp = val + base * B + lane;
  const int64_t row = s * 32 + lane;
  const bool own = diff && row < A.n;
  const float xi0 = own ? x[3 * row] : 0.f, xi1 = own ? x[3 * row + 1] : 0.f,
              xi2 = own ? x[3 * row + 2] : 0.f;
#pragma unroll 2
  for (int k = 0; k < len; ++k) {
    const int64_t j = __ldcs(cp + (int64_t)k * 32);
    const float* bp = vp + (int64_t)k * (32 * B);
    const float x0 = __fsub_rn(__ldg(x + 3 * j), xi0), x1 = __fsub_rn(__ldg(x + 3 * j + 1), xi1),
                x2 = __fsub_rn(__ldg(x + 3 * j + 2), xi2);
    float w[B];
#pragma unroll
    for (int e = 0; e < B; ++e) w[e] = __ldcs(bp + e * 32);
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      acc[a].add(w[blk<B>(a, 0)], x0);
      acc[a].add(w[blk<B>(a, 1)], x1);
      acc[a].add(w[blk<B>(a, 2)], x2);
    }
  }
}

// Work unit of the SELL kernels for schedule VAR: one slice per warp (VAR 0, 1), or half a slice
// per warp with two lanes per row (VAR 2).  unit_row() gives, for this lane, the slice, the SELL
// lane of its row, and the first neighbour and stride it handles.
template <int VAR>
__device__ __forceinline__ void unit_row(int64_t u, int lane, int64_t& s, int& sl, int& k0,
                                         int& kstep) {
  if (VAR == 2) {
    s = u >> 1;
    sl = (int)(u & 1) * 16 + (lane & 15);
    k0 = lane >> 4;
    kstep = 2;
  } else {
    s = u;
    sl = lane;
    k0 = 0;
    kstep = 1;
  }
}
// minimum resident blocks per SM a schedule is compiled for (register cap)
template <int VAR>
constexpr int min_blocks() {
  return VAR == 3 ? 3 : 1;
}
template <int VAR>
__device__ __forceinline__ int units_per_slice() {
  return VAR == 2 ? 2 : 1;
}
// combine the two partial row results of VAR 2 (lanes l and l+16); true on the lane that owns
// the row's result
template <int VAR, typename Acc, int N>
__device__ __forceinline__ bool unit_combine(Acc (&acc)[N], int lane) {
  if (VAR != 2) return true;
#pragma unroll
  for (int a = 0; a < N; ++a) acc[a] += __shfl_xor_sync(kFull, acc[a], 16);
  return lane < 16;
}

}  // namespace

}  // namespace gspm
