// A whole CG loop as one kernel: the iterations of one solve run in a persistent cooperative grid
// (at most one block per SM) instead of three to seven launches each.
//
// Why: on the sizes whose operators fit the L2, an iteration's kernels take about 8 us each however
// small their work is (launch, wait for the grid before, block reductions, the last item's sum), so
// a solve is a serial chain of latencies.  Here a block keeps its rows for the whole solve, their
// r, q, p, x and D^-1 stay in its shared memory as far as they fit, and the blocks exchange only
// what others need.
//
// Exchanges.  Values travel as packets of two 64-bit words, each half a value and half the
// exchange's number, so a reader recognises a fresh word by itself: no fence and no counter.  What
// costs is the hop (store to seen: about 1400 cycles between any two SMs) and polling by many: the
// same packets polled by all 152 blocks take 8000 cycles, a line that one block polls 1400.  So
//  - partial sums go to the mesh's leader (its first block), which sums them in block order, takes
//    the decisions and writes the scalars to one line per block (two hops);
//  - the restricted residual goes to a few server blocks, which apply the dense coarse inverse and
//    post each aggregate's correction for the blocks that hold its rows.  r.z and the mean of z
//    come from the parts, r.D^-1 r + r_c.e_c, so no block waits for z itself;
//  - p, gathered by neighbours in bulk, is published as packets too, so a gather waits by itself
//    for exactly the rows it needs.  The gather reads twice the bytes, from L2; with plain values
//    and a barrier (one counter, one polling thread per block: 2400 cycles) a step took 27.0 against
//    24.8 ms at 198,400 nodes and 54.9 against 51.2 ms at 524,288.
// A slot is written again only after its readers have answered (argued at each).  Every wait is
// bounded (LoopPart::polls): a block that gives up sets *err and returns, so do the others once their
// own waits run out, and the loops that are queued behind return at once, until the host has taken
// the context off the fused loops.
//
// Meshes of a batch are independent groups of blocks: they neither wait for one another nor stop
// together.  Their exchange numbers drift apart, so their packets lie in ranges of their own
// (looplayout.h; ex and line are per block).
//
// Measured, separate kernels -> fused: three mixed steps at 19,305 nodes 44.0 -> 16.4 ms, at 65,536
// 56.4 -> 20.4; two FP64 steps at 65,536 hexahedra 44.9 -> 25.0; an elastic solve at 152,969 nodes
// 14.9 -> 7.2 ms; larger sizes at kLoopRows.  Cycles of a K^mech iteration (clock64 in the leader's and a
// server's first thread, mean of a solve):
//                            19,305 mixed   65,536 mixed   152,969 mixed   65,536 hexahedra FP64
//   product                        6,650         13,700          31,700          86,400
//   p.q at the leader, summed      6,200          7,100           8,400          11,300
//   alpha, lines to the blocks     3,350          3,400           3,150           3,750
//   vectors, pieces                3,430          3,750           6,650          16,100
//   server: pieces arrive          3,700          3,850           4,050           5,100
//     gather, inverse x pieces     8,800          5,050           5,200           6,300
//   leader: sums arrive            4,350          6,200           4,800           5,500
//     decisions                    2,600          3,050           3,100           2,800
//   beta, correction received      2,350          1,600           2,400           2,700
//   p                                900          1,300           2,700           2,900
// (a hop between two SMs is 1,400).  So up to 65,536 nodes the serial sections of the leader and the
// servers and the hops between them bound it, not bandwidth; in FP64 the product does, by the FP64 pipe
// (27 x 9 multiply-adds per row at two per clock and SM).  The kernels spill (128 registers per thread at
// 512 threads: 596 bytes loaded in the mixed K^mech loop, 380 in FP64, none in the plain scalar ones).
// Tried, no faster: clusters of 4 to 16 blocks with the sums in distributed shared memory (12.4 to
// 14.7 ms for four FP64 steps at 1,024 nodes that took 12.4 without, 29.7 for three mixed ones at 65,536
// that took 21.0: fewer SMs hold clusters), helper functions out of line, and warps waiting by
// nanosleep instead of at the barrier.
#include <cuda_runtime.h>

#include <cstdint>

#include "device.cuh"
#include "kernels.cuh"
#include "looplayout.h"
#include "sum3.h"

namespace gspm {

namespace {

constexpr int kNW = kLoopThreads / 32;
constexpr int kPolls = kLoopMaxBlocks / 32;  // packets per lane

enum { kExPq = 0, kExRr = 1, kExCo = 2 };    // sums to the leader: p.q, of the residual, of servers
enum { kLnAlpha = 0, kLnBeta = 1, kLnPin = 2 };  // lines from the leader

// ---- packets ---------------------------------------------------------------------------------
__device__ __forceinline__ void st_pair(ulonglong2* p, uint64_t a, uint64_t b) {
  asm volatile("st.relaxed.gpu.global.v2.b64 [%0], {%1, %2};" ::"l"(p), "l"(a), "l"(b) : "memory");
}
__device__ __forceinline__ ulonglong2 ld_pair(const ulonglong2* p) {
  ulonglong2 v;
  asm volatile("ld.relaxed.gpu.global.v2.b64 {%0, %1}, [%2];"
               : "=l"(v.x), "=l"(v.y) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void st_word(uint64_t* p, uint64_t a) {
  asm volatile("st.relaxed.gpu.global.b64 [%0], %1;" ::"l"(p), "l"(a) : "memory");
}
__device__ __forceinline__ uint64_t ld_word(const uint64_t* p) {
  uint64_t v;
  asm volatile("ld.relaxed.gpu.global.b64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ uint64_t word(uint32_t ep, uint32_t v) { return (uint64_t)ep << 32 | v; }
__device__ __forceinline__ bool fresh(uint64_t w, uint32_t ep) { return (uint32_t)(w >> 32) == ep; }
__device__ __forceinline__ bool fresh(const ulonglong2& w, uint32_t ep) {
  return fresh(w.x, ep) && fresh(w.y, ep);
}
// an FP64 value, or an unevaluated FP32 sum hi + lo
__device__ __forceinline__ void post(ulonglong2* s, double v, uint32_t ep) {
  const uint64_t b = (uint64_t)__double_as_longlong(v);
  st_pair(s, word(ep, (uint32_t)b), word(ep, (uint32_t)(b >> 32)));
}
__device__ __forceinline__ void post(ulonglong2* s, double hi, double lo, uint32_t ep) {
  post(s, hi + lo, ep);
}
__device__ __forceinline__ void post(ulonglong2* s, float hi, float lo, uint32_t ep) {
  st_pair(s, word(ep, __float_as_uint(hi)), word(ep, __float_as_uint(lo)));
}
__device__ __forceinline__ double value(const ulonglong2& w) {
  return __longlong_as_double((long long)((w.x & 0xffffffffull) | (w.y << 32)));
}
__device__ __forceinline__ void pair_of(const ulonglong2& w, float& h, float& l) {
  h = __uint_as_float((uint32_t)w.x);
  l = __uint_as_float((uint32_t)w.y);
}
__device__ __forceinline__ void pair_of(const ulonglong2& w, double& h, double& l) {
  h = value(w);
  l = 0.0;
}
// ---- sums ------------------------------------------------------------------------------------
// (h, l) += (bh, bl): double-float in FP32, plain in FP64 (l unused)
__device__ __forceinline__ void pair_add(float& h, float& l, float bh, float bl) {
  df_add(h, l, bh, bl);
}
__device__ __forceinline__ void pair_add(double& h, double&, double bh, double) { h += bh; }

__host__ __device__ constexpr int pow2(int v) { return v <= 1 ? 1 : (v <= 2 ? 2 : (v <= 4 ? 4 : 8)); }

template <typename T>
struct RedBuf {
  T hi[8][kNW], lo[8][kNW];
};

// Per-thread sums hi + lo of V values to one pair per warp in R.  The lanes halve the values among
// themselves as they halve the distance (V = 8: 4 + 2 + 1 + 1 + 1 additions instead of 8 x 5): with
// every warp of the block in it the additions are what it costs, in FP64 16 cycles each.  A warp
// that holds no rows (idle) only writes its zeros.
template <typename T, int V>
__device__ __forceinline__ void warp_partials(const T (&hi)[V], const T (&lo)[V], RedBuf<T>& R,
                                              bool idle) {
  constexpr int VP = pow2(V);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (idle) {
    if (lane < V) R.hi[lane][warp] = R.lo[lane][warp] = T(0);
    return;
  }
  T h[VP], l[VP];
#pragma unroll
  for (int v = 0; v < VP; ++v) {
    h[v] = v < V ? hi[v] : T(0);
    l[v] = v < V ? lo[v] : T(0);
    if (sizeof(T) == 8) {
      h[v] += l[v];
      l[v] = T(0);
    }
  }
  int idx = 0, o = 16;
#pragma unroll
  for (int half = VP / 2; half >= 1; half >>= 1, o >>= 1) {
    const bool up = lane & o;
    if (up) idx += half;
#pragma unroll
    for (int i = 0; i < half; ++i) {
      const T sh = up ? h[i] : h[i + half], sl = up ? l[i] : l[i + half];
      T kh = up ? h[i + half] : h[i], kl = up ? l[i + half] : l[i];
      const T bh = __shfl_xor_sync(kFull, sh, o);
      const T bl = sizeof(T) == 4 ? __shfl_xor_sync(kFull, sl, o) : T(0);
      pair_add(kh, kl, bh, bl);
      h[i] = kh;
      l[i] = kl;
    }
  }
  for (; o >= 1; o >>= 1) {
    const T bh = __shfl_xor_sync(kFull, h[0], o);
    const T bl = sizeof(T) == 4 ? __shfl_xor_sync(kFull, l[0], o) : T(0);
    pair_add(h[0], l[0], bh, bl);
  }
  if ((lane & (32 / VP - 1)) == 0 && idx < V) {
    R.hi[idx][warp] = h[0];
    R.lo[idx][warp] = l[0];
  }
}

// The block's V sums (one warp, after a barrier that follows warp_partials) posted for the leader:
// value v of block slot b at ex[v * kLoopMaxBlocks + b].
template <typename T, int V>
__device__ __forceinline__ void post_sums(ulonglong2* ex, int b, uint32_t ep, const RedBuf<T>& R) {
  constexpr int VP = pow2(V), LPV = 32 / VP;  // lanes per value
  constexpr int PER = (kNW + LPV - 1) / LPV;  // warps per lane
  const int lane = threadIdx.x & 31, v = lane / LPV, j = lane % LPV;
  T h = T(0), l = T(0);
#pragma unroll
  for (int k = 0; k < PER; ++k) {
    const int w = j * PER + k;
    if (v < V && w < kNW) pair_add(h, l, R.hi[v][w], R.lo[v][w]);
  }
#pragma unroll
  for (int o = LPV / 2; o >= 1; o >>= 1) {
    const T bh = __shfl_down_sync(kFull, h, o, LPV);
    const T bl = sizeof(T) == 4 ? __shfl_down_sync(kFull, l, o, LPV) : T(0);
    pair_add(h, l, bh, bl);
  }
  if (j == 0 && v < V) post(ex + v * kLoopMaxBlocks + b, h, l, ep);
}

// Leader, one warp: the sum of the n packets at ex, in *out.  False: gave up.  The sum has FP64's
// precision, from FP64 additions or, for FP32 pairs, from Sum3: converted to FP64 the pairs of twelve
// values take 300 instructions of the FP64 pipe (16 cycles each), steps at 65,536 nodes 22.1 ms instead
// of 20.0 (double-float sums, of some 44 bits, 20.4).
template <typename T>
__device__ __forceinline__ bool sum_posts(const ulonglong2* ex, int n, uint32_t ep, uint32_t polls,
                                          double* out) {
  const int lane = threadIdx.x & 31;
  ulonglong2 w[kPolls];
  bool ok;
  do {
    ok = true;
#pragma unroll
    for (int u = 0; u < kPolls; ++u)
      if (lane + 32 * u < n) w[u] = ld_pair(ex + lane + 32 * u);
#pragma unroll
    for (int u = 0; u < kPolls; ++u)
      if (lane + 32 * u < n) ok = ok && fresh(w[u], ep);
  } while (!ok && --polls);
  if constexpr (sizeof(T) == 8) {
    double sum = 0.0;
#pragma unroll
    for (int u = 0; u < kPolls; ++u)
      if (lane + 32 * u < n) sum += value(w[u]);
    __syncwarp();
#pragma unroll
    for (int o = 16; o >= 1; o >>= 1) sum += __shfl_xor_sync(kFull, sum, o);
    if (lane == 0) *out = sum;
  } else {
    Sum3 t;
#pragma unroll
    for (int u = 0; u < kPolls; ++u)
      if (lane + 32 * u < n) {
        float h, l;
        pair_of(w[u], h, l);
        t.add(h, l, 0.f);
      }
    __syncwarp();
#pragma unroll
    for (int o = 16; o >= 1; o >>= 1)
      t.add(__shfl_xor_sync(kFull, t.s, o), __shfl_xor_sync(kFull, t.e, o),
            __shfl_xor_sync(kFull, t.f, o));
    if (lane == 0) *out = t.value();
  }
  return __all_sync(kFull, ok);
}

// One warp: payload k of a line into ln[k], k < n.  False: gave up.
__device__ __forceinline__ bool wait_line(const ulonglong2* line, int k, int n, uint32_t ep,
                                          uint32_t polls, uint2* ln) {
  bool ok = k >= n;
  if (!ok) {
    ulonglong2 w;
    do {
      w = ld_pair(line + k);
      ok = fresh(w, ep);
    } while (!ok && --polls);
    if (ok) ln[k] = make_uint2((uint32_t)w.x, (uint32_t)w.y);
  }
  __syncwarp();
  return ok;
}

// Values of n coarse packets from thread k0 on, every step-th, into dst (FP32: the high words; the low
// ones are posted as zero).  False: gave up.
template <typename T>
__device__ __forceinline__ bool wait_coarse(const ulonglong2* src, int k0, int step, int n, uint32_t ep,
                                            uint32_t polls, T* dst) {
  bool ok = true;
#pragma unroll 1
  for (int k = k0; ok && k < n; k += 4 * step) {
    ulonglong2 w[4];
    bool got;
    uint32_t left = polls;
    do {
      got = true;
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (k + u * step < n) w[u] = ld_pair(src + k + u * step);
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (k + u * step < n) got = got && fresh(w[u], ep);
    } while (!got && --left);
    ok = ok && got;
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (k + u * step < n) {
        T l;
        pair_of(w[u], dst[k + u * step], l);
      }
  }
  __syncwarp();
  return ok;
}

// Leader: the n payloads of out to the line of each of the nb blocks
__device__ __forceinline__ void send_lines(ulonglong2* lines, int nb, int n, uint32_t ep,
                                           const uint2* out) {
  for (int t = threadIdx.x; t < nb; t += kLoopThreads)
    for (int v = 0; v < n; ++v)
      st_pair(lines + (int64_t)t * 8 + v, word(ep, out[v].x), word(ep, out[v].y));
}

// Scalars in a line: FP32 values travel in pairs with the flags, FP64 values alone.
template <typename T, int NR, bool KS>
struct LineFormat;
template <int NR, bool KS>
struct LineFormat<float, NR, KS> {
  static constexpr int NA = NR, NB = NR + (KS ? 2 : 0);
  __device__ __forceinline__ static void put(uint2* o, int k, double v, uint32_t flags) {
    o[k] = make_uint2(__float_as_uint((float)v), flags);
  }
  __device__ __forceinline__ static void put_sub(uint2* o, const double (&s)[3]) {
    o[NR] = make_uint2(__float_as_uint((float)s[0]), __float_as_uint((float)s[1]));
    o[NR + 1] = make_uint2(__float_as_uint((float)s[2]), 0u);
  }
  __device__ __forceinline__ static float get(const uint2* l, int k) {
    return __uint_as_float(l[k].x);
  }
  __device__ __forceinline__ static uint32_t flags(const uint2* l) { return l[0].y; }
  __device__ __forceinline__ static float sub(const uint2* l, int c) {
    return __uint_as_float(c == 0 ? l[NR].x : (c == 1 ? l[NR].y : l[NR + 1].x));
  }
};
template <int NR, bool KS>
struct LineFormat<double, NR, KS> {
  static constexpr int NA = NR + 1, NB = NR + 1 + (KS ? 3 : 0);
  __device__ __forceinline__ static uint2 bits(double v) {
    return make_uint2((uint32_t)__double2loint(v), (uint32_t)__double2hiint(v));
  }
  __device__ __forceinline__ static double dbl(uint2 u) {
    return __hiloint2double((int)u.y, (int)u.x);
  }
  __device__ __forceinline__ static void put(uint2* o, int k, double v, uint32_t flags) {
    o[k] = bits(v);
    if (k == 0) o[NR] = make_uint2(flags, 0u);
  }
  __device__ __forceinline__ static void put_sub(uint2* o, const double (&s)[3]) {
    for (int c = 0; c < 3; ++c) o[NR + 1 + c] = bits(s[c]);
  }
  __device__ __forceinline__ static double get(const uint2* l, int k) { return dbl(l[k]); }
  __device__ __forceinline__ static uint32_t flags(const uint2* l) { return l[NR].x; }
  __device__ __forceinline__ static double sub(const uint2* l, int c) { return dbl(l[NR + 1 + c]); }
};

// All blocks of the group have published their global stores before any passes: arrivals counted in
// *count, which reaches `target`.  False: gave up.
__device__ __forceinline__ bool group_barrier(uint32_t* count, uint32_t target, uint32_t polls) {
  __syncthreads();
  bool ok = true;
  if (threadIdx.x == 0) {
    asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(count) : "memory");
    do {
      uint32_t v;
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(count) : "memory");
      ok = (int32_t)(v - target) >= 0;
    } while (!ok && --polls);
  }
  return __syncthreads_and(ok);
}

// ---- rows ------------------------------------------------------------------------------------
// rows of one block in a vector: element (c, local row) of [n][3] (AOS) or component-major storage,
// in shared or global memory
template <typename T, bool AOS>
struct Rows {
  T* b;
  int64_t cs;
  __device__ __forceinline__ T& at(int c, int64_t lr) const {
    return AOS ? b[3 * lr + c] : b[c * cs + lr];
  }
};

// p as packets: FP32 one word per value, FP64 two
__device__ __forceinline__ void put_p(void* pp, int64_t i, float v, uint32_t ep) {
  st_word(static_cast<uint64_t*>(pp) + i, word(ep, __float_as_uint(v)));
}
__device__ __forceinline__ void put_p(void* pp, int64_t i, double v, uint32_t ep) {
  post(static_cast<ulonglong2*>(pp) + i, v, ep);
}
template <typename T> struct PWord;
template <> struct PWord<float> {
  using W = uint64_t;
  __device__ __forceinline__ static W ld(const void* pp, int64_t i) {
    return ld_word(static_cast<const uint64_t*>(pp) + i);
  }
  __device__ __forceinline__ static float val(W w) { return __uint_as_float((uint32_t)w); }
};
template <> struct PWord<double> {
  using W = ulonglong2;
  __device__ __forceinline__ static W ld(const void* pp, int64_t i) {
    return ld_pair(static_cast<const ulonglong2*>(pp) + i);
  }
  __device__ __forceinline__ static double val(const W& w) { return value(w); }
};

// Part of one SELL row's product with p, neighbours k0, k0 + ks, ...: a round's columns and values
// are all loaded before its gathers.  p is read as packets of exchange ep; a lane past the
// mesh's last row (not valid: its columns point at itself) reads none.  False: gave up.
template <typename T, int B, int NR, bool DIFF>
__device__ __forceinline__ bool row_part(const DSell& A, const T* __restrict__ val, int64_t s,
                                         int lane, const void* pp, uint32_t ep, uint32_t polls,
                                         const T (&xi)[B == 1 ? NR : 3], unsigned skip,
                                         bool valid, T (&acc)[B == 1 ? NR : 3], int k0, int ks) {
  constexpr int NV = B == 1 ? NR : 3;
  const int64_t base = A.sptr[s];
  const int len = A.slen[s];
  const int32_t* cp = A.col + base + lane;
  const T* vp = val + base * B + lane;
#pragma unroll
  for (int c = 0; c < NV; ++c) acc[c] = T(0);
  // neighbours per round: what the registers hold (FP64 packets take four each)
  constexpr int U = sizeof(T) == 4 ? (B == 1 && NR < 3 ? 8 : 5) : (B == 1 && NR == 1 ? 5 : 2);
  using PW = PWord<T>;
  for (int kb = k0; kb < len; kb += U * ks) {
    int j[U];
    T w[U][B];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      // past the row's end (k is the same for the whole warp): entry kb again, not used
      const int k = kb + u * ks < len ? kb + u * ks : kb;
      j[u] = __ldcs(cp + (int64_t)k * 32);
      const T* bp = vp + (int64_t)k * (32 * B);
#pragma unroll
      for (int e = 0; e < B; ++e) w[u][e] = __ldcs(bp + e * 32);
    }
    typename PW::W x[U][NV];
    for (uint32_t left = polls;;) {
      bool ok = true;
#pragma unroll
      for (int u = 0; u < U; ++u)
#pragma unroll
        for (int c = 0; c < NV; ++c) {
          const int64_t i = B != 1 ? p_packet3(j[u], c) : (NR == 1 ? p_packet1(j[u]) : p_packet1(j[u], c));
          if (B != 1 || !(skip >> c & 1)) x[u][c] = PW::ld(pp, i);
        }
#pragma unroll
      for (int u = 0; u < U; ++u)
#pragma unroll
        for (int c = 0; c < NV; ++c)
          if (B != 1 || !(skip >> c & 1)) ok &= fresh(x[u][c], ep);
      if (__all_sync(kFull, ok || !valid)) break;
      if (!--left) return false;
    }
    auto get = [&](int u, int c) -> T {
      const T v = PW::val(x[u][c]);
      return DIFF ? v - xi[c] : v;
    };
#pragma unroll
    for (int u = 0; u < U; ++u)
      if (kb + u * ks < len) {
        if constexpr (B == 1) {
#pragma unroll
          for (int c = 0; c < NV; ++c)
            if (!(skip >> c & 1)) acc[c] += w[u][0] * get(u, c);
        } else {
          const T v[3] = {get(u, 0), get(u, 1), get(u, 2)};
#pragma unroll
          for (int a = 0; a < 3; ++a)
            acc[a] += w[u][blk<B>(a, 0)] * v[0] + w[u][blk<B>(a, 1)] * v[1] +
                      w[u][blk<B>(a, 2)] * v[2];
        }
      }
  }
  return true;
}

template <typename S>
struct FullPack;
template <>
struct FullPack<uint16_t> {
  static constexpr int W = 8;
  __device__ __forceinline__ static float dot(const uint16_t* a, const float* x) {
    const uint4 u = __ldg(reinterpret_cast<const uint4*>(a));
    const float4 v[2] = {reinterpret_cast<const float4*>(x)[0],
                         reinterpret_cast<const float4*>(x)[1]};
    const uint32_t w[4] = {u.x, u.y, u.z, u.w};
    const float xv[8] = {v[0].x, v[0].y, v[0].z, v[0].w, v[1].x, v[1].y, v[1].z, v[1].w};
    float s = 0.f;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      s += __uint_as_float(w[k] << 16) * xv[2 * k];  // bfloat16 -> float is exact
      s += __uint_as_float(w[k] & 0xffff0000u) * xv[2 * k + 1];
    }
    return s;
  }
};
template <>
struct FullPack<double> {
  static constexpr int W = 2;
  __device__ __forceinline__ static double dot(const double* a, const double* x) {
    const double2 u = __ldg(reinterpret_cast<const double2*>(a));
    return u.x * x[0] + u.y * x[1];
  }
};

// The loop.  PC 0: plain CG (KS: K^ms / K^mech, pinned or projected singular; else a GSPM system),
// 1: two-level preconditioner, 2: Jacobi (GSPM systems).  The scalars and decisions are those of
// k_cg_spmv, k_cg_update, k_pcg_z and k_cg_pupdate.
template <typename T, int B, int NR, int PC, bool KS>
__global__ void __launch_bounds__(kLoopThreads, 1) k_cg_loop(CgLoop<T> a) {
  constexpr int NC = B == 1 ? 1 : 3;        // components per row of one right-hand side
  constexpr int NV = B == 1 ? NR : 3;       // values per row
  constexpr bool AOS = B != 1;
  constexpr bool DIFF = KS && kDiff<T>;
  // sums of the residual: r.r; two-level and projected: sums of r; r.D^-1 r; two-level: of D^-1 r
  constexpr int VR = PC == 1 ? 2 + 2 * NC : (PC == 2 ? 2 * NR : (KS ? 1 + NC : NR));
  using S = typename CoarseStore<T>::type;
  using LF = LineFormat<T, NR, KS>;
  extern __shared__ __align__(16) unsigned char dyn[];
  __shared__ RedBuf<T> R, RC;
  __shared__ CGState s;                     // leader: the mesh's CG scalars
  __shared__ double tot[8], totc[4];
  __shared__ uint2 out[8];                  // leader: the line being sent
  __shared__ uint2 ln[8];                   // the last line from the leader
  __shared__ int s_fail;

  const LoopPart& P = a.part;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int blk = blockIdx.x, seg = P.seg[blk];
  const int b0 = P.seg_b0[seg], nb = P.seg_b0[seg + 1] - b0;
  const bool leader = blk == b0;
  const int sl0 = P.sl0[blk], nsl = P.sl1[blk] - sl0;
  const int64_t row0 = (int64_t)sl0 * 32;
  const int64_t rend = a.G.seg_row0[seg] + a.G.seg_nrow[seg];
  const int64_t pin = a.pinned ? a.G.seg_pin[seg] : -1;
  uint32_t ep = P.epoch[2 * seg], bars = P.epoch[2 * seg + 1];
  // few slices per block: `split` warps share a slice, each taking every split-th neighbour
  int split = 1;
  while (2 * split * nsl <= kNW) split *= 2;
  const int my0 = split == 1 ? warp : (warp % split == 0 ? warp / split : nsl);
  const int mystep = split == 1 ? kNW : nsl;
  const bool idle = my0 >= nsl;

  // shared memory: the layout of loop_smem
  const LoopSmem M = loop_smem<T>(NC, NR, PC, a.place, P);
  T* comb = reinterpret_cast<T*>(dyn + M.comb);
  T* psum = reinterpret_cast<T*>(dyn + M.psum);
  T* pieces = reinterpret_cast<T*>(dyn + M.pieces);
  T* rcs = reinterpret_cast<T*>(dyn + M.rc);
  T* ecl = reinterpret_cast<T*>(dyn + M.ec);
  int* prow = reinterpret_cast<int*>(dyn + M.prow);
  const int64_t gofs = AOS ? 3 * row0 : row0;
  auto place = [&](int k, T* g) {
    return k < a.place ? Rows<T, AOS>{reinterpret_cast<T*>(dyn + M.vec[k]), P.max_rows}
                       : Rows<T, AOS>{g + gofs, a.ld};
  };
  const Rows<T, AOS> r = place(0, a.r), q = place(1, a.q), p = place(2, a.p), x = place(3, a.x);
  const Rows<T, AOS> gp{a.p + gofs, a.ld}, gx{a.x + gofs, a.ld}, gr{a.r + gofs, a.ld};
  const Rows<T, AOS> gd{const_cast<T*>(a.dinv) + gofs, a.ld};
  const Rows<T, AOS> di = PC == 0 ? gd : place(4, const_cast<T*>(a.dinv));
  void* const pp = B == 1 && NR == 1 ? P.pp1 : P.pp;
  auto publish = [&](int c, int64_t lr, T v) {  // v is row lr's new p
    p.at(c, lr) = v;
    const int row = (int)(row0 + lr);
    put_p(pp, AOS ? p_packet3(row, c) : (NR == 1 ? p_packet1(row) : p_packet1(row, c)), v, ep);
  };
  ulonglong2* line = P.line + (int64_t)blk * 8;  // + kLn* * kLoopLines

  // aggregates of this block's rows, and the coarse rows it serves
  constexpr int CI = NC == 3 ? 0 : 1;
  const int pc0 = PC == 1 ? P.pc0[blk] : 0, np = PC == 1 ? P.pc0[blk + 1] - pc0 : 0;
  const int agg0 = PC == 1 ? a.C.seg_agg0[seg] : 0;
  const int nagg = PC == 1 ? a.C.seg_agg0[seg + 1] - agg0 : 0;
  const int segp0 = PC == 1 ? P.ap[agg0] : 0, segp = PC == 1 ? P.ap[agg0 + nagg] - segp0 : 0;
  const int la0 = PC == 1 ? a.C.agg_of_row[row0] : 0;
  const int ldc = PC == 1 ? P.inv_ld[CI][seg] : 0;
  int ns = 0, g0 = 0, g1 = 0;  // servers of the mesh, coarse rows of this block
  if (PC == 1) {
    const int64_t nc = (int64_t)nagg * NC;
    const int64_t want = nc * nc / kLoopServe<T>;
    ns = (int)(want < 1 ? 1 : (want < nb ? want : nb));
    if (blk - b0 < ns) {
      g0 = (int)((blk - b0) * nc / ns);
      g1 = (int)((blk - b0 + 1) * nc / ns);
    }
  }
  if (tid == 0) {
    s = a.st[seg];
    s_fail = *(const volatile int*)P.err;
  }
  if (PC == 1) {
    for (int k = tid; k <= np; k += kLoopThreads)
      prow[k] = (int)(k < np ? P.pc_row[pc0 + k] - row0 : (int64_t)nsl * 32);
    for (int k = tid; k < ldc; k += kLoopThreads) rcs[k] = T(0);
  }
  __syncthreads();
  // a loop before this one gave up: its exchange numbers are not to be met again
  if (s_fail) return;
  const bool active = s.active;
  const bool proj = KS && s.proj;
  unsigned skip = 0;  // right-hand sides that are done, by value of a row
  if (!AOS)
#pragma unroll
    for (int k = 0; k < NR; ++k) skip |= s.r[k].done ? 1u << k : 0u;
  const double inv_n = leader && tid == 0 ? 1.0 / (double)a.G.seg_nrow[seg] : 0.0;
  if (active) {
    if (PC != 1) ++ep;
    for (int ls = my0; ls < nsl; ls += mystep) {
      const int64_t lr = (int64_t)ls * 32 + lane;
      const bool ok = row0 + lr < rend;
#pragma unroll
      for (int c = 0; c < NV; ++c) {
        if (a.place > 0) r.at(c, lr) = ok ? gr.at(c, lr) : T(0);
        if (a.place > 3 && ok) x.at(c, lr) = gx.at(c, lr);
        if (PC != 1 && ok) publish(c, lr, gp.at(c, lr));
      }
      if (PC != 0 && a.place > 4 && ok) {
#pragma unroll
        for (int c = 0; c < NC; ++c) di.at(c, lr) = gd.at(c, lr);
      }
    }
    __syncthreads();  // warps that share a slice read its rows of p
  }
  bool first = PC == 1;
  bool failed = false;
  while (active) {
    if (!first) {
      // q = A p, p.q
      T pq[NR], pl[NR];
#pragma unroll
      for (int k = 0; k < NR; ++k) pq[k] = pl[k] = T(0);
      auto finish = [&](int64_t lr, T (&acc)[NV]) {
        const int64_t row = row0 + lr;
        if (row >= rend) return;
        if (KS && row == pin) {
#pragma unroll
          for (int c = 0; c < NV; ++c) acc[c] = T(0);
        }
        if (AOS) {
          T t = T(0);
#pragma unroll
          for (int c = 0; c < NV; ++c) {
            q.at(c, lr) = acc[c];
            t += p.at(c, lr) * acc[c];
          }
          kahan_add(pq[0], pl[0], t);
        } else {
#pragma unroll
          for (int k = 0; k < NR; ++k)
            if (!(skip >> k & 1)) {
              q.at(k, lr) = acc[k];
              kahan_add(pq[k], pl[k], p.at(k, lr) * acc[k]);
            }
        }
      };
      bool ok = true;
      auto part = [&](int ls, int k0, int ks, T (&acc)[NV]) {
        const int64_t lr = (int64_t)ls * 32 + lane;
        T xi[NV];
#pragma unroll
        for (int c = 0; c < NV; ++c) xi[c] = DIFF && row0 + lr < rend ? p.at(c, lr) : T(0);
        ok = ok && row_part<T, B, NR, DIFF>(a.A, a.val, sl0 + ls, lane, pp, ep, P.polls, xi,
                                            skip, row0 + lr < rend, acc, k0, ks);
      };
      if (split == 1) {
        for (int ls = warp; ls < nsl; ls += kNW) {
          T acc[NV];
          part(ls, 0, 1, acc);
          finish((int64_t)ls * 32 + lane, acc);
        }
      } else {
        const int ls = warp / split, sub = warp % split;
        T acc[NV];
        if (ls < nsl) {
          part(ls, sub, split, acc);
          if (sub)
#pragma unroll
            for (int c = 0; c < NV; ++c) comb[(warp * NV + c) * 32 + lane] = acc[c];
        }
        __syncthreads();
        if (ls < nsl && sub == 0) {
          for (int w = 1; w < split; ++w)
#pragma unroll
            for (int c = 0; c < NV; ++c) acc[c] += comb[((warp + w) * NV + c) * 32 + lane];
          finish((int64_t)ls * 32 + lane, acc);
        }
      }
      if (!ok) s_fail = 1;
#pragma unroll
      for (int k = 0; k < NR; ++k) pl[k] = -pl[k];
      warp_partials<T, NR>(pq, pl, R, idle);
      __syncthreads();
      ++ep;
      if (warp == 0) post_sums<T, NR>(P.ex + kExPq * kLoopExStride, blk, ep, R);
      if (leader) {
        if (warp < NR && !sum_posts<T>(P.ex + kExPq * kLoopExStride + warp * kLoopMaxBlocks + b0, nb,
                                       ep, P.polls, tot + warp))
          s_fail = 1;
        __syncthreads();
        if (warp == 0) {
          if (lane < NR) {
            CGRhs& c = s.r[lane];
            if (!c.done) {
              c.pq = tot[lane];
              if (c.pq > 0.0) {
                c.alpha = (PC != 0 ? c.rz : c.rr) / c.pq;
              } else {  // p = 0: nothing left to reduce
                c.alpha = 0.0;
                c.done = 1;
              }
            }
          }
          __syncwarp();
          const unsigned mask = __ballot_sync(kFull, lane < NR && s.r[lane < NR ? lane : 0].done);
          if (lane < NR) LF::put(out, lane, s.r[lane].alpha, mask);
        }
        __syncthreads();
        send_lines(P.line + kLnAlpha * kLoopLines + (int64_t)b0 * 8, nb, LF::NA, ep, out);
      }
      if (warp == 0 && !wait_line(line + kLnAlpha * kLoopLines, lane, LF::NA, ep, P.polls, ln))
        s_fail = 1;
      __syncthreads();
      if (s_fail) {
        failed = true;
        break;
      }
    }
    // x += alpha p, r -= alpha q, sums of the residual, restriction
    T hi[VR], lo[VR];
#pragma unroll
    for (int v = 0; v < VR; ++v) hi[v] = lo[v] = T(0);
    if (PC == 1) {
      for (int k = lane; k < np * NC; k += 32) psum[((k / NC) * kNW + warp) * NC + k % NC] = T(0);
      __syncwarp();
    }
    {
      T al[NR];
      const unsigned done = first ? 0u : LF::flags(ln);
#pragma unroll
      for (int k = 0; k < NR; ++k) al[k] = first ? T(0) : LF::get(ln, k);
      if (!AOS) skip = first ? skip : done;
      const bool stop = AOS && (done & 1);
      T comp = T(0);
      int pcur = 0;
      for (int ls = my0; ls < nsl; ls += mystep) {
        const int64_t lr = (int64_t)ls * 32 + lane;
        const bool ok = row0 + lr < rend;
        T rv[NV], t = T(0);
#pragma unroll
        for (int c = 0; c < NV; ++c) rv[c] = T(0);
        if (ok && !stop) {
#pragma unroll
          for (int c = 0; c < NV; ++c) {
            const int k = AOS ? 0 : c;
            if (skip >> c & 1) continue;
            rv[c] = r.at(c, lr);
            if (!first) {
              x.at(c, lr) += al[k] * p.at(c, lr);
              rv[c] -= al[k] * q.at(c, lr);
              r.at(c, lr) = rv[c];
            }
            hi[k] += rv[c] * rv[c];
            if (PC == 2) hi[NR + k] += rv[c] * di.at(0, lr) * rv[c];
            if (KS && PC != 2) hi[1 + (AOS ? c : 0)] += rv[c];
            if (PC == 1) {
              const T z = di.at(c, lr) * rv[c];
              t += rv[c] * z;
              hi[2 + NC + c] += z;
            }
          }
        }
        if (PC == 1) {
          kahan_add(hi[1 + NC], comp, t);
          const int beg = ls * 32, end = beg + 32;
          while (pcur + 1 < np && prow[pcur + 1] <= beg) ++pcur;
          for (int k = pcur; k < np && prow[k] < end; ++k) {
            const bool in = ok && lr >= prow[k] && lr < prow[k + 1];
#pragma unroll
            for (int c = 0; c < NC; ++c) {
              T v = in ? rv[c] : T(0);
#pragma unroll
              for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(kFull, v, o);
              if (lane == 0) psum[(k * kNW + warp) * NC + c] += v;
            }
          }
        }
      }
      if (PC == 1) lo[1 + NC] = -comp;
    }
    warp_partials<T, VR>(hi, lo, R, idle);
    __syncthreads();
    ++ep;
    if (warp == 0) {
      post_sums<T, VR>(P.ex + kExRr * kLoopExStride, blk, ep, R);
    } else if (PC == 1) {
      // this block's pieces of the restricted residual (read by the servers, which answer before
      // the leader's next line)
      for (int k = tid - 32; k < np * NC; k += kLoopThreads - 32) {
        T v = T(0);
#pragma unroll
        for (int w = 0; w < kNW; ++w) v += psum[((k / NC) * kNW + w) * NC + k % NC];
        post(P.rcx + coarse_packet(segp0, pc0, NC, k), v, T(0), ep);
      }
    }
    if (PC == 1 && g1 > g0) {
      // server: its rows of the dense inverse times the restricted residual; r_c.e_c and the sums of
      // P e_c for the leader
      if (!wait_coarse<T>(P.rcx + coarse_packet(segp0, segp0, NC, 0), tid, kLoopThreads, segp * NC, ep,
                          P.polls, pieces))
        s_fail = 1;
      __syncthreads();
      for (int k = tid; k < nagg * NC; k += kLoopThreads) {
        const int I = agg0 + k / NC;
        T v = T(0);
        for (int e = P.ap[I] - segp0; e < P.ap[I + 1] - segp0; ++e) v += pieces[e * NC + k % NC];
        rcs[k] = v;
      }
      __syncthreads();
      const S* inv = static_cast<const S*>(P.inv[CI]) + P.inv_off[CI][seg];
      T ch[1 + NC], cl[1 + NC];
#pragma unroll
      for (int v = 0; v < 1 + NC; ++v) ch[v] = cl[v] = T(0);
      for (int g = g0 + warp; g < g1; g += kNW) {
        const S* arow = inv + (int64_t)g * ldc;
        T t = T(0);
#pragma unroll 4
        for (int k = lane; k < ldc / FullPack<S>::W; k += 32)
          t += FullPack<S>::dot(arow + k * FullPack<S>::W, rcs + k * FullPack<S>::W);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) t += __shfl_down_sync(kFull, t, o);
        if (lane == 0) {
          // (read by the blocks of this aggregate's rows, which post their next pieces after it)
          post(P.ecx + coarse_packet(agg0, agg0, NC, g), t, T(0), ep);
          const int I = agg0 + g / NC;
          const T cnt = (T)(a.C.agg_ptr[I + 1] - a.C.agg_ptr[I]);
          pair_add(ch[0], cl[0], t * rcs[g], T(0));
#pragma unroll
          for (int c = 0; c < NC; ++c)
            if (g % NC == c) pair_add(ch[1 + c], cl[1 + c], cnt * t, T(0));
        }
      }
      if (lane == 0)
#pragma unroll
        for (int v = 0; v < 1 + NC; ++v) {
          RC.hi[v][warp] = ch[v];
          RC.lo[v][warp] = cl[v];
        }
      __syncthreads();
      if (warp == 0) post_sums<T, 1 + NC>(P.ex + kExCo * kLoopExStride, blk, ep, RC);
    }
    if (leader) {
      if (warp < VR) {
        if (!sum_posts<T>(P.ex + kExRr * kLoopExStride + warp * kLoopMaxBlocks + b0, nb, ep,
                          P.polls, tot + warp))
          s_fail = 1;
      } else if (PC == 1 && warp >= 8 && warp < 9 + NC) {
        if (!sum_posts<T>(P.ex + kExCo * kLoopExStride + (warp - 8) * kLoopMaxBlocks + b0, ns, ep,
                          P.polls, totc + warp - 8))
          s_fail = 1;
      }
      __syncthreads();
      if (tid == 0) {
        int any = first, mask = 0;
        double sub[3] = {0.0, 0.0, 0.0};
        for (int k = 0; k < NR; ++k) {
          CGRhs& c = s.r[k];
          if (!c.done && !first) {
            c.iters += 1;
            double rr = tot[k];
            if (proj) {
              // r.r without r's constant part; plain CG subtracts r's mean from its direction
              double s2 = 0.0;
              for (int d = 0; d < NC; ++d) {
                s.sr[d] = tot[1 + d];
                s2 += s.sr[d] * s.sr[d];
                if (PC == 0) sub[d] = s.sr[d] * inv_n;
              }
              rr -= s2 * inv_n;
              rr = rr > 0.0 ? rr : 0.0;
            }
            if (PC == 0) {
              c.beta = rr / c.rr;
            } else if (PC == 2) {
              c.beta = c.rz != 0.0 ? tot[NR + k] / c.rz : 0.0;
              c.rz = tot[NR + k];
            }
            c.rr = rr;
            if (rr < c.tol2) {
              c.done = 1;
            } else if (c.iters >= s.max_iter) {
              c.done = 1;
              s.noconv += 1;
            }
            any |= !c.done;
          }
          if (PC == 1 && any) {
            // r.z and the mean of z = D^-1 r + P e_c; z projected off the constants: r.(z - zbar 1)
            double rz = tot[1 + NC] + totc[0];
            if (proj)
              for (int d = 0; d < NC; ++d) {
                sub[d] = (tot[2 + NC + d] + totc[1 + d]) * inv_n;
                rz -= sub[d] * s.sr[d];
              }
            if (!first) c.beta = c.rz != 0.0 ? rz / c.rz : 0.0;
            c.rz = rz;
          }
          mask |= c.done ? 1 << k : 0;
        }
        s.active = any;
        for (int k = 0; k < NR; ++k) LF::put(out, k, first ? 0.0 : s.r[k].beta, mask | any << 8);
        if (KS) {
          for (int d = 0; d < 3; ++d) s.sub[d] = sub[d];
          LF::put_sub(out, sub);
        }
      }
      __syncthreads();
      send_lines(P.line + kLnBeta * kLoopLines + (int64_t)b0 * 8, nb, LF::NB, ep, out);
    }
    {
      bool ok = true;
      if (warp == 0)
        ok = wait_line(line + kLnBeta * kLoopLines, lane, LF::NB, ep, P.polls, ln);
      else if (PC == 1)
        ok = wait_coarse<T>(P.ecx + coarse_packet(agg0, la0, NC, 0), tid - 32, kLoopThreads - 32, np * NC, ep,
                            P.polls, ecl);
      if (!ok) s_fail = 1;
    }
    __syncthreads();
    if (s_fail) {
      failed = true;
      break;
    }
    const unsigned flags = LF::flags(ln);
    if (!(flags >> 8)) break;
    // p = (D^-1 r + P e_c, D^-1 r or r) - mean + beta p, published to the group
    ++ep;
    if (!AOS) skip = flags & 0xff;
    {
      T be[NR], sub[NC];
#pragma unroll
      for (int k = 0; k < NR; ++k) be[k] = LF::get(ln, k);
#pragma unroll
      for (int c = 0; c < NC; ++c) sub[c] = KS ? LF::sub(ln, c) : T(0);
      for (int ls = my0; ls < nsl; ls += mystep) {
        const int64_t lr = (int64_t)ls * 32 + lane;
        if (row0 + lr >= rend) continue;
        const T* e = PC == 1 ? ecl + (a.C.agg_of_row[row0 + lr] - la0) * NC : nullptr;
#pragma unroll
        for (int c = 0; c < NV; ++c) {
          const int k = AOS ? 0 : c;
          if (skip >> c & 1) continue;
          T z = r.at(c, lr);
          if (PC != 0) z *= di.at(AOS ? c : 0, lr);
          if (PC == 1) z += e[c];
          if (KS) z -= sub[AOS ? c : 0];
          publish(c, lr, first ? z : z + be[k] * p.at(c, lr));
        }
      }
    }
    first = false;
    __syncthreads();  // warps that share a slice read its rows of p
  }
  if (failed) {
    if (tid == 0) atomicExch(P.err, 1);
    return;
  }
  // the solution: zero where b vanished, moved to zero at the pinned node (singular systems)
  const bool in_smem = active && a.place > 3;
  const bool zero = KS && s.zero_x;
  auto xval = [&](int c, int64_t lr) {
    return zero ? T(0) : (in_smem ? x.at(c, lr) : gx.at(c, lr));
  };
  ++ep;
  if (KS && a.shift) {
    __syncthreads();
    const int pb = P.pin_blk[seg];
    ulonglong2* slot = P.line + kLnPin * kLoopLines + (int64_t)b0 * 8;
    if (warp == 0) {
      if (blk == pb && lane < NC) post(slot + lane, (double)xval(lane, a.G.seg_pin[seg] - row0), ep);
      if (!wait_line(slot, lane, NC, ep, P.polls, ln))
        s_fail = 1;
    }
    __syncthreads();
    if (s_fail) {
      if (tid == 0) atomicExch(P.err, 1);
      return;
    }
  }
  double pinv[3] = {0.0, 0.0, 0.0};
  if (KS && a.shift)
#pragma unroll
    for (int c = 0; c < NC; ++c) pinv[c] = __hiloint2double((int)ln[c].y, (int)ln[c].x);
  if (in_smem || zero || (KS && a.shift)) {
    for (int ls = my0; ls < nsl; ls += mystep) {
      const int64_t lr = (int64_t)ls * 32 + lane;
      if (row0 + lr >= rend) continue;
#pragma unroll
      for (int c = 0; c < NV; ++c) {
        T v = xval(c, lr);
        if (KS && a.shift) v = (T)((double)v - pinv[c]);
        gx.at(c, lr) = v;
      }
    }
  }
  // A mesh that had nothing to solve exchanged the pinned value at most: the others may not have
  // read their exchange numbers yet.  (Otherwise the leader has heard from every block.)
  if (!active) {
    ++bars;
    if (!group_barrier(P.count + seg, bars * (uint32_t)nb, P.polls)) {
      if (tid == 0) atomicExch(P.err, 1);
      return;
    }
  }
  if (leader && tid == 0) {
    if (active) a.st[seg] = s;
    P.epoch[2 * seg] = ep;
    P.epoch[2 * seg + 1] = bars;
    int it = 0;
    for (int k = 0; k < s.nr; ++k)
      it = a.kind == 2 ? it + s.r[k].iters : (s.r[k].iters > it ? s.r[k].iters : it);
    a.acc[4 * seg + a.kind] += it;
    a.acc[4 * seg + 3] += s.noconv;
  }
}

template <typename T>
using LoopKernel = void (*)(CgLoop<T>);

// the instantiation of a solve (see launch_cg_loop), or NULL
template <typename T>
LoopKernel<T> loop_kernel(int kind, int B, int nr, int pc) {
  if (B == 6) return pc == 1 ? k_cg_loop<T, 6, 1, 1, true> : k_cg_loop<T, 6, 1, 0, true>;
  if (B != 1) return nullptr;
  if (kind != 2) return pc == 1 ? k_cg_loop<T, 1, 1, 1, true> : k_cg_loop<T, 1, 1, 0, true>;
  switch (pc == 2 ? nr : -nr) {
    case 1: return k_cg_loop<T, 1, 1, 2, false>;
    case 2: return k_cg_loop<T, 1, 2, 2, false>;
    case 3: return k_cg_loop<T, 1, 3, 2, false>;
    case -1: return k_cg_loop<T, 1, 1, 0, false>;
    case -2: return k_cg_loop<T, 1, 2, 0, false>;
    case -3: return k_cg_loop<T, 1, 3, 0, false>;
  }
  return nullptr;
}
}  // namespace

template <typename T>
cudaError_t loop_dynamic_limit(int kind, int B, int nr, int pc, size_t* bytes) {
  *bytes = 0;
  const LoopKernel<T> k = loop_kernel<T>(kind, B, nr, pc);
  if (!k) return cudaErrorInvalidValue;
  int dev = 0, optin = 0, resident = 0;
  cudaFuncAttributes fa;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess)
    e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  if (e == cudaSuccess) e = cudaFuncGetAttributes(&fa, k);
  if (e != cudaSuccess) return e;
  if ((size_t)optin <= fa.sharedSizeBytes) return cudaSuccess;
  const size_t most = (size_t)optin - fa.sharedSizeBytes;
  // (one value for every context: a smaller one set by another thread would refuse this one's launch)
  e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)most);
  if (e == cudaSuccess)
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&resident, k, kLoopThreads, most);
  if (e == cudaSuccess && resident > 0) *bytes = most;
  return e;
}

template <typename T>
cudaError_t launch_cg_loop(const Launch& L, const CgLoop<T>& a, int B, int nr, int pc) {
  (*L.counter) += 1;
  const LoopKernel<T> k = loop_kernel<T>(a.kind, B, nr, pc);
  if (!k) return cudaErrorInvalidValue;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)a.part.nblocks);
  cfg.blockDim = dim3(kLoopThreads);
  cfg.dynamicSmemBytes = loop_smem<T>(B == 1 ? 1 : 3, nr, pc, a.place, a.part).total;
  cfg.stream = L.stream;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeCooperative;  // the blocks wait for one another
  at[0].val.cooperative = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k, a);
}

template cudaError_t loop_dynamic_limit<float>(int, int, int, int, size_t*);
template cudaError_t loop_dynamic_limit<double>(int, int, int, int, size_t*);
template cudaError_t launch_cg_loop<float>(const Launch&, const CgLoop<float>&, int, int, int);
template cudaError_t launch_cg_loop<double>(const Launch&, const CgLoop<double>&, int, int, int);

}  // namespace gspm
