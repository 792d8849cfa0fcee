// Learned warm start of the mechanical CG: a three-layer message-passing network over the mesh
// (hidden width 64) that predicts the displacement correction on top of linear extrapolation.
//
// Forward layers run on the Blackwell tensor cores (tcgen05.mma kind::f16, BF16 operands, FP32
// accumulator in tensor memory) with the element-message aggregation z_i = sum_j A_ij h_j fused
// into the tile load: a block owns 128 rows, gathers [h_i, z_i] into shared memory as BF16 and
// multiplies by the layer's weights held in shared memory.  Training (backward and Adam) runs in FP32 on CUDA cores with
// deterministic block partials.  The network definition (features, aggregation, loss) is the
// one documented in include/gspm.h (gspm_mpnn_*).
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cstdint>

#include "kernels.cuh"
#include "mpnn.cuh"

namespace gspm {

namespace {

constexpr int kRows = 128;      // rows per tile (8 warps x 16)
constexpr int kThreads = 256;
constexpr int kGather = 8;      // neighbour feature loads in flight per lane in k_tc_layer

__device__ __forceinline__ int64_t tid() { return (int64_t)blockIdx.x * blockDim.x + threadIdx.x; }
__device__ __forceinline__ int64_t tstride() { return (int64_t)gridDim.x * blockDim.x; }

__device__ __forceinline__ uint32_t pack2(__nv_bfloat16 a, __nv_bfloat16 b) {
  return (uint32_t)__bfloat16_as_ushort(a) | ((uint32_t)__bfloat16_as_ushort(b) << 16);
}

// ---------------------------------------------------------------------------------------------
// Blackwell tensor cores: tcgen05.mma with the FP32 accumulator in tensor memory (TMEM)
// ---------------------------------------------------------------------------------------------
// A layer's GEMM is one 128 x 64 tile per block and K step: A = the block's 128 rows of [h, z]
// (or of the 16 input features), B = W^T (64 x K), both K-major in shared memory with the
// 128-byte swizzle (rows of 64 bf16, eight-row groups 1024 bytes apart, 16-byte chunk c of row r
// stored at chunk c ^ (r mod 8)).  One thread issues the K / 16 MMAs and commits them to an
// mbarrier; the accumulator (row i in TMEM lane i, column j in TMEM column j) is read back with
// tcgen05.ld by all eight warps (warp w: lanes 32 (w mod 4) .., columns 32 (w / 4) ..).
constexpr int kTileA = kRows * 128;   // bytes of one 64-wide K-block of A
constexpr int kTileB = kHid * 128;    // bytes of one 64-wide K-block of B
constexpr int kTmemCols = 64;         // TMEM columns of the 128 x 64 FP32 accumulator
constexpr size_t kTcSmem = 2 * kTileA + 2 * kTileB + kHid * 4 + 16 + 1024;  // + alignment slack
// spin limit of the accumulator wait (each try_wait may also suspend for a while): far beyond the
// microsecond an MMA group takes, so reaching it means the tensor-core work never completed
constexpr uint32_t kSpinLimit = 1u << 22;
// instruction descriptor of kind::f16: FP32 accumulator (bits 4-5 = 1), A and B bf16 (bits 7-9,
// 10-12 = 1), both K-major (bits 15, 16 = 0), N >> 3 at bits 17-22, M >> 4 at bits 24-28
constexpr uint32_t kIdesc = (1u << 4) | (1u << 7) | (1u << 10) |
                            ((uint32_t)(kHid >> 3) << 17) | ((uint32_t)(kRows >> 4) << 24);

__device__ __forceinline__ uint32_t smem_addr(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
// byte offset of 16-byte chunk c (0..7) of row r in a 128-byte-swizzled K-block
__device__ __forceinline__ uint32_t sw128(int r, int c) {
  return (uint32_t)(r * 128 + ((c ^ (r & 7)) << 4));
}
// shared-memory matrix descriptor: start address >> 4 (bits 0-13), leading byte offset >> 4
// (bits 16-29; not used by a swizzled K-major operand), stride byte offset >> 4 = 1024 >> 4
// between eight-row groups (bits 32-45), the fixed 0b001 at bits 46-48, 128-byte swizzle (2 at
// bits 61-63).  The K-block starts on a 1024-byte boundary, so the base offset is 0 and a K step
// inside the block advances the start address by 32 bytes.
__device__ __forceinline__ uint64_t sw128_desc(uint32_t addr) {
  return (uint64_t)((addr & 0x3FFFFu) >> 4) | ((uint64_t)1 << 16) | ((uint64_t)(1024 >> 4) << 32) |
         ((uint64_t)1 << 46) | ((uint64_t)2 << 61);
}
__device__ __forceinline__ void tc_mma(uint32_t tmem, uint64_t adesc, uint64_t bdesc,
                                       uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(tmem),
      "l"(adesc), "l"(bdesc), "r"(kIdesc), "r"(accumulate)
      : "memory");
}
__device__ __forceinline__ void tc_commit(uint32_t mbar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                   mbar)
               : "memory");
}
__device__ __forceinline__ void tc_fence_before() {
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_after() {
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void async_proxy_fence() {
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}
// true once the mbarrier phase of parity `phase` has completed; false after kSpinLimit polls
__device__ __forceinline__ bool mbar_wait(uint32_t mbar, uint32_t phase) {
  for (uint32_t it = 0; it < kSpinLimit; ++it) {
    uint32_t done;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}\n"
        : "=r"(done)
        : "r"(mbar), "r"(phase)
        : "memory");
    if (done) return true;
  }
  return false;
}
// 32 consecutive FP32 columns of this thread's TMEM lane
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&v)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,"
      "%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
      : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]),
        "=r"(v[7]), "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]),
        "=r"(v[14]), "=r"(v[15]), "=r"(v[16]), "=r"(v[17]), "=r"(v[18]), "=r"(v[19]),
        "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]), "=r"(v[24]), "=r"(v[25]),
        "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
      : "r"(taddr)
      : "memory");
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

// ---------------------------------------------------------------------------------------------
// features: m (3), E0(m) Voigt / lambda_s (6), u_prev / u_s (3), (u_prev - u_prev2) / u_s (3), 1
// ---------------------------------------------------------------------------------------------
template <typename T>
__global__ void k_features(int64_t n, const T* __restrict__ m, int64_t ld,
                           const uint8_t* __restrict__ mag, const T* __restrict__ up,
                           const T* __restrict__ up2, double l100, double l111,
                           double inv_ls, double inv_us, __nv_bfloat16* __restrict__ F) {
  for (int64_t i = tid(); i < n; i += tstride()) {
    float f[kFeat];
    const double m0 = m[i], m1 = m[ld + i], m2 = m[2 * ld + i];
    f[0] = (float)m0;
    f[1] = (float)m1;
    f[2] = (float)m2;
    if (mag[i]) {
      const double a = 1.5 * l100 * inv_ls, b = 1.5 * l111 * inv_ls;
      f[3] = (float)(a * (m0 * m0 - 1.0 / 3.0));
      f[4] = (float)(a * (m1 * m1 - 1.0 / 3.0));
      f[5] = (float)(a * (m2 * m2 - 1.0 / 3.0));
      f[6] = (float)(b * m1 * m2);
      f[7] = (float)(b * m0 * m2);
      f[8] = (float)(b * m0 * m1);
    } else {
      for (int c = 3; c < 9; ++c) f[c] = 0.f;
    }
    for (int c = 0; c < 3; ++c) {
      const double p = up ? (double)up[3 * i + c] : 0.0, q = up2 ? (double)up2[3 * i + c] : 0.0;
      f[9 + c] = (float)(p * inv_us);
      f[12 + c] = (float)((p - q) * inv_us);
    }
    f[15] = 1.f;
    uint32_t* o = reinterpret_cast<uint32_t*>(F + i * kFeat);
    for (int c = 0; c < kFeat / 2; ++c)
      o[c] = pack2(__float2bfloat16_rn(f[2 * c]), __float2bfloat16_rn(f[2 * c + 1]));
  }
}

// One forward layer on the tensor cores.  MODE 0: h0 = relu(F W_in + b_in) (K = 16, the node
// features); MODE 1: h_out = relu([h, A h] W + b) (K = 128) with the element-message aggregation
// z = A h gathered into the A tile (z optionally saved for the backward pass).  A block owns
// 128 rows per round; TMEM holds its 128 x 64 accumulator.  err (device int) is set when the
// accumulator wait gives up; the block then waits once more (bounded) for its MMAs, frees its
// TMEM and returns.
template <int MODE>
__global__ void __launch_bounds__(kThreads) k_tc_layer(int64_t n, DSell S,
                                                       const float* __restrict__ Aw,
                                                       const __nv_bfloat16* __restrict__ Hin,
                                                       const __nv_bfloat16* __restrict__ WT,
                                                       const float* __restrict__ bias,
                                                       __nv_bfloat16* __restrict__ Hout,
                                                       __nv_bfloat16* __restrict__ Zout,
                                                       int* __restrict__ err) {
  constexpr int K = MODE == 0 ? kFeat : 2 * kHid;
  constexpr int KC = K / 8;  // 16-byte chunks per row
  extern __shared__ unsigned char smem_raw[];
  const uint32_t raw = smem_addr(smem_raw);
  unsigned char* sm = smem_raw + (((raw + 1023u) & ~1023u) - raw);
  unsigned char* As = sm;                  // K-blocks 0 (h or F) and 1 (z)
  unsigned char* Bs = sm + 2 * kTileA;     // W^T, K-blocks 0 and 1
  float* bs = reinterpret_cast<float*>(Bs + 2 * kTileB);
  uint64_t* mbar = reinterpret_cast<uint64_t*>(bs + kHid);
  uint32_t* tslot = reinterpret_cast<uint32_t*>(mbar + 1);
  __shared__ int s_fail;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (int t = threadIdx.x; t < kHid * KC; t += blockDim.x) {
    const int o = t / KC, cc = t % KC;
    const uint4 v = *reinterpret_cast<const uint4*>(WT + (int64_t)o * K + cc * 8);
    *reinterpret_cast<uint4*>(Bs + (cc >> 3) * kTileB + sw128(o, cc & 7)) = v;
  }
  for (int k = threadIdx.x; k < kHid; k += blockDim.x) bs[k] = bias[k];
  if (threadIdx.x == 0) {
    s_fail = 0;
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_addr(mbar)) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_addr(tslot)),
                 "r"(kTmemCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  async_proxy_fence();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tslot;
  const uint32_t bar = smem_addr(mbar);
  uint32_t phase = 0;
  int inflight = 0;
  for (int64_t base = (int64_t)blockIdx.x * kRows; base < n; base += (int64_t)gridDim.x * kRows) {
    if (MODE == 0) {
      // 128 rows x 2 chunks of the features, one 16-byte load per thread
      for (int t = threadIdx.x; t < kRows * KC; t += blockDim.x) {
        const int r = t / KC, c = t % KC;
        const int64_t i = base + r;
        const uint4 v = i < n ? *reinterpret_cast<const uint4*>(Hin + i * kFeat + c * 8)
                              : make_uint4(0u, 0u, 0u, 0u);
        *reinterpret_cast<uint4*>(As + sw128(r, c)) = v;
      }
    } else {
      // each warp fills its 16 rows (half a SELL slice) four at a time: lane group g = lane / 8
      // takes row 4 rr + g, lane q = lane % 8 its features 8 q .. 8 q + 7 (one 16-byte chunk);
      // the neighbours go in batches of kGather, all their column loads before their feature
      // loads, so a lane has kGather gathers in flight.  z sums the neighbours in column order.
      const int grp = lane >> 3, q = lane & 7;
      const int64_t s0 = (base + 16 * warp) >> 5;
      const int64_t sb = s0 < S.nslices ? S.sptr[s0] : 0;
      const int len = s0 < S.nslices ? S.slen[s0] : 0;
      for (int rr = 0; rr < 4; ++rr) {
        const int r = 16 * warp + 4 * rr + grp;
        const int64_t i = base + r;
        float z[8];
#pragma unroll
        for (int c = 0; c < 8; ++c) z[c] = 0.f;
        uint4 hi = make_uint4(0u, 0u, 0u, 0u);
        if (i < n) {
          hi = *reinterpret_cast<const uint4*>(Hin + i * kHid + 8 * q);
          const int64_t li = i & 31;
          for (int k0 = 0; k0 < len; k0 += kGather) {
            int64_t j[kGather];
            float a[kGather];
#pragma unroll
            for (int u = 0; u < kGather; ++u) {
              // past the row's end: entry k0 (k0 < len) again, weight 0; no load leaves the slice
              const bool ok = k0 + u < len;
              const int64_t e = sb + (int64_t)(ok ? k0 + u : k0) * 32 + li;
              j[u] = (int64_t)S.col[e];
              const float av = Aw[e];
              a[u] = ok ? av : 0.f;
            }
            uint4 hj[kGather];
#pragma unroll
            for (int u = 0; u < kGather; ++u)
              hj[u] = *reinterpret_cast<const uint4*>(Hin + j[u] * kHid + 8 * q);
#pragma unroll
            for (int u = 0; u < kGather; ++u) {
              const uint32_t w[4] = {hj[u].x, hj[u].y, hj[u].z, hj[u].w};
#pragma unroll
              for (int c = 0; c < 4; ++c) {
                z[2 * c] += a[u] * __bfloat162float(__ushort_as_bfloat16((unsigned short)(w[c] & 0xffffu)));
                z[2 * c + 1] += a[u] * __bfloat162float(__ushort_as_bfloat16((unsigned short)(w[c] >> 16)));
              }
            }
          }
        }
        uint4 zp;
        zp.x = pack2(__float2bfloat16_rn(z[0]), __float2bfloat16_rn(z[1]));
        zp.y = pack2(__float2bfloat16_rn(z[2]), __float2bfloat16_rn(z[3]));
        zp.z = pack2(__float2bfloat16_rn(z[4]), __float2bfloat16_rn(z[5]));
        zp.w = pack2(__float2bfloat16_rn(z[6]), __float2bfloat16_rn(z[7]));
        *reinterpret_cast<uint4*>(As + sw128(r, q)) = hi;
        *reinterpret_cast<uint4*>(As + kTileA + sw128(r, q)) = zp;
        if (Zout && i < n) *reinterpret_cast<uint4*>(Zout + i * kHid + 8 * q) = zp;
      }
    }
    // the A tile written by every thread becomes visible to the tensor cores; one thread issues
    // the K / 16 MMAs of the tile and commits them to the mbarrier
    async_proxy_fence();
    __syncthreads();
    if (threadIdx.x == 0) {
      tc_fence_after();
      const uint32_t a0 = smem_addr(As), b0 = smem_addr(Bs);
#pragma unroll
      for (int ks = 0; ks < K / 16; ++ks) {
        const uint32_t koff = (uint32_t)((ks & 3) * 32);
        tc_mma(tmem, sw128_desc(a0 + (ks >> 2) * kTileA + koff),
               sw128_desc(b0 + (ks >> 2) * kTileB + koff), ks > 0 ? 1u : 0u);
      }
      tc_commit(bar);
    }
    inflight = 1;
    if (!mbar_wait(bar, phase)) s_fail = 1;
    __syncthreads();
    if (s_fail) break;
    inflight = 0;
    phase ^= 1u;
    tc_fence_after();
    // epilogue: warp w reads lanes 32 (w mod 4) .. + 31 (its rows), columns 32 (w / 4) .. + 31
    const int lg = warp & 3, ch = warp >> 2;
    uint32_t v[32];
    tmem_ld32(tmem + ((uint32_t)(32 * lg) << 16) + (uint32_t)(32 * ch), v);
    const int64_t row = base + 32 * lg + lane;
    if (row < n) {
      uint32_t pk[16];
#pragma unroll
      for (int c = 0; c < 16; ++c) {
        const int col = 32 * ch + 2 * c;
        pk[c] = pack2(__float2bfloat16_rn(fmaxf(__uint_as_float(v[2 * c]) + bs[col], 0.f)),
                      __float2bfloat16_rn(fmaxf(__uint_as_float(v[2 * c + 1]) + bs[col + 1], 0.f)));
      }
      uint4* dst = reinterpret_cast<uint4*>(Hout + row * kHid + 32 * ch);
#pragma unroll
      for (int c = 0; c < 4; ++c) dst[c] = make_uint4(pk[4 * c], pk[4 * c + 1], pk[4 * c + 2], pk[4 * c + 3]);
    }
    // the accumulator and the A tile are consumed before the next round overwrites them
    tc_fence_before();
    __syncthreads();
  }
  if (s_fail) {
    if (threadIdx.x == 0) atomicExch(err, 1);
    if (inflight) mbar_wait(bar, phase);  // bounded: give the MMAs a last chance to finish
  }
  __syncthreads();
  if (warp == 0) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                 "r"(kTmemCols)
                 : "memory");
  }
}

// y = h3 W_out + b_out; mode 0: Y = y (float [n][3]); mode 1: x0 = 2 u_prev - u_prev2 + u_s y
template <typename T>
__global__ void k_output(int64_t n, const __nv_bfloat16* __restrict__ H,
                         const float* __restrict__ Wout, const float* __restrict__ bout, int mode,
                         float* __restrict__ Y, const T* __restrict__ up,
                         const T* __restrict__ up2, double us, T* __restrict__ x0) {
  __shared__ float w[kHid * 3 + 3];
  for (int k = threadIdx.x; k < kHid * 3; k += blockDim.x) w[k] = Wout[k];
  if (threadIdx.x < 3) w[kHid * 3 + threadIdx.x] = bout[threadIdx.x];
  __syncthreads();
  for (int64_t i = tid(); i < n; i += tstride()) {
    float y0 = w[kHid * 3], y1 = w[kHid * 3 + 1], y2 = w[kHid * 3 + 2];
    const uint32_t* hp = reinterpret_cast<const uint32_t*>(H + i * kHid);
    for (int c = 0; c < kHid / 2; ++c) {
      const uint32_t v = hp[c];
      const float a = __bfloat162float(__ushort_as_bfloat16((unsigned short)(v & 0xffffu)));
      const float b = __bfloat162float(__ushort_as_bfloat16((unsigned short)(v >> 16)));
      y0 += a * w[3 * (2 * c)] + b * w[3 * (2 * c + 1)];
      y1 += a * w[3 * (2 * c) + 1] + b * w[3 * (2 * c + 1) + 1];
      y2 += a * w[3 * (2 * c) + 2] + b * w[3 * (2 * c + 1) + 2];
    }
    if (mode == 0) {
      Y[3 * i] = y0;
      Y[3 * i + 1] = y1;
      Y[3 * i + 2] = y2;
    } else {
      const float y[3] = {y0, y1, y2};
      for (int c = 0; c < 3; ++c) {
        const double p = up ? (double)up[3 * i + c] : 0.0, q = up2 ? (double)up2[3 * i + c] : 0.0;
        x0[3 * i + c] = (T)(2.0 * p - q + us * (double)y[c]);
      }
    }
  }
}

// ---------------------------------------------------------------------------------------------
// training (FP32)
// ---------------------------------------------------------------------------------------------
__device__ __forceinline__ float bf(const __nv_bfloat16* p) { return __bfloat162float(*p); }

// dY = 2 (Y - T) / (3n); dH3 = dY W_out^T; block partials of dW_out (h3^T dY), db_out, loss
__global__ void __launch_bounds__(kThreads) k_out_bwd(int64_t n, const float* __restrict__ Y,
                                                      const float* __restrict__ T,
                                                      const __nv_bfloat16* __restrict__ H,
                                                      const float* __restrict__ Wout,
                                                      float* __restrict__ dH,
                                                      float* __restrict__ part) {
  // part per block: [kHid*3 dW_out][3 db_out][1 loss]
  __shared__ float acc[kHid * 3 + 4];
  __shared__ float w[kHid * 3];
  for (int k = threadIdx.x; k < kHid * 3 + 4; k += blockDim.x) acc[k] = 0.f;
  for (int k = threadIdx.x; k < kHid * 3; k += blockDim.x) w[k] = Wout[k];
  __syncthreads();
  const float scale = 2.f / (3.f * (float)n);
  // one warp per row: lanes own features 2*lane, 2*lane+1
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  float pw[2][3] = {{0, 0, 0}, {0, 0, 0}}, pb[3] = {0, 0, 0}, pl = 0.f;
  const int64_t nwarps = tstride() >> 5;
  for (int64_t i = tid() >> 5; i < n; i += nwarps) {
    float dy[3];
    for (int c = 0; c < 3; ++c) {
      const float d = Y[3 * i + c] - T[3 * i + c];
      dy[c] = scale * d;
      if (lane == 0) {
        pb[c] += dy[c];
        pl += d * d;
      }
    }
    const float h0 = bf(H + i * kHid + 2 * lane), h1 = bf(H + i * kHid + 2 * lane + 1);
    for (int c = 0; c < 3; ++c) {
      pw[0][c] += h0 * dy[c];
      pw[1][c] += h1 * dy[c];
    }
    dH[i * kHid + 2 * lane] = dy[0] * w[3 * (2 * lane)] + dy[1] * w[3 * (2 * lane) + 1] +
                             dy[2] * w[3 * (2 * lane) + 2];
    dH[i * kHid + 2 * lane + 1] = dy[0] * w[3 * (2 * lane + 1)] +
                                 dy[1] * w[3 * (2 * lane + 1) + 1] +
                                 dy[2] * w[3 * (2 * lane + 1) + 2];
  }
  // fixed-order block accumulation: warps in turn
  for (int wv = 0; wv < (int)(blockDim.x >> 5); ++wv) {
    if (warp == wv) {
      for (int c = 0; c < 3; ++c) {
        acc[3 * (2 * lane) + c] += pw[0][c];
        acc[3 * (2 * lane + 1) + c] += pw[1][c];
      }
      if (lane == 0) {
        for (int c = 0; c < 3; ++c) acc[kHid * 3 + c] += pb[c];
        acc[kHid * 3 + 3] += pl;
      }
    }
    __syncthreads();
  }
  for (int k = threadIdx.x; k < kHid * 3 + 4; k += blockDim.x)
    part[(int64_t)blockIdx.x * (kHid * 3 + 4) + k] = acc[k];
}

// Rows of a backward tile and the padded row lengths of its shared arrays (multiples of four floats,
// so that rows of consecutive lanes start four banks apart: 16-byte accesses without conflicts)
constexpr int kBwdRows = 64;
constexpr int kPitch = kHid + 4, kPitch2 = 2 * kHid + 4;

// 16 consecutive bf16 values
__device__ __forceinline__ void load16(const __nv_bfloat16* p, float (&v)[16]) {
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const uint4 u = *reinterpret_cast<const uint4*>(p + 8 * h);
    const uint32_t w[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      v[8 * h + 2 * k] = __uint_as_float(w[k] << 16);
      v[8 * h + 2 * k + 1] = __uint_as_float(w[k] & 0xffff0000u);
    }
  }
}
__device__ __forceinline__ void store16(float* p, const float (&v)[16]) {
#pragma unroll
  for (int k = 0; k < 4; ++k)
    *reinterpret_cast<float4*>(p + 4 * k) =
        make_float4(v[4 * k], v[4 * k + 1], v[4 * k + 2], v[4 * k + 3]);
}
// dA = dH (.) [h > 0], 16 columns from c0 of row i (zero past the last row)
__device__ __forceinline__ void load_da(int64_t n, int64_t i, int c0, const float* __restrict__ dH,
                                        const __nv_bfloat16* __restrict__ H, float (&v)[16]) {
#pragma unroll
  for (int k = 0; k < 16; ++k) v[k] = 0.f;
  if (i >= n) return;
  float h[16];
  load16(H + i * kHid + c0, h);
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const float4 d = *reinterpret_cast<const float4*>(dH + i * kHid + c0 + 4 * k);
    v[4 * k] = h[4 * k] > 0.f ? d.x : 0.f;
    v[4 * k + 1] = h[4 * k + 1] > 0.f ? d.y : 0.f;
    v[4 * k + 2] = h[4 * k + 2] > 0.f ? d.z : 0.f;
    v[4 * k + 3] = h[4 * k + 3] > 0.f ? d.w : 0.f;
  }
}

// For one layer: dA = dH (.) [h > 0]; block partials of dW (X^T dA, X = [h_prev, z]) and db;
// dX = dA W^T: columns 0..63 -> dHprev, 64..127 -> dZ.  Both products of a tile of 64 rows are
// register-tiled FP32 (32 outputs per thread from three 16-byte shared loads per step; a tile's part
// of dW is summed by itself before it joins the block's running sum).  The FP32 pipe bounds it: 29 us
// at 65,536 rows, of which the 1,024 tiles fill 304 blocks in four rounds where 3.4 would do; it takes
// 63 us, against 209 us with two shared loads per multiply-add.
__global__ void __launch_bounds__(kThreads, 2) k_layer_bwd(int64_t n, const float* __restrict__ dH,
                                                           const __nv_bfloat16* __restrict__ Hcur,
                                                           const __nv_bfloat16* __restrict__ Hprev,
                                                           const __nv_bfloat16* __restrict__ Z,
                                                           const float* __restrict__ W,  // [128][64]
                                                           float* __restrict__ dHprev,
                                                           float* __restrict__ dZ,
                                                           float* __restrict__ part) {
  // part per block: [128*64 dW][64 db]
  extern __shared__ __align__(16) unsigned char smem[];
  float* WT = reinterpret_cast<float*>(smem);  // [64][kPitch2]: WT[c][f] = W[f][c]
  float* X = WT + kHid * kPitch2;              // [rows][kPitch2]
  float* D = X + kBwdRows * kPitch2;           // [rows][kPitch]   dA
  float* DT = D + kBwdRows * kPitch;           // [64][kPitch]     its transpose
  const int t = threadIdx.x;
  for (int k = t; k < 2 * kHid * kHid; k += kThreads) WT[(k % kHid) * kPitch2 + k / kHid] = W[k];
  const int lr = t % kBwdRows, lc = 16 * (t / kBwdRows);  // loads: row and first column
  const int tx = 4 * (t % 16), ty = 4 * (t / 16);
  float w[2][4][4] = {}, db = 0.f;  // dW[64 h + ty + i][tx + j]
  for (int64_t base = (int64_t)blockIdx.x * kBwdRows; base < n;
       base += (int64_t)gridDim.x * kBwdRows) {
    const int64_t i = base + lr;
    float v[16];
    load_da(n, i, lc, dH, Hcur, v);
    __syncthreads();  // the tile before has been read
    store16(D + lr * kPitch + lc, v);
#pragma unroll
    for (int k = 0; k < 16; ++k) DT[(lc + k) * kPitch + lr] = v[k];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      if (i < n) {
        load16((h ? Z : Hprev) + i * kHid + lc, v);
      } else {
#pragma unroll
        for (int k = 0; k < 16; ++k) v[k] = 0.f;
      }
      store16(X + lr * kPitch2 + h * kHid + lc, v);
    }
    __syncthreads();
    // dX[ty + r][64 h + tx + j] = sum_c dA[ty + r][c] W[64 h + tx + j][c], c ascending
    float x[2][4][4] = {};
#pragma unroll 4
    for (int c = 0; c < kHid; ++c) {
      const float4 d4 = *reinterpret_cast<const float4*>(DT + c * kPitch + ty);
      const float d[4] = {d4.x, d4.y, d4.z, d4.w};
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const float4 f4 = *reinterpret_cast<const float4*>(WT + c * kPitch2 + h * kHid + tx);
        const float f[4] = {f4.x, f4.y, f4.z, f4.w};
#pragma unroll
        for (int r = 0; r < 4; ++r)
#pragma unroll
          for (int j = 0; j < 4; ++j) x[h][r][j] += d[r] * f[j];
      }
    }
#pragma unroll
    for (int r = 0; r < 4; ++r)
      if (base + ty + r < n) {
        const int64_t o = (base + ty + r) * kHid + tx;
        *reinterpret_cast<float4*>(dHprev + o) = make_float4(x[0][r][0], x[0][r][1], x[0][r][2], x[0][r][3]);
        *reinterpret_cast<float4*>(dZ + o) = make_float4(x[1][r][0], x[1][r][1], x[1][r][2], x[1][r][3]);
      }
    // dW[64 h + ty + i][tx + j] += sum over the tile's rows of X[row][64 h + ty + i] dA[row][tx + j]
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
      for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int j = 0; j < 4; ++j) x[h][r][j] = 0.f;
#pragma unroll 4
    for (int row = 0; row < kBwdRows; ++row) {
      const float4 d4 = *reinterpret_cast<const float4*>(D + row * kPitch + tx);
      const float d[4] = {d4.x, d4.y, d4.z, d4.w};
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const float4 f4 = *reinterpret_cast<const float4*>(X + row * kPitch2 + h * kHid + ty);
        const float f[4] = {f4.x, f4.y, f4.z, f4.w};
#pragma unroll
        for (int r = 0; r < 4; ++r)
#pragma unroll
          for (int j = 0; j < 4; ++j) x[h][r][j] += f[r] * d[j];
      }
    }
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
      for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int j = 0; j < 4; ++j) w[h][r][j] += x[h][r][j];
    if (t < kHid) {
      float b = 0.f;
#pragma unroll 8
      for (int row = 0; row < kBwdRows; ++row) b += D[row * kPitch + t];
      db += b;
    }
  }
  float* pp = part + (int64_t)blockIdx.x * (2 * kHid * kHid + kHid);
#pragma unroll
  for (int h = 0; h < 2; ++h)
#pragma unroll
    for (int r = 0; r < 4; ++r)
      *reinterpret_cast<float4*>(pp + (h * kHid + ty + r) * kHid + tx) =
          make_float4(w[h][r][0], w[h][r][1], w[h][r][2], w[h][r][3]);
  if (t < kHid) pp[2 * kHid * kHid + t] = db;
}

// dH_prev += A^T dZ (SELL with transposed weights), 64-wide, warp per row.  A block takes runs of 64
// consecutive rows, whose neighbours are largely the same rows of dZ (read from L1); the lanes load
// the row's columns and weights together and hand them round, and eight rows of dZ are in flight.
// 252 MB gathered at 65,536 rows: 35.5 us (47 us one neighbour at a time).
__global__ void __launch_bounds__(kThreads) k_agg_t(int64_t n, DSell S, const float* __restrict__ At,
                                                    const float* __restrict__ dZ,
                                                    float* __restrict__ dH) {
  constexpr int U = 8, kRun = 64;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int64_t base = (int64_t)blockIdx.x * kRun; base < n; base += (int64_t)gridDim.x * kRun)
    for (int64_t i = base + warp; i < base + kRun && i < n; i += kThreads / 32) {
      const int64_t s = i >> 5, li = i & 31;
      const int64_t sb = S.sptr[s];
      const int len = S.slen[s];
      float2* o = reinterpret_cast<float2*>(dH + i * kHid + 2 * lane);
      const float2 h = *o;
      float2 acc = make_float2(0.f, 0.f);
      for (int kb = 0; kb < len; kb += 32) {
        const bool ok = kb + lane < len;
        const int64_t e = sb + (int64_t)(kb + lane) * 32 + li;
        const int cj = ok ? S.col[e] : (int)i;
        const float ca = ok ? At[e] : 0.f;
        const int m = len - kb < 32 ? len - kb : 32;
        for (int k0 = 0; k0 < m; k0 += U) {
          float2 z[U];
          float a[U];
#pragma unroll
          for (int u = 0; u < U; ++u) {
            // past the row's end (k0 + u < 32 still): the row itself with weight 0
            const int j = __shfl_sync(0xffffffffu, cj, k0 + u);
            a[u] = __shfl_sync(0xffffffffu, ca, k0 + u);
            z[u] = *reinterpret_cast<const float2*>(dZ + (int64_t)j * kHid + 2 * lane);
          }
#pragma unroll
          for (int u = 0; u < U; ++u) {
            acc.x += a[u] * z[u].x;
            acc.y += a[u] * z[u].y;
          }
        }
      }
      *o = make_float2(h.x + acc.x, h.y + acc.y);
    }
}

// input layer backward: block partials of dW_in (F^T dA0) and db_in, tiles of 64 rows as above (four
// outputs per thread): 22 us at 65,536 rows, 131 us with a block per row
__global__ void __launch_bounds__(kThreads) k_in_bwd(int64_t n, const float* __restrict__ dH,
                                                     const __nv_bfloat16* __restrict__ H0,
                                                     const __nv_bfloat16* __restrict__ F,
                                                     float* __restrict__ part) {
  // part per block: [16*64 dW_in][64 db_in]
  __shared__ __align__(16) float D[kBwdRows * kPitch];
  __shared__ __align__(16) float X[kBwdRows * (kFeat + 4)];
  const int t = threadIdx.x;
  const int lr = t % kBwdRows, lc = 16 * (t / kBwdRows);
  const int tx = 4 * (t % 16), f = t / 16;
  float w[4] = {}, db = 0.f;
  for (int64_t base = (int64_t)blockIdx.x * kBwdRows; base < n;
       base += (int64_t)gridDim.x * kBwdRows) {
    const int64_t i = base + lr;
    float v[16];
    load_da(n, i, lc, dH, H0, v);
    __syncthreads();
    store16(D + lr * kPitch + lc, v);
    if (lc == 0) {
      if (i < n) {
        load16(F + i * kFeat, v);
      } else {
#pragma unroll
        for (int k = 0; k < 16; ++k) v[k] = 0.f;
      }
      store16(X + lr * (kFeat + 4), v);
    }
    __syncthreads();
    float x[4] = {}, b = 0.f;
#pragma unroll 8
    for (int row = 0; row < kBwdRows; ++row) {
      const float4 d = *reinterpret_cast<const float4*>(D + row * kPitch + tx);
      const float a = X[row * (kFeat + 4) + f];
      x[0] += a * d.x;
      x[1] += a * d.y;
      x[2] += a * d.z;
      x[3] += a * d.w;
    }
    if (t < kHid)
#pragma unroll 8
      for (int row = 0; row < kBwdRows; ++row) b += D[row * kPitch + t];
#pragma unroll
    for (int j = 0; j < 4; ++j) w[j] += x[j];
    db += b;
  }
  float* pp = part + (int64_t)blockIdx.x * (kFeat * kHid + kHid);
  *reinterpret_cast<float4*>(pp + f * kHid + tx) = make_float4(w[0], w[1], w[2], w[3]);
  if (t < kHid) pp[kFeat * kHid + t] = db;
}

// The block partials of one gradient: out[k] = sum over blocks b < nblocks of part[b][k], k < count,
// and part[b][count] to *last where there is one.  first: its first block of k_reduce_parts.
struct Parts {
  int nblocks, count, stride, first;
  const float* part;
  float *out, *last;
};
constexpr int kPartSets = kLayers + 2;  // W_out (with the loss), the layers, W_in
struct PartList {
  Parts p[kPartSets];
};

// A block sums 32 values: eight groups of threads take every eighth partial, eight loads in flight,
// then the groups in order (13 us for 304 partials of 8,256 values; one thread per value 57 us).
// All gradients in one launch: bound by the latency of its longest sum (1,024 partials of W_out's
// 196 values, 12 us), which alone or beside the layers' takes the same time; a launch per gradient
// took 41 us of device time.  Loss and gradients at 65,536 nodes: 513 -> 495 us.
__global__ void __launch_bounds__(kThreads) k_reduce_parts(PartList PL) {
  __shared__ float sm[8][32];
  int set = 0;
#pragma unroll
  for (int i = 1; i < kPartSets; ++i)
    if ((int)blockIdx.x >= PL.p[i].first) set = i;
  const Parts& P = PL.p[set];
  const int nblocks = P.nblocks, count = P.count, stride = P.stride;
  const float* __restrict__ part = P.part;
  float *grad = P.out, *last = P.last;
  const int lane = threadIdx.x & 31, g = threadIdx.x >> 5;
  const int k = ((int)blockIdx.x - P.first) * 32 + lane;
  const bool ok = k < count + (last ? 1 : 0);
  float s = 0.f;
  for (int b = g; ok && b < nblocks; b += 64) {
    float v[8];
#pragma unroll
    for (int u = 0; u < 8; ++u)
      v[u] = b + 8 * u < nblocks ? part[(int64_t)(b + 8 * u) * stride + k] : 0.f;
#pragma unroll
    for (int u = 0; u < 8; ++u) s += v[u];
  }
  sm[g][lane] = s;
  __syncthreads();
  if (g == 0 && ok) {
#pragma unroll
    for (int u = 1; u < 8; ++u) s += sm[u][lane];
    *(k < count ? grad + k : last) = s;
  }
}

__global__ void k_adam(int64_t count, float* __restrict__ w, const float* __restrict__ g,
                       float* __restrict__ m, float* __restrict__ v, float lr, float b1, float b2,
                       float eps, float c1, float c2) {
  for (int64_t k = tid(); k < count; k += tstride()) {
    const float gk = g[k];
    const float mk = b1 * m[k] + (1.f - b1) * gk;
    const float vk = b2 * v[k] + (1.f - b2) * gk * gk;
    m[k] = mk;
    v[k] = vk;
    w[k] -= lr * (mk / c1) / (sqrtf(vk / c2) + eps);
  }
}

// bf16 transposed weight copies for the tensor-core layers: dst[o][i] = src[i][o]
__global__ void k_transpose_bf16(int rows, int cols, const float* __restrict__ src,
                                 __nv_bfloat16* __restrict__ dst) {
  for (int64_t k = tid(); k < (int64_t)rows * cols; k += tstride()) {
    const int i = (int)(k / cols), o = (int)(k % cols);
    dst[(int64_t)o * rows + i] = __float2bfloat16_rn(src[k]);
  }
}

}  // namespace

// ---------------------------------------------------------------------------------------------
// host-side launchers
// ---------------------------------------------------------------------------------------------
static inline int grid_rows(const Launch& L, int64_t n) {
  int64_t b = (n + kRows - 1) / kRows;
  const int64_t cap = (int64_t)L.max_blocks;
  return (int)(b < 1 ? 1 : (b > cap ? cap : b));
}

size_t mpnn_layer_smem() { return kTcSmem; }
size_t mpnn_layer_bwd_smem() {
  return (size_t)(kHid * kPitch2 + kBwdRows * kPitch2 + kBwdRows * kPitch + kHid * kPitch) * 4;
}
// backward tiles: a block per tile, at most two per SM (each then keeps its sums over its tiles)
static inline int grid_bwd(const Launch& L, int64_t n) {
  const int64_t b = (n + kBwdRows - 1) / kBwdRows, cap = 2 * (int64_t)L.sms;
  return (int)(b > cap ? cap : b);
}
template <typename T>
cudaError_t mpnn_features(const Launch& L, int64_t n, const T* m, int64_t ld, const uint8_t* mag,
                          const T* up, const T* up2, double l100, double l111,
                          double ls, double us, __nv_bfloat16* F) {
  (*L.counter) += 1;
  k_features<T><<<L.blocks_for(n), kBlock, 0, L.stream>>>(n, m, ld, mag, up, up2, l100, l111,
                                                          1.0 / ls, 1.0 / us, F);
  return cudaGetLastError();
}
template cudaError_t mpnn_features<double>(const Launch&, int64_t, const double*, int64_t,
                                           const uint8_t*, const double*, const double*, double,
                                           double, double, double, __nv_bfloat16*);
template cudaError_t mpnn_features<float>(const Launch&, int64_t, const float*, int64_t,
                                          const uint8_t*, const float*, const float*, double,
                                          double, double, double, __nv_bfloat16*);

cudaError_t mpnn_forward(const Launch& L, int64_t n, const DSell& S, const MpnnDev& W,
                         const __nv_bfloat16* F, __nv_bfloat16* const H[4],
                         __nv_bfloat16* const Z[3]) {
  const int g = grid_rows(L, n);
  const size_t sm = mpnn_layer_smem();
  (*L.counter) += 1;
  k_tc_layer<0><<<g, kThreads, sm, L.stream>>>(n, S, W.A, F, W.WinT, W.b_in, H[0], nullptr,
                                               W.err);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  for (int l = 0; l < kLayers; ++l) {
    (*L.counter) += 1;
    k_tc_layer<1><<<g, kThreads, sm, L.stream>>>(n, S, W.A, H[l], W.WT[l], W.b[l], H[l + 1],
                                                 Z ? Z[l] : nullptr, W.err);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

template <typename T>
cudaError_t mpnn_output(const Launch& L, int64_t n, const MpnnDev& W, const __nv_bfloat16* H3,
                        int mode, float* Y, const T* up, const T* up2, double us, T* x0) {
  (*L.counter) += 1;
  k_output<T><<<L.blocks_for(n), kBlock, 0, L.stream>>>(n, H3, W.Wout, W.bout, mode, Y, up, up2,
                                                      us, x0);
  return cudaGetLastError();
}

template cudaError_t mpnn_output<double>(const Launch&, int64_t, const MpnnDev&,
                                         const __nv_bfloat16*, int, float*, const double*,
                                         const double*, double, double*);
template cudaError_t mpnn_output<float>(const Launch&, int64_t, const MpnnDev&,
                                        const __nv_bfloat16*, int, float*, const float*,
                                        const float*, double, float*);

cudaError_t mpnn_backward(const Launch& L, int64_t n, const DSell& S, const MpnnDev& W,
                          const __nv_bfloat16* F, __nv_bfloat16* const H[4],
                          __nv_bfloat16* const Z[3], const float* Y, const float* T, float* dHa,
                          float* dHb, float* dZ, float* part, float* grad, float* loss) {
  // grad layout = parameter layout: W_in, b_in, {W_l, b_l} x 3, W_out, b_out
  const int gb = grid_rows(L, n), gt = grid_bwd(L, n);
  cudaError_t e;
  // every gradient's block partials stay until the one reduction at the end: gb rows of W_out, b_out
  // and the loss, then gt rows per layer and of W_in, less than max_blocks rows of a layer in all
  // (gb <= max_blocks = 8 SMs, gt <= 2 SMs)
  const int wout = kHid * 3 + 4, wl = 2 * kHid * kHid + kHid, wi = kFeat * kHid + kHid;
  static_assert(8 * (kHid * 3 + 4) + 2 * kLayers * (2 * kHid * kHid + kHid) +
                        2 * (kFeat * kHid + kHid) <= 8 * (2 * kHid * kHid + kHid),
                "partials exceed the scratch");
  PartList PL;
  int set = 0, blocks = 0;
  float* pp = part;
  auto add = [&](int nblocks, int count, int stride, float* out, float* last) {
    PL.p[set++] = Parts{nblocks, count, stride, blocks, pp, out, last};
    blocks += (count + (last ? 1 : 0) + 31) / 32;
    float* at = pp;
    pp += (int64_t)nblocks * stride;
    return at;
  };
  (*L.counter) += 1;
  k_out_bwd<<<gb, kThreads, 0, L.stream>>>(n, Y, T, H[kLayers], W.Wout, dHa,
                                           add(gb, wout - 1, wout, grad + kOffWout, loss));
  float* dH = dHa;
  float* dHp = dHb;
  const size_t sm = mpnn_layer_bwd_smem();
  for (int l = kLayers - 1; l >= 0; --l) {
    (*L.counter) += 2;
    k_layer_bwd<<<gt, kThreads, sm, L.stream>>>(n, dH, H[l + 1], H[l], Z[l], W.Wf[l], dHp, dZ,
                                                add(gt, wl, wl, grad + kOffW[l], nullptr));
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    k_agg_t<<<L.blocks_for(n * (kThreads / 64)), kThreads, 0, L.stream>>>(n, S, W.At, dZ, dHp);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    float* t = dH;
    dH = dHp;
    dHp = t;
  }
  (*L.counter) += 2;
  k_in_bwd<<<gt, kThreads, 0, L.stream>>>(n, dH, H[0], F, add(gt, wi, wi, grad, nullptr));
  k_reduce_parts<<<blocks, kThreads, 0, L.stream>>>(PL);
  return cudaGetLastError();
}

cudaError_t mpnn_adam(const Launch& L, float* w, const float* g, float* m, float* v, float lr,
                      int t) {
  const float b1 = 0.9f, b2 = 0.999f;
  const float c1 = 1.f - powf(b1, (float)t), c2 = 1.f - powf(b2, (float)t);
  (*L.counter) += 1;
  k_adam<<<L.blocks_for(kParams), kBlock, 0, L.stream>>>(kParams, w, g, m, v, lr, b1, b2, 1e-8f,
                                                         c1, c2);
  return cudaGetLastError();
}

cudaError_t mpnn_refresh_bf16(const Launch& L, __nv_bfloat16* WinT, __nv_bfloat16* const WT[3],
                              const float* params) {
  (*L.counter) += 1 + kLayers;
  k_transpose_bf16<<<8, 256, 0, L.stream>>>(kFeat, kHid, params + kOffWin, WinT);
  for (int l = 0; l < kLayers; ++l)
    k_transpose_bf16<<<32, 256, 0, L.stream>>>(2 * kHid, kHid, params + kOffW[l], WT[l]);
  return cudaGetLastError();
}

cudaError_t mpnn_setup_smem() {
  cudaError_t e = cudaFuncSetAttribute(k_tc_layer<0>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)mpnn_layer_smem());
  if (e != cudaSuccess) return e;
  e = cudaFuncSetAttribute(k_tc_layer<1>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)mpnn_layer_smem());
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(k_layer_bwd, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)mpnn_layer_bwd_smem());
}

}  // namespace gspm
