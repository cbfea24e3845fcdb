// kpz_mlp.cu -- the learned surrogate: a 4-128-128-128-1 GELU MLP with
// bfloat16 weights and float32 arithmetic, trained with Adam by the kernels
// below (forward and backward in one kernel on the tcgen05 tensor cores,
// gradient reduction and update in another).
//
// The paper has no learned component. The network maps the features of a
// realisation and a time (log2 L, log t, p, q, scaled) to log W^2; the
// ensemble batcher uses its curves to estimate saturation times. Parameters
// are one flat vector: W1 (128x4 row-major), b1, W2 (128x128), b2, W3, b3,
// w4 (128), b4. Gradients are reduced in a fixed order, so training is
// deterministic for a given data order.
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>
#include <new>
#include <vector>

#include "kpz.h"
#include "kpz_host.h"
#include "kpz_internal.h"

namespace kpz {
namespace mlp {

constexpr int kW = 128, kIn = 4;
constexpr int oW1 = 0, oB1 = oW1 + kW * kIn, oW2 = oB1 + kW, oB2 = oW2 + kW * kW, oW3 = oB2 + kW,
              oB3 = oW3 + kW * kW, oW4 = oB3 + kW, oB4 = oW4 + kW, kParams = oB4 + 1;
static_assert(kParams == 33793, "parameter count");
constexpr int kPart = kParams + 3;   // partial of one block: gradient, squared-error sum; 16-byte multiple
static_assert(kPart % 4 == 0 && oW2 % 4 == 0 && oW3 % 4 == 0, "16-byte stores of the weight gradients");

__device__ __forceinline__ float bf(const __nv_bfloat16* p, int i) { return __bfloat162float(p[i]); }

// ---------------------------------------------------------------------------
// Forward and backward pass on the 5th-generation tensor cores (tcgen05). A
// tile is 32 samples; units are the rows of every product (M = 128), samples
// its columns, so one thread owns a unit and 8 samples of it: 16 warps, warp w
// reads tensor-memory lanes 32 (w % 4) onwards and columns 8 (w / 4) onwards.
// What bounds a minibatch is the chain of products and activations, not work:
// a small tile spreads 128 samples over four SMs and leaves a thread 8
// activations a layer (128-sample tiles with 32 took 19 us forward and 113 us
// backward on one SM), and forward and backward share one kernel, which keeps
// the activations' derivatives in registers instead of writing pre-activations
// out and evaluating them three times over. Larger inputs loop over tiles in a
// block per SM, with the weights staged once and the weight gradients
// accumulated in tensor memory.
// Whole calls from host arrays, before (forward, backward, reduction and Adam
// in four kernels with 128-sample tiles, four copies): loss_grad of 128 samples
// 217 -> 40 us, of 300000 2860 -> 470; predict of 251 47 -> 23 us, of 300000
// 332 -> 240; 24 training steps of 128 samples 4.3 -> 0.64 ms.
//
// Operands are bfloat16 in shared memory without swizzle, core matrices of 8
// rows x 16 bytes. The weights are bfloat16 already; activations h and errors
// dz are split into a high and a low part, hi = bf16(a), lo = bf16(a - hi), and
// every product takes the chains that matter (hi, lo with weights; hi.hi,
// hi.lo, lo.hi between activations and errors), which agrees with the float32
// product to about 2^-16 relative. One copy of each operand serves all its
// products, as K-major or MN-major matrix:
//   W [unit][k]        forward: A, K-major; input gradient: A = W^T, MN-major
//   h, dz [unit][sample] (8 samples = 16 bytes): B, MN-major, of those two;
//                      weight gradient dz h^T: A and B, K-major (K = samples).
// One thread issues the products and commits them to an mbarrier; every wait
// on one is bounded in time (a timeout sets *err and the host reports it).
namespace tc {

constexpr int kS = 32;                                // samples per tile
constexpr int kThreads = 512;
constexpr uint32_t kWBytes = (uint32_t)kW * kW * 2;   // a weight matrix
constexpr uint32_t kHBytes = (uint32_t)kW * kS * 2;   // a high or low part of h or dz
// Instruction descriptor of tcgen05.mma kind::f16: float32 accumulator, both
// operands bfloat16, transpose bits (MN-major A, B), N / 8, M / 16.
constexpr uint32_t idesc(bool ta, bool tb, int n) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((ta ? 1u : 0u) << 15) | ((tb ? 1u : 0u) << 16) |
         ((uint32_t)(n >> 3) << 17) | ((uint32_t)(kW >> 4) << 24);
}
constexpr uint64_t kWaitNs = 1000000000ull;           // bound of every wait

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// Shared-memory matrix descriptor: start address, byte offsets between core
// matrices along the leading dimension (K) and the other one, version 1 (bit
// 46), no swizzle.
__device__ __forceinline__ uint64_t sdesc(uint32_t addr, uint32_t along_k, uint32_t along_mn) {
  return (uint64_t)((addr >> 4) & 0x3FFFu) | ((uint64_t)(along_k >> 4) << 16) | ((uint64_t)(along_mn >> 4) << 32) |
         (1ull << 46);
}
__device__ __forceinline__ void mma(uint32_t d, uint64_t a, uint64_t b, uint32_t id, bool acc) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(d),
      "l"(a), "l"(b), "r"(id), "r"((uint32_t)acc));
}
__device__ __forceinline__ void commit(uint32_t mbar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(mbar) : "memory");
}
// D[j][s] = sum_k W[j][k] h[k][s].
__device__ __forceinline__ void mma_forward(uint32_t d, uint32_t w, uint32_t hi, uint32_t lo) {
#pragma unroll
  for (int i = 0; i < 2 * (kW / 16); ++i) {
    const int kk = i & 7;
    mma(d, sdesc(w + kk * 256u, 128u, 2048u), sdesc((i < 8 ? hi : lo) + kk * 1024u, 512u, 128u), idesc(false, true, kS),
        i != 0);
  }
}
// D[k][s] = sum_u W[u][k] dz[u][s].
__device__ __forceinline__ void mma_input(uint32_t d, uint32_t w, uint32_t hi, uint32_t lo) {
#pragma unroll
  for (int i = 0; i < 2 * (kW / 16); ++i) {
    const int kk = i & 7;
    mma(d, sdesc(w + kk * 4096u, 2048u, 128u), sdesc((i < 8 ? hi : lo) + kk * 1024u, 512u, 128u), idesc(true, true, kS),
        i != 0);
  }
}
// D[u][k] (+)= sum_s dz[u][s] h[k][s].
__device__ __forceinline__ void mma_weight(uint32_t d, uint32_t dzhi, uint32_t dzlo, uint32_t hhi, uint32_t hlo, bool acc) {
#pragma unroll
  for (int i = 0; i < 6; ++i) {
    const uint32_t a = (i >= 4 ? dzlo : dzhi) + (i & 1) * 256u, b = ((i & 6) == 2 ? hlo : hhi) + (i & 1) * 256u;
    mma(d, sdesc(a, 128u, 512u), sdesc(b, 128u, 512u), idesc(false, false, kW), acc || i != 0);
  }
}

__device__ __forceinline__ uint64_t gtimer() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
// Wait until phase `parity` of the mbarrier has completed; false on timeout.
__device__ __forceinline__ bool wait_phase(uint32_t mbar, uint32_t parity) {
  uint64_t t0 = 0;
  for (uint32_t it = 0;; ++it) {
    uint32_t done;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.b32 %0, 1, 0, p;\n}\n"
        : "=r"(done)
        : "r"(mbar), "r"(parity)
        : "memory");
    if (done) break;
    if (it == 0) t0 = gtimer();
    else if (gtimer() - t0 > kWaitNs) return false;
  }
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  return true;
}

// 8 and 32 consecutive float32 columns of this warp's 32 tensor-memory lanes.
// The aligned forms are only defined for a converged warp; lanes leave the wait
// before one at a time.
__device__ __forceinline__ void ld8(uint32_t ta, float (&v)[8]) {
  uint32_t r[8];
  __syncwarp();
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "r"(ta));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 8; ++i) v[i] = __uint_as_float(r[i]);
}
__device__ __forceinline__ void ld32(uint32_t ta, float (&v)[32]) {
  uint32_t r[32];
  __syncwarp();
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
      "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
        "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
        "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(ta));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
}

// Eight values of unit u and sample group g, as high and low parts.
__device__ __forceinline__ void put8(unsigned char* Xhi, unsigned char* Xlo, int u, int g, const float (&v)[8]) {
  __align__(16) __nv_bfloat16 hi[8], lo[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    hi[i] = __float2bfloat16_rn(v[i]);
    lo[i] = __float2bfloat16_rn(v[i] - __bfloat162float(hi[i]));
  }
  const uint32_t at = (uint32_t)(((u >> 3) * 4 + g) * 128 + (u & 7) * 16);
  *reinterpret_cast<uint4*>(Xhi + at) = *reinterpret_cast<const uint4*>(hi);
  *reinterpret_cast<uint4*>(Xlo + at) = *reinterpret_cast<const uint4*>(lo);
}

// W (128 x 128 bfloat16, row = output unit, K contiguous): 8-row x 16-byte core
// matrices, 128 bytes apart along K, 2048 along the rows.
__device__ __forceinline__ void stage_w(unsigned char* Bs, const __nv_bfloat16* W, int t) {
  uint4 v[kW * kW / 8 / kThreads];
#pragma unroll
  for (int i = 0; i < kW * kW / 8 / kThreads; ++i) v[i] = *reinterpret_cast<const uint4*>(W + (t + i * kThreads) * 8);
#pragma unroll
  for (int i = 0; i < kW * kW / 8 / kThreads; ++i) {
    const int q = t + i * kThreads, row = q >> 4, k8 = q & 15;
    *reinterpret_cast<uint4*>(Bs + ((row >> 3) * 16 + k8) * 128 + (row & 7) * 16) = v[i];
  }
}

// Shared-memory writes of all threads visible to the tensor cores.
__device__ __forceinline__ void fence_to_mma() {
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}

// gelu(z) and, for training, its derivative (sharing the error function).
template <bool kGrad>
__device__ __forceinline__ float gelu(float z, float& d) {
  const float c = 0.5f * (1.0f + erff(z * 0.70710678118654752f));
  if (kGrad) d = c + z * 0.39894228040143268f * expf(-0.5f * z * z);
  return z * c;
}

constexpr size_t kSmemPredict = 2 * (size_t)kWBytes + 2 * (size_t)kHBytes;   // W2, W3, h hi, h lo
constexpr size_t kSmemGrad = 2 * (size_t)kWBytes + 8 * (size_t)kHBytes;      // h1, h2, dz3, dz2, hi and lo

}  // namespace tc

// kGrad = false: y[i] = network(x[i]). kGrad = true: the gradient of the mean
// squared error over the block's tiles (block b takes tiles b, b + gridDim.x,
// ...) and the sum of squared errors into its slot of gpart. x, t and y may be
// host memory the device reaches; the next tile's samples are read ahead.
template <bool kGrad>
__global__ void __launch_bounds__(tc::kThreads, kGrad ? 1 : 2)
    net_kernel(const __nv_bfloat16* __restrict__ P, const float* __restrict__ x, const float* __restrict__ t, int n,
               float inv_n, float* __restrict__ y, float* __restrict__ gpart, int* err) {
  extern __shared__ __align__(1024) unsigned char smem_tc[];
  unsigned char* Wb[2] = {smem_tc, smem_tc + tc::kWBytes};
  unsigned char* Hb = smem_tc + 2 * tc::kWBytes;
  // h1, h2 (predict: one pair of buffers, h2 replaces h1), dz3, dz2; hi and lo
  auto buf = [&](int i) { return Hb + (size_t)i * tc::kHBytes; };
  constexpr int iH1 = 0, iH2 = kGrad ? 2 : 0, iD3 = 4, iD2 = 6;
  constexpr uint32_t kCols = kGrad ? 512u : 32u;   // tensor memory: products 0..31, dW3 32.., dW2 160..
  __shared__ __align__(8) uint64_t mbar[2];
  __shared__ uint32_t taddr_s;
  __shared__ float xs[tc::kS * kIn], ts[tc::kS], part[4][tc::kS];
  __shared__ float red[4][kW][kIn + 1];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int u = (warp & 3) * 32 + lane, g = warp >> 2, s0 = 8 * g;
  const int ntiles = (n + tc::kS - 1) / tc::kS;
  // Samples of a tile, one value a thread: inputs (threads 0..127), targets (128..159).
  auto fetch = [&](int tile) -> float {
    const long long i = (long long)tile * tc::kS;
    if (tile >= ntiles) return 0.f;
    if (tid < tc::kS * kIn) return i + (tid >> 2) < n ? x[i * kIn + tid] : 0.f;
    if (kGrad && tid < tc::kS * (kIn + 1)) return i + (tid - tc::kS * kIn) < n ? t[i + (tid - tc::kS * kIn)] : 0.f;
    return 0.f;
  };
  float ahead = fetch(blockIdx.x);
  tc::stage_w(Wb[0], P + oW2, tid);
  tc::stage_w(Wb[1], P + oW3, tid);
  float w1[kIn];
#pragma unroll
  for (int c = 0; c < kIn; ++c) w1[c] = bf(P + oW1, u * kIn + c);
  const float b1 = bf(P + oB1, u), b2 = bf(P + oB2, u), b3 = bf(P + oB3, u), w4 = bf(P + oW4, u), b4 = bf(P + oB4, 0);
  if (tid == 0) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(tc::smem_u32(&mbar[0])));
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(tc::smem_u32(&mbar[1])));
  }
  if (warp == 0) {
    __syncwarp();
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(tc::smem_u32(&taddr_s)),
                 "n"(kCols));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  tc::fence_to_mma();
  const uint32_t taddr = taddr_s, lanes = taddr + ((uint32_t)((warp & 3) * 32) << 16);
  const uint32_t mz = tc::smem_u32(&mbar[0]), mw = tc::smem_u32(&mbar[1]);
  const uint32_t w2a = tc::smem_u32(Wb[0]), w3a = tc::smem_u32(Wb[1]);
  uint32_t phase = 0, wphase = 0;
  bool ok = true;
  float gw1[kIn] = {0.f, 0.f, 0.f, 0.f}, gb1 = 0.f, gb2 = 0.f, gb3 = 0.f, gw4 = 0.f, gb4 = 0.f, gsq = 0.f;
  bool first = true;
#pragma unroll 1
  for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
    if (tid < tc::kS * kIn) xs[tid] = ahead;
    else if (kGrad && tid < tc::kS * (kIn + 1)) ts[tid - tc::kS * kIn] = ahead;
    __syncthreads();
    ahead = fetch(tile + (int)gridDim.x);
    float h[8], d1[8], d2[8], d3[8], z[8];
    // Layer 1 (K = 4) on the CUDA cores.
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      float v = b1;
#pragma unroll
      for (int c = 0; c < kIn; ++c) v += w1[c] * xs[(s0 + i) * kIn + c];
      h[i] = tc::gelu<kGrad>(v, d1[i]);
    }
    tc::put8(buf(iH1), buf(iH1 + 1), u, g, h);
    tc::fence_to_mma();
    if (tid == 0) {
      tc::mma_forward(taddr, w2a, tc::smem_u32(buf(iH1)), tc::smem_u32(buf(iH1 + 1)));
      tc::commit(mz);
    }
    ok = tc::wait_phase(mz, phase) && ok;
    phase ^= 1u;
    tc::ld8(lanes + (uint32_t)s0, z);
#pragma unroll
    for (int i = 0; i < 8; ++i) h[i] = tc::gelu<kGrad>(z[i] + b2, d2[i]);
    tc::put8(buf(iH2), buf(iH2 + 1), u, g, h);
    tc::fence_to_mma();
    if (tid == 0) {
      tc::mma_forward(taddr, w3a, tc::smem_u32(buf(iH2)), tc::smem_u32(buf(iH2 + 1)));
      tc::commit(mz);
    }
    ok = tc::wait_phase(mz, phase) && ok;
    phase ^= 1u;
    tc::ld8(lanes + (uint32_t)s0, z);
#pragma unroll
    for (int i = 0; i < 8; ++i) h[i] = tc::gelu<kGrad>(z[i] + b3, d3[i]);
    // Output: sum over the units, 32 by shuffles, then the four warps of a sample group.
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      float o = w4 * h[i];
#pragma unroll
      for (int d = 16; d > 0; d >>= 1) o += __shfl_xor_sync(0xffffffffu, o, d);
      if (lane == i) part[warp & 3][s0 + i] = o;
    }
    __syncthreads();
    if (!kGrad) {
      const int s = tile * tc::kS + tid;
      if (tid < tc::kS && s < n) y[s] = ((part[0][tid] + part[1][tid]) + part[2][tid]) + part[3][tid] + b4;
      __syncthreads();   // part is written again by the next tile
      continue;
    }
    float dy[8];
    float sg4 = 0.f;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int s = s0 + i;
      const float o = ((part[0][s] + part[1][s]) + part[2][s]) + part[3][s] + b4;
      const float r = tile * tc::kS + s < n ? o - ts[s] : 0.f;
      dy[i] = 2.f * r * inv_n;
      sg4 += dy[i];
      gsq += r * r;
    }
    gb4 += sg4;
    // Layer 3: dz3 = dy w4 gelu'(z3); its products with h2 and W3.
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      gw4 += dy[i] * h[i];
      h[i] = dy[i] * w4 * d3[i];
      gb3 += h[i];
    }
    tc::put8(buf(iD3), buf(iD3 + 1), u, g, h);
    tc::fence_to_mma();
    if (tid == 0) {
      tc::mma_input(taddr, w3a, tc::smem_u32(buf(iD3)), tc::smem_u32(buf(iD3 + 1)));
      tc::commit(mz);
      tc::mma_weight(taddr + 32u, tc::smem_u32(buf(iD3)), tc::smem_u32(buf(iD3 + 1)), tc::smem_u32(buf(iH2)),
                     tc::smem_u32(buf(iH2 + 1)), !first);
    }
    ok = tc::wait_phase(mz, phase) && ok;
    phase ^= 1u;
    tc::ld8(lanes + (uint32_t)s0, z);
    // Layer 2: dz2 = dh2 gelu'(z2).
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      h[i] = z[i] * d2[i];
      gb2 += h[i];
    }
    tc::put8(buf(iD2), buf(iD2 + 1), u, g, h);
    tc::fence_to_mma();
    if (tid == 0) {
      tc::mma_input(taddr, w2a, tc::smem_u32(buf(iD2)), tc::smem_u32(buf(iD2 + 1)));
      tc::commit(mz);
      tc::mma_weight(taddr + 160u, tc::smem_u32(buf(iD2)), tc::smem_u32(buf(iD2 + 1)), tc::smem_u32(buf(iH1)),
                     tc::smem_u32(buf(iH1 + 1)), !first);
      tc::commit(mw);
    }
    ok = tc::wait_phase(mz, phase) && ok;
    phase ^= 1u;
    tc::ld8(lanes + (uint32_t)s0, z);
    // Layer 1: dz1 = dh1 gelu'(z1).
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const float d = z[i] * d1[i];
      gb1 += d;
#pragma unroll
      for (int c = 0; c < kIn; ++c) gw1[c] += d * xs[(s0 + i) * kIn + c];
    }
    ok = tc::wait_phase(mw, wphase) && ok;   // the operands of the weight products are free again
    wphase ^= 1u;
    first = false;
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();   // xs, ts and part are written again by the next tile
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  }
  if (kGrad) {
    float* o = gpart + (size_t)blockIdx.x * kPart;
    // Sums over the four sample groups, in a fixed order.
    auto combine = [&](int c) -> float { return ((red[0][u][c] + red[1][u][c]) + red[2][u][c]) + red[3][u][c]; };
#pragma unroll
    for (int c = 0; c < kIn; ++c) red[g][u][c] = gw1[c];
    red[g][u][kIn] = gb1;
    __syncthreads();
    if (g == 0) {
#pragma unroll
      for (int c = 0; c < kIn; ++c) o[oW1 + u * kIn + c] = combine(c);
      o[oB1 + u] = combine(kIn);
    }
    __syncthreads();
    red[g][u][0] = gb2;
    red[g][u][1] = gb3;
    red[g][u][2] = gw4;
    red[g][u][3] = gb4;   // the same for every unit of a group
    red[g][u][4] = gsq;
    __syncthreads();
    if (g == 0) {
      o[oB2 + u] = combine(0);
      o[oB3 + u] = combine(1);
      o[oW4 + u] = combine(2);
      if (u == 0) {
        o[oB4] = combine(3);
        o[kParams] = combine(4);
      }
    }
    // Weight gradients: row u, columns 32 g .. 32 g + 31 of each matrix.
#pragma unroll
    for (int m = 0; m < 2; ++m) {
      float v[32];
      tc::ld32(lanes + (m ? 160u : 32u) + 32u * (uint32_t)g, v);
      float4* dst = reinterpret_cast<float4*>(o + (m ? oW2 : oW3) + u * kW + 32 * g);
#pragma unroll
      for (int i = 0; i < 8; ++i) dst[i] = make_float4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
    }
  }
  if (!ok) {
    *(volatile int*)err = 1;
    __threadfence_system();
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "n"(kCols));
}

// Sum over the blocks' partials, in order (deterministic).
__device__ __forceinline__ float reduce_one(const float* __restrict__ gpart, int nparts, int i) {
  float s = 0.f;
  int b = 0;
  for (; b + 8 <= nparts; b += 8) {
    float v[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) v[k] = gpart[(size_t)(b + k) * kPart + i];
#pragma unroll
    for (int k = 0; k < 8; ++k) s += v[k];
  }
  for (; b < nparts; ++b) s += gpart[(size_t)b * kPart + i];
  return s;
}

// grad[i] (may be null) and the sum of squared errors; both may be host memory.
__global__ void reduce_kernel(const float* __restrict__ gpart, int nparts, float* __restrict__ grad, float* sq) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i > kParams || (i < kParams && !grad)) return;
  const float s = reduce_one(gpart, nparts, i);
  if (i < kParams) grad[i] = s;
  else *sq = s;
}

// Reduction and Adam (Kingma and Ba): master weights in float32, bfloat16 copy for the passes.
__global__ void adam_kernel(const float* __restrict__ gpart, int nparts, float* __restrict__ theta, float* __restrict__ m,
                            float* __restrict__ v, __nv_bfloat16* __restrict__ P, float* sq, float lr, float b1, float b2,
                            float c1, float c2, float eps) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i > kParams) return;
  const float gi = reduce_one(gpart, nparts, i);
  if (i == kParams) {
    *sq = gi;
    return;
  }
  const float mi = b1 * m[i] + (1.f - b1) * gi;
  const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
  m[i] = mi;
  v[i] = vi;
  const float th = theta[i] - lr * (mi / c1) / (sqrtf(vi / c2) + eps);
  theta[i] = th;
  P[i] = __float2bfloat16_rn(th);
}

__global__ void to_bf16_kernel(const float* __restrict__ theta, __nv_bfloat16* __restrict__ P) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < kParams) P[i] = __float2bfloat16_rn(theta[i]);
}

}  // namespace mlp
}  // namespace kpz

using namespace kpz;
using namespace kpz::mlp;

struct kpz_mlp {
  int device = 0;
  int sms = 0;
  bool direct_host = false;     // the GPU reads and writes pageable host memory itself
  cudaStream_t stream = nullptr;
  float* theta = nullptr;       // master parameters
  float* m = nullptr;
  float* v = nullptr;
  __nv_bfloat16* P = nullptr;   // bfloat16 copy
  uint64_t step = 0;
  // per-call buffers: data (x, t, y) for `cap` samples, partials of `pcap` blocks, a gradient
  float *x = nullptr, *t = nullptr, *y = nullptr, *gpart = nullptr, *grad = nullptr;
  size_t cap = 0, pcap = 0;
  // Set when a tensor-core wait timed out; sum of squared errors. The kernels
  // write them here where the GPU reaches pageable memory, else to device memory.
  struct Out { int err; float sq; };
  alignas(64) Out result = {};
  Out* out = nullptr;
};

namespace {

void mlp_release(kpz_mlp* m) {
  float* ptrs[] = {m->theta, m->m, m->v, m->grad, m->x, m->t, m->y, m->gpart};
  for (float* p : ptrs) if (p) cudaFree(p);
  if (m->P) cudaFree(m->P);
  if (m->out && m->out != &m->result) cudaFree(m->out);
}

// Synchronises the stream; KPZ_ETIMEOUT when a kernel's tensor-core wait ran
// out (the flag is then cleared).
kpz_status finish(kpz_mlp* m) {
  if (m->out != &m->result &&
      cudaMemcpyAsync(&m->result, m->out, sizeof(m->result), cudaMemcpyDeviceToHost, m->stream) != cudaSuccess)
    return KPZ_ECUDA;
  if (cudaStreamSynchronize(m->stream) != cudaSuccess) return KPZ_ECUDA;
  volatile kpz_mlp::Out* h = &m->result;
  if (h->err) {
    h->err = 0;
    if (m->out != &m->result) cudaMemsetAsync(&m->out->err, 0, sizeof(int), m->stream);
    return KPZ_ETIMEOUT;
  }
  return KPZ_OK;
}

// Device buffers for n samples.
kpz_status ensure_data(kpz_mlp* m, size_t n) {
  if (n <= m->cap) return KPZ_OK;
  float** bufs[] = {&m->x, &m->t, &m->y};
  for (float** p : bufs) {
    if (*p) cudaFree(*p);
    *p = nullptr;
  }
  m->cap = 0;
  if (cudaMalloc(&m->x, n * kIn * 4) != cudaSuccess || cudaMalloc(&m->t, n * 4) != cudaSuccess ||
      cudaMalloc(&m->y, n * 4) != cudaSuccess) {
    cudaGetLastError();
    return KPZ_ENOMEM;
  }
  m->cap = n;
  return KPZ_OK;
}

int tiles_of(size_t n) { return (int)((n + tc::kS - 1) / tc::kS); }
int grad_blocks(const kpz_mlp* m, size_t n) { return std::min(tiles_of(n), m->sms); }

// The kernels count samples in 32 bits, a tile beyond the last one included; a
// call for more is refused before any of its arrays is touched.
constexpr uint32_t kMaxSamples = 0x7FFFFFFFu - (uint32_t)(tc::kS - 1);

// Partials for gradients over n samples.
kpz_status ensure_parts(kpz_mlp* m, size_t n) {
  const size_t b = (size_t)grad_blocks(m, n);
  if (b <= m->pcap) return KPZ_OK;
  if (m->gpart) cudaFree(m->gpart);
  m->gpart = nullptr;
  m->pcap = 0;
  if (cudaMalloc(&m->gpart, b * kPart * 4) != cudaSuccess) {
    cudaGetLastError();
    return KPZ_ENOMEM;
  }
  m->pcap = b;
  return KPZ_OK;
}

// Partial gradients of the mean squared error over n samples; returns the
// number of partials.
int queue_grad(kpz_mlp* m, const float* x, const float* t, int n) {
  const int blocks = grad_blocks(m, (size_t)n);
  net_kernel<true><<<blocks, tc::kThreads, tc::kSmemGrad, m->stream>>>(m->P, x, t, n, 1.f / (float)n, nullptr, m->gpart,
                                                                      &m->out->err);
  count_launch();
  return blocks;
}

constexpr unsigned kReduceBlocks = (kParams + 1 + 255) / 256;

}  // namespace

extern "C" {

kpz_status kpz_mlp_create(kpz_mlp** out, const float* params, void* stream) {
  if (!out || !params) return KPZ_EINVAL;
  *out = nullptr;
  int ndev = 0;
  if (cudaGetDeviceCount(&ndev) != cudaSuccess || ndev == 0) return KPZ_ENODEV;
  kpz_mlp* m = new (std::nothrow) kpz_mlp();
  if (!m) return KPZ_ENOMEM;
  cudaGetDevice(&m->device);
  cudaDeviceGetAttribute(&m->sms, cudaDevAttrMultiProcessorCount, m->device);
  m->sms = std::max(m->sms, 1);
  m->direct_host = reaches_pageable(m->device);
  if (m->direct_host) m->out = &m->result;
  m->stream = (cudaStream_t)stream;
  if (cudaMalloc(&m->theta, kParams * 4) != cudaSuccess || cudaMalloc(&m->m, kParams * 4) != cudaSuccess ||
      cudaMalloc(&m->v, kParams * 4) != cudaSuccess || cudaMalloc(&m->grad, kParams * 4) != cudaSuccess ||
      cudaMalloc(&m->P, kParams * 2) != cudaSuccess ||
      (!m->direct_host && cudaMalloc(&m->out, sizeof(*m->out)) != cudaSuccess)) {
    cudaGetLastError();
    mlp_release(m);
    delete m;
    return KPZ_ENOMEM;
  }
  if (cudaFuncSetAttribute(net_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)tc::kSmemGrad) !=
          cudaSuccess ||
      cudaFuncSetAttribute(net_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)tc::kSmemPredict) !=
          cudaSuccess ||
      cudaMemcpyAsync(m->theta, params, kParams * 4, cudaMemcpyHostToDevice, m->stream) != cudaSuccess ||
      cudaMemsetAsync(m->m, 0, kParams * 4, m->stream) != cudaSuccess ||
      cudaMemsetAsync(m->v, 0, kParams * 4, m->stream) != cudaSuccess ||
      (!m->direct_host && cudaMemsetAsync(m->out, 0, sizeof(*m->out), m->stream) != cudaSuccess)) {
    mlp_release(m);
    delete m;
    return KPZ_ECUDA;
  }
  to_bf16_kernel<<<(kParams + 255) / 256, 256, 0, m->stream>>>(m->theta, m->P);
  count_launch();
  if (cudaStreamSynchronize(m->stream) != cudaSuccess) {
    mlp_release(m);
    delete m;
    return KPZ_ECUDA;
  }
  *out = m;
  return KPZ_OK;
}

kpz_status kpz_mlp_params(kpz_mlp* m, float* params) {
  if (!m || !params) return KPZ_EINVAL;
  if (cudaMemcpyAsync(params, m->theta, kParams * 4, cudaMemcpyDeviceToHost, m->stream) != cudaSuccess ||
      cudaStreamSynchronize(m->stream) != cudaSuccess)
    return KPZ_ECUDA;
  return KPZ_OK;
}

// Where the GPU reaches pageable host memory (its pages touched before it
// writes them), predict and loss_grad read and write the caller's arrays in the
// kernels: a launch or two and one synchronisation instead of four copies.
// Arrays that are not aligned, or an output that overlaps an input, are copied.
kpz_status kpz_mlp_predict(kpz_mlp* m, const float* x, uint32_t n, float* y) {
  if (!m || !x || !y) return KPZ_EINVAL;
  if (n == 0) return KPZ_OK;
  if (n > kMaxSamples) return KPZ_ENOMEM;
  const float* xin = x;
  float* yout = y;
  const HostSpan in = {x, (size_t)n * kIn * 4};
  const bool direct = m->direct_host && usable_in_place(&in, 1, HostSpan{y, (size_t)n * 4});
  if (direct) {
    touch_pages(y, (size_t)n * 4);
  } else {
    kpz_status st = ensure_data(m, n);
    if (st) return st;
    if (cudaMemcpyAsync(m->x, x, (size_t)n * kIn * 4, cudaMemcpyHostToDevice, m->stream) != cudaSuccess) return KPZ_ECUDA;
    xin = m->x;
    yout = m->y;
  }
  net_kernel<false><<<std::min(tiles_of(n), 2 * m->sms), tc::kThreads, tc::kSmemPredict, m->stream>>>(
      m->P, xin, nullptr, (int)n, 0.f, yout, nullptr, &m->out->err);
  count_launch();
  if (cudaGetLastError() != cudaSuccess ||
      (!direct && cudaMemcpyAsync(y, m->y, (size_t)n * 4, cudaMemcpyDeviceToHost, m->stream) != cudaSuccess))
    return KPZ_ECUDA;
  return finish(m);
}

kpz_status kpz_mlp_loss_grad(kpz_mlp* m, const float* x, const float* t, uint32_t n, float* loss, float* grad) {
  if (!m || !x || !t || n == 0) return KPZ_EINVAL;
  if (n > kMaxSamples) return KPZ_ENOMEM;
  kpz_status st = ensure_parts(m, n);
  if (st) return st;
  const float *xin = x, *tin = t;
  float* gout = grad;
  const HostSpan in[2] = {{x, (size_t)n * kIn * 4}, {t, (size_t)n * 4}};
  const bool direct = m->direct_host && usable_in_place(in, 2, HostSpan{grad, (size_t)kParams * 4});
  if (direct) {
    if (grad) touch_pages(grad, kParams * 4);
  } else {
    if ((st = ensure_data(m, n)) != KPZ_OK) return st;
    if (cudaMemcpyAsync(m->x, x, (size_t)n * kIn * 4, cudaMemcpyHostToDevice, m->stream) != cudaSuccess ||
        cudaMemcpyAsync(m->t, t, (size_t)n * 4, cudaMemcpyHostToDevice, m->stream) != cudaSuccess)
      return KPZ_ECUDA;
    xin = m->x;
    tin = m->t;
    gout = grad ? m->grad : nullptr;
  }
  const int parts = queue_grad(m, xin, tin, (int)n);
  reduce_kernel<<<kReduceBlocks, 256, 0, m->stream>>>(m->gpart, parts, gout, &m->out->sq);
  count_launch();
  if (cudaGetLastError() != cudaSuccess ||
      (grad && !direct &&
       cudaMemcpyAsync(grad, m->grad, kParams * 4, cudaMemcpyDeviceToHost, m->stream) != cudaSuccess))
    return KPZ_ECUDA;
  st = finish(m);
  if (loss) *loss = *(volatile float*)&m->result.sq / (float)n;
  return st;
}

kpz_status kpz_mlp_train(kpz_mlp* m, const float* x, const float* t, uint32_t n, const uint32_t* order,
                         uint32_t steps, uint32_t batch, float lr, float* last_loss) {
  if (!m || !x || !t || !order || n == 0 || batch == 0 || !(lr > 0.f)) return KPZ_EINVAL;
  if (batch > kMaxSamples) return KPZ_ENOMEM;
  // Upload the minibatches already gathered in the order the caller chose:
  // step s uses samples order[s*batch .. s*batch + batch - 1] (indices < n).
  const size_t total = (size_t)steps * batch;
  for (size_t i = 0; i < total; ++i) if (order[i] >= n) return KPZ_EINVAL;
  kpz_status st = ensure_data(m, total);
  if (st == KPZ_OK) st = ensure_parts(m, batch);
  if (st) return st;
  std::vector<float> xg(total * kIn), tg(total);
  for (size_t i = 0; i < total; ++i) {
    for (int c = 0; c < kIn; ++c) xg[i * kIn + c] = x[(size_t)order[i] * kIn + c];
    tg[i] = t[order[i]];
  }
  if (cudaMemcpyAsync(m->x, xg.data(), total * kIn * 4, cudaMemcpyHostToDevice, m->stream) != cudaSuccess ||
      cudaMemcpyAsync(m->t, tg.data(), total * 4, cudaMemcpyHostToDevice, m->stream) != cudaSuccess)
    return KPZ_ECUDA;
  const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
  m->result.sq = 0.f;   // the loss of no step at all
  if (m->out != &m->result && cudaMemsetAsync(&m->out->sq, 0, sizeof(float), m->stream) != cudaSuccess) return KPZ_ECUDA;
  for (uint32_t s = 0; s < steps; ++s) {
    ++m->step;
    const float c1 = 1.f - std::pow(b1, (float)m->step), c2 = 1.f - std::pow(b2, (float)m->step);
    const int parts = queue_grad(m, m->x + (size_t)s * batch * kIn, m->t + (size_t)s * batch, (int)batch);
    adam_kernel<<<kReduceBlocks, 256, 0, m->stream>>>(m->gpart, parts, m->theta, m->m, m->v, m->P, &m->out->sq, lr, b1, b2,
                                                      c1, c2, eps);
    count_launch();
  }
  if (cudaGetLastError() != cudaSuccess) return KPZ_ECUDA;
  st = finish(m);
  if (last_loss) *last_loss = *(volatile float*)&m->result.sq / (float)batch;
  return st;
}

void kpz_mlp_free(kpz_mlp* m) {
  if (!m) return;
  cudaSetDevice(m->device);
  cudaStreamSynchronize(m->stream);
  mlp_release(m);
  delete m;
}

}  // extern "C"
