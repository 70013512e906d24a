// The learned warm start: a small fully convolutional network (3x3 convolutions
// cin -> 32 -> 32 -> 32 -> 2, GELU after the first three) that maps the forcing sampled on
// the streamfunction control grid plus log10(sigma/nu) to a scaled streamfunction and a
// scaled pressure; the exact discrete curl of the first seeds the V-cycle with a
// divergence-free velocity, the second with a pressure.
//
// Weights are held in BF16 for every product (FP32 master copy for the optimizer);
// accumulation is FP32.  Forward, backward (data and weights), the masked mean-squared loss and
// Adam are hand-written kernels.  Training keeps FP32 activations: tiles of 16 x 16 pixels per
// block with the input tile (plus halo) and the layer's weights staged in shared memory.  Inference
// hands BF16 activations from layer to layer and runs the 32 -> 32 layers on the tensor cores,
// over tiles of 128 consecutive pixels whose neighbourhoods are gathered from global memory.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cmath>
#include <cstdlib>
#include <cstdint>
#include <cstring>
#include <string>
#include <vector>

#include "igamg.h"

namespace {

constexpr int TILE = 16;
constexpr int NT = TILE * TILE;       // threads per block
template <int DIL> struct Halo { static constexpr int value = TILE + 2 * DIL; };

__device__ __forceinline__ float gelu_f(float z) { return 0.5f * z * (1.0f + erff(z * 0.70710678118654752f)); }
__device__ __forceinline__ float gelu_grad_f(float z) {
  return 0.5f * (1.0f + erff(z * 0.70710678118654752f)) + z * 0.39894228040143268f * expf(-0.5f * z * z);
}

enum Epi { EPI_GELU = 0, EPI_LINEAR = 1, EPI_DGELU = 2 };

// out[b,o,p] = bias[o] + sum_{c,tap} w[o,c,tap] in[b,c,p+DIL*tap] (zero padding; taps in
// {-1,0,1}^2, spread by the dilation DIL), then
//   EPI_GELU:   z = out, a = gelu(z)          (z -> outz, a -> outa)
//   EPI_LINEAR: z = out                        (-> outz)
//   EPI_DGELU:  out * gelu'(aux[b,o,p])        (-> outz; backward through an activation)
// w: the layer's BF16 weights as floats, [c][tap][o].  What bounds the 32-output layers is the data the
// shared memory returns to registers (128 bytes a cycle, broadcast or not): one pixel by 32 outputs
// per thread took 33 words per 32 multiply-adds and 36 us a tile; four pixels by eight outputs
// take 12 (58 us a layer of 8 inputs of 66 x 66, 75 before).
template <int CIN, int COUT, int DIL>
__global__ void __launch_bounds__(NT) k_conv(int H, int W, int tiles_x, int tiles_y, const float* __restrict__ in,
                                             const float* __restrict__ w, const float* __restrict__ bias,
                                             const float* __restrict__ aux, float* __restrict__ outz,
                                             float* __restrict__ outa, int epi) {
  constexpr int HALO = Halo<DIL>::value;
  extern __shared__ __align__(16) float smf[];
  float* ws = smf;                                  // COUT * CIN * 9
  float* tile = smf + COUT * CIN * 9;               // CIN * HALO * HALO
  const int tid = threadIdx.x;
  const int tpi = tiles_x * tiles_y;
  const int b = blockIdx.x / tpi, t = blockIdx.x - b * tpi;
  const int y0 = (t / tiles_x) * TILE, x0 = (t % tiles_x) * TILE;
  for (int i = tid; i < COUT * CIN * 9; i += NT) ws[i] = w[i];
  const float* inb = in + (size_t)b * CIN * H * W;
  for (int i = tid; i < CIN * HALO * HALO; i += NT) {
    int c = i / (HALO * HALO), r = i - c * HALO * HALO;
    int yy = y0 + r / HALO - DIL, xx = x0 + r % HALO - DIL;
    tile[i] = (yy >= 0 && yy < H && xx >= 0 && xx < W) ? inb[((size_t)c * H + yy) * W + xx] : 0.0f;
  }
  __syncthreads();
  if constexpr (COUT == 32) {
    // four pixels (rows ty + 4 k) by eight outputs (o0 ..) per thread: 12 shared words per 32 multiply-adds
    const int tx = tid % TILE, ty = tid / TILE % 4, o0 = tid / 64 * 8;
    float acc[4][8];
#pragma unroll
    for (int k = 0; k < 4; ++k)
#pragma unroll
      for (int o = 0; o < 8; ++o) acc[k][o] = 0.0f;
    for (int c = 0; c < CIN; ++c) {
#pragma unroll
      for (int tap = 0; tap < 9; ++tap) {
        const float* wk = ws + (c * 9 + tap) * COUT + o0;
        const float4 q0 = *reinterpret_cast<const float4*>(wk), q1 = *reinterpret_cast<const float4*>(wk + 4);
        const float* tp = tile + c * HALO * HALO + (ty + DIL * (tap / 3)) * HALO + tx + DIL * (tap % 3);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const float v = tp[4 * k * HALO];
          acc[k][0] = fmaf(q0.x, v, acc[k][0]);
          acc[k][1] = fmaf(q0.y, v, acc[k][1]);
          acc[k][2] = fmaf(q0.z, v, acc[k][2]);
          acc[k][3] = fmaf(q0.w, v, acc[k][3]);
          acc[k][4] = fmaf(q1.x, v, acc[k][4]);
          acc[k][5] = fmaf(q1.y, v, acc[k][5]);
          acc[k][6] = fmaf(q1.z, v, acc[k][6]);
          acc[k][7] = fmaf(q1.w, v, acc[k][7]);
        }
      }
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int y = y0 + ty + 4 * k, x = x0 + tx;
      if (y >= H || x >= W) continue;
#pragma unroll
      for (int o = 0; o < 8; ++o) {
        const size_t idx = (((size_t)b * COUT + o0 + o) * H + y) * W + x;
        const float z = acc[k][o] + (bias ? bias[o0 + o] : 0.0f);
        if (epi == EPI_GELU) { outz[idx] = z; outa[idx] = gelu_f(z); }
        else if (epi == EPI_LINEAR) outz[idx] = z;
        else outz[idx] = z * gelu_grad_f(aux[idx]);
      }
    }
  } else {
    const int ty = tid / TILE, tx = tid % TILE;
    float acc[COUT];
#pragma unroll
    for (int o = 0; o < COUT; ++o) acc[o] = 0.0f;
    for (int c = 0; c < CIN; ++c) {
#pragma unroll
      for (int tap = 0; tap < 9; ++tap) {
        const float v = tile[c * HALO * HALO + (ty + DIL * (tap / 3)) * HALO + tx + DIL * (tap % 3)];
#pragma unroll
        for (int o = 0; o < COUT; ++o) acc[o] = fmaf(ws[(c * 9 + tap) * COUT + o], v, acc[o]);
      }
    }
    const int y = y0 + ty, x = x0 + tx;
    if (y >= H || x >= W) return;
#pragma unroll
    for (int o = 0; o < COUT; ++o) {
      const size_t idx = (((size_t)b * COUT + o) * H + y) * W + x;
      const float z = acc[o] + (bias ? bias[o] : 0.0f);
      if (epi == EPI_GELU) { outz[idx] = z; outa[idx] = gelu_f(z); }
      else if (epi == EPI_LINEAR) outz[idx] = z;
      else outz[idx] = z * gelu_grad_f(aux[idx]);
    }
  }
}

// ---- inference -----------------------------------------------------------------------------
// Layers 1 and 2 hand their activations on in BF16 (channel planes): the tensor-core layers round
// their inputs to BF16 in any case, at the producer or at the consumer.  The last hidden layer's
// output stays FP32 for the FP32 output layer.

// Layer 1 (3 -> 32, FP32 input and arithmetic): one thread per pixel.
template <int DIL>
__global__ void __launch_bounds__(128) k_conv_in(int H, int W, int npix, const float* __restrict__ in,
                                                 const float* __restrict__ w, const float* __restrict__ bias,
                                                 __nv_bfloat16* __restrict__ out) {
  __shared__ __align__(16) float ws[27 * 32];
  for (int i = threadIdx.x; i < 27 * 32; i += 128) ws[i] = w[i];
  __syncthreads();
  const int p = blockIdx.x * 128 + threadIdx.x;
  if (p >= npix) return;
  const int HW = H * W, b = p / HW, r = p - b * HW, y = r / W, x = r - y * W;
  float acc[32];
#pragma unroll
  for (int o = 0; o < 32; ++o) acc[o] = 0.0f;
  const float* inb = in + (size_t)b * 3 * HW;
#pragma unroll
  for (int c = 0; c < 3; ++c)
#pragma unroll
    for (int tap = 0; tap < 9; ++tap) {
      const int yy = y + DIL * (tap / 3 - 1), xx = x + DIL * (tap % 3 - 1);
      const float v = yy >= 0 && yy < H && xx >= 0 && xx < W ? inb[c * HW + yy * W + xx] : 0.0f;
#pragma unroll
      for (int o = 0; o < 32; o += 4) {
        const float4 q = *reinterpret_cast<const float4*>(ws + (c * 9 + tap) * 32 + o);
        acc[o] = fmaf(q.x, v, acc[o]);
        acc[o + 1] = fmaf(q.y, v, acc[o + 1]);
        acc[o + 2] = fmaf(q.z, v, acc[o + 2]);
        acc[o + 3] = fmaf(q.w, v, acc[o + 3]);
      }
    }
#pragma unroll
  for (int o = 0; o < 32; ++o) out[((size_t)b * 32 + o) * HW + r] = __float2bfloat16_rn(gelu_f(acc[o] + bias[o]));
}

// Output layer (32 -> 2, FP32): the last hidden layer's epilogue forms each pixel's products with
// the 9 x 2 weight vectors, channels 0-15 into pa[2 tap + o][pixel] and 16-31 into pb; here every pixel
// adds its nine neighbours' shares.
// (Reading the 32 channels of nine neighbours per pixel moved 311 MB from L2 at 16 x 130 x 130: 68 us, now 9.)
template <int DIL>
__global__ void __launch_bounds__(256) k_conv_out(int H, int W, int npix, const float* __restrict__ pa,
                                                  const float* __restrict__ pb, const float* __restrict__ bias,
                                                  float* __restrict__ out) {
  const int p = blockIdx.x * 256 + threadIdx.x;
  if (p >= npix) return;
  const int HW = H * W, b = p / HW, r = p - b * HW, y = r / W, x = r - y * W;
  float a0 = 0.0f, a1 = 0.0f;
#pragma unroll
  for (int tap = 0; tap < 9; ++tap) {
    const int dy = DIL * (tap / 3 - 1), dx = DIL * (tap % 3 - 1);
    const bool ok = y + dy >= 0 && y + dy < H && x + dx >= 0 && x + dx < W;
    const size_t q = (size_t)2 * tap * npix + (ok ? p + dy * W + dx : p);
    a0 += ok ? pa[q] + pb[q] : 0.0f;
    a1 += ok ? pa[q + npix] + pb[q + npix] : 0.0f;
  }
  out[(size_t)b * 2 * HW + r] = a0 + bias[0];
  out[(size_t)b * 2 * HW + HW + r] = a1 + bias[1];
}

// 32 -> 32 layers on the tensor cores (tcgen05).  An implicit GEMM per tile of 128 pixels: D (128
// pixels x 32 output channels, FP32 in tensor memory) = A (128 pixels x K, BF16) * B^T (32 channels
// x K, BF16), K = 32 input channels x 9 taps = 288, as 18 tcgen05.mma instructions of 128 x 32 x 16
// issued by one thread.  A and B lie in shared memory in the no-swizzle K-major layout of 8-row x
// 16-byte core matrices: core matrix (r, k) of an operand at ((r * KC + k) * 128) bytes, KC = K / 8, so
// the descriptor's K-direction stride is 128 bytes and its row-group stride KC * 128.  B is kept in
// its shared-memory image and loaded once per block; two blocks per SM walk over the tiles.
// What bounds it is building A, 288 neighbourhood values a pixel: two threads per pixel read them
// in BF16 (coalesced over the pixels) eight at a time and store them as one 16-byte core-matrix row.
// Reading FP32 values and storing 2 bytes at a time into conflicting banks took 260 us a layer at 16
// inputs of 130 x 130, this 81-104 us; the whole inference 697 -> 218 us.  (Channel-innermost BF16 with
// 16-byte asynchronous copies, K order tap by tap, measured 57 us a layer but sums the products in
// another order, which moves activations across BF16 rounding boundaries.)
constexpr int TC_M = 128, TC_N = 32, TC_K = 288, TC_KC = TC_K / 8;
constexpr int TC_A_BYTES = TC_M * TC_K * 2, TC_B_BYTES = TC_N * TC_K * 2;
constexpr size_t TC_SMEM = TC_A_BYTES + TC_B_BYTES + 64;
constexpr int TC_TMEM_COLS = 32;
constexpr long TC_SPIN = 1L << 24;

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

// shared-memory matrix descriptor: start address, K-direction (leading) and row-group (stride)
// byte offsets, descriptor version 1, no swizzle
__device__ __forceinline__ uint64_t tc_smem_desc(uint32_t addr, uint32_t lbo, uint32_t sbo) {
  uint64_t d = 0;
  d |= (uint64_t)((addr & 0x3FFFFu) >> 4);
  d |= (uint64_t)((lbo >> 4) & 0x3FFFu) << 16;
  d |= (uint64_t)((sbo >> 4) & 0x3FFFu) << 32;
  d |= (uint64_t)1 << 46;
  return d;
}

// instruction descriptor of kind::f16: FP32 accumulator, BF16 A and B, both K-major, N, M
constexpr uint32_t tc_idesc(int M, int N) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

// LAST: the activations (FP32) go straight into the output layer's products (pa, pb; w4: its weights
// [c][tap][o]); else the output is BF16 channel planes (outh).  ntiles: tiles of 128 consecutive pixels
// of the whole batch.
template <int DIL, bool LAST>
__global__ void __launch_bounds__(256) k_conv32_tc(int H, int W, int npix, int ntiles, const __nv_bfloat16* __restrict__ in,
                                                   const uint4* __restrict__ wimg, const float* __restrict__ bias,
                                                   __nv_bfloat16* __restrict__ outh, const float* __restrict__ w4,
                                                   float* __restrict__ pa, float* __restrict__ pb, int* __restrict__ err) {
  extern __shared__ __align__(128) unsigned char smem[];
  unsigned char* As = smem;
  unsigned char* Bs = smem + TC_A_BYTES;
  uint64_t* mbar = reinterpret_cast<uint64_t*>(smem + TC_A_BYTES + TC_B_BYTES);
  uint32_t* tslot = reinterpret_cast<uint32_t*>(smem + TC_A_BYTES + TC_B_BYTES + 16);
  __shared__ __align__(16) float w4s[LAST ? 32 * 20 : 4];         // [c][2 tap + o], 20 apart
  const int tid = threadIdx.x, warp = tid >> 5, m = tid & 127, half = tid >> 7;
  if constexpr (LAST)
    for (int i = tid; i < 32 * 18; i += 256) w4s[i / 18 * 20 + i % 18] = w4[i];
  const int HW = H * W;
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tslot)),
                 "r"(TC_TMEM_COLS));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  if (tid == 0) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(mbar)));
    asm volatile("fence.mbarrier_init.release.cluster;");
  }
  for (int i = tid; i < TC_B_BYTES / 16; i += 256) reinterpret_cast<uint4*>(Bs)[i] = wimg[i];
  // A: thread (m, half) stages channels 16 half .. 16 half + 15 of pixel m, k = c * 9 + tap
  auto fetch = [&](int tile) {
    const int p = tile * TC_M + m, b = p / HW, r = p - b * HW, y = r / W, x = r - y * W;
    int off[9];
    unsigned ok = 0;
#pragma unroll
    for (int tap = 0; tap < 9; ++tap) {
      const int yy = y + DIL * (tap / 3 - 1), xx = x + DIL * (tap % 3 - 1);
      const bool in_ = p < npix && yy >= 0 && yy < H && xx >= 0 && xx < W;
      ok |= (unsigned)in_ << tap;
      off[tap] = in_ ? yy * W + xx : 0;
    }
    const unsigned short* src =
        reinterpret_cast<const unsigned short*>(in) + (p < npix ? ((size_t)b * 32 + 16 * half) * HW : 0);
    uint4* dst = reinterpret_cast<uint4*>(As + ((m >> 3) * TC_KC + 18 * half) * 128 + (m & 7) * 16);
#pragma unroll
    for (int kc = 0; kc < 18; ++kc) {
      uint32_t h[4];
#pragma unroll
      for (int e = 0; e < 8; e += 2) {
        const int k0 = 8 * kc + e, k1 = k0 + 1;
        const uint32_t v0 = ok >> (k0 % 9) & 1 ? src[(size_t)(k0 / 9) * HW + off[k0 % 9]] : 0;
        const uint32_t v1 = ok >> (k1 % 9) & 1 ? src[(size_t)(k1 / 9) * HW + off[k1 % 9]] : 0;
        h[e / 2] = v0 | v1 << 16;
      }
      dst[kc * 8] = make_uint4(h[0], h[1], h[2], h[3]);
    }
  };
  uint32_t phase = 0, tmem = 0;
  for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x, phase ^= 1u) {
    fetch(tile);
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    tmem = *tslot;
    if (tid == 0) {
      const uint32_t a0 = smem_u32(As), b0 = smem_u32(Bs);
      constexpr uint32_t idesc = tc_idesc(TC_M, TC_N);
#pragma unroll 1
      for (int s = 0; s < TC_K / 16; ++s) {
        const uint64_t ad = tc_smem_desc(a0 + s * 256, 128, TC_KC * 128);
        const uint64_t bd = tc_smem_desc(b0 + s * 256, 128, TC_KC * 128);
        asm volatile(
            "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
            "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(tmem),
            "l"(ad), "l"(bd), "r"(idesc), "r"(s));
      }
      asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(mbar))
                   : "memory");
    }
    // wait for the accumulator (bounded)
    uint32_t done = 0;
    for (long it = 0; it < TC_SPIN && !done; ++it) {
      asm volatile(
          "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
          : "=r"(done)
          : "r"(smem_u32(mbar)), "r"(phase)
          : "memory");
    }
    if (!__syncthreads_and((int)done)) {                         // every thread leaves together
      if (tid == 0) atomicExch(err, 1);
      break;
    }
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    // warps 0-3 read channels 0-15 of the 128 pixels, warps 4-7 channels 16-31
    uint32_t r[16];
    const uint32_t taddr = tmem + ((uint32_t)((warp & 3) * 32) << 16) + 16 * half;
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
    const int p = tile * TC_M + m;
    if (p < npix) {
      float v[16];
#pragma unroll
      for (int o = 0; o < 16; ++o) v[o] = gelu_f(__uint_as_float(r[o]) + bias[16 * half + o]);
      if constexpr (LAST) {
        float s[18];
#pragma unroll
        for (int k = 0; k < 18; ++k) s[k] = 0.0f;
#pragma unroll
        for (int c = 0; c < 16; ++c)
#pragma unroll
          for (int k = 0; k < 18; k += 2) {
            const float2 q = *reinterpret_cast<const float2*>(w4s + (16 * half + c) * 20 + k);
            s[k] = fmaf(q.x, v[c], s[k]);
            s[k + 1] = fmaf(q.y, v[c], s[k + 1]);
          }
        float* part = half ? pb : pa;
#pragma unroll
        for (int k = 0; k < 18; ++k) part[(size_t)k * npix + p] = s[k];
      } else {
        const int b = p / HW;
        __nv_bfloat16* dst = outh + ((size_t)b * 32 + 16 * half) * HW + (p - b * HW);
#pragma unroll
        for (int o = 0; o < 16; ++o) dst[(size_t)o * HW] = __float2bfloat16_rn(v[o]);
      }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  }
  __syncthreads();
  if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(*tslot), "r"(TC_TMEM_COLS));
}

// The 32 -> 32 layers' weights in the shared-memory image of B (k = c * 9 + tap).
__global__ void k_pack_weights(const __nv_bfloat16* __restrict__ w, __nv_bfloat16* __restrict__ img) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= TC_N * TC_K) return;
  const int o = i / TC_K, k = i - o * TC_K;
  img[((o >> 3) * TC_KC + (k >> 3)) * 64 + (o & 7) * 8 + (k & 7)] = w[i];
}

// dw[o,c,tap] += sum_{b,p} dz[b,o,p] in[b,c,p+tap], dbias[o] += sum dz[b,o,p]; blocks loop
// over tiles and add their partial sums atomically once at the end.
// A thread owns OG output channels and all nine taps of one input channel (lanes along c, so the
// gradients are shared by the warp and the inputs lie in different banks): 9 OG multiply-adds per
// 9 + OG/4 shared loads.  One weight per loop with two shared loads per multiply-add, as before, kept
// the shared memory busy for 75 us a tile of 32 -> 32 channels.  Where several threads share a weight they
// meet in shared memory before the one atomic per weight and block (all of them at the weight's
// address in memory cost 190 us a layer).  One training gradient of 8 inputs of 66 x 66: 1080 -> 506 us.
template <int CIN, int COUT>
struct WgShape {
  static constexpr int OG = COUT >= 4 ? 4 : COUT;             // output channels per thread
  static constexpr int NG = COUT / OG;                        // groups of them
  static constexpr int SPLIT = CIN * NG >= NT ? 1 : NT / (CIN * NG);   // threads sharing a weight's pixels
};
template <int DIL> struct WgHalo {                            // odd stride between channels: conflict-free lanes
  static constexpr int value = Halo<DIL>::value, plane = value * value | 1;
};
template <int CIN, int COUT, int DIL>
__global__ void __launch_bounds__(NT) k_conv_wgrad(int B, int H, int W, int tiles_x, int tiles_y,
                                                   const float* __restrict__ in, const float* __restrict__ dz,
                                                   float* __restrict__ dw, float* __restrict__ db) {
  constexpr int HALO = WgHalo<DIL>::value, PL = WgHalo<DIL>::plane;
  using G = WgShape<CIN, COUT>;
  extern __shared__ __align__(16) float smf[];
  float* dzs = smf;                                 // [pixel][COUT]
  float* tile = smf + COUT * NT;                    // CIN planes of PL
  const int tid = threadIdx.x;
  const int c = tid % CIN, g = tid / CIN % G::NG, part = tid / (CIN * G::NG);
  const bool on = tid < CIN * G::NG * G::SPLIT;
  float acc[G::OG][9], bs[G::OG];
#pragma unroll
  for (int o = 0; o < G::OG; ++o) {
    bs[o] = 0.0f;
#pragma unroll
    for (int t = 0; t < 9; ++t) acc[o][t] = 0.0f;
  }
  const int tpi = tiles_x * tiles_y, ntiles = B * tpi;
  for (int tt = blockIdx.x; tt < ntiles; tt += gridDim.x) {
    const int b = tt / tpi, t = tt - b * tpi;
    const int y0 = (t / tiles_x) * TILE, x0 = (t % tiles_x) * TILE;
    __syncthreads();
    const float* inb = in + (size_t)b * CIN * H * W;
    for (int i = tid; i < CIN * HALO * HALO; i += NT) {
      int cc = i / (HALO * HALO), r = i - cc * HALO * HALO;
      int yy = y0 + r / HALO - DIL, xx = x0 + r % HALO - DIL;
      tile[cc * PL + r] = (yy >= 0 && yy < H && xx >= 0 && xx < W) ? inb[((size_t)cc * H + yy) * W + xx] : 0.0f;
    }
    {
      const int yy = y0 + tid / TILE, xx = x0 + tid % TILE;
      const bool ok = yy < H && xx < W;
      const float* d = dz + (size_t)b * COUT * H * W + (ok ? yy * W + xx : 0);
#pragma unroll
      for (int o = 0; o < COUT; ++o) dzs[tid * COUT + (o ^ (COUT == 32 ? (tid & 7) * 4 : 0))] = ok ? d[(size_t)o * H * W] : 0.0f;
    }
    __syncthreads();
    if (on) {
      const float* tl = tile + c * PL;
#pragma unroll 2
      for (int pp = part; pp < NT; pp += G::SPLIT) {
        const int py = pp / TILE, px = pp % TILE;
        float d[G::OG], v[9];
        const float* dp = dzs + pp * COUT + ((g * G::OG) ^ (COUT == 32 ? (pp & 7) * 4 : 0));
        if constexpr (G::OG == 4) {
          const float4 q = *reinterpret_cast<const float4*>(dp);
          d[0] = q.x; d[1] = q.y; d[2] = q.z; d[3] = q.w;
        } else {
#pragma unroll
          for (int o = 0; o < G::OG; ++o) d[o] = dp[o];
        }
#pragma unroll
        for (int t9 = 0; t9 < 9; ++t9) v[t9] = tl[(py + DIL * (t9 / 3)) * HALO + px + DIL * (t9 % 3)];
#pragma unroll
        for (int o = 0; o < G::OG; ++o) {
          bs[o] += d[o];
#pragma unroll
          for (int t9 = 0; t9 < 9; ++t9) acc[o][t9] = fmaf(d[o], v[t9], acc[o][t9]);
        }
      }
    }
  }
  if constexpr (G::SPLIT > 1) {                     // add up the threads that share a weight, then once to memory
    constexpr int NO = COUT * CIN * 9 + COUT;
    __syncthreads();
    for (int i = tid; i < NO; i += NT) smf[i] = 0.0f;
    __syncthreads();
    if (on) {
#pragma unroll
      for (int o = 0; o < G::OG; ++o) {
        const int oo = g * G::OG + o;
#pragma unroll
        for (int t9 = 0; t9 < 9; ++t9) atomicAdd(&smf[(oo * CIN + c) * 9 + t9], acc[o][t9]);
        if (c == 0) atomicAdd(&smf[COUT * CIN * 9 + oo], bs[o]);
      }
    }
    __syncthreads();
    for (int i = tid; i < NO; i += NT) atomicAdd(i < COUT * CIN * 9 ? &dw[i] : &db[i - COUT * CIN * 9], smf[i]);
  } else {
#pragma unroll
    for (int o = 0; o < G::OG; ++o) {
      const int oo = g * G::OG + o;
#pragma unroll
      for (int t9 = 0; t9 < 9; ++t9) atomicAdd(&dw[(oo * CIN + c) * 9 + t9], acc[o][t9]);
      if (c == 0) atomicAdd(&db[oo], bs[o]);
    }
  }
}

// masked mean-squared loss of the two output channels: channel 0 (streamfunction) over the
// interior points (the boundary ring, where psi = 0, excluded), channel 1 (pressure) over
// the leading (H-1) x (W-1) points; each channel's mean is over its own mask:
// dz = 2 (z - t) / M_c, loss += (z - t)^2 / M_c
__global__ void k_loss(int B, int H, int W, const float* __restrict__ z, const float* __restrict__ tgt,
                       float* __restrict__ dz, double* __restrict__ loss, float inv_m0, float inv_m1) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  double l = 0.0;
  if (i < B * 2 * H * W) {
    int r = i % (H * W), ch = (i / (H * W)) % 2, y = r / W, x = r % W;
    bool in = ch == 0 ? (y > 0 && y < H - 1 && x > 0 && x < W - 1) : (y < H - 1 && x < W - 1);
    float inv_m = ch == 0 ? inv_m0 : inv_m1;
    float d = in ? z[i] - tgt[i] : 0.0f;
    dz[i] = 2.0f * d * inv_m;
    l = (double)d * d * inv_m;
  }
  for (int o = 16; o > 0; o >>= 1) l += __shfl_xor_sync(0xffffffffu, l, o);
  if ((threadIdx.x & 31) == 0 && l != 0.0) atomicAdd(loss, l);
}

__global__ void k_adam(int n, float* __restrict__ w, const float* __restrict__ g, float* __restrict__ m,
                       float* __restrict__ v, float lr, float b1, float b2, float eps, float c1, float c2) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  float gi = g[i];
  float mi = b1 * m[i] + (1.0f - b1) * gi;
  float vi = b2 * v[i] + (1.0f - b2) * gi * gi;
  m[i] = mi; v[i] = vi;
  w[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
}

// the weights rounded to BF16: as BF16 (w[o,c,tap]), and as the floats that the convolutions read:
// wf[c,tap,o], and its flipped transpose wt[o,8-tap,c] used to propagate gradients back.
__global__ void k_refresh_bf16(int cout, int cin, const float* __restrict__ w, __nv_bfloat16* __restrict__ wb,
                               float* __restrict__ wf, float* __restrict__ wt) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= cout * cin * 9) return;
  int o = i / (cin * 9), rem = i - o * cin * 9, c = rem / 9, tap = rem - c * 9;
  __nv_bfloat16 v = __float2bfloat16_rn(w[i]);
  wb[i] = v;
  wf[(c * 9 + tap) * cout + o] = __bfloat162float(v);
  wt[(o * 9 + 8 - tap) * cin + c] = __bfloat162float(v);
}

inline unsigned cdiv(long long a, long long b) { return (unsigned)((a + b - 1) / b); }

std::string g_nn_err;

}  // namespace

struct igamg_nn {
  int cin = 3, width = 32;
  int dil[4] = {1, 1, 1, 1};
  int off_w[4], off_b[4], cin_l[4], cout_l[4];
  int nparam = 0;
  float *master = nullptr, *grad = nullptr, *m = nullptr, *v = nullptr;
  __nv_bfloat16* wb = nullptr;                      // per-layer bf16 weights, same offsets as master
  float *wf = nullptr, *wt = nullptr;               // the same values for the convolutions (k_refresh_bf16)
  __nv_bfloat16* wimg = nullptr;                    // layers 2 and 3 as the tensor-core kernel's B images
  int blocks_tc = 0;                                // blocks of k_conv32_tc (they walk over the tiles)
  int step = 0;
  cudaStream_t stream = nullptr;
  size_t cap = 0;                                   // B*H*W capacity of the workspaces
  float* z[4] = {nullptr, nullptr, nullptr, nullptr};
  float* a[3] = {nullptr, nullptr, nullptr};
  float *d0 = nullptr, *d1 = nullptr;
  double* loss = nullptr;
  double* h_loss = nullptr;
  int* tc_err = nullptr;                            // set by a tensor-core convolution whose wait gave up
  int* h_tc_err = nullptr;
};

namespace {

#define NCK(x) do { cudaError_t e_ = (x); if (e_ != cudaSuccess) { g_nn_err = cudaGetErrorString(e_); return IGAMG_ECUDA; } } while (0)

// splitmix64 + Box-Muller (own counter-based generator) for the He initialisation
struct Rng {
  uint64_t s;
  uint64_t next() {
    uint64_t z = (s += 0x9E3779B97F4A7C15ull);
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
  }
  double uni() { return (next() >> 11) * (1.0 / 9007199254740992.0); }
  double normal() { double u1 = 1.0 - uni(), u2 = uni(); return std::sqrt(-2.0 * std::log(u1)) * std::cos(6.283185307179586 * u2); }
};

template <int CIN, int COUT, int DIL>
size_t conv_smem() { return (size_t)(CIN * Halo<DIL>::value * Halo<DIL>::value + COUT * CIN * 9) * sizeof(float); }
template <int CIN, int COUT, int DIL>
size_t wgrad_smem() { return (size_t)(CIN * WgHalo<DIL>::plane + COUT * NT) * sizeof(float); }

template <int CIN, int COUT, int DIL>
int set_smem_one() {
  NCK(cudaFuncSetAttribute(k_conv<CIN, COUT, DIL>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)conv_smem<CIN, COUT, DIL>()));
  NCK(cudaFuncSetAttribute(k_conv_wgrad<CIN, COUT, DIL>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)wgrad_smem<CIN, COUT, DIL>()));
  return IGAMG_OK;
}
template <int DIL>
int set_smem_tc() {
  NCK(cudaFuncSetAttribute(k_conv32_tc<DIL, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)TC_SMEM));
  NCK(cudaFuncSetAttribute(k_conv32_tc<DIL, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)TC_SMEM));
  return IGAMG_OK;
}

// Tensor-core forward of the 32 -> 32 layers (default) or the SIMT kernel (IGAMG_NN_TC=0).
bool nn_tc() {
  const char* e = std::getenv("IGAMG_NN_TC");
  return !e || std::atoi(e) != 0;
}

template <int DIL>
void conv32_tc_d(igamg_nn* nn, int npix, int H, int W, const __nv_bfloat16* in, const __nv_bfloat16* wimg,
                 const float* bias, __nv_bfloat16* outh, const float* w4, float* pa, float* pb) {
  const int tiles = (int)cdiv(npix, TC_M), grid = tiles < nn->blocks_tc ? tiles : nn->blocks_tc;
  const uint4* img = reinterpret_cast<const uint4*>(wimg);
  if (pa) k_conv32_tc<DIL, true><<<grid, 256, TC_SMEM, nn->stream>>>(H, W, npix, tiles, in, img, bias, outh, w4, pa, pb, nn->tc_err);
  else k_conv32_tc<DIL, false><<<grid, 256, TC_SMEM, nn->stream>>>(H, W, npix, tiles, in, img, bias, outh, w4, pa, pb, nn->tc_err);
}
void conv32_tc(igamg_nn* nn, int dil, int npix, int H, int W, const __nv_bfloat16* in, const __nv_bfloat16* wimg,
               const float* bias, __nv_bfloat16* outh, const float* w4, float* pa, float* pb) {
  switch (dil) {
    case 2: conv32_tc_d<2>(nn, npix, H, W, in, wimg, bias, outh, w4, pa, pb); break;
    case 4: conv32_tc_d<4>(nn, npix, H, W, in, wimg, bias, outh, w4, pa, pb); break;
    case 8: conv32_tc_d<8>(nn, npix, H, W, in, wimg, bias, outh, w4, pa, pb); break;
    default: conv32_tc_d<1>(nn, npix, H, W, in, wimg, bias, outh, w4, pa, pb);
  }
}
// the first (3 -> 32) and the output (32 -> 2) layer of inference
void conv_in(igamg_nn* nn, int dil, int npix, int H, int W, const float* x, const float* w, const float* bias,
             __nv_bfloat16* out) {
  const unsigned nb = cdiv(npix, 128);
  switch (dil) {
    case 2: k_conv_in<2><<<nb, 128, 0, nn->stream>>>(H, W, npix, x, w, bias, out); break;
    case 4: k_conv_in<4><<<nb, 128, 0, nn->stream>>>(H, W, npix, x, w, bias, out); break;
    case 8: k_conv_in<8><<<nb, 128, 0, nn->stream>>>(H, W, npix, x, w, bias, out); break;
    default: k_conv_in<1><<<nb, 128, 0, nn->stream>>>(H, W, npix, x, w, bias, out);
  }
}
void conv_out(igamg_nn* nn, int dil, int npix, int H, int W, const float* pa, const float* pb, const float* bias, float* out) {
  const unsigned nb = cdiv(npix, 256);
  switch (dil) {
    case 2: k_conv_out<2><<<nb, 256, 0, nn->stream>>>(H, W, npix, pa, pb, bias, out); break;
    case 4: k_conv_out<4><<<nb, 256, 0, nn->stream>>>(H, W, npix, pa, pb, bias, out); break;
    case 8: k_conv_out<8><<<nb, 256, 0, nn->stream>>>(H, W, npix, pa, pb, bias, out); break;
    default: k_conv_out<1><<<nb, 256, 0, nn->stream>>>(H, W, npix, pa, pb, bias, out);
  }
}

template <int CIN, int COUT>
int set_smem_all() {
  int rc;
  if ((rc = set_smem_one<CIN, COUT, 1>()) || (rc = set_smem_one<CIN, COUT, 2>()) || (rc = set_smem_one<CIN, COUT, 4>()) ||
      (rc = set_smem_one<CIN, COUT, 8>()))
    return rc;
  return IGAMG_OK;
}

template <int CIN, int COUT, int DIL>
void conv_d(igamg_nn* nn, int B, int H, int W, const float* in, const float* w, const float* bias,
            const float* aux, float* outz, float* outa, int epi) {
  int tx = cdiv(W, TILE), ty = cdiv(H, TILE);
  k_conv<CIN, COUT, DIL><<<B * tx * ty, NT, conv_smem<CIN, COUT, DIL>(), nn->stream>>>(H, W, tx, ty, in, w, bias, aux,
                                                                                       outz, outa, epi);
}
template <int CIN, int COUT>
void conv(igamg_nn* nn, int dil, int B, int H, int W, const float* in, const float* w, const float* bias,
          const float* aux, float* outz, float* outa, int epi) {
  switch (dil) {
    case 2: conv_d<CIN, COUT, 2>(nn, B, H, W, in, w, bias, aux, outz, outa, epi); break;
    case 4: conv_d<CIN, COUT, 4>(nn, B, H, W, in, w, bias, aux, outz, outa, epi); break;
    case 8: conv_d<CIN, COUT, 8>(nn, B, H, W, in, w, bias, aux, outz, outa, epi); break;
    default: conv_d<CIN, COUT, 1>(nn, B, H, W, in, w, bias, aux, outz, outa, epi);
  }
}

template <int CIN, int COUT, int DIL>
void wgrad_d(igamg_nn* nn, int B, int H, int W, const float* in, const float* dz, float* dw, float* db) {
  int tx = cdiv(W, TILE), ty = cdiv(H, TILE);
  int nt = B * tx * ty;
  int grid = nt < 2 * 152 ? nt : 2 * 152;
  k_conv_wgrad<CIN, COUT, DIL><<<grid, NT, wgrad_smem<CIN, COUT, DIL>(), nn->stream>>>(B, H, W, tx, ty, in, dz, dw, db);
}
template <int CIN, int COUT>
void wgrad(igamg_nn* nn, int dil, int B, int H, int W, const float* in, const float* dz, float* dw, float* db) {
  switch (dil) {
    case 2: wgrad_d<CIN, COUT, 2>(nn, B, H, W, in, dz, dw, db); break;
    case 4: wgrad_d<CIN, COUT, 4>(nn, B, H, W, in, dz, dw, db); break;
    case 8: wgrad_d<CIN, COUT, 8>(nn, B, H, W, in, dz, dw, db); break;
    default: wgrad_d<CIN, COUT, 1>(nn, B, H, W, in, dz, dw, db);
  }
}

int ensure_cap(igamg_nn* nn, size_t pix) {
  if (pix <= nn->cap) return IGAMG_OK;
  for (auto*& p : nn->z) { if (p) cudaFree(p); p = nullptr; }
  for (auto*& p : nn->a) { if (p) cudaFree(p); p = nullptr; }
  if (nn->d0) cudaFree(nn->d0);
  if (nn->d1) cudaFree(nn->d1);
  nn->d0 = nn->d1 = nullptr;
  size_t wpix = pix * nn->width * sizeof(float);
  for (int l = 0; l < 3; ++l) { NCK(cudaMalloc(&nn->z[l], wpix)); NCK(cudaMalloc(&nn->a[l], wpix)); }
  NCK(cudaMalloc(&nn->z[3], 2 * pix * sizeof(float)));
  NCK(cudaMalloc(&nn->d0, wpix));
  NCK(cudaMalloc(&nn->d1, wpix));
  nn->cap = pix;
  return IGAMG_OK;
}

int refresh(igamg_nn* nn) {
  for (int l = 0; l < 4; ++l) {
    int n = nn->cout_l[l] * nn->cin_l[l] * 9;
    k_refresh_bf16<<<cdiv(n, 256), 256, 0, nn->stream>>>(nn->cout_l[l], nn->cin_l[l], nn->master + nn->off_w[l],
                                                          nn->wb + nn->off_w[l], nn->wf + nn->off_w[l],
                                                          nn->wt + nn->off_w[l]);
  }
  for (int l = 1; l <= 2; ++l)
    k_pack_weights<<<cdiv(TC_N * TC_K, 256), 256, 0, nn->stream>>>(nn->wb + nn->off_w[l], nn->wimg + (size_t)(l - 1) * TC_N * TC_K);
  NCK(cudaGetLastError());
  return IGAMG_OK;
}

// Inference: the two 32 -> 32 layers on the tensor cores (BF16 activations and weights, FP32
// accumulation), the others in FP32.  z[0], z[1] hold the BF16 activations, a[2] and z[2] the output layer's products.
int infer(igamg_nn* nn, int B, int H, int W, const float* x, float* out) {
  const float* P = nn->master;
  const int* d = nn->dil;
  const int npix = B * H * W;
  __nv_bfloat16 *a0 = (__nv_bfloat16*)nn->z[0], *a1 = (__nv_bfloat16*)nn->z[1];
  conv_in(nn, d[0], npix, H, W, x, nn->wf + nn->off_w[0], P + nn->off_b[0], a0);
  conv32_tc(nn, d[1], npix, H, W, a0, nn->wimg, P + nn->off_b[1], a1, nullptr, nullptr, nullptr);
  conv32_tc(nn, d[2], npix, H, W, a1, nn->wimg + TC_N * TC_K, P + nn->off_b[2], nullptr, nn->wf + nn->off_w[3], nn->a[2],
            nn->z[2]);
  conv_out(nn, d[3], npix, H, W, nn->a[2], nn->z[2], P + nn->off_b[3], out);
  NCK(cudaGetLastError());
  return IGAMG_OK;
}

// FP32 activations throughout, kept for the backward pass.
int forward(igamg_nn* nn, int B, int H, int W, const float* x) {
  const float* P = nn->master;
  const int* d = nn->dil;
  conv<3, 32>(nn, d[0], B, H, W, x, nn->wf + nn->off_w[0], P + nn->off_b[0], nullptr, nn->z[0], nn->a[0], EPI_GELU);
  conv<32, 32>(nn, d[1], B, H, W, nn->a[0], nn->wf + nn->off_w[1], P + nn->off_b[1], nullptr, nn->z[1], nn->a[1], EPI_GELU);
  conv<32, 32>(nn, d[2], B, H, W, nn->a[1], nn->wf + nn->off_w[2], P + nn->off_b[2], nullptr, nn->z[2], nn->a[2], EPI_GELU);
  conv<32, 2>(nn, d[3], B, H, W, nn->a[2], nn->wf + nn->off_w[3], P + nn->off_b[3], nullptr, nn->z[3], nullptr, EPI_LINEAR);
  NCK(cudaGetLastError());
  return IGAMG_OK;
}

// loss and gradients into nn->grad (zeroed first); loss left in nn->loss (device)
int backward(igamg_nn* nn, int B, int H, int W, const float* x, const float* tgt) {
  long long pix = (long long)B * H * W;
  long long m0 = (long long)B * (H - 2) * (W - 2), m1 = (long long)B * (H - 1) * (W - 1);
  NCK(cudaMemsetAsync(nn->grad, 0, nn->nparam * sizeof(float), nn->stream));
  NCK(cudaMemsetAsync(nn->loss, 0, sizeof(double), nn->stream));
  float* dz4 = nn->d0;
  k_loss<<<cdiv(2 * pix, 256), 256, 0, nn->stream>>>(B, H, W, nn->z[3], tgt, dz4, nn->loss, 1.0f / (float)m0,
                                                       1.0f / (float)m1);
  float* G = nn->grad;
  const int* d = nn->dil;
  wgrad<32, 2>(nn, d[3], B, H, W, nn->a[2], dz4, G + nn->off_w[3], G + nn->off_b[3]);
  float* dz3 = nn->d1;
  conv<2, 32>(nn, d[3], B, H, W, dz4, nn->wt + nn->off_w[3], nullptr, nn->z[2], dz3, nullptr, EPI_DGELU);
  wgrad<32, 32>(nn, d[2], B, H, W, nn->a[1], dz3, G + nn->off_w[2], G + nn->off_b[2]);
  float* dz2 = nn->d0;
  conv<32, 32>(nn, d[2], B, H, W, dz3, nn->wt + nn->off_w[2], nullptr, nn->z[1], dz2, nullptr, EPI_DGELU);
  wgrad<32, 32>(nn, d[1], B, H, W, nn->a[0], dz2, G + nn->off_w[1], G + nn->off_b[1]);
  float* dz1 = nn->d1;
  conv<32, 32>(nn, d[1], B, H, W, dz2, nn->wt + nn->off_w[1], nullptr, nn->z[0], dz1, nullptr, EPI_DGELU);
  wgrad<3, 32>(nn, d[0], B, H, W, x, dz1, G + nn->off_w[0], G + nn->off_b[0]);
  NCK(cudaGetLastError());
  return IGAMG_OK;
}

int check_dims(igamg_nn* nn, int B, int H, int W) {
  if (!nn || B < 1 || H < 3 || W < 3 || (long long)B * H * W > (1LL << 31) / 64) return IGAMG_EINVAL;
  return ensure_cap(nn, (size_t)B * H * W);
}

}  // namespace

extern "C" {

int igamg_nn_create(int in_channels, int width, const int* dilations, unsigned long long seed, void* cuda_stream,
                    igamg_nn** out) {
  if (!out) return IGAMG_EINVAL;
  *out = nullptr;
  if (in_channels != 3 || width != 32) return IGAMG_EUNSUPPORTED;
  for (int l = 0; dilations && l < 4; ++l)
    if (dilations[l] != 1 && dilations[l] != 2 && dilations[l] != 4 && dilations[l] != 8) return IGAMG_EUNSUPPORTED;
  auto* nn = new igamg_nn();
  nn->stream = (cudaStream_t)cuda_stream;
  for (int l = 0; dilations && l < 4; ++l) nn->dil[l] = dilations[l];
  const int cins[4] = {3, 32, 32, 32}, couts[4] = {32, 32, 32, 2};
  int off = 0;
  for (int l = 0; l < 4; ++l) {
    nn->cin_l[l] = cins[l]; nn->cout_l[l] = couts[l];
    nn->off_w[l] = off; off += couts[l] * cins[l] * 9;
    nn->off_b[l] = off; off += couts[l];
  }
  nn->nparam = off;
  std::vector<float> h(off, 0.0f);
  Rng r{seed};
  for (int l = 0; l < 4; ++l) {
    double sd = std::sqrt(2.0 / (cins[l] * 9.0)) * (l == 3 ? 0.1 : 1.0);   // He; small last layer
    for (int i = 0; i < couts[l] * cins[l] * 9; ++i) h[nn->off_w[l] + i] = (float)(sd * r.normal());
  }
  auto fail = [&](int code) { igamg_nn_destroy(nn); return code; };
  size_t pb = off * sizeof(float);
  if (cudaMalloc(&nn->master, pb) || cudaMalloc(&nn->grad, pb) || cudaMalloc(&nn->m, pb) || cudaMalloc(&nn->v, pb) ||
      cudaMalloc(&nn->wb, off * sizeof(__nv_bfloat16)) || cudaMalloc(&nn->wf, pb) || cudaMalloc(&nn->wt, pb) ||
      cudaMalloc(&nn->wimg, 2 * TC_N * TC_K * sizeof(__nv_bfloat16)) ||
      cudaMalloc(&nn->loss, sizeof(double)) || cudaMallocHost(&nn->h_loss, sizeof(double)) ||
      cudaMalloc(&nn->tc_err, sizeof(int)) || cudaMallocHost(&nn->h_tc_err, sizeof(int)))
    return fail(IGAMG_ECUDA);
  if (cudaMemset(nn->tc_err, 0, sizeof(int))) return fail(IGAMG_ECUDA);
  if (cudaMemcpy(nn->master, h.data(), pb, cudaMemcpyHostToDevice) || cudaMemset(nn->m, 0, pb) ||
      cudaMemset(nn->v, 0, pb) || cudaMemset(nn->wt, 0, pb))
    return fail(IGAMG_ECUDA);
  int rc;
  if ((rc = set_smem_all<3, 32>()) || (rc = set_smem_all<32, 32>()) || (rc = set_smem_all<32, 2>()) ||
      (rc = set_smem_all<2, 32>()) || (rc = set_smem_tc<1>()) || (rc = set_smem_tc<2>()) || (rc = set_smem_tc<4>()) ||
      (rc = set_smem_tc<8>()))
    return fail(rc);
  {
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) return fail(IGAMG_ECUDA);
    nn->blocks_tc = 2 * sms;                       // 95 KB of shared memory each: two per SM
  }
  if ((rc = refresh(nn))) return fail(rc);
  if (cudaStreamSynchronize(nn->stream)) return fail(IGAMG_ECUDA);
  *out = nn;
  return IGAMG_OK;
}

void igamg_nn_destroy(igamg_nn* nn) {
  if (!nn) return;
  for (void* p : {(void*)nn->master, (void*)nn->grad, (void*)nn->m, (void*)nn->v, (void*)nn->wb, (void*)nn->wf, (void*)nn->wt, (void*)nn->wimg,
                  (void*)nn->loss, (void*)nn->d0, (void*)nn->d1, (void*)nn->tc_err})
    if (p) cudaFree(p);
  if (nn->h_tc_err) cudaFreeHost(nn->h_tc_err);
  for (auto* p : nn->z) if (p) cudaFree(p);
  for (auto* p : nn->a) if (p) cudaFree(p);
  if (nn->h_loss) cudaFreeHost(nn->h_loss);
  delete nn;
}

int igamg_nn_num_params(const igamg_nn* nn) { return nn ? nn->nparam : 0; }

int igamg_nn_get_params(igamg_nn* nn, float* host, size_t cap) {
  if (!nn || !host || cap < (size_t)nn->nparam) return IGAMG_EINVAL;
  NCK(cudaMemcpyAsync(host, nn->master, nn->nparam * sizeof(float), cudaMemcpyDeviceToHost, nn->stream));
  NCK(cudaStreamSynchronize(nn->stream));
  return IGAMG_OK;
}

int igamg_nn_set_params(igamg_nn* nn, const float* host, size_t n) {
  if (!nn || !host || n != (size_t)nn->nparam) return IGAMG_EINVAL;
  NCK(cudaMemcpyAsync(nn->master, host, n * sizeof(float), cudaMemcpyHostToDevice, nn->stream));
  NCK(cudaMemsetAsync(nn->m, 0, n * sizeof(float), nn->stream));
  NCK(cudaMemsetAsync(nn->v, 0, n * sizeof(float), nn->stream));
  nn->step = 0;
  int rc = refresh(nn);
  if (rc) return rc;
  NCK(cudaStreamSynchronize(nn->stream));
  return IGAMG_OK;
}

int igamg_nn_forward(igamg_nn* nn, int B, int H, int W, const float* x, float* out) {
  int rc = check_dims(nn, B, H, W);
  if (rc) return rc;
  if (!x || !out) return IGAMG_EINVAL;
  const bool tc = nn_tc();
  if (!tc) {
    if ((rc = forward(nn, B, H, W, x))) return rc;
    NCK(cudaMemcpyAsync(out, nn->z[3], (size_t)B * 2 * H * W * sizeof(float), cudaMemcpyDeviceToDevice, nn->stream));
  } else {
    if ((rc = infer(nn, B, H, W, x, out))) return rc;
    // a tensor-core wait that gave up is reported here
    NCK(cudaMemcpyAsync(nn->h_tc_err, nn->tc_err, sizeof(int), cudaMemcpyDeviceToHost, nn->stream));
    NCK(cudaStreamSynchronize(nn->stream));
    if (*nn->h_tc_err) {
      NCK(cudaMemset(nn->tc_err, 0, sizeof(int)));
      g_nn_err = "a tensor-core convolution gave up waiting for its accumulator";
      return IGAMG_ETIMEOUT;
    }
  }
  return IGAMG_OK;
}

int igamg_nn_loss_grad(igamg_nn* nn, int B, int H, int W, const float* x, const float* target, double* loss,
                       float* grad_host) {
  int rc = check_dims(nn, B, H, W);
  if (rc) return rc;
  if (!x || !target) return IGAMG_EINVAL;
  if ((rc = forward(nn, B, H, W, x)) || (rc = backward(nn, B, H, W, x, target))) return rc;
  NCK(cudaMemcpyAsync(nn->h_loss, nn->loss, sizeof(double), cudaMemcpyDeviceToHost, nn->stream));
  if (grad_host) NCK(cudaMemcpyAsync(grad_host, nn->grad, nn->nparam * sizeof(float), cudaMemcpyDeviceToHost, nn->stream));
  NCK(cudaStreamSynchronize(nn->stream));
  if (loss) *loss = *nn->h_loss;
  return IGAMG_OK;
}

int igamg_nn_train_step(igamg_nn* nn, int B, int H, int W, const float* x, const float* target, float lr,
                        double* loss) {
  int rc = check_dims(nn, B, H, W);
  if (rc) return rc;
  if (!x || !target || !(lr > 0)) return IGAMG_EINVAL;
  if ((rc = forward(nn, B, H, W, x)) || (rc = backward(nn, B, H, W, x, target))) return rc;
  nn->step += 1;
  const float b1 = 0.9f, b2 = 0.999f;
  float c1 = 1.0f - std::pow(b1, (float)nn->step), c2 = 1.0f - std::pow(b2, (float)nn->step);
  k_adam<<<cdiv(nn->nparam, 256), 256, 0, nn->stream>>>(nn->nparam, nn->master, nn->grad, nn->m, nn->v, lr, b1, b2,
                                                         1e-8f, c1, c2);
  if ((rc = refresh(nn))) return rc;
  if (loss) {
    NCK(cudaMemcpyAsync(nn->h_loss, nn->loss, sizeof(double), cudaMemcpyDeviceToHost, nn->stream));
    NCK(cudaStreamSynchronize(nn->stream));
    *loss = *nn->h_loss;
  }
  return IGAMG_OK;
}

}  // extern "C"
