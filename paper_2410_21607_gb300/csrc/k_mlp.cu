// Learned refinement flags: per-element features, a 3-layer MLP (136-128-128-3)
// with bfloat16 tensor-core forward products and float32 accumulation, its
// backward pass and Adam.
//
// The paper's velocity criterion (Sec. 3.1) fires only once intensification
// has started (Sec. 5); the network predicts the criterion's flags some steps
// ahead from the current state, so that adaptation can run less often while
// the criterion stays the fallback.
//
// Precision contract (shared with the CPU oracle): inputs, weights and the two
// hidden activations enter their products rounded to bfloat16 (nearest even);
// products accumulate in float32; the backward pass is float32 on the same
// rounded values (the gradient of the loss with respect to the rounded
// weights); master weights and Adam moments are float32.
#include <algorithm>
#include <cstring>
#include <string>
#include <vector>
#include <cuda_bf16.h>

#include "sem_internal.h"
#include "tcgen05.cuh"

namespace sem {
namespace {

constexpr int IN = 136, HID = 128, OUT = 3;
constexpr int OFF_W1 = 0, OFF_B1 = OFF_W1 + IN * HID, OFF_W2 = OFF_B1 + HID;
constexpr int OFF_B2 = OFF_W2 + HID * HID, OFF_W3 = OFF_B2 + HID, OFF_B3 = OFF_W3 + HID * OUT;
constexpr int NPARAM = OFF_B3 + OUT;
// transposed bfloat16 weights for the tensor-core B operands, padded strides
// (in bfloat16 elements) that keep the fragment loads free of bank conflicts
constexpr int K1P = 152, K2P = 136;
constexpr int W1T_SZ = HID * K1P, W2T_SZ = HID * K2P, W3T_SZ = 8 * K2P;

__device__ __forceinline__ unsigned pack_bf16(float lo, float hi) {
  __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<unsigned*>(&v);
}
__device__ __forceinline__ float bf16r(float x) { return __bfloat162float(__float2bfloat16_rn(x)); }

__device__ __forceinline__ void mma_bf16(float (&d)[4], const unsigned (&a)[4], unsigned b0, unsigned b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
      "{%0,%1,%2,%3};\n"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// refresh the transposed bfloat16 weights and the rounded float32 copies
__global__ void mlp_refresh(const float* __restrict__ P, __nv_bfloat16* __restrict__ w1t,
                            __nv_bfloat16* __restrict__ w2t, __nv_bfloat16* __restrict__ w3t,
                            float* __restrict__ R) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < W1T_SZ + W2T_SZ + W3T_SZ;
       i += gridDim.x * blockDim.x) {
    float v = 0.f;
    if (i < W1T_SZ) {
      const int n = i / K1P, k = i % K1P;
      if (k < IN) v = P[OFF_W1 + k * HID + n];
      w1t[i] = __float2bfloat16_rn(v);
    } else if (i < W1T_SZ + W2T_SZ) {
      const int r = i - W1T_SZ, n = r / K2P, k = r % K2P;
      if (k < HID) v = P[OFF_W2 + k * HID + n];
      w2t[r] = __float2bfloat16_rn(v);
    } else {
      const int r = i - W1T_SZ - W2T_SZ, n = r / K2P, k = r % K2P;
      if (k < HID && n < OUT) v = P[OFF_W3 + k * OUT + n];
      w3t[r] = __float2bfloat16_rn(v);
    }
  }
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < NPARAM; i += gridDim.x * blockDim.x)
    R[i] = bf16r(P[i]);
}

// Forward pass.  One warp per 16 rows, 4 warps per CTA.  Writes the class
// probabilities, and in training mode the rounded activations.
constexpr int FWD_ROWS = 64;
constexpr size_t FWD_SMEM = (size_t)(W1T_SZ + W2T_SZ + W3T_SZ) * 2 + (2 * HID + 8) * 4;

__global__ void __launch_bounds__(128)
mlp_forward(const float* __restrict__ X, int n, const __nv_bfloat16* __restrict__ w1t,
            const __nv_bfloat16* __restrict__ w2t, const __nv_bfloat16* __restrict__ w3t,
            const float* __restrict__ P, float* __restrict__ prob, __nv_bfloat16* __restrict__ H1r,
            __nv_bfloat16* __restrict__ H2r, int8_t* __restrict__ flags) {
  extern __shared__ __align__(16) unsigned char sm[];
  __nv_bfloat16* s1 = reinterpret_cast<__nv_bfloat16*>(sm);
  __nv_bfloat16* s2 = s1 + W1T_SZ;
  __nv_bfloat16* s3 = s2 + W2T_SZ;
  float* sb = reinterpret_cast<float*>(s3 + W3T_SZ);   // b1 | b2 | b3
  {
    const uint4* src = reinterpret_cast<const uint4*>(w1t);
    uint4* dst = reinterpret_cast<uint4*>(s1);
    for (int i = threadIdx.x; i < (W1T_SZ + W2T_SZ + W3T_SZ) / 8; i += blockDim.x) dst[i] = src[i];
    for (int i = threadIdx.x; i < HID; i += blockDim.x) {
      sb[i] = P[OFF_B1 + i];
      sb[HID + i] = P[OFF_B2 + i];
    }
    if (threadIdx.x < 8) sb[2 * HID + threadIdx.x] = threadIdx.x < OUT ? P[OFF_B3 + threadIdx.x] : 0.f;
  }
  __syncthreads();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int gid = lane >> 2, tig = lane & 3;
  const int row0 = blockIdx.x * FWD_ROWS + warp * 16;
  const int ra = row0 + gid, rb = row0 + gid + 8;
  // A fragments of the input rows, 9 k-steps of 16 (136 padded to 144)
  unsigned a[9][4];
#pragma unroll
  for (int s = 0; s < 9; ++s) {
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int c = 16 * s + 8 * h + 2 * tig;
      float x0 = 0.f, x1 = 0.f, y0 = 0.f, y1 = 0.f;
      if (ra < n && c < IN) { x0 = X[(long long)ra * IN + c]; x1 = X[(long long)ra * IN + c + 1]; }
      if (rb < n && c < IN) { y0 = X[(long long)rb * IN + c]; y1 = X[(long long)rb * IN + c + 1]; }
      a[s][2 * h + 0] = pack_bf16(x0, x1);
      a[s][2 * h + 1] = pack_bf16(y0, y1);
    }
  }
  // layer 1: 16 column tiles of 8; results become layer 2's A fragments
  unsigned h1[8][4];
#pragma unroll
  for (int t = 0; t < 16; ++t) {
    float d[4] = {0.f, 0.f, 0.f, 0.f};
    const __nv_bfloat16* wb = s1 + (8 * t + gid) * K1P + 2 * tig;
#pragma unroll
    for (int s = 0; s < 9; ++s) {
      const unsigned b0 = *reinterpret_cast<const unsigned*>(wb + 16 * s);
      const unsigned b1 = *reinterpret_cast<const unsigned*>(wb + 16 * s + 8);
      mma_bf16(d, a[s], b0, b1);
    }
    const int c = 8 * t + 2 * tig;
    const float v0 = fmaxf(d[0] + sb[c], 0.f), v1 = fmaxf(d[1] + sb[c + 1], 0.f);
    const float v2 = fmaxf(d[2] + sb[c], 0.f), v3 = fmaxf(d[3] + sb[c + 1], 0.f);
    h1[t >> 1][(t & 1) * 2 + 0] = pack_bf16(v0, v1);
    h1[t >> 1][(t & 1) * 2 + 1] = pack_bf16(v2, v3);
    if (H1r) {
      if (ra < n) *reinterpret_cast<unsigned*>(H1r + (long long)ra * HID + c) = h1[t >> 1][(t & 1) * 2 + 0];
      if (rb < n) *reinterpret_cast<unsigned*>(H1r + (long long)rb * HID + c) = h1[t >> 1][(t & 1) * 2 + 1];
    }
  }
  // layer 2
  unsigned h2[8][4];
#pragma unroll
  for (int t = 0; t < 16; ++t) {
    float d[4] = {0.f, 0.f, 0.f, 0.f};
    const __nv_bfloat16* wb = s2 + (8 * t + gid) * K2P + 2 * tig;
#pragma unroll
    for (int s = 0; s < 8; ++s) {
      const unsigned b0 = *reinterpret_cast<const unsigned*>(wb + 16 * s);
      const unsigned b1 = *reinterpret_cast<const unsigned*>(wb + 16 * s + 8);
      mma_bf16(d, h1[s], b0, b1);
    }
    const int c = 8 * t + 2 * tig;
    const float v0 = fmaxf(d[0] + sb[HID + c], 0.f), v1 = fmaxf(d[1] + sb[HID + c + 1], 0.f);
    const float v2 = fmaxf(d[2] + sb[HID + c], 0.f), v3 = fmaxf(d[3] + sb[HID + c + 1], 0.f);
    h2[t >> 1][(t & 1) * 2 + 0] = pack_bf16(v0, v1);
    h2[t >> 1][(t & 1) * 2 + 1] = pack_bf16(v2, v3);
    if (H2r) {
      if (ra < n) *reinterpret_cast<unsigned*>(H2r + (long long)ra * HID + c) = h2[t >> 1][(t & 1) * 2 + 0];
      if (rb < n) *reinterpret_cast<unsigned*>(H2r + (long long)rb * HID + c) = h2[t >> 1][(t & 1) * 2 + 1];
    }
  }
  // layer 3: one column tile (3 of 8 used)
  float d[4] = {0.f, 0.f, 0.f, 0.f};
  {
    const __nv_bfloat16* wb = s3 + gid * K2P + 2 * tig;
#pragma unroll
    for (int s = 0; s < 8; ++s) {
      const unsigned b0 = *reinterpret_cast<const unsigned*>(wb + 16 * s);
      const unsigned b1 = *reinterpret_cast<const unsigned*>(wb + 16 * s + 8);
      mma_bf16(d, h2[s], b0, b1);
    }
  }
  // logits of rows ra (d0, d1 at columns 2 tig, 2 tig + 1) and rb (d2, d3);
  // columns 0..2 live in lanes tig = 0, 1 of each quad
  const float za0 = d[0] + sb[2 * HID + 2 * tig], za1 = d[1] + sb[2 * HID + 2 * tig + 1];
  const float zb0 = d[2] + sb[2 * HID + 2 * tig], zb1 = d[3] + sb[2 * HID + 2 * tig + 1];
  const int q0 = lane & ~3;
  const float a00 = __shfl_sync(0xffffffffu, za0, q0), a01 = __shfl_sync(0xffffffffu, za1, q0);
  const float a02 = __shfl_sync(0xffffffffu, za0, q0 + 1);
  const float b00 = __shfl_sync(0xffffffffu, zb0, q0), b01 = __shfl_sync(0xffffffffu, zb1, q0);
  const float b02 = __shfl_sync(0xffffffffu, zb0, q0 + 1);
  if (tig == 0) {
    const float zs[2][3] = {{a00, a01, a02}, {b00, b01, b02}};
    const int rows[2] = {ra, rb};
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      if (rows[h] >= n) continue;
      const float m = fmaxf(zs[h][0], fmaxf(zs[h][1], zs[h][2]));
      const float e0 = expf(zs[h][0] - m), e1 = expf(zs[h][1] - m), e2 = expf(zs[h][2] - m);
      const float inv = 1.f / (e0 + e1 + e2);
      if (prob) {
        prob[(long long)rows[h] * OUT + 0] = e0 * inv;
        prob[(long long)rows[h] * OUT + 1] = e1 * inv;
        prob[(long long)rows[h] * OUT + 2] = e2 * inv;
      }
      if (flags) {
        int cls = 0;
        if (zs[h][1] > zs[h][cls]) cls = 1;
        if (zs[h][2] > zs[h][cls]) cls = 2;
        flags[rows[h]] = (int8_t)(cls - 1);
      }
    }
  }
}

// Forward pass on the fifth-generation tensor cores (tcgen05), the
// default: persistent CTAs of 256 threads (two per SM) keep the weights in
// shared memory and walk over tiles of 128 rows, threads t and t + 128 owning
// the halves of row t of a tile (tensor memory lane t).  A thread asks for all
// of its share of a tile at once, and for the next tile's while this one is
// computed: the inputs (544 B a row) are what the pass cannot do without, and
// with 128 threads loading and rounding in turn their latency was most of its
// time (65536 rows: 54 us, now 28).  The three layers are GEMMs of M = 128 rows by N = 128 (16
// for the 3 logits) by K = 144 (the 136 inputs padded) or 128, as
// tcgen05.mma.cta_group::1.kind::f16 with bfloat16 operands from shared memory
// (K-major, no swizzle: core matrices of 8 rows x 8 bfloat16) and float32
// accumulators in tensor memory (256 columns: layer 1 at 0, layer 2 at 128,
// layer 3 at 0 again).  Each thread reads its row's accumulators back
// (tcgen05.ld), adds the bias, applies ReLU, rounds to bfloat16 and writes the
// next layer's A operand over the previous one (the MMAs that read it have
// completed).  Same precision contract as mlp_forward; waits on the MMA
// completion barrier are bounded, a wait that runs out leaves the outputs of
// the CTA unwritten and sets *err.
constexpr int TC_ROWS = 128;
constexpr int TC_X_BYTES = TC_ROWS * 144 * 2;                  // A operand (X, then H1, H2)
constexpr int TC_W1_BYTES = HID * 144 * 2, TC_W2_BYTES = HID * HID * 2, TC_W3_BYTES = 16 * HID * 2;
constexpr size_t TC_SMEM = (size_t)TC_X_BYTES + TC_W1_BYTES + TC_W2_BYTES + TC_W3_BYTES +
                           (2 * HID + 16) * sizeof(float) + 16;

// byte offset of element (row r, k) of a K-major bfloat16 operand with kc
// core matrices (8 bfloat16 each) along K
__device__ __forceinline__ int boff(int r, int k, int kc) {
  return (r & 7) * 16 + (k & 7) * 2 + (k >> 3) * 128 + (r >> 3) * (kc * 128);
}

constexpr int TC_T = 256, TC_XV = TC_ROWS * (IN / 4) / TC_T;   // threads; float4 of a tile per thread
static_assert(TC_T == 256 && TC_XV * TC_T == TC_ROWS * (IN / 4), "a tile divides evenly");
// The j-th float4 (row r, columns k..k+3) of a 128 x 136 tile for this thread
// of WARPS warps: half a warp takes 8 rows x 32 bytes, whose rounded values fill one
// core matrix (no bank conflicts; a row's worth of neighbouring lanes would
// fall on the same banks).
template <int WARPS>
__device__ __forceinline__ void input_at(int j, int& r, int& k) {
  const int lane = threadIdx.x & 31, unit = (j * WARPS + (int)(threadIdx.x >> 5)) * 2 + (lane >> 4);
  const int g = unit / (IN / 8), c = unit - g * (IN / 8);
  r = g * 8 + ((lane >> 1) & 7);
  k = c * 8 + (lane & 1) * 4;
}
__global__ void __launch_bounds__(TC_T, 2)
mlp_forward_tc(const float* __restrict__ X, int n, const __nv_bfloat16* __restrict__ w1t,
               const __nv_bfloat16* __restrict__ w2t, const __nv_bfloat16* __restrict__ w3t,
               const float* __restrict__ P, float* __restrict__ prob, __nv_bfloat16* __restrict__ H1r,
               __nv_bfloat16* __restrict__ H2r, int8_t* __restrict__ flags, int* err) {
  extern __shared__ __align__(1024) unsigned char sm_tc[];
  unsigned char* sA = sm_tc;
  unsigned char* sW1 = sA + TC_X_BYTES;
  unsigned char* sW2 = sW1 + TC_W1_BYTES;
  unsigned char* sW3 = sW2 + TC_W2_BYTES;
  float* sb = reinterpret_cast<float*>(sW3 + TC_W3_BYTES);   // b1 | b2 | b3 (16)
  uint64_t* mbar = reinterpret_cast<uint64_t*>(sb + 2 * HID + 16);
  uint32_t* taddr_s = reinterpret_cast<uint32_t*>(mbar + 1);
  const int t = threadIdx.x, warp = t >> 5, rl = t & 127, half = t >> 7;
  const int ntiles = (n + TC_ROWS - 1) / TC_ROWS;
  // inputs: float4 loads, 8 rows x 64 contiguous bytes per warp
  float4 xv[TC_XV];
  auto load = [&](int tile) {
    const long long row0 = (long long)tile * TC_ROWS;
#pragma unroll
    for (int j = 0; j < TC_XV; ++j) {
      int r, k;
      input_at<TC_T / 32>(j, r, k);
      xv[j] = row0 + r < n ? __ldg(reinterpret_cast<const float4*>(X + (row0 + r) * IN + k))
                           : make_float4(0.f, 0.f, 0.f, 0.f);
    }
  };
  load(blockIdx.x);
  // weights: 8 bfloat16 (16 bytes) per core-matrix row; the transposed
  // arrays hold row n of W^T with k contiguous (zero beyond the inputs)
#pragma unroll
  for (int i = t; i < HID * 18; i += TC_T) {
    const int nn = i / 18, c = i % 18;
    *reinterpret_cast<uint4*>(sW1 + boff(nn, 8 * c, 18)) = *reinterpret_cast<const uint4*>(w1t + nn * K1P + 8 * c);
  }
#pragma unroll
  for (int i = t; i < HID * 16; i += TC_T) {
    const int nn = i / 16, c = i % 16;
    *reinterpret_cast<uint4*>(sW2 + boff(nn, 8 * c, 16)) = *reinterpret_cast<const uint4*>(w2t + nn * K2P + 8 * c);
  }
  for (int i = t; i < 16 * 16; i += TC_T) {
    const int nn = i / 16, c = i % 16;
    const uint4 z = make_uint4(0u, 0u, 0u, 0u);
    *reinterpret_cast<uint4*>(sW3 + boff(nn, 8 * c, 16)) =
        nn < 8 ? *reinterpret_cast<const uint4*>(w3t + nn * K2P + 8 * c) : z;
  }
  for (int i = t; i < HID; i += TC_T) {
    sb[i] = P[OFF_B1 + i];
    sb[HID + i] = P[OFF_B2 + i];
  }
  if (t < 16) sb[2 * HID + t] = t < OUT ? P[OFF_B3 + t] : 0.f;
  if (warp == 0) tcg::alloc(taddr_s, 256);
  if (t == 0) tcg::mbar_init(tcg::smem_u32(mbar), 1);
  tcg::fence_before();
  __syncthreads();
  tcg::fence_after();
  const uint32_t taddr = *taddr_s, bar = tcg::smem_u32(mbar);
  const uint32_t aA = tcg::smem_u32(sA), a1 = tcg::smem_u32(sW1), a2 = tcg::smem_u32(sW2), a3 = tcg::smem_u32(sW3);
  const uint32_t lane_addr = taddr + ((uint32_t)(32 * (warp & 3)) << 16);
  bool ok = true;
  uint32_t phase = 0;   // completions of the barrier so far (three per tile)
  // persistent: the CTA keeps the weights and walks over tiles of 128 rows
  for (int tile = blockIdx.x; tile < ntiles && ok; tile += gridDim.x) {
  const long long row0 = (long long)tile * TC_ROWS;
#pragma unroll
  for (int j = 0; j < TC_XV; ++j) {
    int r, k;
    input_at<TC_T / 32>(j, r, k);
    *reinterpret_cast<uint2*>(sA + boff(r, k, 18)) =
        make_uint2(pack_bf16(xv[j].x, xv[j].y), pack_bf16(xv[j].z, xv[j].w));
  }
  if (half == 0) *reinterpret_cast<uint4*>(sA + boff(rl, IN, 18)) = make_uint4(0u, 0u, 0u, 0u);   // k = 136..143
  if (tile + (int)gridDim.x < ntiles) load(tile + gridDim.x);
  tcg::fence_async_smem();
  tcg::fence_before();
  __syncthreads();
  tcg::fence_after();
  const long long row = row0 + rl;
  // layer 1: 9 steps of K = 16 (two core matrices each)
  if (t == 0) {
    for (int ks = 0; ks < 9; ++ks)
      tcg::mma_f16(taddr, tcg::sdesc(aA + 256 * ks, 128, 18 * 128), tcg::sdesc(a1 + 256 * ks, 128, 18 * 128),
                   tcg::idesc_bf16(128, 128), ks > 0);
    tcg::commit(bar);
  }
  ok = __syncthreads_and(tcg::mbar_wait(bar, phase & 1));   // the same answer in every thread
  ++phase;
  tcg::fence_after();
  // hidden layers: bias, ReLU, bfloat16, written as the next A operand
  auto hidden = [&](uint32_t col0, const float* bias, __nv_bfloat16* Hr) {
#pragma unroll 1
    for (int c0 = 64 * half; c0 < 64 * half + 64; c0 += 16) {
      float v[16];
      tcg::ld16(lane_addr + col0 + c0, v);
      tcg::wait_ld();
#pragma unroll
      for (int q = 0; q < 16; ++q) v[q] = bf16r(fmaxf(v[q] + bias[c0 + q], 0.f));
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const uint4 w = make_uint4(pack_bf16(v[8 * h + 0], v[8 * h + 1]), pack_bf16(v[8 * h + 2], v[8 * h + 3]),
                                   pack_bf16(v[8 * h + 4], v[8 * h + 5]), pack_bf16(v[8 * h + 6], v[8 * h + 7]));
        *reinterpret_cast<uint4*>(sA + boff(rl, c0 + 8 * h, 16)) = w;
        if (Hr && row < n) *reinterpret_cast<uint4*>(Hr + row * HID + c0 + 8 * h) = w;
      }
    }
  };
  if (ok) hidden(0, sb, H1r);
  tcg::fence_async_smem();
  tcg::fence_before();
  __syncthreads();
  tcg::fence_after();
  if (ok && t == 0) {
    for (int ks = 0; ks < 8; ++ks)
      tcg::mma_f16(taddr + 128, tcg::sdesc(aA + 256 * ks, 128, 16 * 128), tcg::sdesc(a2 + 256 * ks, 128, 16 * 128),
                   tcg::idesc_bf16(128, 128), ks > 0);
    tcg::commit(bar);
  }
  ok = __syncthreads_and(ok && tcg::mbar_wait(bar, phase & 1));
  ++phase;
  tcg::fence_after();
  if (ok) hidden(128, sb + HID, H2r);
  tcg::fence_async_smem();
  tcg::fence_before();
  __syncthreads();
  tcg::fence_after();
  if (ok && t == 0) {
    for (int ks = 0; ks < 8; ++ks)
      tcg::mma_f16(taddr, tcg::sdesc(aA + 256 * ks, 128, 16 * 128), tcg::sdesc(a3 + 256 * ks, 128, 16 * 128),
                   tcg::idesc_bf16(128, 16), ks > 0);
    tcg::commit(bar);
  }
  ok = __syncthreads_and(ok && tcg::mbar_wait(bar, phase & 1));
  ++phase;
  tcg::fence_after();
  if (ok && half == 0) {
    float z[16];
    tcg::ld16(lane_addr, z);
    tcg::wait_ld();
    if (row < n) {
      const float z0 = z[0] + sb[2 * HID], z1 = z[1] + sb[2 * HID + 1], z2 = z[2] + sb[2 * HID + 2];
      const float m = fmaxf(z0, fmaxf(z1, z2));
      const float e0 = expf(z0 - m), e1 = expf(z1 - m), e2 = expf(z2 - m);
      const float inv = 1.f / (e0 + e1 + e2);
      if (prob) {
        prob[row * OUT + 0] = e0 * inv;
        prob[row * OUT + 1] = e1 * inv;
        prob[row * OUT + 2] = e2 * inv;
      }
      if (flags) {
        int cls = 0;
        if (z1 > z0) cls = 1;
        if (z2 > (cls == 1 ? z1 : z0)) cls = 2;
        flags[row] = (int8_t)(cls - 1);
      }
    }
  } else if (!ok && (t & 31) == 0) {
    atomicOr(err, 4);
  }
  // the next tile overwrites the A operand and the accumulators: every
  // thread has read its rows
  tcg::fence_before();
  __syncthreads();
  tcg::fence_after();
  }
  tcg::fence_before();
  __syncthreads();
  if (warp == 0) tcg::dealloc(taddr, 256);
}

// sum of the rows' class weights into acc[1]
__global__ void mlp_wsum(const int8_t* __restrict__ y, int n, float w0, float w1, float w2,
                         double* __restrict__ acc) {
  __shared__ double red[256];
  double s = 0.0;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const int c = y[i];
    s += c == 0 ? w0 : (c == 1 ? w1 : w2);
  }
  red[threadIdx.x] = s;
  __syncthreads();
  for (int o = 128; o > 0; o >>= 1) {
    if (threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) atomicAdd(acc + 1, red[0]);
}

// Backward pass, float32 on the CUDA cores:
//   dZ3 = w_y (p - onehot) / sum(w_y),  dZ2 = (dZ3 W3^T) [H2 > 0],
//   dZ1 = (dZ2 W2^T) [H1 > 0],  gW = (input of the layer)^T dZ,  gb = colsum dZ.
// Every sum runs over its terms in a fixed order of fused multiply-adds: a
// weight gradient over the rows of a split one after another, then over the
// splits in order (back_splits), so the results do not depend on how the work
// is laid out.  That matters beyond rounding: Adam divides a gradient by its own
// size, and a weight or activation that rounds to another bfloat16 moves every
// gradient of the next iteration by 1e-4.  (On the tensor cores, with the
// gradients as three bfloat16 parts, the pass took 68 us at no larger error, but
// not with these sums.)
//   back_rows: dZ3, dZ2 and dZ1 of 64 rows per CTA, W2^T in shared memory; a
//     thread owns 8 rows x 8 features.
//   back_grads: gW1 and gW2, a block of one of them for one split of the rows
//     per CTA.
//   back_tail: gW3 and the bias gradients.
// The products of two columns at a time are packed (fma.rn.f32x2), which halves
// the instructions the schedulers have to issue.  65536 rows: back_rows 80 us,
// back_grads 150, back_tail 73 (the float32 rate would allow 26 and 55 for the
// first two; they wait for loads and shared memory); as 32x32 tiles of 2x2
// products per thread with a pass over memory for each product, mask and bias
// sum it took 980 us.
__host__ __device__ inline int back_splits(int n, int& chunk) {
  int s = n / 512;
  s = s < 1 ? 1 : (s > 64 ? 64 : s);
  chunk = ((n + s - 1) / s + 31) / 32 * 32;
  return (n + chunk - 1) / chunk;
}
__device__ __forceinline__ float2 bf2(unsigned pair) {
  return make_float2(__uint_as_float(pair << 16), __uint_as_float(pair & 0xffff0000u));
}
// v where the bfloat16 activation is positive (neither zero nor NaN), else 0
__device__ __forceinline__ float masked(unsigned pair, int i, float v) {
  const unsigned b = (pair >> (16 * (i & 1))) & 0xffffu;
  return b - 1u < 0x7f80u ? v : 0.f;
}

constexpr int BR_ROWS = 64, BR_T = 128, BR_LD = HID + 4;
constexpr size_t BR_SMEM = sizeof(float) * (HID * BR_LD + HID * (BR_ROWS + 4) + HID * OUT + BR_ROWS * 4);
__global__ void __launch_bounds__(BR_T)
back_rows(const int8_t* __restrict__ y, int n, float w0, float w1, float w2, const float* __restrict__ prob,
          const __nv_bfloat16* __restrict__ H1, const __nv_bfloat16* __restrict__ H2,
          const __nv_bfloat16* __restrict__ w2t, const float* __restrict__ R, double* __restrict__ acc, int want_loss,
          float* __restrict__ dz3, float* __restrict__ dz2,
          float* __restrict__ dz1) {
  extern __shared__ __align__(16) float sb[];
  float* sW = sb;                              // [j][i] = W2[i][j]
  float* sA = sW + HID * BR_LD;                // [j][row] dZ2
  float* sW3 = sA + HID * (BR_ROWS + 4);       // [j][3]
  float* sD3 = sW3 + HID * OUT;                // [row][4]
  const int t = threadIdx.x;
  const long long row0 = (long long)blockIdx.x * BR_ROWS;
#pragma unroll
  for (int u = t; u < HID * HID / 8; u += BR_T) {
    const int j = u >> 4, i = 8 * (u & 15);
    const uint4 w = *reinterpret_cast<const uint4*>(w2t + j * K2P + i);
    const float2 a = bf2(w.x), b = bf2(w.y), c = bf2(w.z), d = bf2(w.w);
    *reinterpret_cast<float4*>(sW + j * BR_LD + i) = make_float4(a.x, a.y, b.x, b.y);
    *reinterpret_cast<float4*>(sW + j * BR_LD + i + 4) = make_float4(c.x, c.y, d.x, d.y);
  }
  for (int i = t; i < HID * OUT; i += BR_T) sW3[i] = R[OFF_W3 + i];
  const float inv = (float)(1.0 / acc[1]);
  double loss = 0.0;
  if (t < BR_ROWS) {
    float d[3] = {0.f, 0.f, 0.f};
    const long long row = row0 + t;
    if (row < n) {
      const int c = y[row];
      const float w = c == 0 ? w0 : (c == 1 ? w1 : w2);
#pragma unroll
      for (int k = 0; k < OUT; ++k) {
        d[k] = w * inv * (prob[row * OUT + k] - (k == c ? 1.f : 0.f));
        dz3[row * OUT + k] = d[k];
      }
      if (want_loss) loss = (double)w * -log((double)prob[row * OUT + c]);
    }
#pragma unroll
    for (int k = 0; k < OUT; ++k) sD3[t * 4 + k] = d[k];
    if (want_loss) {
      for (int o = 16; o > 0; o >>= 1) loss += __shfl_xor_sync(0xffffffffu, loss, o);
      if ((t & 31) == 0) atomicAdd(acc, loss);
    }
  }
  __syncthreads();
  // dZ2, 8 features of a row at a time
  for (int u = t; u < BR_ROWS * (HID / 8); u += BR_T) {
    const int r = u & (BR_ROWS - 1), k = 8 * (u / BR_ROWS);
    const long long row = row0 + r;
    uint4 h = make_uint4(0u, 0u, 0u, 0u);
    if (row < n) h = *reinterpret_cast<const uint4*>(H2 + row * HID + k);
    const unsigned hw[4] = {h.x, h.y, h.z, h.w};
    const float d0 = sD3[r * 4], d1 = sD3[r * 4 + 1], d2 = sD3[r * 4 + 2];
    float v[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const float* w = sW3 + (k + i) * OUT;
      v[i] = masked(hw[i >> 1], i, fmaf(d2, w[2], fmaf(d1, w[1], d0 * w[0])));
      sA[(k + i) * (BR_ROWS + 4) + r] = v[i];
    }
    if (row < n) {
      float4* o = reinterpret_cast<float4*>(dz2 + row * HID + k);
      o[0] = make_float4(v[0], v[1], v[2], v[3]);
      o[1] = make_float4(v[4], v[5], v[6], v[7]);
    }
  }
  __syncthreads();
  // dZ1: thread (rows 4 ty.. and 32 + 4 ty.., features 4 tx.. and 64 + 4 tx..),
  // terms in the order of the features of dZ2
  const int tx = t & 15, ty = t >> 4;
  float2 c[8][4];
#pragma unroll
  for (int a = 0; a < 8; ++a)
#pragma unroll
    for (int b = 0; b < 4; ++b) c[a][b] = make_float2(0.f, 0.f);
#pragma unroll 4
  for (int j = 0; j < HID; ++j) {
    const float4 x = *reinterpret_cast<const float4*>(sA + j * (BR_ROWS + 4) + 4 * ty);
    const float4 z = *reinterpret_cast<const float4*>(sA + j * (BR_ROWS + 4) + 32 + 4 * ty);
    const float4 p = *reinterpret_cast<const float4*>(sW + j * BR_LD + 4 * tx);
    const float4 q = *reinterpret_cast<const float4*>(sW + j * BR_LD + 64 + 4 * tx);
    const float xs[8] = {x.x, x.y, x.z, x.w, z.x, z.y, z.z, z.w};
    const float2 w[4] = {make_float2(p.x, p.y), make_float2(p.z, p.w), make_float2(q.x, q.y), make_float2(q.z, q.w)};
#pragma unroll
    for (int a = 0; a < 8; ++a)
#pragma unroll
      for (int b = 0; b < 4; ++b) c[a][b] = __ffma2_rn(make_float2(xs[a], xs[a]), w[b], c[a][b]);
  }
#pragma unroll
  for (int a = 0; a < 8; ++a) {
    const long long row = row0 + (a >> 2) * 32 + 4 * ty + (a & 3);
    if (row >= n) continue;
#pragma unroll
    for (int g = 0; g < 2; ++g) {
      const uint2 h = *reinterpret_cast<const uint2*>(H1 + row * HID + 64 * g + 4 * tx);
      *reinterpret_cast<float4*>(dz1 + row * HID + 64 * g + 4 * tx) =
          make_float4(masked(h.x, 0, c[a][2 * g].x), masked(h.x, 1, c[a][2 * g].y), masked(h.y, 0, c[a][2 * g + 1].x),
                      masked(h.y, 1, c[a][2 * g + 1].y));
    }
  }
}

// One 64 x 64 block of a weight gradient over one split of the rows: blockIdx.y
// selects gW1 (inputs x dZ1) or gW2 (H1 x dZ2) and the block of 2 x 2; gW1's
// blocks have 68 rows, the last four spread over all threads.  A thread owns
// 4 x 8 gradients; four warps per scheduler cover the loads of the next 32 rows
// (8 x 8 per thread, half the warps: 225 us against 144 us).
constexpr int BG_K = 32, BG_T = 128;
constexpr int PSTRIDE = (NPARAM + 3) / 4 * 4;   // a split's sums: 16-byte aligned rows
static_assert(OFF_W1 % 4 == 0 && OFF_W2 % 4 == 0, "weight blocks are stored 16 bytes at a time");
template <int WHICH>
__device__ __forceinline__ void grad_block(const float* __restrict__ X, const __nv_bfloat16* __restrict__ H1,
                                           const float* __restrict__ Z, int n, int chunk, int mb, int nb,
                                           float* __restrict__ part, float (*sA)[BG_K][72], float (*sB)[BG_K][64]) {
  constexpr int MT = WHICH == 0 ? 68 : 64, QA = MT / 4, NA = (BG_K * QA + BG_T - 1) / BG_T;
  const int t = threadIdx.x, tx = t & 7, ty = t >> 3, m0 = mb * MT;
  const long long k0 = (long long)blockIdx.x * chunk, k1 = min((long long)n, k0 + chunk);
  float4 ra[NA], rb[BG_K * 16 / BG_T];
  auto load = [&](long long kb) {
#pragma unroll
    for (int i = 0; i < NA; ++i) {
      const int u = t + i * BG_T, r = u / QA, m = 4 * (u - r * QA);
      ra[i] = make_float4(0.f, 0.f, 0.f, 0.f);
      if (u < BG_K * QA && kb + r < k1) {
        if (WHICH == 0) {
          const float* p = X + (kb + r) * IN + m0 + m;
          ra[i] = make_float4(bf16r(__ldg(p)), bf16r(__ldg(p + 1)), bf16r(__ldg(p + 2)), bf16r(__ldg(p + 3)));
        } else {
          const uint2 h = __ldg(reinterpret_cast<const uint2*>(H1 + (kb + r) * HID + m0 + m));
          const float2 lo = bf2(h.x), hi = bf2(h.y);
          ra[i] = make_float4(lo.x, lo.y, hi.x, hi.y);
        }
      }
    }
#pragma unroll
    for (int i = 0; i < BG_K * 16 / BG_T; ++i) {
      const int u = t + i * BG_T, r = u >> 4, c = 4 * (u & 15);
      rb[i] = make_float4(0.f, 0.f, 0.f, 0.f);
      if (kb + r < k1) rb[i] = __ldg(reinterpret_cast<const float4*>(Z + (kb + r) * HID + nb * 64 + c));
    }
  };
  auto store = [&](int buf) {
#pragma unroll
    for (int i = 0; i < NA; ++i) {
      const int u = t + i * BG_T, r = u / QA, m = 4 * (u - r * QA);
      if (u < BG_K * QA) *reinterpret_cast<float4*>(&sA[buf][r][m]) = ra[i];
    }
#pragma unroll
    for (int i = 0; i < BG_K * 16 / BG_T; ++i) {
      const int u = t + i * BG_T;
      *reinterpret_cast<float4*>(&sB[buf][u >> 4][4 * (u & 15)]) = rb[i];
    }
  };
  // rows 4 ty..; columns 4 tx.., 32 + 4 tx..; rows 64, 65 (66, 67 for t >= 64) of column t mod 64
  float2 c[4][4], e = make_float2(0.f, 0.f);
  const int et = t & 63, er = 64 + 2 * (t >> 6);
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int b = 0; b < 4; ++b) c[a][b] = make_float2(0.f, 0.f);
  load(k0);
  store(0);
  __syncthreads();
  int buf = 0;
  for (long long kb = k0; kb < k1; kb += BG_K, buf ^= 1) {
    const bool more = kb + BG_K < k1;
    if (more) load(kb + BG_K);
#pragma unroll 8
    for (int k = 0; k < BG_K; ++k) {
      const float4 x = *reinterpret_cast<const float4*>(&sA[buf][k][4 * ty]);
      const float4 p = *reinterpret_cast<const float4*>(&sB[buf][k][4 * tx]);
      const float4 q = *reinterpret_cast<const float4*>(&sB[buf][k][32 + 4 * tx]);
      const float xs[4] = {x.x, x.y, x.z, x.w};
      const float2 w[4] = {make_float2(p.x, p.y), make_float2(p.z, p.w), make_float2(q.x, q.y), make_float2(q.z, q.w)};
#pragma unroll
      for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) c[a][b] = __ffma2_rn(make_float2(xs[a], xs[a]), w[b], c[a][b]);
      if (WHICH == 0) {
        const float wz = sB[buf][k][et];
        e = __ffma2_rn(*reinterpret_cast<const float2*>(&sA[buf][k][er]), make_float2(wz, wz), e);
      }
    }
    if (more) store(buf ^ 1);
    __syncthreads();
  }
  float* G = part + (size_t)blockIdx.x * PSTRIDE + (WHICH == 0 ? OFF_W1 : OFF_W2) + (size_t)m0 * HID + nb * 64;
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int g = 0; g < 2; ++g)
      *reinterpret_cast<float4*>(G + (4 * ty + a) * HID + 32 * g + 4 * tx) =
          make_float4(c[a][2 * g].x, c[a][2 * g].y, c[a][2 * g + 1].x, c[a][2 * g + 1].y);
  if (WHICH == 0) {
    G[er * HID + et] = e.x;
    G[(er + 1) * HID + et] = e.y;
  }
}
__global__ void __launch_bounds__(BG_T)
back_grads(const float* __restrict__ X, const __nv_bfloat16* __restrict__ H1, const float* __restrict__ dz1,
           const float* __restrict__ dz2, int n, int chunk, float* __restrict__ part) {
  __shared__ __align__(16) float sA[2][BG_K][72], sB[2][BG_K][64];
  const int mb = (blockIdx.y >> 1) & 1, nb = blockIdx.y & 1;
  if (blockIdx.y < 4) grad_block<0>(X, H1, dz1, n, chunk, mb, nb, part, sA, sB);
  else grad_block<1>(X, H1, dz2, n, chunk, mb, nb, part, sA, sB);
}

// gW3 over the splits' rows and the bias gradients over chunks of 1024 rows:
// serial sums over the rows of 32 columns per CTA.  Eight warps load 128 rows at
// a time (16 independent loads per thread), the first one adds them up from
// shared memory while the others load the next 128.
constexpr int BT_T = 256, BT_S = 128;
__global__ void __launch_bounds__(BT_T)
back_tail(const __nv_bfloat16* __restrict__ H2, const float* __restrict__ dz1, const float* __restrict__ dz2,
          const float* __restrict__ dz3, int n, int chunk, int splits, float* __restrict__ part,
          float* __restrict__ bpart) {
  __shared__ __align__(16) float sV[2][BT_S][32], sD[2][BT_S][4];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const bool w3 = (int)blockIdx.x < 4 * splits;
  // bias: 4 CTAs for dZ1, 4 for dZ2 and one for dZ3 per chunk
  const int u = w3 ? (int)blockIdx.x : (int)blockIdx.x - 4 * splits, ch = w3 ? u >> 2 : u / 9, sl = w3 ? u & 3 : u - 9 * ch;
  const int len = w3 ? chunk : 1024, cols = !w3 && sl == 8 ? OUT : HID, col = (sl & 3) * 32 + lane;
  const float* Z = sl < 4 ? dz1 : (sl < 8 ? dz2 : dz3);
  const long long r0 = (long long)ch * len, r1 = min((long long)n, r0 + len);
  const bool in = cols == HID || lane < OUT;
  auto stage = [&](int buf, long long rb) {
    float v[BT_S / 8];
#pragma unroll
    for (int i = 0; i < BT_S / 8; ++i) {
      const long long r = rb + warp + 8 * i;
      v[i] = 0.f;
      if (r < r1 && in) v[i] = w3 ? __bfloat162float(H2[r * HID + col]) : __ldg(Z + r * cols + (cols == HID ? col : lane));
    }
    if (w3 && threadIdx.x < BT_S) {
      const long long r = rb + threadIdx.x;
#pragma unroll
      for (int j = 0; j < OUT; ++j) sD[buf][threadIdx.x][j] = r < r1 ? __ldg(dz3 + r * OUT + j) : 0.f;
    }
#pragma unroll
    for (int i = 0; i < BT_S / 8; ++i) sV[buf][warp + 8 * i][lane] = v[i];
  };
  float g[3] = {0.f, 0.f, 0.f};
  stage(0, r0);
  __syncthreads();
  int buf = 0;
  for (long long rb = r0; rb < r1; rb += BT_S, buf ^= 1) {
    if (warp == 0) {
      if (w3) {
#pragma unroll 8
        for (int i = 0; i < BT_S; ++i) {
          const float h = sV[buf][i][lane];
          const float4 d = *reinterpret_cast<const float4*>(sD[buf][i]);
          g[0] = fmaf(h, d.x, g[0]);
          g[1] = fmaf(h, d.y, g[1]);
          g[2] = fmaf(h, d.z, g[2]);
        }
      } else {
#pragma unroll 16
        for (int i = 0; i < BT_S; ++i) g[0] += sV[buf][i][lane];
      }
    }
    if (rb + BT_S < r1) stage(buf ^ 1, rb + BT_S);
    __syncthreads();
  }
  if (warp != 0) return;
  if (w3) {
#pragma unroll
    for (int j = 0; j < OUT; ++j) part[(size_t)ch * PSTRIDE + OFF_W3 + col * OUT + j] = g[j];
  } else if (in) {
    bpart[(size_t)ch * 260 + (sl < 8 ? sl * 32 : 2 * HID) + lane] = g[0];
  }
}

// gradients: the splits' (and chunks') sums added in order
__global__ void __launch_bounds__(128) back_sum(const float* __restrict__ part, int splits, const float* __restrict__ bpart,
                                                int bchunks, float* __restrict__ G) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= NPARAM) return;
  const int b = (i >= OFF_B1 && i < OFF_W2) ? i - OFF_B1
                : ((i >= OFF_B2 && i < OFF_W3) ? HID + i - OFF_B2 : (i >= OFF_B3 ? 2 * HID + i - OFF_B3 : -1));
  const float* p = b >= 0 ? bpart + b : part + i;
  const size_t ld = b >= 0 ? 260 : PSTRIDE;
  const int m = b >= 0 ? bchunks : splits;
  float s = 0.f;
#pragma unroll 16
  for (int k = 0; k < m; ++k) s += p[(size_t)k * ld];
  G[i] = s;
}

__global__ void adam_kernel(float* __restrict__ P, const float* __restrict__ G, float* __restrict__ m,
                            float* __restrict__ v, int count, float lr, float b1, float b2, float eps,
                            float c1, float c2) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < count; i += gridDim.x * blockDim.x) {
    const float g = G[i];
    const float mi = b1 * m[i] + (1.f - b1) * g;
    const float vi = b2 * v[i] + (1.f - b2) * g * g;
    m[i] = mi;
    v[i] = vi;
    P[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
  }
}

// features: the state at the 27 points {-1, 0, 1}^3 of every element
__constant__ double c_fw[kMaxN + 1][3][kMaxN + 1];   // h_m at -1, 0, 1

// (float)(v / s) for a float64 v and a float32 s, bit for bit, on the float32
// and integer pipes (a float64 division per value kept the float64 pipe 87 %
// busy): with the significands m = hi + lo of v (hi its leading 24 bits, lo
// the next 29 rounded to float32) and t of s, one residual correction
// c = (hi - q0 t + lo) / t of the quotient q0 with the residual exact in an
// FMA (Markstein), q = q0 + c, then the exponents.  c is below three units in
// the last place of q0 and within 2^-20 of one of its value, so q is the
// rounded quotient unless what q0 + c leaves over (exact by Fast2Sum) is within
// 2^-17 of a unit of the midpoint between two float32 numbers; those values
// (one in 10^5), quotients outside 2^-110 .. 2^120, infinities and NaN take the
// float64 division.  Quotients below half of float32's smallest value give a
// signed zero.
struct Divisor {
  float s, t, rt;   // s, its significand with s's sign in 1 <= |t| < 2, 1 / t
  int e;            // exponent of s; beyond the table's range for a special s
};
__device__ __forceinline__ Divisor divisor(float s) {
  const unsigned b = __float_as_uint(s);
  const int eb = (int)((b >> 23) & 0xffu);
  Divisor d;
  d.s = s;
  d.t = __uint_as_float((b & 0x807fffffu) | (127u << 23));
  d.rt = 1.0f / d.t;
  d.e = (eb == 0 || eb == 255) ? -(1 << 20) : eb - 127;
  return d;
}
__device__ __forceinline__ float div_to_f32(double v, const Divisor& D) {
  const unsigned vh = (unsigned)__double2hiint(v), vl = (unsigned)__double2loint(v);
  const int e = (int)((vh >> 20) & 0x7ffu) - 1023 - D.e;   // exponent of v / s, or one above it
  const unsigned sign = vh & 0x80000000u;
  if (e < -153) return __uint_as_float(sign ^ (__float_as_uint(D.t) & 0x80000000u));
  const float hi = __uint_as_float(sign | (127u << 23) | ((vh & 0xfffffu) << 3) | (vl >> 29));
  const float lo = __uint_as_float(__float_as_uint((float)(vl & 0x1fffffffu) * 0x1p-52f) | sign);
  const float q0 = hi * D.rt;
  const float c = __fmul_rn(fmaf(-q0, D.t, hi) + lo, D.rt);
  const float q = q0 + c, left = fabsf((q0 - q) + c);
  // half a unit of q, a quarter below a power of two
  const unsigned qb = __float_as_uint(q);
  const float half = __uint_as_float(qb & 0x7f800000u) * ((qb & 0x7fffffu) ? 0x1p-24f : 0x1p-25f);
  if (e < -110 || e > 120 || left >= half * (1.f - 0x1p-16f)) return (float)(v / (double)D.s);
  return q * __uint_as_float((unsigned)(e + 127) << 23);
}

// Features of a column's layers [k0, k0 + KL): one CTA.  First the values of
// the 9 horizontal points at every level that a point needs (even N: nodes
// (a, b) in {0, N/2, N}^2 and every N/2-th level; odd N: horizontal
// interpolation in float64 at every level), the lanes running along a
// z-line, so the loads are contiguous; then the rows, written in the order in
// which they lie in memory.  Bound by DRAM (the sampled lines and the 544 B
// rows); the sampled values of neighbouring layers are formed once.  64x64x16,
// N = 4: 30 us; 1071 us as one thread per point (27 scattered loads per element,
// 64-bit index arithmetic, a float64 division per value).
template <int N>
__global__ void __launch_bounds__(256)
mlp_features_kernel(const double* __restrict__ q, const int* __restrict__ hmap,
                    const int* __restrict__ hang_h, const double* __restrict__ hang_w,
                    const int* __restrict__ col_level, int nz, int NZ, long long NG, int KL, float s0,
                    float s1, float s2, float s3, float s4, float* __restrict__ F) {
  constexpr int n1 = N + 1, Nq = n1 * n1;
  constexpr bool EVEN = N % 2 == 0;
  constexpr int ST = EVEN ? N / 2 : 1;      // level stride of the staged values
  extern __shared__ __align__(16) unsigned char smf[];
  const int col = blockIdx.x;
  const int LD = KL * (N / ST) + 1;         // staged level stride of (field, point)
  float* sv = reinterpret_cast<float*>(smf);            // even N: [5][9][LD] scaled values
  double* sd = reinterpret_cast<double*>(smf);          // odd N: [5][9][LD] values
  const float sc[kFields] = {s0, s1, s2, s3, s4};
  Divisor dv[kFields];
#pragma unroll
  for (int f = 0; f < kFields; ++f) dv[f] = divisor(sc[f]);
  auto line = [&](int ab, int kz, double (&v)[kFields]) {
    const int hm = hmap[(long long)col * Nq + ab];
    if (hm >= 0) {
      const double* p = q + (long long)hm * NZ + kz;
#pragma unroll
      for (int f = 0; f < kFields; ++f) v[f] = __ldg(p + f * NG);
    } else {
      const int hk = -1 - hm;
#pragma unroll
      for (int f = 0; f < kFields; ++f) v[f] = 0.0;
      for (int m = 0; m < n1; ++m) {
        const double w = hang_w[hk * n1 + m];
        const double* p = q + (long long)hang_h[hk * n1 + m] * NZ + kz;
#pragma unroll
        for (int f = 0; f < kFields; ++f) v[f] += w * __ldg(p + f * NG);
      }
    }
  };
  for (int k0 = blockIdx.y * KL; k0 < nz; k0 += gridDim.y * KL) {
  const int kl = min(KL, nz - k0), nlev = kl * (N / ST) + 1;
  for (int it = threadIdx.x; it < 9 * nlev; it += blockDim.x) {
    const int pt = it / nlev, lv = it - pt * nlev, kz = k0 * N + lv * ST;
    const int pa = pt % 3, pb = pt / 3;
    double v[kFields];
    if (EVEN) {
      line(pa * ST + n1 * (pb * ST), kz, v);
#pragma unroll
      for (int f = 0; f < kFields; ++f) sv[(f * 9 + pt) * LD + lv] = div_to_f32(v[f], dv[f]);
    } else {
      double acc[kFields] = {0, 0, 0, 0, 0};
      for (int j = 0; j < n1; ++j) {
        const double wj = c_fw[N][pb][j];
        if (wj == 0.0) continue;
        for (int i = 0; i < n1; ++i) {
          const double wi = c_fw[N][pa][i];
          if (wi == 0.0) continue;
          line(i + n1 * j, kz, v);
#pragma unroll
          for (int f = 0; f < kFields; ++f) acc[f] += wi * wj * v[f];
        }
      }
#pragma unroll
      for (int f = 0; f < kFields; ++f) sd[(f * 9 + pt) * LD + lv] = acc[f];
    }
  }
  __syncthreads();
  const float level = (float)col_level[col];
  float* out = F + ((long long)col * nz + k0) * IN;
  for (int i = threadIdx.x; i < kl * IN; i += blockDim.x) {
    const int k = i / IN, j = i - k * IN;
    float r = level;
    if (j < IN - 1) {
      const int f = j / 27, pnt = j - f * 27, pc = pnt / 9, pt = pnt - 9 * pc;
      const int at = (f * 9 + pt) * LD;
      if (EVEN) {
        r = sv[at + 2 * k + pc];
      } else {
        double a = 0.0;
        if (pc != 1) {
          a = sd[at + k * N + (pc == 0 ? 0 : N)];
        } else {
          for (int c = 0; c < n1; ++c) a += c_fw[N][1][c] * sd[at + k * N + c];
        }
        r = div_to_f32(a, divisor(f == 0 ? s0 : (f == 1 ? s1 : (f == 2 ? s2 : (f == 3 ? s3 : s4)))));
      }
    }
    out[i] = r;
  }
  __syncthreads();   // the next chunk overwrites the staged values
  }
}

}  // namespace

struct MlpImpl {
  float* P = nullptr;      // master parameters
  float* R = nullptr;      // bfloat16-rounded parameters (float32 storage)
  float* G = nullptr;      // gradients
  float* M1 = nullptr;     // Adam moments
  float* M2 = nullptr;
  __nv_bfloat16* wt = nullptr;  // transposed bfloat16 weights (W1T | W2T | W3T)
  int max_rows = 0;
  __nv_bfloat16 *H1 = nullptr, *H2 = nullptr;   // hidden activations of the backward pass's forward
  float *prob = nullptr, *dz3 = nullptr, *dz2 = nullptr, *dz1 = nullptr;
  float *part = nullptr, *bpart = nullptr;      // splits' weight gradients [64][PSTRIDE], chunks' bias sums [..][260]
  double* acc = nullptr;   // loss, weight sum
  int* err = nullptr;      // bit 4: a bounded wait of the tensor-core forward ran out
  int step = 0;
  int dev = -1;
  int forward_tc = 1;      // 1: tcgen05 forward (mlp_forward_tc), 0: mma.sync forward
};

int mlp_create(unsigned long long seed, int max_rows, void** out) {
  MlpImpl* m = new MlpImpl();
  m->max_rows = max_rows;
  cudaGetDevice(&m->dev);
  const size_t rows = (size_t)std::max(max_rows, 1);
  cudaError_t e = cudaSuccess;
  auto A = [&](void** p, size_t bytes) { if (e == cudaSuccess) e = cudaMalloc(p, bytes); };
  A((void**)&m->P, NPARAM * 4);
  A((void**)&m->R, NPARAM * 4);
  A((void**)&m->G, NPARAM * 4);
  A((void**)&m->M1, NPARAM * 4);
  A((void**)&m->M2, NPARAM * 4);
  A((void**)&m->wt, (size_t)(W1T_SZ + W2T_SZ + W3T_SZ) * 2);
  A((void**)&m->H1, rows * HID * 2);
  A((void**)&m->H2, rows * HID * 2);
  A((void**)&m->prob, rows * OUT * 4);
  A((void**)&m->dz3, rows * OUT * 4);
  A((void**)&m->dz2, rows * HID * 4);
  A((void**)&m->dz1, rows * HID * 4);
  A((void**)&m->part, (size_t)64 * PSTRIDE * 4);
  A((void**)&m->bpart, ((rows + 1023) / 1024) * 260 * 4);
  A((void**)&m->acc, 2 * sizeof(double));
  A((void**)&m->err, sizeof(int));
  if (e == cudaSuccess) e = cudaMemset(m->err, 0, sizeof(int));
  if (e == cudaSuccess) e = cudaMemset(m->M1, 0, NPARAM * 4);
  if (e == cudaSuccess) e = cudaMemset(m->M2, 0, NPARAM * 4);
  if (e == cudaSuccess) e = cudaMemset(m->G, 0, NPARAM * 4);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(mlp_forward, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)FWD_SMEM);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(mlp_forward_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)TC_SMEM);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(back_rows, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)BR_SMEM);
  if (e == cudaSuccess) {
    // Uniform(-1/sqrt(fan_in), 1/sqrt(fan_in)) weights from splitmix64 of
    // (seed, index), zero biases
    std::vector<float> h(NPARAM, 0.f);
    auto u01 = [&](unsigned long long i) {
      unsigned long long z = seed * 0x9E3779B97F4A7C15ull + i + 0x9E3779B97F4A7C15ull;
      z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
      z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
      z ^= z >> 31;
      return (double)(z >> 11) * (1.0 / 9007199254740992.0);
    };
    const int offs[3] = {OFF_W1, OFF_W2, OFF_W3}, sz[3] = {IN * HID, HID * HID, HID * OUT}, fan[3] = {IN, HID, HID};
    for (int l = 0; l < 3; ++l)
      for (int i = 0; i < sz[l]; ++i) h[offs[l] + i] = (float)((2.0 * u01(offs[l] + i) - 1.0) / std::sqrt((double)fan[l]));
    e = cudaMemcpy(m->P, h.data(), NPARAM * 4, cudaMemcpyHostToDevice);
  }
  if (e != cudaSuccess) {
    std::string msg = cudaGetErrorString(e);
    void* ps[] = {m->P, m->R, m->G, m->M1, m->M2, m->wt, m->H1, m->H2, m->prob, m->dz3, m->dz2, m->dz1, m->part, m->bpart, m->acc, m->err};
    for (void* p : ps)
      if (p) cudaFree(p);
    delete m;
    return fail(SEM_ERR_CUDA, "mlp allocation: " + msg);
  }
  mlp_refresh<<<64, 256>>>(m->P, m->wt, m->wt + W1T_SZ, m->wt + W1T_SZ + W2T_SZ, m->R);
  SEM_CUDA_TRY(cudaDeviceSynchronize());
  *out = m;
  return SEM_OK;
}

void mlp_destroy(void* h) {
  MlpImpl* m = (MlpImpl*)h;
  if (!m) return;
  void* ps[] = {m->P, m->R, m->G, m->M1, m->M2, m->wt, m->H1, m->H2, m->prob, m->dz3, m->dz2, m->dz1, m->part, m->bpart, m->acc, m->err};
  for (void* p : ps)
    if (p) cudaFree(p);
  delete m;
}

int mlp_params(void* h, float* host, int set, int which) {
  MlpImpl* m = (MlpImpl*)h;
  float* d = which == 0 ? m->P : (which == 1 ? m->G : m->R);
  if (set) {
    SEM_CUDA_TRY(cudaMemcpy(d, host, NPARAM * 4, cudaMemcpyHostToDevice));
    if (which == 0) {
      mlp_refresh<<<64, 256>>>(m->P, m->wt, m->wt + W1T_SZ, m->wt + W1T_SZ + W2T_SZ, m->R);
      SEM_CUDA_TRY(cudaDeviceSynchronize());
    }
  } else {
    SEM_CUDA_TRY(cudaMemcpy(host, d, NPARAM * 4, cudaMemcpyDeviceToHost));
  }
  return SEM_OK;
}

int mlp_param_count() { return NPARAM; }

static void launch_forward(MlpImpl* m, const float* X, int n, float* prob, __nv_bfloat16* H1, __nv_bfloat16* H2,
                           int8_t* flags, cudaStream_t st) {
  if (m->forward_tc) {
    ProfScope ps("mlp_forward_tc", st);
    int dev = 0, nsm = 152;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    const int tiles = (n + TC_ROWS - 1) / TC_ROWS;
    mlp_forward_tc<<<std::min(tiles, 2 * nsm), TC_T, TC_SMEM, st>>>(
        X, n, m->wt, m->wt + W1T_SZ, m->wt + W1T_SZ + W2T_SZ, m->P, prob, H1, H2, flags, m->err);
    return;
  }
  const int grid = (n + FWD_ROWS - 1) / FWD_ROWS;
  ProfScope ps("mlp_forward", st);
  mlp_forward<<<grid, 128, FWD_SMEM, st>>>(X, n, m->wt, m->wt + W1T_SZ, m->wt + W1T_SZ + W2T_SZ, m->P, prob, H1,
                                            H2, flags);
}

int mlp_select_forward(void* h, int tc) {
  MlpImpl* m = (MlpImpl*)h;
  if (tc != 0 && tc != 1) return fail(SEM_ERR_ARG, "forward: 0 (mma.sync) or 1 (tcgen05)");
  m->forward_tc = tc;
  return SEM_OK;
}

int mlp_status(void* h, int* status, cudaStream_t st) {
  MlpImpl* m = (MlpImpl*)h;
  int v = 0;
  SEM_CUDA_TRY(cudaMemcpyAsync(&v, m->err, sizeof(int), cudaMemcpyDeviceToHost, st));
  SEM_CUDA_TRY(cudaMemsetAsync(m->err, 0, sizeof(int), st));
  SEM_CUDA_TRY(cudaStreamSynchronize(st));
  *status = v ? SEM_ERR_TIMEOUT : SEM_OK;
  return SEM_OK;
}

int mlp_forward_api(void* h, const float* X, int n, float* prob, int8_t* flags, cudaStream_t st) {
  MlpImpl* m = (MlpImpl*)h;
  if (n <= 0) return SEM_OK;
  launch_forward(m, X, n, prob, nullptr, nullptr, flags, st);
  SEM_CUDA_TRY(cudaGetLastError());
  return SEM_OK;
}

int mlp_backward_api(void* h, const float* X, const int8_t* y, const float* cw, int n, double* loss_host,
                     cudaStream_t st) {
  MlpImpl* m = (MlpImpl*)h;
  if (n <= 0 || n > m->max_rows) return fail(SEM_ERR_ARG, "row count outside 1..max_rows");
  launch_forward(m, X, n, m->prob, m->H1, m->H2, nullptr, st);
  SEM_CUDA_TRY(cudaMemsetAsync(m->acc, 0, 2 * sizeof(double), st));
  mlp_wsum<<<std::min(256, (n + 255) / 256), 256, 0, st>>>(y, n, cw[0], cw[1], cw[2], m->acc);
  ProfScope ps("mlp_backward", st);
  back_rows<<<(n + BR_ROWS - 1) / BR_ROWS, BR_T, BR_SMEM, st>>>(y, n, cw[0], cw[1], cw[2], m->prob, m->H1, m->H2,
                                                               m->wt + W1T_SZ, m->R, m->acc, loss_host != nullptr, m->dz3, m->dz2, m->dz1);
  int chunk = 0;
  const int splits = back_splits(n, chunk), bchunks = (n + 1023) / 1024;
  back_grads<<<dim3(splits, 8), BG_T, 0, st>>>(X, m->H1, m->dz1, m->dz2, n, chunk, m->part);
  back_tail<<<4 * splits + 9 * bchunks, BT_T, 0, st>>>(m->H2, m->dz1, m->dz2, m->dz3, n, chunk, splits, m->part,
                                                       m->bpart);
  back_sum<<<(NPARAM + 127) / 128, 128, 0, st>>>(m->part, splits, m->bpart, bchunks, m->G);
  SEM_CUDA_TRY(cudaGetLastError());
  if (loss_host) {
    double a[2];
    SEM_CUDA_TRY(cudaMemcpyAsync(a, m->acc, sizeof(a), cudaMemcpyDeviceToHost, st));
    SEM_CUDA_TRY(cudaStreamSynchronize(st));
    *loss_host = a[0] / a[1];
  }
  return SEM_OK;
}

int mlp_adam_api(void* h, float lr, cudaStream_t st) {
  MlpImpl* m = (MlpImpl*)h;
  m->step += 1;
  const float b1 = 0.9f, b2 = 0.999f;
  const float c1 = (float)(1.0 - std::pow(0.9, m->step)), c2 = (float)(1.0 - std::pow(0.999, m->step));
  adam_kernel<<<(NPARAM + 255) / 256, 256, 0, st>>>(m->P, m->G, m->M1, m->M2, NPARAM, lr, b1, b2, 1e-8f, c1, c2);
  mlp_refresh<<<64, 256, 0, st>>>(m->P, m->wt, m->wt + W1T_SZ, m->wt + W1T_SZ + W2T_SZ, m->R);
  SEM_CUDA_TRY(cudaGetLastError());
  return SEM_OK;
}

int mlp_features_api(Mesh& mesh, const double* q, const float* scales, float* F, cudaStream_t st) {
  // the interpolation rows of the current device (uploaded on its first use)
  static DeviceOnce once;
  int rc = device_once(once, [] {
    double fw[kMaxN + 1][3][kMaxN + 1] = {};
    for (int N = 2; N <= kMaxN; ++N) {
      const Basis1D& B = basis(N);
      const double pts[3] = {-1.0, 0.0, 1.0};
      for (int p = 0; p < 3; ++p)
        for (int mm = 0; mm <= N; ++mm) {
          double v = lagrange(B.xi, mm, pts[p]);
          for (int r = 0; r <= N; ++r)
            if (pts[p] == B.xi[r]) v = (r == mm) ? 1.0 : 0.0;
          fw[N][p][mm] = v;
        }
    }
    SEM_CUDA_TRY(cudaMemcpyToSymbol(c_fw, fw, sizeof(fw)));
    return SEM_OK;
  });
  if (rc) return rc;
  DeviceTables& D = *mesh.dev;
  // layers per CTA: 16 (a 16-layer column of the benchmark per CTA); 4 when
  // that leaves fewer than two CTAs per SM
  int dev = 0, nsm = 152;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  const long long ncol = mesh.Ncol();
  int KL = std::min(16, mesh.nz);
  if (ncol * ((mesh.nz + KL - 1) / KL) < 2LL * nsm) KL = std::min(4, mesh.nz);
  const int chunks = (mesh.nz + KL - 1) / KL;
  const dim3 grid((unsigned)ncol, (unsigned)std::min(chunks, 65535));
  ProfScope ps("mlp_features", st);
  auto go = [&](auto kern, int N) {
    const size_t sm = N % 2 == 0 ? sizeof(float) * 45 * (2 * KL + 1) : sizeof(double) * 45 * (N * KL + 1);
    kern<<<grid, 256, sm, st>>>(q, D.hmap, D.hang_h, D.hang_w, D.col_level, mesh.nz, mesh.NZ, mesh.NG, KL,
                                scales[0], scales[1], scales[2], scales[3], scales[4], F);
  };
  switch (mesh.N) {
    case 2: go(mlp_features_kernel<2>, 2); break;
    case 3: go(mlp_features_kernel<3>, 3); break;
    case 4: go(mlp_features_kernel<4>, 4); break;
    case 5: go(mlp_features_kernel<5>, 5); break;
    case 6: go(mlp_features_kernel<6>, 6); break;
    default: return fail(SEM_ERR_UNSUPPORTED, "order N not compiled");
  }
  SEM_CUDA_TRY(cudaGetLastError());
  return SEM_OK;
}

}  // namespace sem
