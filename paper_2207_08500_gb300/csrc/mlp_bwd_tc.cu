// Gradient of the classifier's training loss on the tensor cores: the mean
// binary cross entropy of Eq. (Crossentropy) over the S = 4 sigmoid outputs of
// the 6-64-32-16-8-4 ReLU network of Sec. 3.1, with respect to all 3228
// parameters, for mixed-precision handles (bf16 or fp16 operands, FP32
// accumulation in tensor memory).
//
// Persistent CTAs of 128 threads, two per SM, one 128-sample tile per
// iteration; thread t owns sample row t (MMA row t, TMEM lane t).
//   forward   layers 1-4 by tcgen05.mma exactly as the inference kernel
//             (16-bit activations in TMEM, biases of layers 1-2 on the
//             tensor cores, layer 5 in FP32); every hidden layer's ReLU
//             output is also written, transposed, into shared memory and
//             its ReLU mask kept in registers;
//   deltas    D5 = sigma(z) - y (the 1/(n S) of the mean is applied once, in
//             FP32, to the summed gradient: 16-bit operands then stay in
//             their normal range), D4 and D3 in FP32 on the CUDA cores,
//             D2 = (D3 W3) * relu' and D1 = (D2 W2) * relu' by tcgen05.mma
//             against the transposed weights;
//   gradients dW_l^T (or dW_1) = H_{l-1}^T D_l as tcgen05.mma with K = the
//             tile's 128 samples, accumulated over all of a CTA's tiles in
//             FP32 in tensor memory; a row of ones in each A operand gives
//             the bias gradient sum_s D_l in the same MMA.
// The weight-gradient MMAs run M = 128 rows of which only the first few are
// meaningful: the rows past them read whatever follows in shared memory and
// only fill accumulator rows that are never read.  Per-CTA partial sums go
// to a fixed-order reduction, which applies the 1/(n S).
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "internal.h"
#include "mlp_tc.cuh"
#include "tc.cuh"

namespace neno6 {
namespace {

using namespace tc;
using namespace tcmlp;

constexpr int kT = 128;
// Activations and deltas of a tile lie in shared memory by groups of eight
// units: group g of a buffer is 128 samples x 16 bytes (eight 16-bit values), so
// a thread stores its sample's eight units with one 16-byte store, without bank
// conflicts.  One buffer serves two operands: M (or N) = units, K = samples
// ("MN-major": the core matrix's 16-byte rows run along M) for the weight
// gradients, M = samples, K = units (K-major) for the deltas, with the strides
// between core matrices along units and samples
constexpr int kGroup = 2048;
constexpr uint32_t kUnits = kGroup, kSamples = 128;
// shared memory (bytes): images, then the weight-gradient A operands (each
// read as 16 groups = 32 KB from its start), then the rest
constexpr int kOffNet = 0;
constexpr int kOffBwd = kOffNet + kNetImageBytes;
constexpr int kOffH1 = kOffBwd + kBwdImageBytes;  // H1 (64 units), then 1 in unit 64: 9 groups
// H2, H3 and H4 follow one another, and D3, D4 and D5: one product of the two
// runs holds the gradients of layers 3, 4 and 5 in its diagonal blocks (the rest
// is not read), in a third of the MMAs and of the tensor memory
constexpr int kOffH2 = kOffH1 + 9 * kGroup;       // H2 (32), 1 in unit 32: 5 groups
constexpr int kOffH3 = kOffH2 + 5 * kGroup;       // H3 (16), 1 in unit 16: 3 groups
constexpr int kOffH4 = kOffH3 + 3 * kGroup;       // H4 (8), 1 in unit 8: 2 groups
constexpr int kOffD1 = kOffH4 + 2 * kGroup;       // D1 (64): 8 groups
constexpr int kOffD2 = kOffD1 + 8 * kGroup;       // D2 (32): 4 groups
constexpr int kOffD3 = kOffD2 + 4 * kGroup;       // D3 (16): 2 groups
constexpr int kOffD4 = kOffD3 + 2 * kGroup;       // D4 (8)
constexpr int kOffD5 = kOffD4 + kGroup;           // D5 (4 of 8)
constexpr int kOffX0 = kOffD5 + kGroup;           // layer-1 input, 128 x 16, K-major (store_input_row)
constexpr int kOffXs = kOffX0 + 128 * 16 * 2;     // the next tile's stencils, 128 x 6 doubles
constexpr int kOffBar = kOffXs + 128 * 48;        // mbarrier, TMEM address, timeout flag, stencils' mbarrier
constexpr int kOffLoss = kOffBar + 32;            // kT doubles
// rows of the combined product's units
constexpr int kRowH3 = 40, kRowH4 = 64;
static_assert(kOffH3 - kOffH2 == kRowH3 / 8 * kGroup && kOffH4 - kOffH2 == kRowH4 / 8 * kGroup, "combined product");
constexpr int kSmem = ((kOffLoss + kT * 8) + 127) / 128 * 128;
static_assert(kOffH1 % 128 == 0 && kOffX0 % 128 == 0, "alignment");
static_assert(kOffD1 + 16 * kGroup <= kSmem, "the last weight-gradient A operand's 128 rows are addressable");
// two CTAs per SM (2 x 256 TMEM columns)
static_assert(2 * (kSmem + 1024) <= 228 * 1024, "two CTAs per SM");
// TMEM columns: forward / backward working area [0, 64), the weight-gradient
// accumulators from column 128
constexpr uint32_t kAcc1 = 128, kAcc2 = 144, kAcc3 = 176;  // kAcc3: layers 3, 4, 5

// Eight 16-bit units (group g of the buffer) of sample t.
__device__ __forceinline__ void st_group(uint8_t* base, int g, int t, uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
  asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(smem_u32(base + g * kGroup + t * 16)), "r"(a), "r"(b),
               "r"(c), "r"(d)
               : "memory");
}

// D[col] (+)= A (units x samples) * B (units x samples)^T over the tile's 128
// samples, both MN-major: unit groups a_mn / b_mn bytes apart, groups of eight
// samples a_k / b_k; issued by this thread.
__device__ __forceinline__ void mma_grad(uint32_t d_tmem, const uint8_t* A, const uint8_t* B, uint32_t b_mn,
                                         uint32_t b_k, int N, bool bf16, bool acc0) {
  const uint32_t idesc = idesc_f16(128, N, bf16) | (1u << 15) | (1u << 16);
  const uint32_t a0 = smem_u32(A), b0 = smem_u32(B);
#pragma unroll
  for (int ks = 0; ks < 8; ++ks)
    mma_f16(d_tmem, smem_desc(a0 + 2u * kSamples * ks, kSamples, kUnits), smem_desc(b0 + 2u * b_k * ks, b_k, b_mn),
            idesc, (ks > 0 || acc0) ? 1u : 0u);
}
// D[col] = A (128 samples x K units, K-major) * W^T (N x K image at B): a layer's
// forward pass or its delta.
__device__ __forceinline__ void mma_layer(uint32_t d_tmem, const uint8_t* A, const uint8_t* B, uint32_t b_sbo, int K,
                                          int N, bool bf16) {
  const uint32_t idesc = idesc_f16(128, N, bf16);
  const uint32_t a0 = smem_u32(A), b0 = smem_u32(B);
#pragma unroll
  for (int ks = 0; ks < K / 16; ++ks)
    mma_f16(d_tmem, smem_desc(a0 + 2u * kUnits * ks, kUnits, kSamples), smem_desc(b0 + 256u * ks, 128u, b_sbo), idesc,
            ks > 0 ? 1u : 0u);
}

template <bool BF16>
__global__ void __launch_bounds__(kT, 2) mlp_bwd_tc_kernel(const double* __restrict__ X,
                                                           const uint8_t* __restrict__ y, long long n,
                                                           const uint8_t* __restrict__ net_image,
                                                           const uint8_t* __restrict__ bwd_image,
                                                           float* __restrict__ partial,
                                                           double* __restrict__ partial_loss, int* status) {
  extern __shared__ __align__(1024) uint8_t smem[];
  uint8_t* s_net = smem + kOffNet;
  const uint8_t* s_bwd = smem + kOffBwd;
  uint64_t* bar = reinterpret_cast<uint64_t*>(smem + kOffBar);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + kOffBar + 8);
  int* fail = reinterpret_cast<int*>(smem + kOffBar + 12);
  double* s_loss = reinterpret_cast<double*>(smem + kOffLoss);
  const int t = threadIdx.x;
  const uint32_t lane = (uint32_t)(t & ~31) << 16;

  // images; every operand buffer zeroed, then the constant units of one
  for (int i = t; i < kNetImageBytes / 16; i += kT)
    reinterpret_cast<uint4*>(s_net)[i] = reinterpret_cast<const uint4*>(net_image)[i];
  for (int i = t; i < kBwdImageBytes / 16; i += kT)
    reinterpret_cast<uint4*>(smem + kOffBwd)[i] = reinterpret_cast<const uint4*>(bwd_image)[i];
  for (int i = t; i < (kOffXs - kOffH1) / 16; i += kT)
    reinterpret_cast<uint4*>(smem + kOffH1)[i] = make_uint4(0u, 0u, 0u, 0u);
  __syncthreads();
  st_group(smem + kOffH1, 8, t, one0<BF16>(), 0u, 0u, 0u);
  st_group(smem + kOffH2, 4, t, one0<BF16>(), 0u, 0u, 0u);
  st_group(smem + kOffH3, 2, t, one0<BF16>(), 0u, 0u, 0u);
  st_group(smem + kOffH4, 1, t, one0<BF16>(), 0u, 0u, 0u);
  TileRows rows{X, n, reinterpret_cast<double*>(smem + kOffXs), reinterpret_cast<uint64_t*>(smem + kOffBar + 16), 0u,
                (reinterpret_cast<uintptr_t>(X) & 15u) == 0};
  if (t == 0) {
    mbar_init(bar, 1);
    mbar_init(rows.bar, 1);
    fence_mbar_init();
    *fail = 0;
    rows.fetch(blockIdx.x);
  }
  if (t < 32) {
    tmem_alloc(tmem_slot, 256);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  MlpCtx mc{s_net, smem + kOffX0, bar, tmem, 0u, BF16, fail};
  const float* fbias = reinterpret_cast<const float*>(s_net + kNetImageBias);  // b3 at 0, b4 at 16, b5 at 24
  const float* W4 = reinterpret_cast<const float*>(s_bwd + kBwdW4);          // [8][16]
  const float* W5 = reinterpret_cast<const float*>(s_bwd + kBwdW5);          // [4][8]
  double loss = 0.0;
  const long long tiles = (n + kT - 1) / kT;
  bool first = true;
  for (long long tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
    const long long s = tile * kT + t;
    const bool live = s < n;
    // ---- Eq. (normalizainput) in FP32
    const unsigned lab = live ? y[s] : 0u;
    float x0[6], m = 1.0f;
    const bool got = rows.get(tile, x0);
    if (!got) *fail = 1;
#pragma unroll
    for (int j = 0; j < 6; ++j) m = fmaxf(m, fabsf(x0[j]));
#pragma unroll
    for (int j = 0; j < 6; ++j) x0[j] = x0[j] / m;
    // the previous tile's weight-gradient MMAs read the operand buffers
    if (!first) wait_layer(mc);
    store_input_row<BF16>(smem + kOffX0, t, x0);
    fence_async_smem();
    tc_fence_before();
    __syncthreads();
    // ---- layer 1 (bias on the ones columns) -> H1
    if (t == 0) {
      issue_layer<BF16>(mc, smem + kOffX0, 16, kNetImageB1, 64, (int)kColD1);
      if (got) rows.fetch(tile + gridDim.x);
    }
    wait_layer(mc);
    uint32_t mask1[2] = {0u, 0u};
#pragma unroll
    for (int c32 = 0; c32 < 2; ++c32) {
      uint32_t r[16], q[16];
      tmem_ld16(tmem + lane + kColD1 + 32u * c32, r);
      tmem_ld16(tmem + lane + kColD1 + 32u * c32 + 16u, q);
      tmem_ld_wait();
      uint32_t pk[16];
#pragma unroll
      for (int i = 0; i < 16; ++i) {
        const float z0 = __uint_as_float(i < 8 ? r[2 * i] : q[2 * i - 16]);
        const float z1 = __uint_as_float(i < 8 ? r[2 * i + 1] : q[2 * i - 15]);
        mask1[c32] |= (z0 > 0.0f ? 1u : 0u) << (2 * i);
        mask1[c32] |= (z1 > 0.0f ? 1u : 0u) << (2 * i + 1);
        pk[i] = relu_pack2<BF16>(z0, z1);
      }
#pragma unroll
      for (int g = 0; g < 4; ++g)
        st_group(smem + kOffH1, 4 * c32 + g, t, pk[4 * g], pk[4 * g + 1], pk[4 * g + 2], pk[4 * g + 3]);
    }
    fence_async_smem();
    tc_fence_before();
    __syncthreads();
    // ---- layer 2 (bias K-step on the layer-1 input tile) -> H2
    if (t == 0) {
      tc_fence_after();
      mma_layer(tmem + kColD2, smem + kOffH1, s_net + kNetImageB2, 1024u, 64, 32, BF16);
      mma_f16(tmem + kColD2, smem_desc(smem_u32(smem + kOffX0), 128u, 256u),
              smem_desc(smem_u32(s_net + kNetImageB2b), 128u, 256u), idesc_f16(128, 32, BF16), 1u);
      mma_commit(bar);
    }
    wait_layer(mc);
    uint32_t mask2 = 0u;
    {
      uint32_t r[16], q[16];
      tmem_ld16(tmem + lane + kColD2, r);
      tmem_ld16(tmem + lane + kColD2 + 16u, q);
      tmem_ld_wait();
      uint32_t pk[16];
#pragma unroll
      for (int i = 0; i < 16; ++i) {
        const float z0 = __uint_as_float(i < 8 ? r[2 * i] : q[2 * i - 16]);
        const float z1 = __uint_as_float(i < 8 ? r[2 * i + 1] : q[2 * i - 15]);
        mask2 |= (z0 > 0.0f ? 1u : 0u) << (2 * i);
        mask2 |= (z1 > 0.0f ? 1u : 0u) << (2 * i + 1);
        pk[i] = relu_pack2<BF16>(z0, z1);
      }
#pragma unroll
      for (int g = 0; g < 4; ++g) st_group(smem + kOffH2, g, t, pk[4 * g], pk[4 * g + 1], pk[4 * g + 2], pk[4 * g + 3]);
    }
    fence_async_smem();
    tc_fence_before();
    __syncthreads();
    // ---- layer 3 (+ b3 in FP32) -> H3
    if (t == 0) {
      tc_fence_after();
      mma_layer(tmem + kColD3, smem + kOffH2, s_net + kNetImageB3, 512u, 32, 16, BF16);
      mma_commit(bar);
    }
    wait_layer(mc);
    uint32_t mask3 = 0u;
    {
      uint32_t r[16];
      tmem_ld16(tmem + lane + kColD3, r);
      tmem_ld_wait();
      uint32_t pk[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const float z0 = __uint_as_float(r[2 * i]) + fbias[2 * i];
        const float z1 = __uint_as_float(r[2 * i + 1]) + fbias[2 * i + 1];
        mask3 |= (z0 > 0.0f ? 1u : 0u) << (2 * i);
        mask3 |= (z1 > 0.0f ? 1u : 0u) << (2 * i + 1);
        pk[i] = relu_pack2<BF16>(z0, z1);
      }
#pragma unroll
      for (int g = 0; g < 2; ++g) st_group(smem + kOffH3, g, t, pk[4 * g], pk[4 * g + 1], pk[4 * g + 2], pk[4 * g + 3]);
    }
    fence_async_smem();
    tc_fence_before();
    __syncthreads();
    // ---- layer 4 (+ b4 in FP32) -> H4; layer 5 in FP32; deltas D5, D4, D3
    if (t == 0) {
      tc_fence_after();
      mma_layer(tmem + kColD4, smem + kOffH3, s_net + kNetImageB4, 256u, 16, 16, BF16);
      mma_commit(bar);
    }
    wait_layer(mc);
    float h4[8];
    uint32_t mask4 = 0u;
    {
      uint32_t r[16];
      tmem_ld16(tmem + lane + kColD4, r);
      tmem_ld_wait();
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const float z = __uint_as_float(r[i]) + fbias[16 + i];
        mask4 |= (z > 0.0f ? 1u : 0u) << i;
        h4[i] = fmaxf(z, 0.0f);
      }
      st_group(smem + kOffH4, 0, t, pack2<BF16>(h4[0], h4[1]), pack2<BF16>(h4[2], h4[3]), pack2<BF16>(h4[4], h4[5]),
               pack2<BF16>(h4[6], h4[7]));
    }
    float d5[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      float z = fbias[24 + k];
#pragma unroll
      for (int i = 0; i < 8; ++i) z = fmaf(W5[k * 8 + i], h4[i], z);
      const float yk = (float)((lab >> k) & 1u);
      // -[y log s + (1-y) log(1-s)] = softplus(z) - y z
      if (live) loss += (double)(fmaxf(z, 0.0f) + log1pf(__expf(-fabsf(z))) - yk * z);
      d5[k] = live ? 1.0f / (1.0f + __expf(-z)) - yk : 0.0f;
    }
    st_group(smem + kOffD5, 0, t, pack2<BF16>(d5[0], d5[1]), pack2<BF16>(d5[2], d5[3]), 0u, 0u);
    float d4[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      float a = 0.0f;
#pragma unroll
      for (int k = 0; k < 4; ++k) a = fmaf(W5[k * 8 + i], d5[k], a);
      d4[i] = (mask4 >> i) & 1u ? a : 0.0f;
    }
    st_group(smem + kOffD4, 0, t, pack2<BF16>(d4[0], d4[1]), pack2<BF16>(d4[2], d4[3]), pack2<BF16>(d4[4], d4[5]),
             pack2<BF16>(d4[6], d4[7]));
    float d3[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      float a = 0.0f;
#pragma unroll
      for (int k = 0; k < 8; ++k) a = fmaf(W4[k * 16 + i], d4[k], a);
      d3[i] = (mask3 >> i) & 1u ? a : 0.0f;
    }
#pragma unroll
    for (int g = 0; g < 2; ++g)
      st_group(smem + kOffD3, g, t, pack2<BF16>(d3[8 * g], d3[8 * g + 1]), pack2<BF16>(d3[8 * g + 2], d3[8 * g + 3]),
               pack2<BF16>(d3[8 * g + 4], d3[8 * g + 5]), pack2<BF16>(d3[8 * g + 6], d3[8 * g + 7]));
    fence_async_smem();
    tc_fence_before();
    __syncthreads();
    // ---- D2 = (D3 W3) * relu'(Z2); gradients of layers 5, 4, 3
    if (t == 0) {
      tc_fence_after();
      mma_layer(tmem + 0u, smem + kOffD3, s_bwd + kBwdBW3, 256u, 16, 32, BF16);
      mma_grad(tmem + kAcc3, smem + kOffH2, smem + kOffD3, kUnits, kSamples, 32, BF16, !first);
      mma_commit(bar);
    }
    wait_layer(mc);
    {
      uint32_t r[16], q[16];
      tmem_ld16(tmem + lane + 0u, r);
      tmem_ld16(tmem + lane + 16u, q);
      tmem_ld_wait();
      float d2[32];
#pragma unroll
      for (int i = 0; i < 32; ++i) {
        const float v = __uint_as_float(i < 16 ? r[i] : q[i - 16]);
        d2[i] = (mask2 >> i) & 1u ? v : 0.0f;
      }
#pragma unroll
      for (int g = 0; g < 4; ++g)
        st_group(smem + kOffD2, g, t, pack2<BF16>(d2[8 * g], d2[8 * g + 1]), pack2<BF16>(d2[8 * g + 2], d2[8 * g + 3]),
                 pack2<BF16>(d2[8 * g + 4], d2[8 * g + 5]), pack2<BF16>(d2[8 * g + 6], d2[8 * g + 7]));
    }
    fence_async_smem();
    tc_fence_before();
    __syncthreads();
    // ---- D1 = (D2 W2) * relu'(Z1); gradient of layer 2
    if (t == 0) {
      tc_fence_after();
      mma_layer(tmem + 0u, smem + kOffD2, s_bwd + kBwdBW2, 512u, 32, 64, BF16);
      mma_grad(tmem + kAcc2, smem + kOffH1, smem + kOffD2, kUnits, kSamples, 32, BF16, !first);
      mma_commit(bar);
    }
    wait_layer(mc);
#pragma unroll
    for (int c32 = 0; c32 < 2; ++c32) {
      uint32_t r[16], q[16];
      tmem_ld16(tmem + lane + 32u * c32, r);
      tmem_ld16(tmem + lane + 32u * c32 + 16u, q);
      tmem_ld_wait();
#pragma unroll
      for (int g = 0; g < 4; ++g) {
        uint32_t w[4];
#pragma unroll
        for (int h = 0; h < 4; ++h) {
          const int i = 8 * g + 2 * h;
          const float a = __uint_as_float(i < 16 ? r[i] : q[i - 16]), b = __uint_as_float(i < 16 ? r[i + 1] : q[i - 15]);
          w[h] = pack2<BF16>((mask1[c32] >> i) & 1u ? a : 0.0f, (mask1[c32] >> (i + 1)) & 1u ? b : 0.0f);
        }
        st_group(smem + kOffD1, 4 * c32 + g, t, w[0], w[1], w[2], w[3]);
      }
    }
    fence_async_smem();
    tc_fence_before();
    __syncthreads();
    // ---- gradient of layer 1 (waited for before the next tile's operands)
    if (t == 0) {
      tc_fence_after();
      // the layer-1 input tile as the N operand: stencil values in columns 0-5,
      // ones from ones_col on; its core matrices lie 128 bytes apart along the
      // columns, 256 along the samples
      mma_grad(tmem + kAcc1, smem + kOffD1, smem + kOffX0, 128u, 256u, 16, BF16, !first);
      mma_commit(bar);
    }
    first = false;
    if (__syncthreads_or(*fail)) break;
  }
  if (!first) wait_layer(mc);
  if (*fail) {
    // a copy may still be in flight: wait for it (bounded) before leaving
    float x[6];
    rows.get(blockIdx.x, x);
  }
  const bool failed = __syncthreads_or(*fail) != 0;
  // ---- this CTA's partial gradients, from the accumulator rows
  float* part = partial + (size_t)blockIdx.x * kNetParams;
  {
    uint32_t r[16];
    tmem_ld16(tmem + lane + kAcc1, r);  // row o of dW1 (o < 64): cols 0..5, db1 in col ones_col
    tmem_ld_wait();
    if (t < 64) {
#pragma unroll
      for (int i = 0; i < 6; ++i) part[t * 6 + i] = __uint_as_float(r[i]);
      part[384 + t] = __uint_as_float(r[ones_col(BF16)]);
    }
  }
#pragma unroll
  for (int c = 0; c < 2; ++c) {  // row i of dW2^T (i < 64), db2 in row 64
    uint32_t r[16];
    tmem_ld16(tmem + lane + kAcc2 + 16u * c, r);
    tmem_ld_wait();
#pragma unroll
    for (int o = 0; o < 16; ++o) {
      if (t < 64) part[448 + (16 * c + o) * 64 + t] = __uint_as_float(r[o]);
      if (t == 64) part[2496 + 16 * c + o] = __uint_as_float(r[o]);
    }
  }
  {
    uint32_t r[16];
    tmem_ld16(tmem + lane + kAcc3, r);  // row i of dW3^T (i < 32), db3 in row 32
    tmem_ld_wait();
#pragma unroll
    for (int o = 0; o < 16; ++o) {
      if (t < 32) part[2528 + o * 32 + t] = __uint_as_float(r[o]);
      if (t == 32) part[3040 + o] = __uint_as_float(r[o]);
    }
    tmem_ld16(tmem + lane + kAcc3 + 16u, r);  // columns of D4 (8), then D5
    tmem_ld_wait();
#pragma unroll
    for (int o = 0; o < 8; ++o) {  // row i of dW4^T, db4 in the row after
      if (t >= kRowH3 && t < kRowH3 + 16) part[3056 + o * 16 + t - kRowH3] = __uint_as_float(r[o]);
      if (t == kRowH3 + 16) part[3184 + o] = __uint_as_float(r[o]);
    }
#pragma unroll
    for (int o = 0; o < 4; ++o) {  // row i of dW5^T, db5 in the row after
      if (t >= kRowH4 && t < kRowH4 + 8) part[3192 + o * 8 + t - kRowH4] = __uint_as_float(r[8 + o]);
      if (t == kRowH4 + 8) part[3224 + o] = __uint_as_float(r[8 + o]);
    }
  }
  // block loss (fixed-order tree)
  s_loss[t] = loss;
  __syncthreads();
  for (int w = kT / 2; w > 0; w >>= 1) {
    if (t < w) s_loss[t] += s_loss[t + w];
    __syncthreads();
  }
  if (t == 0) {
    partial_loss[blockIdx.x] = s_loss[0];
    if (failed) atomicOr(status, 4);
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (t < 32) tmem_dealloc(tmem, 256);
}

}  // namespace

cudaError_t launch_mlp_bwd_tc(const double* X, const uint8_t* y, long long n, const uint8_t* net_image,
                              const uint8_t* bwd_image, bool bf16, float* grad, float* loss, void* scratch,
                              int* status, cudaStream_t s) {
  const long long tiles = (n + kT - 1) / kT;
  const int blocks = (int)(tiles < 2 * 152 ? tiles : 2 * 152);
  float* partial = static_cast<float*>(scratch);
  double* partial_loss =
      reinterpret_cast<double*>(static_cast<char*>(scratch) + (size_t)blocks * kNetParams * sizeof(float));
  auto kern = bf16 ? mlp_bwd_tc_kernel<true> : mlp_bwd_tc_kernel<false>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmem);
  if (e != cudaSuccess) return e;
  kern<<<blocks, kT, kSmem, s>>>(X, y, n, net_image, bwd_image, partial, partial_loss, status);
  e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  return launch_mlp_bwd_reduce(partial, partial_loss, blocks, n, (float)(1.0 / (4.0 * (double)n)), grad, loss, s);
}

}  // namespace neno6
