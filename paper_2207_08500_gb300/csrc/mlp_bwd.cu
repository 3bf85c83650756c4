// Gradient of the classifier's training loss (retraining the NENO6 network):
// the mean binary cross entropy of Eq. (Crossentropy),
//   L = -1/(n S) sum_s sum_k [ y log sigma(z) + (1-y) log(1 - sigma(z)) ],
// S = 4 outputs, with respect to every parameter (w^l, b^l) of the
// 6-64-32-16-8-4 ReLU network of Sec. 3.1, in FP32.
//
// Persistent CTAs of 256 threads take 128-sample tiles.  Every layer's input and
// delta of the tile is staged feature-major in shared memory (rows of 128
// samples), and each layer, forward, delta and weight gradient, is a small
// matrix product over the tile with a register tile per thread:
//  * forward and deltas: a lane takes four samples (one 16-byte load per input
//    row), its warp 1/8 of the layer's outputs (weights broadcast); each output
//    is its bias (or 0), then an FMA chain over its inputs in ascending order;
//  * weight gradients: a warp takes 16 of the tile's samples and all 3228
//    parameters, 8 x 8 of the 32 x 64 layer per lane, summed in registers over
//    all of the CTA's tiles.
// The eight warps' sums are added in order at the end and the CTAs' by a second
// kernel: deterministic.  Bound by the FP32 pipe and shared-memory loads: 2^20
// samples in 0.58 ms (0.23 ms of a full FP32 pipe), against 2.10 ms with one
// thread per sample and per-parameter sums, which took two loads per FMA and
// left four warps per SM.
#include "internal.h"
#include "mlp_fb.cuh"

namespace neno6 {
namespace {

using namespace mlpfb;

constexpr int kS = 128;         // samples per tile
constexpr int kT = 256;         // threads per CTA
constexpr int kWarps = kT / 32;
// row pitch: 16-byte aligned, and rows r..r+7 start in distinct 16-byte bank groups
constexpr int kPitch = kS + 4;
// shared memory in floats: the staged rows, then the weights: transposed
// ([in][out]) for the forward pass, natural for the deltas, and the biases
constexpr int kOffT1 = kRows * kPitch, kOffT2 = kOffT1 + 6 * 64, kOffT3 = kOffT2 + 64 * 32;
constexpr int kOffT4 = kOffT3 + 32 * 16, kOffW2 = kOffT4 + 16 * 8, kOffW3 = kOffW2 + 32 * 64;
constexpr int kOffW4 = kOffW3 + 16 * 32, kOffW5 = kOffW4 + 8 * 16, kOffB = kOffW5 + 4 * 8;  // b1, b2, b3, b4, b5
constexpr int kSmemFloats = kOffB + 64 + 32 + 16 + 8 + 4;
static_assert(kOffT1 % 4 == 0 && kWarps * kNetParams <= kRows * kPitch, "layout");

// NO outputs of one layer for this lane's four samples: out rows o0.., rows of
// the input from `in` on, weights w (row of outputs per input, WP apart), start
// values from `bias` (0 where null).
template <int NIN, int NO, int WP>
__device__ __forceinline__ void rows4(const float* __restrict__ in, const float* __restrict__ w,
                                      const float* __restrict__ bias, float4 (&acc)[NO]) {
  float2 lo[NO], hi[NO];
#pragma unroll
  for (int q = 0; q < NO; ++q) {
    const float b = bias ? bias[q] : 0.0f;
    lo[q] = hi[q] = make_float2(b, b);
  }
#pragma unroll 8
  for (int k = 0; k < NIN; ++k) {
    const float4 h = *reinterpret_cast<const float4*>(in + k * kPitch);
    float wv[NO];
    if (NO % 4 == 0) {
#pragma unroll
      for (int q = 0; q < NO; q += 4) {
        const float4 v = *reinterpret_cast<const float4*>(w + k * WP + q);
        wv[q] = v.x; wv[q + (NO > 1 ? 1 : 0)] = v.y; wv[q + (NO > 2 ? 2 : 0)] = v.z; wv[q + (NO > 3 ? 3 : 0)] = v.w;
      }
    } else {
#pragma unroll
      for (int q = 0; q < NO; ++q) wv[q] = w[k * WP + q];
    }
#pragma unroll
    for (int q = 0; q < NO; ++q) {
      const float2 ww = make_float2(wv[q], wv[q]);
      lo[q] = __ffma2_rn(ww, make_float2(h.x, h.y), lo[q]);
      hi[q] = __ffma2_rn(ww, make_float2(h.z, h.w), hi[q]);
    }
  }
#pragma unroll
  for (int q = 0; q < NO; ++q) acc[q] = make_float4(lo[q].x, lo[q].y, hi[q].x, hi[q].y);
}
__device__ __forceinline__ float4 relu4(float4 a) {
  return make_float4(fmaxf(a.x, 0.0f), fmaxf(a.y, 0.0f), fmaxf(a.z, 0.0f), fmaxf(a.w, 0.0f));
}
// a where the ReLU output h is positive, else 0
__device__ __forceinline__ float4 mask4(float4 a, float4 h) {
  return make_float4(h.x > 0.0f ? a.x : 0.0f, h.y > 0.0f ? a.y : 0.0f, h.z > 0.0f ? a.z : 0.0f,
                     h.w > 0.0f ? a.w : 0.0f);
}
// acc += sum of the products of four samples, in sample order
__device__ __forceinline__ void dot4(float4 a, float4 b, float& acc) {
  acc = fmaf(a.x, b.x, acc);
  acc = fmaf(a.y, b.y, acc);
  acc = fmaf(a.z, b.z, acc);
  acc = fmaf(a.w, b.w, acc);
}

__global__ void __launch_bounds__(kT, 1) mlp_bwd_kernel(const double* __restrict__ X, const uint8_t* __restrict__ y,
                                                        long long n, const float* __restrict__ params,
                                                        float* __restrict__ partial, double* __restrict__ partial_loss) {
  extern __shared__ __align__(16) float sm[];
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  for (int l = 0; l < 5; ++l) {
    const int nin = wid(l), nout = wid(l + 1);
    float* Tr = sm + (l == 0 ? kOffT1 : l == 1 ? kOffT2 : l == 2 ? kOffT3 : kOffT4);
    float* W = sm + (l == 1 ? kOffW2 : l == 2 ? kOffW3 : l == 3 ? kOffW4 : kOffW5);
    float* B = sm + kOffB + (l == 0 ? 0 : l == 1 ? 64 : l == 2 ? 96 : l == 3 ? 112 : 120);
    for (int e = t; e < nin * nout; e += kT) {
      const float w = params[wofs(l) + e];
      if (l < 4) Tr[(e % nin) * nout + e / nin] = w;
      if (l > 0) W[e] = w;
    }
    for (int e = t; e < nout; e += kT) B[e] = params[wofs(l) + nin * nout + e];
  }
  // gradient sums of this warp's samples; lane's elements:
  float g2[8][8];   // W2[o = 4 qo + lane/8][i = 8 qi + lane%8]
  float g3[4][4];   // W3[o = 4 qo + lane/8][i = 8 qi + lane%8]
  float g1[2][7];   // W1 and b1 of units lane, lane + 32
  float g4[4];      // W4[lane/4][4 q + lane%4]
  float g5 = 0.0f;  // W5[lane/8][lane%8]
  float gb2 = 0.0f, gbx = 0.0f;  // b2[lane]; b3, b4, b5 (lanes 0-15, 16-23, 24-27)
#pragma unroll
  for (int a = 0; a < 8; ++a)
#pragma unroll
    for (int b = 0; b < 8; ++b) g2[a][b] = 0.0f;
#pragma unroll
  for (int a = 0; a < 4; ++a) {
    g4[a] = 0.0f;
#pragma unroll
    for (int b = 0; b < 4; ++b) g3[a][b] = 0.0f;
  }
#pragma unroll
  for (int a = 0; a < 2; ++a)
#pragma unroll
    for (int b = 0; b < 7; ++b) g1[a][b] = 0.0f;
  double loss = 0.0;
  const float inv_nS = (float)(1.0 / (4.0 * (double)n));
  const long long tiles = (n + kS - 1) / kS;
  float* col = sm + 4 * lane;  // this lane's four samples in every row
  for (long long tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
    // ---- Eq. (normalizainput); dead samples of the last tile are zeros
    const long long s = tile * kS + t;
    const bool live = t < kS && s < n;
    unsigned lab = 0u;
    __syncthreads();  // the last tile's rows are no longer read
    if (t < kS) {
      float x[6], m = 1.0f;
#pragma unroll
      for (int j = 0; j < 6; ++j) {
        x[j] = live ? (float)X[s * 6 + j] : 0.0f;
        m = fmaxf(m, fabsf(x[j]));
      }
      lab = live ? y[s] : 0u;
#pragma unroll
      for (int j = 0; j < 6; ++j) sm[(kX0 + j) * kPitch + t] = x[j] / m;
    }
    __syncthreads();
    // ---- forward (Eqs. (reconstuction), (activationfunction))
    {
      float4 a[8];
      rows4<6, 8, 64>(col + kX0 * kPitch, sm + kOffT1 + 8 * warp, sm + kOffB + 8 * warp, a);
#pragma unroll
      for (int q = 0; q < 8; ++q) *reinterpret_cast<float4*>(col + (kX1 + 8 * warp + q) * kPitch) = relu4(a[q]);
    }
    __syncthreads();
    {
      float4 a[4];
      rows4<64, 4, 32>(col + kX1 * kPitch, sm + kOffT2 + 4 * warp, sm + kOffB + 64 + 4 * warp, a);
#pragma unroll
      for (int q = 0; q < 4; ++q) *reinterpret_cast<float4*>(col + (kX2 + 4 * warp + q) * kPitch) = relu4(a[q]);
    }
    __syncthreads();
    {
      float4 a[2];
      rows4<32, 2, 16>(col + kX2 * kPitch, sm + kOffT3 + 2 * warp, sm + kOffB + 96 + 2 * warp, a);
#pragma unroll
      for (int q = 0; q < 2; ++q) *reinterpret_cast<float4*>(col + (kX3 + 2 * warp + q) * kPitch) = relu4(a[q]);
    }
    __syncthreads();
    {
      float4 a[1];
      rows4<16, 1, 8>(col + kX3 * kPitch, sm + kOffT4 + warp, sm + kOffB + 112 + warp, a);
      *reinterpret_cast<float4*>(col + (kX4 + warp) * kPitch) = relu4(a[0]);
    }
    __syncthreads();
    // ---- output: loss, dL/dz = (sigma(z) - y) / (n S), and layer 4's delta
    if (t < kS) {
      float h4[8], d5[4];
#pragma unroll
      for (int i = 0; i < 8; ++i) h4[i] = sm[(kX4 + i) * kPitch + t];
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        float z = sm[kOffB + 120 + k];
#pragma unroll
        for (int i = 0; i < 8; ++i) z = fmaf(sm[kOffW5 + k * 8 + i], h4[i], z);
        const float yk = (float)((lab >> k) & 1u);
        const float sig = 1.0f / (1.0f + __expf(-z));
        // -[y log s + (1-y) log(1-s)] = softplus(z) - y z
        if (live) loss += (double)(softplus(z) - yk * z);
        d5[k] = live ? (sig - yk) * inv_nS : 0.0f;
        sm[(kD5 + k) * kPitch + t] = d5[k];
      }
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        float a = 0.0f;
#pragma unroll
        for (int k = 0; k < 4; ++k) a = fmaf(sm[kOffW5 + k * 8 + i], d5[k], a);
        sm[(kD4 + i) * kPitch + t] = h4[i] > 0.0f ? a : 0.0f;
      }
    }
    __syncthreads();
    // ---- deltas: (W_{l+1}^T delta_{l+1}) * relu'
    {
      float4 a[2];
      rows4<8, 2, 16>(col + kD4 * kPitch, sm + kOffW4 + 2 * warp, nullptr, a);
#pragma unroll
      for (int q = 0; q < 2; ++q)
        *reinterpret_cast<float4*>(col + (kD3 + 2 * warp + q) * kPitch) =
            mask4(a[q], *reinterpret_cast<const float4*>(col + (kX3 + 2 * warp + q) * kPitch));
    }
    __syncthreads();
    {
      float4 a[4];
      rows4<16, 4, 32>(col + kD3 * kPitch, sm + kOffW3 + 4 * warp, nullptr, a);
#pragma unroll
      for (int q = 0; q < 4; ++q)
        *reinterpret_cast<float4*>(col + (kD2 + 4 * warp + q) * kPitch) =
            mask4(a[q], *reinterpret_cast<const float4*>(col + (kX2 + 4 * warp + q) * kPitch));
    }
    __syncthreads();
    {
      float4 a[8];
      rows4<32, 8, 64>(col + kD2 * kPitch, sm + kOffW2 + 8 * warp, nullptr, a);
#pragma unroll
      for (int q = 0; q < 8; ++q)
        *reinterpret_cast<float4*>(col + (kD1 + 8 * warp + q) * kPitch) =
            mask4(a[q], *reinterpret_cast<const float4*>(col + (kX1 + 8 * warp + q) * kPitch));
    }
    __syncthreads();
    // ---- parameter gradients over this warp's 16 samples: dW = delta^T x, db = sum delta
    const int hb = lane >> 3, lb = lane & 7;
#pragma unroll 1
    for (int c = 0; c < 16; c += 4) {
      const float* st = sm + 16 * warp + c;
      auto row = [&](int r) { return *reinterpret_cast<const float4*>(st + r * kPitch); };
      {
        float4 d[8];
#pragma unroll
        for (int qo = 0; qo < 8; ++qo) d[qo] = row(kD2 + 4 * qo + hb);
#pragma unroll
        for (int qi = 0; qi < 8; ++qi) {
          const float4 h = row(kX1 + 8 * qi + lb);
#pragma unroll
          for (int qo = 0; qo < 8; ++qo) dot4(d[qo], h, g2[qo][qi]);
        }
      }
      {
        float4 d[4];
#pragma unroll
        for (int qo = 0; qo < 4; ++qo) d[qo] = row(kD3 + 4 * qo + hb);
#pragma unroll
        for (int qi = 0; qi < 4; ++qi) {
          const float4 h = row(kX2 + 8 * qi + lb);
#pragma unroll
          for (int qo = 0; qo < 4; ++qo) dot4(d[qo], h, g3[qo][qi]);
        }
      }
      const float4 one = make_float4(1.0f, 1.0f, 1.0f, 1.0f);
      {
        const float4 d0 = row(kD1 + lane), d1 = row(kD1 + 32 + lane);
#pragma unroll
        for (int i = 0; i < 6; ++i) {
          const float4 x = row(kX0 + i);
          dot4(d0, x, g1[0][i]);
          dot4(d1, x, g1[1][i]);
        }
        dot4(d0, one, g1[0][6]);
        dot4(d1, one, g1[1][6]);
      }
      {
        const float4 d = row(kD4 + (lane >> 2));
#pragma unroll
        for (int q = 0; q < 4; ++q) dot4(d, row(kX3 + 4 * q + (lane & 3)), g4[q]);
      }
      dot4(row(kD5 + hb), row(kX4 + lb), g5);
      dot4(row(kD2 + lane), one, gb2);
      dot4(row(lane < 16 ? kD3 + lane : lane < 24 ? kD4 + lane - 16 : kD5 + (lane & 3)), one, gbx);
    }
  }
  // ---- the warps' sums, added in warp order
  __syncthreads();
  {
    float* w = sm + warp * kNetParams;
    const int hb = lane >> 3, lb = lane & 7;
#pragma unroll
    for (int qo = 0; qo < 8; ++qo)
#pragma unroll
      for (int qi = 0; qi < 8; ++qi) w[wofs(1) + (4 * qo + hb) * 64 + 8 * qi + lb] = g2[qo][qi];
#pragma unroll
    for (int qo = 0; qo < 4; ++qo)
#pragma unroll
      for (int qi = 0; qi < 4; ++qi) w[wofs(2) + (4 * qo + hb) * 32 + 8 * qi + lb] = g3[qo][qi];
#pragma unroll
    for (int a = 0; a < 2; ++a) {
#pragma unroll
      for (int i = 0; i < 6; ++i) w[(lane + 32 * a) * 6 + i] = g1[a][i];
      w[384 + lane + 32 * a] = g1[a][6];
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) w[wofs(3) + (lane >> 2) * 16 + 4 * q + (lane & 3)] = g4[q];
    w[wofs(4) + lane] = g5;
    w[wofs(1) + 2048 + lane] = gb2;
    if (lane < 28) w[lane < 16 ? wofs(2) + 512 + lane : lane < 24 ? wofs(3) + 128 + lane - 16 : wofs(4) + 32 + lane - 24] = gbx;
  }
  __syncthreads();
  for (int p = t; p < kNetParams; p += kT) {
    float a = 0.0f;
#pragma unroll
    for (int w = 0; w < kWarps; ++w) a += sm[w * kNetParams + p];
    partial[(size_t)blockIdx.x * kNetParams + p] = a;
  }
  // block loss (fixed-order tree in shared memory)
  __shared__ double sl[kS];
  if (t < kS) sl[t] = loss;
  __syncthreads();
  for (int w = kS / 2; w > 0; w >>= 1) {
    if (t < w) sl[t] += sl[t + w];
    __syncthreads();
  }
  if (t == 0) partial_loss[blockIdx.x] = sl[0];
}

// grad[p] = scale * sum_b partial[b][p], loss likewise, in a fixed order
// (deterministic): eight runs of consecutive CTAs, each in order, then the runs
// in order.  scale is 1 for partial sums of deltas that carry the 1/(n S) of the
// mean, 1/(n S) for sums of unscaled deltas.  Latency-bound on its loads: eight
// threads per parameter with several loads in flight each, against one thread
// adding up to 304 values in turn.
constexpr int kRedP = 32, kRedR = 8;  // parameters and runs per CTA
__global__ void __launch_bounds__(kRedP * kRedR)
    mlp_bwd_reduce_kernel(const float* __restrict__ partial, const double* __restrict__ partial_loss, int blocks,
                          long long n, float scale, float* __restrict__ grad, float* loss) {
  __shared__ float run[kRedR][kRedP];
  __shared__ double lrun[kRedR];
  const int q = threadIdx.x % kRedP, r = threadIdx.x / kRedP;
  const int p = blockIdx.x * kRedP + q;
  const int per = (blocks + kRedR - 1) / kRedR;
  const int b0 = min(r * per, blocks), b1 = min(b0 + per, blocks);
  float a = 0.0f;
  if (p < kNetParams) {
#pragma unroll 8
    for (int b = b0; b < b1; ++b) a += partial[(size_t)b * kNetParams + p];
  }
  run[r][q] = a;
  if (blockIdx.x == 0 && q == 0) {
    double l = 0.0;
#pragma unroll 8
    for (int b = b0; b < b1; ++b) l += partial_loss[b];
    lrun[r] = l;
  }
  __syncthreads();
  if (r == 0 && p < kNetParams) {
    float g = 0.0f;
#pragma unroll
    for (int w = 0; w < kRedR; ++w) g += run[w][q];
    grad[p] = g * scale;
  }
  if (blockIdx.x == 0 && threadIdx.x == 0 && loss) {
    double l = 0.0;
#pragma unroll
    for (int w = 0; w < kRedR; ++w) l += lrun[w];
    *loss = (float)(l / (4.0 * (double)n));
  }
}

}  // namespace

int mlp_bwd_blocks(long long n) {
  const long long tiles = (n + kS - 1) / kS;
  return (int)(tiles < 152 ? tiles : 152);
}

// Partial sums of up to 2 x 152 CTAs (the tensor-core kernel runs two per SM).
size_t mlp_bwd_scratch_bytes(long long n) {
  const long long tiles = (n + kS - 1) / kS;
  const size_t b = (size_t)(tiles < 2 * 152 ? tiles : 2 * 152);
  return b * kNetParams * sizeof(float) + b * sizeof(double);
}

cudaError_t launch_mlp_bwd(const double* X, const uint8_t* y, long long n, const float* params, float* grad,
                           float* loss, void* scratch, cudaStream_t s) {
  const int blocks = mlp_bwd_blocks(n);
  float* partial = static_cast<float*>(scratch);
  double* partial_loss = reinterpret_cast<double*>(static_cast<char*>(scratch) +
                                                   (size_t)blocks * kNetParams * sizeof(float));
  const size_t smem = (size_t)kSmemFloats * sizeof(float);
  cudaError_t e = cudaFuncSetAttribute(mlp_bwd_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  mlp_bwd_kernel<<<blocks, kT, smem, s>>>(X, y, n, params, partial, partial_loss);
  e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  return launch_mlp_bwd_reduce(partial, partial_loss, blocks, n, 1.0f, grad, loss, s);
}

cudaError_t launch_mlp_bwd_reduce(const float* partial, const double* partial_loss, int blocks, long long n,
                                  float scale, float* grad, float* loss, cudaStream_t s) {
  mlp_bwd_reduce_kernel<<<(kNetParams + kRedP - 1) / kRedP, kRedP * kRedR, 0, s>>>(partial, partial_loss, blocks, n,
                                                                                   scale, grad, loss);
  return cudaGetLastError();
}

}  // namespace neno6
