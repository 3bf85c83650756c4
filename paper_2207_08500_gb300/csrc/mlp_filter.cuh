// Certified evaluation of the 6-64-32-16-8-4 classifier (Sec. 3.1) for the FP64
// paths.  Those paths need the classifier for four bits only -- the signs of the
// logits that the binary64 network yields in the canonical order -- and GB300's
// FP32 and tensor pipes run at 61 and several hundred times its FP64 pipe's
// rate.  So the network is evaluated in FP32 (layer 1) and in split 16-bit
// products with FP32 accumulation (layers 2 to 5), together with a bound on the
// distance of its logits from the binary64 ones; a logit beyond the bound has
// the binary64 logit's sign, and every other row is evaluated again in binary64
// in the canonical order (mlp64_warp / mlp64_rows below).  The bits are the
// binary64 network's, always.
//
// Each FP32 value v of layers 2 to 5 (weights and inputs) is split into two
// binary16 terms, v = hi + lo + d, and a product is hi hi' + lo hi' + hi lo':
// warp-level matrix instructions (16 rows x 8 outputs x 16 inputs, three per block
// of 16 inputs), whose operands and results stay in registers.  They fit this
// kernel: a warp's 64 rows (32 faces, two sides) need no barrier, no tensor memory
// and no wait on other warps, and at 2 clocks per instruction and SM they take a
// quarter of the FP64 time beside which they run.  2048^2 RHS: 11.70 ms, against
// 13.8 ms with every layer in FP32 on the CUDA cores (weights by broadcast loads,
// which bound it).
//
// The bound (forward error analysis, Higham, "Accuracy and Stability of
// Numerical Algorithms", ch. 3), u = 2^-24.  Layer 1: a bias and six FMAs on
// weights rounded to FP32 differ from the exact value of the same inputs x by at
// most
//   sum_j (6 - j + 2) u |w_j| |x_j| + 7 u |b|,   j = 1..6.
// A layer above takes its inputs in blocks of 16; a block's sum starts at 0, takes
// the products with a lo term in two instructions, those of the hi terms in a
// third, and is added to the blocks before it, which start at the bias.
//  * Splitting: binary16 keeps 11 bits, so lo is at most 2^-11 |v| and d at most
//    2 u |v| + 2^-25 (hi + lo need not reach 24 bits: 1 + 2^-12 + 2^-23).  Of the
//    weight both are known, |lo| and dw; with s = |hi| + |lo| of the weight a product
//    is off by 2 u s |h| for the input's split, dw |h| for the weight's, and
//    2^-11 |lo| |h| for the dropped lo lo'; besides 2^-25 (s + |lo|).
//  * An instruction sums the accumulator and at most n = 16 products (8 in layer 5),
//    themselves exact.  All that is promised is at least single precision, in any
//    order and with any rounding.  Additions one after the other, cut off at 24 bits,
//    lose 2 u each, n of them.  Sums of a group of addends, aligned to the largest and
//    cut off below its 24 bits, are what has been found (Fasi, Higham, Mikaitis and
//    Pranesh, "Numerical behavior of NVIDIA tensor cores", PeerJ CS 7:e330), in groups
//    of 4, 8 or 16 products and the sum before: the largest is kept whole, the others
//    lose 2 u of it each, and 2 u for the group's result, (2 n + 2 n / 4) u at most.
//    So an instruction loses at most 40 u (20 u) of the magnitudes it sums.  The first
//    two work on magnitudes 2^-10 of the third's: only that one counts.  Were all
//    three to work on the layer's whole sum, as they may, a layer of 64 inputs would
//    lose twelve times as much: three times as many rows would stay undecided (200 x
//    136 with 36 u each: 189 us, 153 with a sum per block).
//  * Of B blocks an addition rounds block k and those before it, B - k times.
// Together the unit is off by at most
//   sum_j ((40 + B - k_j + 2) u s_j + dw_j + 2^-11 |lo_j|) |h_j|
//     + 2^-25 sum_j (s_j + |lo_j|) + (B + 1) u |b|
// up to O(u^2) and relative 2^-8.  ReLU does not enlarge a difference, and layers
// l+1..5 carry one of layer l to logit k multiplied by at most
// G_l = |W5| ... |W_{l+1}|.  Summed over the layers the bound is linear in the
// computed hidden values (all >= 0) and inputs:
//   |error of logit k| <= k0 + sum_j kin_j |x_j| + sum_l sum_i kappa_l,i h_l,i,
// one more FMA per hidden unit.  The coefficients (build_filter_kappa, on the
// host in binary64) take the maximum over the four logits after dividing
// logit k's row of W5 and b5 by its share rho_k of a static bound, which
// changes no sign and makes one bound serve all four.  They include the
// input's conversion (8 u relative: two truncations to 24 bits, a reciprocal
// to 1 ulp and a product), underflow (every |w|, |b| counted as at least
// 2^-125, and 2^-125 for each of a block's four sums) and a factor 1.01 for the
// O(u^2) and 2^-8 terms, the binary64 network's own rounding (2^-28 of the bound)
// and the rounding of the bound itself.
// A row whose inputs leave [0, 2^100], or any of whose logits or whose bound
// is not finite (a value outside the binary16 range makes it so), is never
// certified.
#pragma once

#include <cuda_fp16.h>

#include "fp64_ops.cuh"
#include "internal.h"

namespace neno6 {
namespace filt {

using namespace f64ops;

// Truncate a binary64 value to binary32 on the integer pipe: |result| <= |x|,
// relative error below 2^-23 for 2^-126 <= |x| < 2^127, 0 below; `top`
// collects the largest exponent field (values from 2^100 on, infinities and
// NaN are not certified and need no meaningful result).
__device__ __forceinline__ float trunc32(double x, unsigned& top) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  const unsigned hi = (unsigned)(b >> 32), lo = (unsigned)b;
  const unsigned mag = hi & 0x7fffffffu;
  top = max(top, mag);
  const unsigned f = (((__funnelshift_l(lo, hi, 3)) ^ 0x40000000u) & 0x7fffffffu) | (hi & 0x80000000u);
  return __uint_as_float(mag < (897u << 20) ? 0u : f);
}
constexpr unsigned kTopLimit = (1023u + 100u) << 20;

// FP32 input of the network for the stencil s (Eq. (normalizainput)); false
// when a value is too large to certify.
__device__ __forceinline__ bool filter_input(const double (&s)[6], float (&x)[6]) {
  unsigned top = 0u;
  float m = 1.0f;
#pragma unroll
  for (int j = 0; j < 6; ++j) {
    x[j] = trunc32(s[j], top);
    m = fmaxf(m, fabsf(x[j]));
  }
  float inv;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(inv) : "f"(m));
#pragma unroll
  for (int j = 0; j < 6; ++j) x[j] *= inv;
  return top < kTopLimit;
}

// d += a b: 16 rows x 16 inputs times 16 inputs x 8 outputs, binary16 operands,
// FP32 accumulators.  Lane 4 g + q holds of d: rows g (first two) and g + 8,
// outputs 2 q, 2 q + 1; of a: the pairs of inputs 2 q, 2 q + 1 of rows g and g +
// 8, then the pairs 2 q + 8, 2 q + 9; of b: the same pairs of output g.
__device__ __forceinline__ void mma16(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
// ReLU that keeps NaN: a value outside the binary16 range splits into infinities
// of both signs, whose products are NaN, and reaches the logits as NaN.
__device__ __forceinline__ float relu_nan(float x) {
  float y;
  asm("max.NaN.f32 %0, %1, 0f00000000;" : "=f"(y) : "f"(x));
  return y;
}
// Split a pair of FP32 values into packed binary16 terms.
__device__ __forceinline__ void split16(float x, float y, uint32_t& hi, uint32_t& lo) {
  const __half2 h = __floats2half2_rn(x, y);
  const float2 f = __half22float2(h);
  const __half2 l = __floats2half2_rn(x - f.x, y - f.y);
  hi = *reinterpret_cast<const uint32_t*>(&h);
  lo = *reinterpret_cast<const uint32_t*>(&l);
}
// One block of 16 inputs (pairs p: rows g, g + 8 of inputs 2q.., then of 2q + 8..)
// into NT tiles of 8 outputs of both row tiles: T points at the block's weights,
// per tile and lane hi b0, b1, lo b0, b1.  The block's sum starts at 0 and takes
// the small terms first; see the bound above.
template <int NT>
__device__ __forceinline__ void block16(float (&acc)[2][NT][4], const uint32_t (&hi)[2][4], const uint32_t (&lo)[2][4],
                                        const float* T, int lane) {
  uint4 b[NT];
  float s[NT][2][4];
#pragma unroll
  for (int nt = 0; nt < NT; ++nt) {
    b[nt] = reinterpret_cast<const uint4*>(T)[32 * nt + lane];
#pragma unroll
    for (int mt = 0; mt < 2; ++mt) s[nt][mt][0] = s[nt][mt][1] = s[nt][mt][2] = s[nt][mt][3] = 0.0f;
  }
  // term by term: the instructions on one sum are 2 NT apart
#pragma unroll
  for (int nt = 0; nt < NT; ++nt)
#pragma unroll
    for (int mt = 0; mt < 2; ++mt) mma16(s[nt][mt], lo[mt], b[nt].x, b[nt].y);
#pragma unroll
  for (int nt = 0; nt < NT; ++nt)
#pragma unroll
    for (int mt = 0; mt < 2; ++mt) mma16(s[nt][mt], hi[mt], b[nt].z, b[nt].w);
#pragma unroll
  for (int nt = 0; nt < NT; ++nt)
#pragma unroll
    for (int mt = 0; mt < 2; ++mt) mma16(s[nt][mt], hi[mt], b[nt].x, b[nt].y);
#pragma unroll
  for (int nt = 0; nt < NT; ++nt)
#pragma unroll
    for (int mt = 0; mt < 2; ++mt)
#pragma unroll
      for (int r = 0; r < 4; ++r) acc[mt][nt][r] += s[nt][mt][r];
}
// Accumulators start at the biases of their outputs.
template <int NT>
__device__ __forceinline__ void start16(float (&acc)[2][NT][4], const float* B, int q) {
#pragma unroll
  for (int nt = 0; nt < NT; ++nt) {
    const float2 b = reinterpret_cast<const float2*>(B)[4 * nt + q];
#pragma unroll
    for (int mt = 0; mt < 2; ++mt) {
      acc[mt][nt][0] = acc[mt][nt][2] = b.x;
      acc[mt][nt][1] = acc[mt][nt][3] = b.y;
    }
  }
}
// ReLU of one tile of outputs (8 nt ..) of a layer, its share of the bound, and
// its terms as half (`h` = 0, 1) of the next layer's block of 16 inputs.
template <int NT>
__device__ __forceinline__ void next16(const float (&acc)[2][NT][4], int nt, int h, const float* K, int q,
                                       float (&err)[4], uint32_t (&hi)[2][4], uint32_t (&lo)[2][4]) {
  const float2 k = reinterpret_cast<const float2*>(K)[4 * nt + q];
#pragma unroll
  for (int mt = 0; mt < 2; ++mt)
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      const float x = relu_nan(acc[mt][nt][2 * r]), y = relu_nan(acc[mt][nt][2 * r + 1]);
      err[2 * mt + r] = fmaf(k.x, x, err[2 * mt + r]);
      err[2 * mt + r] = fmaf(k.y, y, err[2 * mt + r]);
      split16(x, y, hi[mt][2 * h + r], lo[mt][2 * h + r]);
    }
}

// The network for a warp's 64 rows: lane l's rows x[0], x[1] (the two sides of
// its face), against the table T in shared memory (the kFilt* layout).  Returns
// per row the eta bits in bits 0-3 and, in bit 4, whether they are certified.
// All 32 lanes call it.
__device__ __forceinline__ void filter_rows(const float* __restrict__ T, const float (&x)[2][6], unsigned (&res)[2]) {
  const int lane = threadIdx.x & 31, g = lane >> 2, q = lane & 3;
#pragma unroll 1
  for (int side = 0; side < 2; ++side) {
    // inputs of rows g, g + 8, g + 16, g + 24 (row = lane of origin)
    float xr[4][6], err[4];
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
      for (int j = 0; j < 6; ++j) xr[r][j] = __shfl_sync(0xffffffffu, side ? x[1][j] : x[0][j], g + 8 * r);
    {
      const float4 e0 = *reinterpret_cast<const float4*>(T + kFiltIn);  // k0, then the six inputs
      const float4 e1 = *reinterpret_cast<const float4*>(T + kFiltIn + 4);
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        float e = fmaf(e0.y, fabsf(xr[r][0]), e0.x);
        e = fmaf(e0.z, fabsf(xr[r][1]), e);
        e = fmaf(e0.w, fabsf(xr[r][2]), e);
        e = fmaf(e1.x, fabsf(xr[r][3]), e);
        e = fmaf(e1.y, fabsf(xr[r][4]), e);
        err[r] = q == 0 ? fmaf(e1.z, fabsf(xr[r][5]), e) : 0.0f;  // the four lanes' shares are added below
      }
    }
    uint32_t hi[2][4], lo[2][4];
    float a2[2][4][4];
    start16<4>(a2, T + kFiltB2, q);
    // layer 1 a block of 16 units at a time, straight into layer 2
#pragma unroll 1
    for (int kb = 0; kb < 4; ++kb) {
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        float v[2][4];  // units 16 kb + 8 h + 2 q + {0, 1} of the four rows
#pragma unroll
        for (int w = 0; w < 2; ++w) {
          const float* W = T + kFiltW1 + 8 * (16 * kb + 8 * h + 2 * q + w);
          const float4 w0 = *reinterpret_cast<const float4*>(W), w1 = *reinterpret_cast<const float4*>(W + 4);
#pragma unroll
          for (int r = 0; r < 4; ++r) {
            float s = fmaf(w0.x, xr[r][0], w1.z);
            s = fmaf(w0.y, xr[r][1], s);
            s = fmaf(w0.z, xr[r][2], s);
            s = fmaf(w0.w, xr[r][3], s);
            s = fmaf(w1.x, xr[r][4], s);
            s = fmaf(w1.y, xr[r][5], s);
            s = relu_nan(s);
            err[r] = fmaf(w1.w, s, err[r]);
            v[w][r] = s;
          }
        }
#pragma unroll
        for (int r = 0; r < 4; ++r) split16(v[0][r], v[1][r], hi[r >> 1][2 * h + (r & 1)], lo[r >> 1][2 * h + (r & 1)]);
      }
      block16<4>(a2, hi, lo, T + kFiltW2 + 512 * kb, lane);
    }
    float a3[2][2][4];
    start16<2>(a3, T + kFiltB3, q);
#pragma unroll
    for (int kb = 0; kb < 2; ++kb) {
      next16<4>(a2, 2 * kb, 0, T + kFiltK2, q, err, hi, lo);
      next16<4>(a2, 2 * kb + 1, 1, T + kFiltK2, q, err, hi, lo);
      block16<2>(a3, hi, lo, T + kFiltW3 + 256 * kb, lane);
    }
    float a4[2][1][4];
    start16<1>(a4, T + kFiltB4, q);
    next16<2>(a3, 0, 0, T + kFiltK3, q, err, hi, lo);
    next16<2>(a3, 1, 1, T + kFiltK3, q, err, hi, lo);
    block16<1>(a4, hi, lo, T + kFiltW4, lane);
    float z[2][1][4];
    start16<1>(z, T + kFiltB5, q);
    next16<1>(a4, 0, 0, T + kFiltK4, q, err, hi, lo);
#pragma unroll
    for (int mt = 0; mt < 2; ++mt) hi[mt][2] = hi[mt][3] = lo[mt][2] = lo[mt][3] = 0u;  // eight inputs only
    block16<1>(z, hi, lo, T + kFiltW5, lane);
    // rows' bits: lane q = 0 holds logits 0, 1 of its rows, q = 1 logits 2, 3
    unsigned w[4];
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      float e = err[r];
      e += __shfl_xor_sync(0xffffffffu, e, 1);
      e += __shfl_xor_sync(0xffffffffu, e, 2);
      const float z0 = z[r >> 1][0][2 * (r & 1)], z1 = z[r >> 1][0][2 * (r & 1) + 1];
      const bool sure = fabsf(z0) > e && fabsf(z0) <= 3.0e38f && fabsf(z1) > e && fabsf(z1) <= 3.0e38f;
      unsigned b = ((z0 > 0.0f ? 1u : 0u) | (z1 > 0.0f ? 2u : 0u)) << (2 * q) | (sure ? 0u : 16u);
      b = q < 2 ? b : 0u;
      b |= __shfl_xor_sync(0xffffffffu, b, 1);
      w[r] = b;  // complete in lanes 4 g and 4 g + 1
    }
    unsigned mine = 0u;
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const unsigned b = __shfl_sync(0xffffffffu, w[r], 4 * (lane & 7));
      if ((lane >> 3) == r) mine = b;
    }
    mine ^= 16u;
    if (side == 0) res[0] = mine;
    else res[1] = mine;
  }
}

// Start copying the table into shared memory (16-byte aligned both sides);
// table_ready() before the barrier that precedes its use.
__device__ __forceinline__ void load_filter(float* dst, const float* __restrict__ src, int t, int nt) {
  const uint32_t d = static_cast<uint32_t>(__cvta_generic_to_shared(dst));
  for (int i = t; i < kFiltFloats / 4; i += nt)
    asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"(d + 16u * i), "l"(src + 4 * i) : "memory");
}
__device__ __forceinline__ void table_ready() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// Binary64 network in the canonical order, one row per thread, weights from
// the transposed copy Wt ([in][out] per layer, then the bias): the sums of a
// layer take each input's weights as consecutive values.
__device__ __forceinline__ unsigned mlp64_rows(const double* __restrict__ Wt, const double (&x)[6]) {
  double a2[32];
#pragma unroll
  for (int o = 0; o < 32; ++o) a2[o] = Wt[2496 + o];
#pragma unroll 1
  for (int i = 0; i < 64; ++i) {
    double h = Wt[384 + i];
#pragma unroll
    for (int k = 0; k < 6; ++k) h = __fma_rn(Wt[k * 64 + i], x[k], h);
    h = relu(h);
#pragma unroll
    for (int o = 0; o < 32; ++o) a2[o] = __fma_rn(Wt[448 + i * 32 + o], h, a2[o]);
  }
  double a3[16];
#pragma unroll
  for (int o = 0; o < 16; ++o) a3[o] = Wt[3040 + o];
#pragma unroll
  for (int i = 0; i < 32; ++i) {
    const double h = relu(a2[i]);
#pragma unroll
    for (int o = 0; o < 16; ++o) a3[o] = __fma_rn(Wt[2528 + i * 16 + o], h, a3[o]);
  }
  double a4[8];
#pragma unroll
  for (int o = 0; o < 8; ++o) a4[o] = Wt[3184 + o];
#pragma unroll
  for (int i = 0; i < 16; ++i) {
    const double h = relu(a3[i]);
#pragma unroll
    for (int o = 0; o < 8; ++o) a4[o] = __fma_rn(Wt[3056 + i * 8 + o], h, a4[o]);
  }
  unsigned eta = 0u;
#pragma unroll
  for (int o = 0; o < 4; ++o) {
    double z = Wt[3224 + o];
#pragma unroll
    for (int i = 0; i < 8; ++i) z = __fma_rn(Wt[3192 + i * 4 + o], relu(a4[i]), z);
    eta |= (gt0(z) ? 1u : 0u) << o;
  }
  return eta;
}

// The same for one row by a whole warp (lane = output, each output's chain in
// the canonical order): 138 dependent FMA issues instead of 3104.  s: the
// row's six raw stencil values, readable by every lane, `sstride` doubles
// apart; ws: 72 doubles of the warp's scratch (64 hidden values, 6 inputs).  Returns the eta bits in all
// lanes.  All 32 lanes call it.
__device__ __forceinline__ unsigned mlp64_warp(const double* __restrict__ Wt, const double* s, int sstride,
                                               double* ws) {
  const int lane = threadIdx.x & 31;
  if (lane == 0) {
    double st[6], x[6];
#pragma unroll
    for (int j = 0; j < 6; ++j) st[j] = s[j * sstride];
    normalise6(st, x);
#pragma unroll
    for (int j = 0; j < 6; ++j) ws[64 + j] = x[j];
  }
  __syncwarp();
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    const int o = lane + 32 * q;
    double h = Wt[384 + o];
#pragma unroll
    for (int k = 0; k < 6; ++k) h = __fma_rn(Wt[k * 64 + o], ws[64 + k], h);
    ws[o] = relu(h);
  }
  __syncwarp();
  // each layer's values replace those two layers below
  double h2 = Wt[2496 + lane];
#pragma unroll 16
  for (int i = 0; i < 64; ++i) h2 = __fma_rn(Wt[448 + i * 32 + lane], ws[i], h2);
  __syncwarp();
  ws[lane] = relu(h2);
  __syncwarp();
  if (lane < 16) {
    double h = Wt[3040 + lane];
#pragma unroll 16
    for (int i = 0; i < 32; ++i) h = __fma_rn(Wt[2528 + i * 16 + lane], ws[i], h);
    ws[32 + lane] = relu(h);
  }
  __syncwarp();
  if (lane < 8) {
    double h = Wt[3184 + lane];
#pragma unroll
    for (int i = 0; i < 16; ++i) h = __fma_rn(Wt[3056 + i * 8 + lane], ws[32 + i], h);
    ws[lane] = relu(h);
  }
  __syncwarp();
  bool bit = false;
  if (lane < 4) {
    double z = Wt[3224 + lane];
#pragma unroll
    for (int i = 0; i < 8; ++i) z = __fma_rn(Wt[3192 + i * 4 + lane], ws[i], z);
    bit = gt0(z);
  }
  const unsigned eta = __ballot_sync(0xffffffffu, bit) & 15u;
  __syncwarp();
  return eta;
}

// Flagged lanes of a warp from which the row-per-thread form wins: it costs
// the warp 3104 FMA issues however many rows it carries, the warp form 138
// per row, and the crossover of the issue counts is at 22.
constexpr int kRowsFrom = 22;

// Binary64 bits of the rows of this warp whose lane has `need` set; the raw
// stencil of lane l starts at s0 + l, its values `sstride` doubles apart.  All
// 32 lanes call it; `eta` of the other lanes is left alone.
__device__ __forceinline__ void settle_rows(const double* __restrict__ Wt, const double* s0, int sstride,
                                            double* ws, bool need, unsigned& eta) {
  unsigned bal = __ballot_sync(0xffffffffu, need);
  if (bal == 0u) return;
  const int lane = threadIdx.x & 31;
  __syncwarp();  // the stencils were written by their own lanes
  if (__popc(bal) >= kRowsFrom) {
    if (need) {
      double st[6], x[6];
#pragma unroll
      for (int j = 0; j < 6; ++j) st[j] = s0[lane + j * sstride];
      normalise6(st, x);
      eta = mlp64_rows(Wt, x);
    }
    __syncwarp();
    return;
  }
  while (bal) {
    const int src = __ffs(bal) - 1;
    bal &= bal - 1;
    const unsigned e = mlp64_warp(Wt, s0 + src, sstride, ws);
    if (lane == src) eta = e;
  }
}

}  // namespace filt
}  // namespace neno6
