// Certified FP32 evaluation of the 6-64-32-16-8-4 classifier (Sec. 3.1) for
// the FP64 paths.  Those paths need the classifier for four bits only -- the
// signs of the logits that the binary64 network yields in the canonical order
// -- and GB300's FP32 pipe runs at 61 times its FP64 pipe's rate.  So the
// network is evaluated in FP32 together with a bound on the distance of its
// logits from the binary64 ones; a logit beyond the bound has the binary64
// logit's sign, and every other row is evaluated again in binary64 in the
// canonical order (mlp64_warp / mlp64_rows below).  The bits are the binary64
// network's, always.
//
// The bound (forward error analysis of a fixed-order FMA chain, Higham,
// "Accuracy and Stability of Numerical Algorithms", ch. 3).  A unit of n
// inputs is its bias followed by n FMAs, on weights rounded to FP32, so with
// u = 2^-24 its computed pre-activation differs from the exact one of the
// same computed inputs h by at most
//   sum_j (n - j + 2) u |w_j| |h_j| + (n + 1) u |b|,    j = 1..n,
// up to O(u^2).  ReLU does not enlarge a difference, and layers l+1..5 carry
// one of layer l to logit k multiplied by at most G_l = |W5| ... |W_{l+1}|.
// Summed over the layers the bound is linear in the computed hidden values
// (all >= 0) and inputs:
//   |error of logit k| <= k0 + sum_j kin_j |x_j| + sum_l sum_i kappa_l,i h_l,i,
// one more FMA per hidden unit.  The coefficients (build_filter_kappa, on the
// host in binary64) take the maximum over the four logits after dividing
// logit k's row of W5 and b5 by its share rho_k of a static bound, which
// changes no sign and makes one bound serve all four.  They include the
// input's conversion (8 u relative: two truncations to 24 bits, a reciprocal
// to 1 ulp and a product), underflow (every |w|, |b| counted as at least
// 2^-125) and a factor 1.01 for the O(u^2) terms, the binary64 network's own
// rounding (2^-29 of the FP32 bound) and the rounding of the bound itself.
// A row whose inputs leave [0, 2^100], or any of whose logits or whose bound
// is not finite, is never certified.
#pragma once

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

// The network of R rows per thread against the table T in shared memory (the
// kFilt* layout; every lane reads the same address).  Outputs packed in pairs
// (fma.rn.f32x2 rounds each half like a scalar FMA).  Returns per row the eta
// bits in bits 0-3 and, in bit 4, whether they are certified.
template <int R>
__device__ __forceinline__ void filter_rows(const float* __restrict__ T, const float (&x)[R][6],
                                            unsigned (&res)[R]) {
  float err[R];
  {
    const float4 e0 = *reinterpret_cast<const float4*>(T + kFiltIn);
    const float4 e1 = *reinterpret_cast<const float4*>(T + kFiltIn + 4);
#pragma unroll
    for (int r = 0; r < R; ++r) {
      float e = e0.x;  // k0, then the six inputs
      e = fmaf(e0.y, fabsf(x[r][0]), e);
      e = fmaf(e0.z, fabsf(x[r][1]), e);
      e = fmaf(e0.w, fabsf(x[r][2]), e);
      e = fmaf(e1.x, fabsf(x[r][3]), e);
      e = fmaf(e1.y, fabsf(x[r][4]), e);
      err[r] = fmaf(e1.z, fabsf(x[r][5]), e);
    }
  }
  float2 a[R][16];
#pragma unroll
  for (int q = 0; q < 16; ++q) {
    const float2 b = reinterpret_cast<const float2*>(T + kFiltB2)[q];
#pragma unroll
    for (int r = 0; r < R; ++r) a[r][q] = b;
  }
  // layers 1 and 2 fused: hidden unit i of layer 1 goes into the 32 sums of
  // layer 2 (each sum's order: bias, then inputs in ascending order).  The
  // weights of the first 16 sums and of layer 1 are loaded one unit ahead, the
  // others while the unit's layer 1 runs: a pass of a warp alone on its SM
  // quarter takes 7.4-8.5 k clocks instead of 10.7 k.
  float4 w0 = *reinterpret_cast<const float4*>(T + kFiltW1);
  float4 w1 = *reinterpret_cast<const float4*>(T + kFiltW1 + 4);  // w4, w5, bias, kappa
  float4 wa[4], wb[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) wa[q] = *reinterpret_cast<const float4*>(T + kFiltW2 + 4 * q);
#pragma unroll 1
  for (int i = 0; i < 64; ++i) {
#pragma unroll
    for (int q = 0; q < 4; ++q) wb[q] = *reinterpret_cast<const float4*>(T + kFiltW2 + 32 * i + 16 + 4 * q);
    float2 h[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
      float v = fmaf(w0.x, x[r][0], w1.z);
      v = fmaf(w0.y, x[r][1], v);
      v = fmaf(w0.z, x[r][2], v);
      v = fmaf(w0.w, x[r][3], v);
      v = fmaf(w1.x, x[r][4], v);
      v = fmaf(w1.y, x[r][5], v);
      v = fmaxf(v, 0.0f);
      err[r] = fmaf(w1.w, v, err[r]);
      h[r] = make_float2(v, v);
    }
    const int nx = min(i + 1, 63);
    w0 = *reinterpret_cast<const float4*>(T + kFiltW1 + 8 * nx);
    w1 = *reinterpret_cast<const float4*>(T + kFiltW1 + 8 * nx + 4);
#pragma unroll
    for (int q = 0; q < 4; ++q)
#pragma unroll
      for (int r = 0; r < R; ++r) {
        a[r][2 * q] = __ffma2_rn(make_float2(wa[q].x, wa[q].y), h[r], a[r][2 * q]);
        a[r][2 * q + 1] = __ffma2_rn(make_float2(wa[q].z, wa[q].w), h[r], a[r][2 * q + 1]);
      }
#pragma unroll
    for (int q = 0; q < 4; ++q) wa[q] = *reinterpret_cast<const float4*>(T + kFiltW2 + 32 * nx + 4 * q);
#pragma unroll
    for (int q = 0; q < 4; ++q)
#pragma unroll
      for (int r = 0; r < R; ++r) {
        a[r][8 + 2 * q] = __ffma2_rn(make_float2(wb[q].x, wb[q].y), h[r], a[r][8 + 2 * q]);
        a[r][9 + 2 * q] = __ffma2_rn(make_float2(wb[q].z, wb[q].w), h[r], a[r][9 + 2 * q]);
      }
  }
  float2 c[R][8];
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    const float2 b = reinterpret_cast<const float2*>(T + kFiltB3)[q];
#pragma unroll
    for (int r = 0; r < R; ++r) c[r][q] = b;
  }
#pragma unroll
  for (int i = 0; i < 32; ++i) {
    float2 h[R];
    const float kap = T[kFiltK2 + i];
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const float v = fmaxf(i & 1 ? a[r][i / 2].y : a[r][i / 2].x, 0.0f);
      err[r] = fmaf(kap, v, err[r]);
      h[r] = make_float2(v, v);
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const float4 w = *reinterpret_cast<const float4*>(T + kFiltW3 + 16 * i + 4 * q);
#pragma unroll
      for (int r = 0; r < R; ++r) {
        c[r][2 * q] = __ffma2_rn(make_float2(w.x, w.y), h[r], c[r][2 * q]);
        c[r][2 * q + 1] = __ffma2_rn(make_float2(w.z, w.w), h[r], c[r][2 * q + 1]);
      }
    }
  }
  float2 d[R][4];
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const float2 b = reinterpret_cast<const float2*>(T + kFiltB4)[q];
#pragma unroll
    for (int r = 0; r < R; ++r) d[r][q] = b;
  }
#pragma unroll
  for (int i = 0; i < 16; ++i) {
    float2 h[R];
    const float kap = T[kFiltK3 + i];
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const float v = fmaxf(i & 1 ? c[r][i / 2].y : c[r][i / 2].x, 0.0f);
      err[r] = fmaf(kap, v, err[r]);
      h[r] = make_float2(v, v);
    }
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const float4 w = *reinterpret_cast<const float4*>(T + kFiltW4 + 8 * i + 4 * q);
#pragma unroll
      for (int r = 0; r < R; ++r) {
        d[r][2 * q] = __ffma2_rn(make_float2(w.x, w.y), h[r], d[r][2 * q]);
        d[r][2 * q + 1] = __ffma2_rn(make_float2(w.z, w.w), h[r], d[r][2 * q + 1]);
      }
    }
  }
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const float4 b = *reinterpret_cast<const float4*>(T + kFiltB5);
    float z[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const float v = fmaxf(i & 1 ? d[r][i / 2].y : d[r][i / 2].x, 0.0f);
      err[r] = fmaf(T[kFiltK4 + i], v, err[r]);
      const float4 w = *reinterpret_cast<const float4*>(T + kFiltW5 + 4 * i);
      z[0] = fmaf(w.x, v, z[0]);
      z[1] = fmaf(w.y, v, z[1]);
      z[2] = fmaf(w.z, v, z[2]);
      z[3] = fmaf(w.w, v, z[3]);
    }
    unsigned eta = 0u;
    bool sure = true;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      eta |= (z[k] > 0.0f ? 1u : 0u) << k;
      sure = sure && fabsf(z[k]) > err[r] && fabsf(z[k]) <= 3.0e38f;
    }
    res[r] = eta | (sure ? 16u : 0u);
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
// apart; ws: 128 doubles of the warp's scratch.  Returns the eta bits in all
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
    for (int j = 0; j < 6; ++j) ws[120 + j] = x[j];
  }
  __syncwarp();
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    const int o = lane + 32 * q;
    double h = Wt[384 + o];
#pragma unroll
    for (int k = 0; k < 6; ++k) h = __fma_rn(Wt[k * 64 + o], ws[120 + k], h);
    ws[o] = relu(h);
  }
  __syncwarp();
  {
    double h = Wt[2496 + lane];
#pragma unroll 16
    for (int i = 0; i < 64; ++i) h = __fma_rn(Wt[448 + i * 32 + lane], ws[i], h);
    ws[64 + lane] = relu(h);
  }
  __syncwarp();
  if (lane < 16) {
    double h = Wt[3040 + lane];
#pragma unroll 16
    for (int i = 0; i < 32; ++i) h = __fma_rn(Wt[2528 + i * 16 + lane], ws[64 + i], h);
    ws[96 + lane] = relu(h);
  }
  __syncwarp();
  if (lane < 8) {
    double h = Wt[3184 + lane];
#pragma unroll
    for (int i = 0; i < 16; ++i) h = __fma_rn(Wt[3056 + i * 8 + lane], ws[96 + i], h);
    ws[112 + lane] = relu(h);
  }
  __syncwarp();
  bool bit = false;
  if (lane < 4) {
    double z = Wt[3224 + lane];
#pragma unroll
    for (int i = 0; i < 8; ++i) z = __fma_rn(Wt[3192 + i * 4 + lane], ws[112 + i], z);
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
