// Classifier training on the GPU (Sec. 3.3, Table 2): mini-batch Adam
// (Kingma & Ba, Algorithm 1: beta1 0.9, beta2 0.999, epsilon 1e-8) on the
// mean binary cross entropy of Eq. (Crossentropy), the batches taken in the
// order of a caller-given permutation of the samples.
//
// Mini-batch Adam is sequential (every step reads the parameters the
// previous step wrote), so one persistent cluster of CTAs runs all the steps
// of a call, sharing each step's batch (below).  No launch per step and no
// global-memory round trip of the parameters; the gradient and the loss are
// reduced in a fixed order, so a call is deterministic.  A step is bound by the
// latency of its chain (four layers forward, four back, the gradient, two
// cluster barriers): 7.1 us per step, 31.7 with four warps per CTA, weights and
// parameter sums loaded a value at a time and the new parameters read back from
// their owners.
#include "internal.h"
#include "mlp_fb.cuh"

namespace neno6 {
namespace {

using namespace mlpfb;

// The training loop on a cluster of kCl CTAs (kCl SMs): every step's batch is
// shared among the CTAs (at most kPerCta samples each).  Eight warps of a CTA
// run its samples' forward and backward pass (lane = sample, a layer's outputs
// split among the warps) and form the partial gradient of all 3228 parameters
// over them; after a cluster barrier, CTA r sums the partials of the parameter
// slice it owns over the kCl CTAs (read from their shared memory, in rank order:
// deterministic), applies Adam to that slice (its moments stay in its shared
// memory for the whole call) and writes the new values into every CTA's copy of
// the parameters; a second barrier ends the step.  A ninth warp stays off the
// chain: it fetches the next step's samples, forms the bias corrections and adds
// up the loss, the step's binary64 work.
constexpr int kCl = 8;
constexpr int kWarps = 8, kCT = 32 * kWarps, kAll = kCT + 32;  // working threads, all threads
constexpr int kPerCta = (kMaxTrainBatch + kCl - 1) / kCl;      // samples per CTA (24)
constexpr int kP = 28;  // row pitch: 16-byte aligned, eight consecutive rows in distinct banks
constexpr int kSlice = (kNetParams + kCl - 1) / kCl;           // 404 parameters per CTA
// floats: W, staged rows, partial gradient, Adam m and v, then two steps' raw
// samples (6 values, label bits and 256 where live) and loss terms, c1 and c2
constexpr int kOffW = 0, kOffSt = kNetParams, kOffPart = kOffSt + kRows * kP;
constexpr int kOffM = kOffPart + kNetParams, kOffV = kOffM + kSlice;
constexpr int kOffRaw = kOffV + kSlice, kRaw = 8 * kPerCta;
constexpr int kOffLoss = kOffRaw + 2 * kRaw, kLoss = 4 * kPerCta;
constexpr int kOffC = kOffLoss + 2 * kLoss;
constexpr int kSmemFloats = kOffC + 4;
static_assert(kPerCta <= kP && kPerCta % 4 == 0 && kSlice <= 2 * kCT, "samples in whole quads, two slice entries per thread");
static_assert(kOffSt % 4 == 0 && kP % 4 == 0 && kNetParams % 4 == 0, "16-byte rows");

__device__ __forceinline__ void cluster_sync() {
  __syncwarp();
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
// address of shared-memory pointer p in the cluster's CTA `rank`
__device__ __forceinline__ uint32_t cluster_addr(const float* p, uint32_t rank) {
  uint32_t local = static_cast<uint32_t>(__cvta_generic_to_shared(p)), remote;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(remote) : "r"(local), "r"(rank));
  return remote;
}
__device__ __forceinline__ float ld_cluster(uint32_t a) {
  float v;
  asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(a) : "memory");
  return v;
}
__device__ __forceinline__ void st_cluster(uint32_t a, float v) {
  asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(a), "f"(v) : "memory");
}
// barrier of the working warps
__device__ __forceinline__ void work_sync() {
  __syncwarp();
  asm volatile("bar.sync 1, %0;" ::"n"(kCT) : "memory");
}

// This warp's share (NOUT / 8 consecutive outputs) of a hidden layer for sample
// column `col`: bias, then an FMA chain over the inputs in ascending order; ReLU.
// Columns without a live sample hold zeros.
template <int L>
__device__ __forceinline__ void layer_fwd(const float* W, float* st, int warp, int col, bool store, bool live) {
  constexpr int NIN = wid(L), NOUT = wid(L + 1), G = NOUT / kWarps;
  constexpr int XIN = L == 0 ? kX0 : L == 1 ? kX1 : L == 2 ? kX2 : kX3;
  constexpr int XOUT = L == 0 ? kX1 : L == 1 ? kX2 : L == 2 ? kX3 : kX4;
  const float* Wl = W + wofs(L);
  const int o0 = warp * G;
  float a[G];
#pragma unroll
  for (int g = 0; g < G; ++g) a[g] = Wl[NOUT * NIN + o0 + g];
  if (L == 0) {
    float x[6];
#pragma unroll
    for (int i = 0; i < 6; ++i) x[i] = st[(XIN + i) * kP + col];
#pragma unroll
    for (int g = 0; g < G; ++g) {
      const float2* w = reinterpret_cast<const float2*>(Wl + (o0 + g) * 6);
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        a[g] = fmaf(w[i].x, x[2 * i], a[g]);
        a[g] = fmaf(w[i].y, x[2 * i + 1], a[g]);
      }
    }
  } else {
#pragma unroll
    for (int i = 0; i < NIN; i += 4) {
      float x[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) x[q] = st[(XIN + i + q) * kP + col];
#pragma unroll
      for (int g = 0; g < G; ++g) {
        const float4 w = *reinterpret_cast<const float4*>(Wl + (o0 + g) * NIN + i);
        a[g] = fmaf(w.x, x[0], a[g]);
        a[g] = fmaf(w.y, x[1], a[g]);
        a[g] = fmaf(w.z, x[2], a[g]);
        a[g] = fmaf(w.w, x[3], a[g]);
      }
    }
  }
  if (store) {
#pragma unroll
    for (int g = 0; g < G; ++g) st[(XOUT + o0 + g) * kP + col] = live ? fmaxf(a[g], 0.0f) : 0.0f;
  }
}

// This warp's share of the delta of layer L's outputs (L = 1..4), from the one
// above it: an FMA chain over the outputs above in ascending order, times relu'.
template <int L>
__device__ __forceinline__ void layer_bwd(const float* W, float* st, int warp, int col, bool store, bool live) {
  constexpr int N = wid(L), NUP = wid(L + 1), G = N / kWarps;
  constexpr int DUP = L == 4 ? kD5 : L == 3 ? kD4 : L == 2 ? kD3 : kD2;
  constexpr int DOUT = L == 4 ? kD4 : L == 3 ? kD3 : L == 2 ? kD2 : kD1;
  constexpr int XACT = L == 4 ? kX4 : L == 3 ? kX3 : L == 2 ? kX2 : kX1;
  const float* Wu = W + wofs(L) + warp * G;  // W_{L+1}[NUP][N]
  float a[G];
#pragma unroll
  for (int g = 0; g < G; ++g) a[g] = 0.0f;
#pragma unroll
  for (int k = 0; k < NUP; ++k) {
    const float d = st[(DUP + k) * kP + col];
    float w[G];
    if (G % 4 == 0) {
#pragma unroll
      for (int g = 0; g < G; g += 4) {
        const float4 v = *reinterpret_cast<const float4*>(Wu + k * N + g);
        w[g] = v.x; w[g + (G > 1 ? 1 : 0)] = v.y; w[g + (G > 2 ? 2 : 0)] = v.z; w[g + (G > 3 ? 3 : 0)] = v.w;
      }
    } else {
#pragma unroll
      for (int g = 0; g < G; ++g) w[g] = Wu[k * N + g];
    }
#pragma unroll
    for (int g = 0; g < G; ++g) a[g] = fmaf(w[g], d, a[g]);
  }
  if (store) {
#pragma unroll
    for (int g = 0; g < G; ++g) {
      const int r = warp * G + g;
      st[(DOUT + r) * kP + col] = live && st[(XACT + r) * kP + col] > 0.0f ? a[g] : 0.0f;
    }
  }
}

// acc += sum of the products of four samples, in sample order
__device__ __forceinline__ void dot4(float4 a, float4 b, float& acc) {
  acc = fmaf(a.x, b.x, acc);
  acc = fmaf(a.y, b.y, acc);
  acc = fmaf(a.z, b.z, acc);
  acc = fmaf(a.w, b.w, acc);
}
// NO x NI gradients sum_s d_o(s) x_i(s) over the CTA's samples (columns without
// a live sample are zeros in both): rows d0 + DO q and x0 + DI q.
template <int NO, int NI>
__device__ __forceinline__ void grad_tile(const float* st, int d0, int DO, int x0, int DI, float (&g)[NO][NI]) {
#pragma unroll
  for (int o = 0; o < NO; ++o)
#pragma unroll
    for (int i = 0; i < NI; ++i) g[o][i] = 0.0f;
#pragma unroll 2
  for (int c = 0; c < kPerCta; c += 4) {
    float4 d[NO];
#pragma unroll
    for (int o = 0; o < NO; ++o) d[o] = *reinterpret_cast<const float4*>(st + (d0 + DO * o) * kP + c);
#pragma unroll
    for (int i = 0; i < NI; ++i) {
      const float4 x = *reinterpret_cast<const float4*>(st + (x0 + DI * i) * kP + c);
#pragma unroll
      for (int o = 0; o < NO; ++o) dot4(d[o], x, g[o][i]);
    }
  }
}
// sum_s d(s): the products with 1 round as the sums do
__device__ __forceinline__ float grad_bias(const float* st, int d0) {
  const float4 one = make_float4(1.0f, 1.0f, 1.0f, 1.0f);
  float g = 0.0f;
#pragma unroll
  for (int c = 0; c < kPerCta; c += 4) dot4(*reinterpret_cast<const float4*>(st + d0 * kP + c), one, g);
  return g;
}

__global__ void __launch_bounds__(kAll, 1) mlp_train_cluster_kernel(const MlpTrainArgs a) {
  extern __shared__ __align__(16) float sm[];
  float* W = sm + kOffW;
  float* st = sm + kOffSt;
  float* part = sm + kOffPart;
  float* mm = sm + kOffM;
  float* vv = sm + kOffV;
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  const uint32_t rank = cluster_rank();
  const int p_lo = (int)rank * kSlice;
  for (int i = t; i < kNetParams; i += kAll) W[i] = a.params[i];
  for (int i = t; i < kRows * kP; i += kAll) st[i] = 0.0f;
  for (int i = t; i < kSlice; i += kAll) {
    const int p = p_lo + i;
    mm[i] = p < kNetParams ? a.m[p] : 0.0f;
    vv[i] = p < kNetParams ? a.v[p] : 0.0f;
  }
  const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
  const float lr = a.lr;
  const long long steps = (a.n_perm + a.batch - 1) / a.batch;
  const bool aux = warp == kWarps;
  double loss_sum = 0.0;
  bool bad_index = false;
  double p1 = 0.0, p2 = 0.0;
  if (aux) {
    p1 = pow(0.9, (double)a.t0);
    p2 = pow(0.999, (double)a.t0);
  }
  // this CTA's samples of a step: [first, first + ns) of its batch of nb
  auto share = [&](long long step, int& nb, int& first, int& ns) {
    nb = (int)min((long long)a.batch, a.n_perm - step * a.batch);
    const int per = (nb + kCl - 1) / kCl;
    first = min((int)rank * per, nb);
    ns = min(per, nb - first);
  };
  // (ninth warp) the raw samples of a step into its buffer
  auto fetch = [&](long long step) {
    int nb, first, ns;
    share(step, nb, first, ns);
    if (lane >= kPerCta) return;
    bool live = lane < ns;
    long long idx = 0;
    if (live) {
      idx = a.perm[step * a.batch + first + lane];
      if (idx < 0 || idx >= a.n) {
        bad_index = true;
        live = false;
        idx = 0;
      }
    }
    float* r = sm + kOffRaw + (int)(step & 1) * kRaw + 8 * lane;
#pragma unroll
    for (int j = 0; j < 6; ++j) r[j] = live ? (float)a.X[idx * 6 + j] : 0.0f;
    r[6] = __uint_as_float(live ? 256u | a.y[idx] : 0u);
  };
  // (ninth warp) the loss terms of a step, per sample in output order
  auto add_loss = [&](long long step) {
    int nb, first, ns;
    share(step, nb, first, ns);
    if (lane >= kPerCta) return;
    const float* l = sm + kOffLoss + (int)(step & 1) * kLoss + 4 * lane;
    double loss = 0.0;
#pragma unroll
    for (int k = 0; k < 4; ++k) loss += (double)l[k];
    loss_sum += loss * (0.25 / (double)nb);
  };
  if (aux) fetch(0);
  // addresses of this thread's slice entries in every CTA: partial sums (read)
  // and parameters (written)
  uint32_t part_at[kCl], w_at[kCl];
#pragma unroll
  for (int r = 0; r < kCl; ++r) {
    part_at[r] = cluster_addr(part + p_lo + t, (uint32_t)r);
    w_at[r] = cluster_addr(W + p_lo + t, (uint32_t)r);
  }
  cluster_sync();
#pragma unroll 1
  for (long long step = 0; step < steps; ++step) {
    if (aux) {
      p1 *= 0.9;
      p2 *= 0.999;
      if (lane == 0) {
        sm[kOffC] = (float)(1.0 / (1.0 - p1));
        sm[kOffC + 1] = (float)(1.0 / (1.0 - p2));
      }
      if (step + 1 < steps) fetch(step + 1);
      if (step > 0) add_loss(step - 1);
    } else {
      int nb, first, ns;
      share(step, nb, first, ns);
      const int col = min(lane, kPerCta - 1);
      const bool store = lane < kPerCta;
      const float* raw = sm + kOffRaw + (int)(step & 1) * kRaw + 8 * col;
      const unsigned lab = __float_as_uint(raw[6]);
      const bool live = (lab & 256u) != 0u;
      // ---- Eq. (normalizainput); warp w < 6 writes value w
      {
        float x[6], m = 1.0f;
#pragma unroll
        for (int j = 0; j < 6; ++j) {
          x[j] = raw[j];
          m = fmaxf(m, fabsf(x[j]));
        }
        float xw = x[0];
#pragma unroll
        for (int j = 1; j < 6; ++j) xw = warp == j ? x[j] : xw;
        if (store && warp < 6) st[(kX0 + warp) * kP + col] = xw / m;
      }
      work_sync();
      // ---- forward (Eqs. (reconstuction), (activationfunction))
      layer_fwd<0>(W, st, warp, col, store, live);
      work_sync();
      layer_fwd<1>(W, st, warp, col, store, live);
      work_sync();
      layer_fwd<2>(W, st, warp, col, store, live);
      work_sync();
      layer_fwd<3>(W, st, warp, col, store, live);
      work_sync();
      // ---- output k by warp k: loss term and dL/dz = (sigma(z) - y) / (n S)
      if (warp < 4) {
        const int k = warp;
        float z = W[wofs(4) + 32 + k];
#pragma unroll
        for (int i = 0; i < 8; ++i) z = fmaf(W[wofs(4) + k * 8 + i], st[(kX4 + i) * kP + col], z);
        const float yk = (float)((lab >> k) & 1u);
        const float sig = 1.0f / (1.0f + __expf(-z));
        // -[y log s + (1-y) log(1-s)] = softplus(z) - y z
        if (store) {
          sm[kOffLoss + (int)(step & 1) * kLoss + 4 * col + k] = live ? softplus(z) - yk * z : 0.0f;
          st[(kD5 + k) * kP + col] = live ? (sig - yk) * (1.0f / (4.0f * (float)nb)) : 0.0f;
        }
      }
      work_sync();
      // ---- deltas
      layer_bwd<4>(W, st, warp, col, store, live);
      work_sync();
      layer_bwd<3>(W, st, warp, col, store, live);
      work_sync();
      layer_bwd<2>(W, st, warp, col, store, live);
      work_sync();
      layer_bwd<1>(W, st, warp, col, store, live);
      work_sync();
      // ---- partial gradient of every parameter over these samples (dW =
      // sum delta x, db = sum delta): W2 by warps 0-3, W3 by warp 4, W1 and b1 by
      // warps 5 and 6, the rest by warp 7
      if (warp < 4) {
        const int ob = t >> 4, ib = t & 15;
        float g[4][4];
        grad_tile<4, 4>(st, kD2 + ob, 8, kX1 + ib, 16, g);
#pragma unroll
        for (int o = 0; o < 4; ++o)
#pragma unroll
          for (int i = 0; i < 4; ++i) part[wofs(1) + (ob + 8 * o) * 64 + ib + 16 * i] = g[o][i];
      } else if (warp == 4) {
        const int ob = lane >> 3, ib = lane & 7;
        float g[4][4];
        grad_tile<4, 4>(st, kD3 + ob, 4, kX2 + ib, 8, g);
#pragma unroll
        for (int o = 0; o < 4; ++o)
#pragma unroll
          for (int i = 0; i < 4; ++i) part[wofs(2) + (ob + 4 * o) * 32 + ib + 8 * i] = g[o][i];
      } else if (warp < 7) {
        const int u = t - 160;
        float g[1][6];
        grad_tile<1, 6>(st, kD1 + u, 0, kX0, 1, g);
#pragma unroll
        for (int i = 0; i < 6; ++i) part[u * 6 + i] = g[0][i];
        part[384 + u] = grad_bias(st, kD1 + u);
      } else {
        float g[1][4], h[1][1];
        grad_tile<1, 4>(st, kD4 + (lane >> 2), 0, kX3 + (lane & 3), 4, g);
#pragma unroll
        for (int i = 0; i < 4; ++i) part[wofs(3) + (lane >> 2) * 16 + (lane & 3) + 4 * i] = g[0][i];
        grad_tile<1, 1>(st, kD5 + (lane >> 3), 0, kX4 + (lane & 7), 0, h);
        part[wofs(4) + lane] = h[0][0];
        part[wofs(1) + 2048 + lane] = grad_bias(st, kD2 + lane);
        if (lane < 28) {
          const int row = lane < 16 ? kD3 + lane : lane < 24 ? kD4 + lane - 16 : kD5 + lane - 24;
          part[lane < 16 ? wofs(2) + 512 + lane : lane < 24 ? wofs(3) + 128 + lane - 16 : wofs(4) + 32 + lane - 24] =
              grad_bias(st, row);
        }
      }
    }
    cluster_sync();
    // ---- this CTA's slice: sum over the CTAs (rank order), Adam, the new
    // values to every CTA
    if (!aux) {
      const float c1 = sm[kOffC], c2 = sm[kOffC + 1];
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        const int i = t + q * kCT, p = p_lo + i;
        if (i < kSlice && p < kNetParams) {
          float gr[kCl];
#pragma unroll
          for (int r = 0; r < kCl; ++r) gr[r] = ld_cluster(part_at[r] + 4u * kCT * q);
          float g = 0.0f;
#pragma unroll
          for (int r = 0; r < kCl; ++r) g += gr[r];
          mm[i] = fmaf(b1, mm[i], (1.0f - b1) * g);
          vv[i] = fmaf(b2, vv[i], (1.0f - b2) * (g * g));
          const float mh = mm[i] * c1, vh = vv[i] * c2;
          const float w = W[p] - lr * mh / (sqrtf(vh) + eps);
#pragma unroll
          for (int r = 0; r < kCl; ++r) st_cluster(w_at[r] + 4u * kCT * q, w);
        }
      }
    }
    cluster_sync();
  }
  if (aux) add_loss(steps - 1);
  // results: every CTA holds the parameters; each writes its own slice and
  // moments
  for (int i = t; i < kSlice; i += kAll) {
    const int p = p_lo + i;
    if (p < kNetParams) {
      a.params[p] = W[p];
      a.m[p] = mm[i];
      a.v[p] = vv[i];
    }
  }
  // loss: per CTA a fixed-order tree over its samples, then the CTAs in rank
  // order
  if (aux) {
#pragma unroll
    for (int w = 16; w > 0; w >>= 1) {
      const double o = __shfl_down_sync(0xffffffffu, loss_sum, w);
      if (lane < w) loss_sum += o;
    }
    if (lane == 0) {  // the CTA's loss as two floats (hi, lo) for the gather
      part[0] = (float)loss_sum;
      part[1] = (float)(loss_sum - (double)(float)loss_sum);
    }
  }
  cluster_sync();
  if (rank == 0 && t == 0 && a.loss_sum) {
    double tot = 0.0;
    for (int r = 0; r < kCl; ++r)
      tot += (double)ld_cluster(cluster_addr(part, (uint32_t)r)) + (double)ld_cluster(cluster_addr(part + 1, (uint32_t)r));
    *a.loss_sum = tot;
  }
  if (bad_index) atomicOr(a.status, 8);
  cluster_sync();  // no CTA leaves while another may still read its memory
}

}  // namespace

cudaError_t launch_mlp_train(const MlpTrainArgs& a, cudaStream_t s) {
  // one cluster of kCl CTAs
  const size_t smem = (size_t)kSmemFloats * sizeof(float);
  cudaError_t e = cudaFuncSetAttribute(mlp_train_cluster_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)smem);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(kCl, 1, 1);
  cfg.blockDim = dim3(kAll, 1, 1);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = kCl;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  e = cudaLaunchKernelEx(&cfg, mlp_train_cluster_kernel, a);
  return e != cudaSuccess ? e : cudaGetLastError();
}

}  // namespace neno6
