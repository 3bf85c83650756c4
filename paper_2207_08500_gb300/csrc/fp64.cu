// FP64 path of the NENO6 Euler right-hand side (Li, Fu & Adams, arXiv
// 2207.08500): one fused kernel per RHS evaluation (optionally with the SSP-RK3
// stage combination as its epilogue), the batched classifier, and the CFL
// reduction.
//
// Every binary64 operation is written with an explicit round-to-nearest
// intrinsic (__dadd_rn, __dmul_rn, __fma_rn, __ddiv_rn, __dsqrt_rn, ...) in the
// fixed order the scheme is specified in, so the compiler can neither contract
// nor reorder it; the classifier masks are therefore a deterministic function
// of the state, identical on any IEEE-754 implementation of that order.
//
// Design (GB300): the binary64 pipe issues two lanes per clock and SM, 1/61 of
// the FP32 pipe's rate, so the classifier (3104 multiply-adds per stencil, 16
// stencils per cell and RHS) is evaluated in FP32 and split 16-bit matrix
// products with a certified bound and in binary64 only where the bound does not
// settle a logit's sign (mlp_filter.cuh).  What stays on the FP64 pipe is the reconstruction itself,
// ~1150 operations per cell, and each is done once: a thread takes a face
// with all its characteristic fields, so the Roe state is formed once per face.
// CTAs take tile after tile of cells: the tile plus a 3-cell halo (periodic
// wrap or zero-gradient copy done in the load) and the per-cell quantities are
// staged in shared memory, the faces' fluxes written back there and
// differenced, with no scratch in global memory.  Comparisons (ReLU, max, |x|)
// run on the integer pipe on the bit patterns.  Measured, 2048^2 RHS: 11.7 ms,
// against 437 ms with every classifier row in binary64 and four lanes per
// face; the FP64 operations alone would take 7.9 ms of a full FP64 pipe.
#include <cuda_fp16.h>

#include <cmath>
#include <cstring>
#include <utility>

#include "fp64_ops.cuh"
#include "internal.h"
#include "mlp_filter.cuh"
#include "tc.cuh"

namespace neno6 {
namespace {

using namespace f64ops;

constexpr int kCflThreads = 128;  // one warp per SM quarter

// Tile of TX x TY cells (TY = 1 in 1D) worked on by NT threads, OCC CTAs per
// SM.  Faces are dealt to warps in runs of 32 of one direction.  SPLIT: a
// warp's item is one characteristic field of 32 faces instead of all of them
// (the Roe state is then formed NV times over).
template <int NDIM_, int TX_, int TY_, int NT_, int OCC_, bool SPLIT_>
struct Tile {
  static constexpr int NDIM = NDIM_, TX = TX_, TY = TY_, NT = NT_, OCC = OCC_;
  static constexpr bool SPLIT = SPLIT_;
  static constexpr unsigned kResident = 152 * OCC;  // CTAs that run at a time
  static constexpr int NV = NDIM == 2 ? 4 : 3;
  static constexpr int HY = NDIM == 2 ? 3 : 0;
  static constexpr int SX = TX + 6, SY = TY + 2 * HY, NC = SX * SY;
  static constexpr int NCELLS = TY * SX + 2 * HY * TX;        // staged cells: no corners
  static constexpr int NXF = TY * (TX + 1);                   // x faces
  static constexpr int NYF = NDIM == 2 ? (TY + 1) * TX : 0;   // y faces
  static constexpr int WX = (NXF + 31) / 32, WY = (NYF + 31) / 32;  // runs of 32 faces
  // staged planes of NC values: U[NV], u, (v,) c, H, sqrt(rho), then the
  // fluxes but the mass flux (which is a momentum): x, then y
  static constexpr int P_U = 0, P_u = NV, P_v = NV + 1, P_c = NV + NDIM, P_H = P_c + 1, P_s = P_c + 2;
  static constexpr int P_F = P_c + 3;
  static constexpr int NPLANES = P_F + NDIM * (NV - 1);
  static constexpr int kPark = 12;  // per thread: the "+" stencil, the mirrored "-" stencil
  static constexpr int kScratch = 72;   // per warp (binary64 classifier)
  // doubles: planes, face fluxes, parked stencils, warp scratch, and for
  // SPLIT the faces' field fluxes and Roe states; dt; then the filter's table
  static constexpr int O_F = NPLANES * NC;
  static constexpr int O_P = O_F + NV * (NXF + NYF);
  static constexpr int O_W = O_P + kPark * NT;
  static constexpr int O_G = O_W + kScratch * (NT / 32);
  static constexpr int O_D = O_G + (SPLIT ? (NV + 5) * (NXF + NYF) : 0);
  static constexpr int O_T = (O_D + 2) / 2 * 2;
  static constexpr size_t SMEM = sizeof(double) * O_T + sizeof(float) * kFiltFloats;
  static_assert(NT % 32 == 0 && OCC * (SMEM + 1024 + 128) <= 228 * 1024, "resident CTAs");
};

// x is 0 or its magnitude lies in [2^-60, 2^60).
__device__ __forceinline__ bool moderate(double x) {
  const unsigned long long b = (unsigned long long)dbits(x) & 0x7fffffffffffffffULL;
  return b == 0ull || (unsigned)(b >> 32) - (963u << 20) < (120u << 20);
}
// Programmatic dependent launch: the next kernel of the stream may be set up
// (and run up to its own wait) while this one runs; the wait returns when every
// earlier kernel of the stream has completed and its writes are visible.
__device__ __forceinline__ void dependents_may_launch() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void wait_for_earlier_kernels() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

__device__ __forceinline__ unsigned long long umax64(unsigned long long a, unsigned long long b) {
  return a > b ? a : b;
}
__device__ __forceinline__ void warp_umax(unsigned long long& x, unsigned long long& y) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    x = umax64(x, __shfl_xor_sync(0xffffffffu, x, o));
    y = umax64(y, __shfl_xor_sync(0xffffffffu, y, o));
  }
}

// x / 2 for x = 0 or |x| >= 2^-1021, infinities and NaN (rows of L where rounding
// leaves a Roe state without a sound speed), on the integer pipe.
__device__ __forceinline__ double half_exact(double x) {
  const int hi = __double2hiint(x);
  const bool scale = (unsigned)(hi & 0x7ff00000) - 0x00100000u < 0x7fe00000u;
  return __hiloint2double(scale ? hi - 0x00100000 : hi, __double2loint(x));
}

// Roe-averaged state of a face (Sec. 4.4).
struct Roe {
  double ut, vt, Ht, ct, ic, b1, b2, qt;
};

// Row m of R applied to the field fluxes g: component n of the face flux.
template <int NDIM>
__device__ __forceinline__ double back_project(const Roe& r, int dir, int n, const double (&g)[4]) {
  constexpr int NV = NDIM == 2 ? 4 : 3;
  double R[4];
  const double ntc = __dmul_rn(dir == 0 ? r.ut : r.vt, r.ct);
  if (NDIM == 1) {
    if (n == 0) { R[0] = 1.0; R[1] = 1.0; R[2] = 1.0; }
    else if (n == 1) { R[0] = __dsub_rn(r.ut, r.ct); R[1] = r.ut; R[2] = __dadd_rn(r.ut, r.ct); }
    else { R[0] = __dsub_rn(r.Ht, ntc); R[1] = __dmul_rn(0.5, r.qt); R[2] = __dadd_rn(r.Ht, ntc); }
    R[3] = 0.0;
  } else if (n == 0) {
    R[0] = 1.0; R[1] = 1.0; R[2] = 0.0; R[3] = 1.0;
  } else if (n == 1) {
    if (dir == 0) { R[0] = __dsub_rn(r.ut, r.ct); R[1] = r.ut; R[2] = 0.0; R[3] = __dadd_rn(r.ut, r.ct); }
    else { R[0] = r.ut; R[1] = r.ut; R[2] = 1.0; R[3] = r.ut; }
  } else if (n == 2) {
    if (dir == 0) { R[0] = r.vt; R[1] = r.vt; R[2] = 1.0; R[3] = r.vt; }
    else { R[0] = __dsub_rn(r.vt, r.ct); R[1] = r.vt; R[2] = 0.0; R[3] = __dadd_rn(r.vt, r.ct); }
  } else {
    R[0] = __dsub_rn(r.Ht, ntc); R[1] = __dmul_rn(0.5, r.qt); R[2] = dir == 0 ? r.vt : r.ut;
    R[3] = __dadd_rn(r.Ht, ntc);
  }
  double F = __dmul_rn(R[0], g[0]);
#pragma unroll
  for (int q = 1; q < NV; ++q) F = __fma_rn(R[q], g[q], F);
  return F;
}

// Row m of L in the Roe/Toro scaling.
template <int NDIM>
__device__ __forceinline__ void left_row(const Roe& r, int dir, int m, double (&L)[4]) {
  const double nt = dir == 0 ? r.ut : r.vt;
  const double nc = __dmul_rn(nt, r.ic);
  const double b1u = __dmul_rn(r.b1, r.ut), hb1 = __dmul_rn(0.5, r.b1);
  L[3] = 0.0;
  if (NDIM == 1) {
    if (m == 0) { L[0] = __dmul_rn(0.5, __dadd_rn(r.b2, nc)); L[1] = __dmul_rn(0.5, __dsub_rn(-b1u, r.ic)); L[2] = hb1; }
    else if (m == 1) { L[0] = __dsub_rn(1.0, r.b2); L[1] = b1u; L[2] = -r.b1; }
    else { L[0] = __dmul_rn(0.5, __dsub_rn(r.b2, nc)); L[1] = __dmul_rn(0.5, __dadd_rn(-b1u, r.ic)); L[2] = hb1; }
    return;
  }
  const double b1v = __dmul_rn(r.b1, r.vt);
  if (m == 1) {
    L[0] = __dsub_rn(1.0, r.b2); L[1] = b1u; L[2] = b1v; L[3] = -r.b1;
  } else if (m == 2) {
    L[0] = dir == 0 ? -r.vt : -r.ut; L[1] = dir == 0 ? 0.0 : 1.0; L[2] = dir == 0 ? 1.0 : 0.0;
  } else {
    // the normal velocity's entry carries -+1/c, the tangential one does not
    const double nb = dir == 0 ? -b1u : -b1v, tb = dir == 0 ? -b1v : -b1u;
    const double ln = __dmul_rn(0.5, m == 0 ? __dsub_rn(nb, r.ic) : __dadd_rn(nb, r.ic));
    const double lt = __dmul_rn(0.5, tb);
    L[0] = __dmul_rn(0.5, m == 0 ? __dadd_rn(r.b2, nc) : __dsub_rn(r.b2, nc));
    L[1] = dir == 0 ? ln : lt; L[2] = dir == 0 ? lt : ln; L[3] = hb1;
  }
}

template <class G>
__global__ void __launch_bounds__(G::NT, G::OCC) rhs_fp64_kernel(const __grid_constant__ RhsArgs a) {
  constexpr int NDIM = G::NDIM, NV = G::NV, TX = G::TX, TY = G::TY, SX = G::SX, NC = G::NC, NT = G::NT;
  extern __shared__ __align__(16) double smem[];
  double* C = smem;
  double* sF = smem + G::O_F;            // x faces [NV][TY][TX+1], then y faces [NV][TY+1][TX]
  double* park0 = smem + G::O_P;         // [kPark][NT]
  float* T = reinterpret_cast<float*>(smem + G::O_T);
  __shared__ __align__(16) uint4 s_next;  // the next tile's answer
  __shared__ __align__(8) uint64_t s_nbar;
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  if (t == 0) {
    tc::mbar_init(&s_nbar, 1);
    tc::fence_mbar_init();
  }
  double* park = park0 + t;
  double* ws = smem + G::O_W + warp * G::kScratch;
  const int nx = a.nx, ny = a.ny;
  const size_t plane = (size_t)nx * ny;
  const double gm1 = a.gm1, gamma = a.gamma;
  const double* __restrict__ Wt = a.net64;
  // a handle's table is never written by the kernels before this one, so it is
  // fetched while they drain (dependent_launch below); what they write, a table
  // laid out on the stream among it, is read after the wait
  if (a.mask_mode == kMaskMLP && !a.net_on_stream) filt::load_filter(T, a.filter, t, NT);
  dependents_may_launch();
  wait_for_earlier_kernels();
  if (a.mask_mode == kMaskMLP && a.net_on_stream) filt::load_filter(T, a.filter, t, NT);

  // dt of an RK3 step (stage 1 computes it from max(|u|+c), max(|v|+c)), by the
  // last warp, which has the fewest cells, into shared memory until step 3.
  double* sdt = smem + G::O_D;
  if (a.stage && warp == NT / 32 - 1) {
    double dt;
    if (a.stage == 1) {
      const double tm = *a.t_dev;
      // maxima over the reduction's CTAs
      unsigned long long mx = 0, my = 0;
      for (int i = lane; i < a.nsmax; i += 32) {
        mx = umax64(mx, a.smax[i]);
        if (NDIM == 2) my = umax64(my, a.smax[kCflBlocks + i]);
      }
      warp_umax(mx, my);
      double s = __ddiv_rn(__longlong_as_double((long long)mx), a.dx);
      if (NDIM == 2) s = __dadd_rn(s, __ddiv_rn(__longlong_as_double((long long)my), a.dy));
      dt = __ddiv_rn(a.cfl, s);
      if (a.t_end > 0.0 && __dadd_rn(tm, dt) > a.t_end) dt = __dsub_rn(a.t_end, tm);
    } else {
      dt = *a.dt_dev;
    }
    if (lane == 0) *sdt = dt;
  }

  const int ntx = (nx + TX - 1) / TX;
  uint32_t nphase = 0u;
  int tile = (int)blockIdx.x;
  do {
    const int i0 = tile % ntx * TX, j0 = tile / ntx * TY;
    if (tile == 0 && a.stage && t == NT - 32) {
      // by whichever CTA has the first tile (block 0 may be one that was handed
      // out), the thread that formed dt
      const double dt = *sdt;
      if (a.stage == 1) {
        *a.dt_dev = dt;
        if (a.dt_user) *a.dt_user = dt;
      }
      if (a.stage == 3) *a.t_dev = __dadd_rn(*a.t_dev, dt);
    }
    // ---- 1. tile + halo (without its corners) and per-cell quantities.
    // `odd`: some value is not 0 or in [2^-60, 2^60), or a cell is not
    // physical; the tile's faces then take every operation of the
    // specification literally (below).
    bool odd = false;
    for (int k = t; k < G::NCELLS; k += NT) {
      // the rows of the tile with their x halo, then the y halo
      int bx = k % SX, by = G::HY + k / SX;
      if (NDIM == 2 && k >= TY * SX) {
        const int h = k - TY * SX, row = h / TX;
        bx = 3 + h % TX;
        by = row < 3 ? row : TY + row;
      }
      const int e = by * SX + bx;
      const int gi = wrap_index(i0 - 3 + bx, nx, a.bcx);
      const int gj = NDIM == 2 ? wrap_index(j0 - 3 + by, ny, a.bcy) : 0;
      const size_t g = (size_t)gj * nx + gi;
      double U[NV];
#pragma unroll
      for (int n = 0; n < NV; ++n) {
        U[n] = a.U[n * plane + g];
        C[(G::P_U + n) * NC + e] = U[n];
        odd |= !moderate(U[n]);
      }
      const double rho = U[0], E = U[NV - 1];
      const double u = __ddiv_rn(U[1], rho);
      double v = 0.0, q;
      if (NDIM == 2) {
        v = __ddiv_rn(U[2], rho);
        q = __fma_rn(v, v, __dmul_rn(u, u));
      } else {
        q = __dmul_rn(u, u);
      }
      const double p = __dmul_rn(gm1, __dsub_rn(E, __dmul_rn(0.5, __dmul_rn(rho, q))));
      const double c = __dsqrt_rn(__ddiv_rn(__dmul_rn(gamma, p), rho));
      const double Ep = __dadd_rn(E, p);
      if (!(rho > 0.0) || !(p > 0.0)) {
        atomicOr(a.status, 1);
        odd = true;
      }
      odd |= !moderate(p);
      C[G::P_u * NC + e] = u;
      C[G::P_c * NC + e] = c;
      C[G::P_H * NC + e] = __ddiv_rn(Ep, rho);
      C[G::P_s * NC + e] = __dsqrt_rn(rho);
      double* F = C + G::P_F * NC + e;
      if (NDIM == 2) {
        C[G::P_v * NC + e] = v;
        if (by >= 3 && by < TY + 3) {
          F[0] = __fma_rn(U[1], u, p);
          F[NC] = __dmul_rn(U[2], u);
          F[2 * NC] = __dmul_rn(Ep, u);
        }
        if (bx >= 3 && bx < TX + 3) {
          F[3 * NC] = __dmul_rn(U[1], v);
          F[4 * NC] = __fma_rn(U[2], v, p);
          F[5 * NC] = __dmul_rn(Ep, v);
        }
      } else {
        F[0] = __fma_rn(U[1], u, p);
        F[NC] = __dmul_rn(Ep, u);
      }
    }
    odd |= !moderate(gm1);
    filt::table_ready();
    odd = __syncthreads_or(odd);

    // ---- 2. faces
    constexpr int kItems = (G::WX + G::WY) * (G::SPLIT ? NV : 1);
#pragma unroll 1
    for (int it = warp; it < kItems; it += NT / 32) {
      const int run = G::SPLIT ? it / NV : it;
      const int dir = NDIM == 2 && run >= G::WX ? 1 : 0;  // warp-uniform
      const int nf = dir == 0 ? G::NXF : G::NYF;
      const int fraw = (run - (dir ? G::WX : 0)) * 32 + lane;
      const int face = min(fraw, nf - 1);
      int cb0, gf, gline;
      const int stride = dir == 0 ? 1 : SX;
      if (dir == 0) {
        const int r = face / (TX + 1), f = face % (TX + 1);
        cb0 = (G::HY + r) * SX + f;
        gf = i0 + f;      // global face index along x, 0..nx
        gline = j0 + r;   // row
      } else {
        const int f = face / TX, c = face % TX;
        cb0 = f * SX + 3 + c;
        gf = j0 + f;
        gline = i0 + c;   // column
      }
      const bool valid = fraw < nf && (dir == 0 ? (gf <= nx && gline < ny) : (gf <= ny && gline < nx));
      if (__ballot_sync(0xffffffffu, valid) == 0u) continue;
      const double* Un = C + (dir == 0 ? G::P_u : G::P_v) * NC;  // normal velocity
      const double* F0 = C + (G::P_U + 1 + dir) * NC;            // mass flux
      const double* F1 = C + (G::P_F + dir * 3) * NC;            // the other fluxes
      const int ca = cb0 + 2 * stride, cb = cb0 + 3 * stride;

      // Roe average of cells i and i+1 (Sec. 4.4).
      Roe r;
      {
        const double sa = C[G::P_s * NC + ca], sb = C[G::P_s * NC + cb];
        const double den = __dadd_rn(sa, sb);
        r.ut = __ddiv_rn(__fma_rn(sb, C[G::P_u * NC + cb], __dmul_rn(sa, C[G::P_u * NC + ca])), den);
        r.Ht = __ddiv_rn(__fma_rn(sb, C[G::P_H * NC + cb], __dmul_rn(sa, C[G::P_H * NC + ca])), den);
        r.vt = 0.0;
        if (NDIM == 2) {
          r.vt = __ddiv_rn(__fma_rn(sb, C[G::P_v * NC + cb], __dmul_rn(sa, C[G::P_v * NC + ca])), den);
          r.qt = __fma_rn(r.vt, r.vt, __dmul_rn(r.ut, r.ut));
        } else {
          r.qt = __dmul_rn(r.ut, r.ut);
        }
        const double c2 = __dmul_rn(gm1, __dsub_rn(r.Ht, __dmul_rn(0.5, r.qt)));
        if (valid && !(c2 > 0.0)) atomicOr(a.status, 2);
        r.ct = __dsqrt_rn(c2);
        r.ic = __ddiv_rn(1.0, r.ct);
        r.b1 = __ddiv_rn(gm1, c2);
        r.b2 = __dmul_rn(0.5, __dmul_rn(r.b1, r.qt));
      }

      double gh[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll 1
      for (int m = G::SPLIT ? it % NV : 0; m < (G::SPLIT ? it % NV + 1 : NV); ++m) {
        // LLF alpha_m: max over the six stencil cells of |lambda_m|.
        double alpha = 0.0;
#pragma unroll
        for (int j = 0; j < 6; ++j) {
          double lam = Un[cb0 + j * stride];
          if (m == 0) lam = __dsub_rn(lam, C[G::P_c * NC + cb0 + j * stride]);
          else if (m == NV - 1) lam = __dadd_rn(lam, C[G::P_c * NC + cb0 + j * stride]);
          alpha = j == 0 ? dabs(lam) : dmax_nn(alpha, dabs(lam));
        }
        // Characteristic projection and LLF split of the six stencil cells,
        // (L F +- alpha L U) / 2 with the "-" side mirrored.  On a moderate
        // tile every intermediate is 0 or far above the subnormal range, so
        // halving the row of L halves every following value exactly and saves
        // the twelve products by 1/2; and the shear row's entries 0 and 1 need
        // no products.
        double L[4], sp[6], sm[6];
        left_row<NDIM>(r, dir, m, L);
        if (!odd) {
          if (NDIM == 2 && m == 2) {
            const double l0 = half_exact(L[0]);
            const double* Ut = C + (G::P_U + 2 - dir) * NC;  // tangential momentum
            const double* Ft = F1 + (1 - dir) * NC;          // and its flux
#pragma unroll
            for (int j = 0; j < 6; ++j) {
              const int cj = cb0 + j * stride;
              const double vv = __fma_rn(0.5, Ut[cj], __dmul_rn(l0, C[G::P_U * NC + cj]));
              const double gg = __fma_rn(0.5, Ft[cj], __dmul_rn(l0, F0[cj]));
              sp[j] = __fma_rn(alpha, vv, gg);
              sm[j] = __fma_rn(-alpha, vv, gg);
            }
          } else {
#pragma unroll
            for (int n = 0; n < NV; ++n) L[n] = half_exact(L[n]);
#pragma unroll
            for (int j = 0; j < 6; ++j) {
              const int cj = cb0 + j * stride;
              double vv = __dmul_rn(L[0], C[G::P_U * NC + cj]);
              double gg = __dmul_rn(L[0], F0[cj]);
#pragma unroll
              for (int n = 1; n < NV; ++n) {
                vv = __fma_rn(L[n], C[(G::P_U + n) * NC + cj], vv);
                gg = __fma_rn(L[n], F1[(n - 1) * NC + cj], gg);
              }
              sp[j] = __fma_rn(alpha, vv, gg);
              sm[j] = __fma_rn(-alpha, vv, gg);
            }
          }
        } else {
#pragma unroll
          for (int j = 0; j < 6; ++j) {
            const int cj = cb0 + j * stride;
            double vv = __dmul_rn(L[0], C[G::P_U * NC + cj]);
            double gg = __dmul_rn(L[0], F0[cj]);
#pragma unroll
            for (int n = 1; n < NV; ++n) {
              vv = __fma_rn(L[n], C[(G::P_U + n) * NC + cj], vv);
              gg = __fma_rn(L[n], F1[(n - 1) * NC + cj], gg);
            }
            sp[j] = __dmul_rn(0.5, __fma_rn(alpha, vv, gg));
            sm[j] = __dmul_rn(0.5, __fma_rn(-alpha, vv, gg));
          }
        }
        double smir[6];
#pragma unroll
        for (int j = 0; j < 6; ++j) {
          smir[j] = sm[5 - j];  // the "-" side is the mirror image
          park[j * NT] = sp[j];
          park[(6 + j) * NT] = smir[j];
        }

        // Classifier bits of both sides.
        unsigned eta_side[2];
        if (a.mask_mode == kMaskMLP) {
          float x[2][6];
          const bool ok0 = filt::filter_input(sp, x[0]);
          const bool ok1 = filt::filter_input(smir, x[1]);
          // the stencils are re-read from shared memory after the classifier
          // rather than kept in registers across it
          asm volatile("" ::: "memory");
          unsigned res[2];
          filt::filter_rows(T, x, res);
          eta_side[0] = res[0] & 15u;
          eta_side[1] = res[1] & 15u;
          filt::settle_rows(Wt, park0 + warp * 32, NT, ws, valid && !(ok0 && (res[0] & 16u)), eta_side[0]);
          filt::settle_rows(Wt, park0 + 6 * NT + warp * 32, NT, ws, valid && !(ok1 && (res[1] & 16u)),
                            eta_side[1]);
          asm volatile("" ::: "memory");
        } else if (a.mask_mode == kMaskTeno) {
          // TENO6-opt selection on the split fluxes themselves (its indicator
          // ratios do not depend on the scale)
          eta_side[0] = teno6_eta(a.teno, sp);
          eta_side[1] = teno6_eta(a.teno, smir);
        } else if (a.mask_mode == kMaskGiven) {
          size_t idx;
          if (dir == 0) idx = ((size_t)m * ny + gline) * (nx + 1) + gf;
          else idx = (size_t)NV * ny * (nx + 1) + ((size_t)m * (ny + 1) + gf) * nx + gline;
          const unsigned b = valid ? a.mask_in[idx] : 0u;
          eta_side[0] = b & 15u;
          eta_side[1] = b >> 4;
        } else {
          eta_side[0] = eta_side[1] = a.mask_mode == kMaskRough ? 15u : 0u;
        }
        if (valid && a.mask_out) {
          size_t idx;
          if (dir == 0) idx = ((size_t)m * ny + gline) * (nx + 1) + gf;
          else idx = (size_t)NV * ny * (nx + 1) + ((size_t)m * (ny + 1) + gf) * nx + gline;
          a.mask_out[idx] = (uint8_t)(eta_side[0] | (eta_side[1] << 4));
        }
        if (!a.out) continue;  // the masks alone
#pragma unroll
        for (int j = 0; j < 6; ++j) {
          sp[j] = park[j * NT];
          smir[j] = park[(6 + j) * NT];
        }
        const double g = __dadd_rn(combine64(a, sp, eta_side[0]), combine64(a, smir, eta_side[1]));
#pragma unroll
        for (int q = 0; q < NV; ++q)
          if (q == m) gh[q] = g;
        if (G::SPLIT) {
          const int fi = (dir == 0 ? 0 : G::NXF) + face;
          double* sG = smem + G::O_G;
          if (fraw < nf) {
            sG[m * (G::NXF + G::NYF) + fi] = g;
            if (m == 0) {
              double* sR = sG + NV * (G::NXF + G::NYF) + fi;
              const double rv[5] = {r.ut, r.vt, r.Ht, r.ct, r.qt};
#pragma unroll
              for (int q = 0; q < 5; ++q) sR[q * (G::NXF + G::NYF)] = rv[q];
            }
          }
        }
      }
      // Back-projection F_n = sum_m R[n][m] gh_m.
      if (!G::SPLIT && a.out && fraw < nf) {
        double* dst = sF + (dir == 0 ? 0 : NV * G::NXF) + face;
#pragma unroll
        for (int n = 0; n < NV; ++n) dst[n * nf] = back_project<NDIM>(r, dir, n, gh);
      }
    }
    __syncthreads();
    // Tiles are handed out: a CTA takes over one that has not been launched yet.
    // Rows evaluated again in binary64 make tiles uneven, and an SM's two CTAs do
    // not advance evenly (2048^2 11.69 ms dealt out beforehand, 11.42 handed out, both
    // before the filter's blocks had sums of their own, 11.67 since).
    if (t == 0 && gridDim.x > G::kResident) tc::try_cancel(&s_next, &s_nbar);
    if (G::SPLIT && a.out) {
      const double* sG = smem + G::O_G;
      for (int e = t; e < NV * (G::NXF + G::NYF); e += NT) {
        const int n = e / (G::NXF + G::NYF), fi = e % (G::NXF + G::NYF);
        const int dir = fi < G::NXF ? 0 : 1;
        double gq[4] = {0.0, 0.0, 0.0, 0.0}, rv[5];
#pragma unroll
        for (int q = 0; q < NV; ++q) gq[q] = sG[q * (G::NXF + G::NYF) + fi];
#pragma unroll
        for (int q = 0; q < 5; ++q) rv[q] = sG[(NV + q) * (G::NXF + G::NYF) + fi];
        Roe r;
        r.ut = rv[0]; r.vt = rv[1]; r.Ht = rv[2]; r.ct = rv[3]; r.qt = rv[4];
        const double F = back_project<NDIM>(r, dir, n, gq);
        if (dir == 0) sF[n * G::NXF + fi] = F;
        else sF[NV * G::NXF + n * G::NYF + fi - G::NXF] = F;
      }
      __syncthreads();
    }

    // ---- 3. conservative difference and (optionally) the RK3 stage update.
    // A division by a power of two is the exact product with its reciprocal.
    const double* sFy = sF + NV * G::NXF;
    const double dt = a.stage ? *sdt : 0.0;
    for (int e = a.out ? t : TX * TY; e < TX * TY; e += NT) {
      const int c = e % TX, rw = e / TX;
      const int gi = i0 + c, gj = j0 + rw;
      if (gi >= nx || gj >= ny) continue;
      const size_t g = (size_t)gj * nx + gi;
      const int bc = (G::HY + rw) * SX + 3 + c;
      double u0[NV];  // loaded before the stores, which may alias it
#pragma unroll
      for (int n = 0; n < NV; ++n) u0[n] = a.stage >= 2 ? a.U0[n * plane + g] : 0.0;
#pragma unroll
      for (int n = 0; n < NV; ++n) {
        const double dF = __dsub_rn(sF[(n * TY + rw) * (TX + 1) + c + 1], sF[(n * TY + rw) * (TX + 1) + c]);
        double rr = -(a.inv_dx != 0.0 ? __dmul_rn(dF, a.inv_dx) : __ddiv_rn(dF, a.dx));
        if (NDIM == 2) {
          const double dG = __dsub_rn(sFy[(n * (TY + 1) + rw + 1) * TX + c], sFy[(n * (TY + 1) + rw) * TX + c]);
          rr = __dsub_rn(rr, a.inv_dy != 0.0 ? __dmul_rn(dG, a.inv_dy) : __ddiv_rn(dG, a.dy));
        }
        double val = rr;
        const double Ucur = C[(G::P_U + n) * NC + bc];
        if (a.stage == 1) {
          val = __fma_rn(dt, rr, Ucur);
        } else if (a.stage == 2) {
          val = __fma_rn(0.75, u0[n], __dmul_rn(0.25, __fma_rn(dt, rr, Ucur)));
        } else if (a.stage == 3) {
          val = __fma_rn(a.third, u0[n], __dmul_rn(a.two_thirds, __fma_rn(dt, rr, Ucur)));
        }
        a.out[n * plane + g] = val;
      }
    }
    if (gridDim.x <= G::kResident) break;
    const bool lost = !tc::mbar_wait(&s_nbar, nphase);
    nphase ^= 1u;
    tile = tc::cancelled_block(&s_next);
    tc::fence_async_smem();
    // the next tile's cells overwrite what the difference reads
    if (__syncthreads_or(lost)) {
      if (t == 0) {
        atomicOr(a.status, 4);
        // the answer may still be on its way into this CTA's memory
        tc::mbar_wait(&s_nbar, nphase ^ 1u);
      }
      break;
    }
  } while (tile >= 0);
}

__global__ void __launch_bounds__(256) classify_fp64_kernel(const __grid_constant__ ClassifyParamsF64 P) {
  const long long r = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (r >= P.n) return;
  double s[6], x[6], z[4];
#pragma unroll
  for (int j = 0; j < 6; ++j) s[j] = P.X[r * 6 + j];
  normalise6(s, x);
  const unsigned eta = mlp64(P.net.p, x, z);
  P.eta[r] = (uint8_t)eta;
  if (P.logits) {
#pragma unroll
    for (int k = 0; k < 4; ++k) P.logits[r * 4 + k] = z[k];
  }
}

// The same for the 6-32-32-32-4 network of the width study.
__global__ void __launch_bounds__(256) classify_fp64_narrow_kernel(const __grid_constant__ ClassifyParamsF64 P) {
  const long long r = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (r >= P.n) return;
  double s[6], x[6], z[4];
#pragma unroll
  for (int j = 0; j < 6; ++j) s[j] = P.X[r * 6 + j];
  normalise6(s, x);
  const unsigned eta = mlp64_narrow(P.net.p, x, z);
  P.eta[r] = (uint8_t)eta;
  if (P.logits) {
#pragma unroll
    for (int k = 0; k < 4; ++k) P.logits[r * 4 + k] = z[k];
  }
}

// max over a CTA's cells of |u|+c (and |v|+c), one value per CTA: bit patterns
// of non-negative doubles order like the values, so integer max gives the exact
// maximum.  The stage-1 kernel takes the maximum over the CTAs: nothing has to
// be cleared before and nothing is contended.
template <int NDIM>
__global__ void __launch_bounds__(kCflThreads) cfl_reduce_kernel(const double* __restrict__ U, int nx, int ny,
                                                         double gamma, unsigned long long* smax,
                                                         int* status) {
  const size_t plane = (size_t)nx * ny;
  const double gm1 = __dsub_rn(gamma, 1.0);
  unsigned long long mx = 0, my = 0;
  dependents_may_launch();
  wait_for_earlier_kernels();
  for (size_t k = (size_t)blockIdx.x * blockDim.x + threadIdx.x; k < plane;
       k += (size_t)gridDim.x * blockDim.x) {
    const double rho = U[k];
    const double E = U[(NDIM == 2 ? 3 : 2) * plane + k];
    const double u = __ddiv_rn(U[plane + k], rho);
    double v = 0.0, q;
    if (NDIM == 2) {
      v = __ddiv_rn(U[2 * plane + k], rho);
      q = __fma_rn(v, v, __dmul_rn(u, u));
    } else {
      q = __dmul_rn(u, u);
    }
    const double p = __dmul_rn(gm1, __dsub_rn(E, __dmul_rn(0.5, __dmul_rn(rho, q))));
    const double c = __dsqrt_rn(__ddiv_rn(__dmul_rn(gamma, p), rho));
    if (!(rho > 0.0) || !(p > 0.0)) atomicOr(status, 1);
    mx = umax64(mx, (unsigned long long)dbits(__dadd_rn(dabs(u), c)));
    if (NDIM == 2) my = umax64(my, (unsigned long long)dbits(__dadd_rn(dabs(v), c)));
  }
  warp_umax(mx, my);
  __shared__ unsigned long long wx[kCflThreads / 32], wy[kCflThreads / 32];
  const int warp = threadIdx.x >> 5;
  if ((threadIdx.x & 31) == 0) {
    wx[warp] = mx;
    wy[warp] = my;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int i = 1; i < kCflThreads / 32; ++i) {
      mx = umax64(mx, wx[i]);
      my = umax64(my, wy[i]);
    }
    smax[blockIdx.x] = mx;
    if (NDIM == 2) smax[kCflBlocks + blockIdx.x] = my;
  }
}

}  // namespace

namespace {

// Launch a kernel that waits for its predecessors itself.  Small grids start
// early (programmatic stream serialisation): of ten 1D 400-cell steps' 835 us
// this takes 50, launch latency and the table's copy.  Grids of more than half
// the SMs do not: their CTAs would be placed beside the running kernel's and end
// up unevenly spread (200 x 136: 241 us per RHS against 191).
template <class... P, class... A>
cudaError_t dependent_launch(void (*kern)(P...), unsigned grid, unsigned block, size_t smem, cudaStream_t s, A&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(block);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr;
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &attr;
  cfg.numAttrs = grid <= 76 ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kern, std::forward<A>(args)...);
}

}  // namespace

namespace {

// Round x to binary16 (nearest even); returns its value.  The table takes 41 us of
// a solver's creation on the GPU's Arm host; the library's host conversions would
// add some 55.
float round16(float x, uint16_t& bits) {
  uint32_t b;
  std::memcpy(&b, &x, 4);
  const uint32_t sign = b >> 16 & 0x8000u, mag = b & 0x7fffffffu;
  if (mag < 0x38800000u) {  // below 2^-14: a multiple of 2^-24
    const float n = std::nearbyint(std::fabs(x) * 16777216.0f);
    bits = (uint16_t)(sign | (uint32_t)n);
    return std::copysign(n * (1.0f / 16777216.0f), x);
  }
  if (mag < 0x477fe000u) {  // up to 65504
    const uint32_t r = (mag + 0xfffu + (mag >> 13 & 1u)) & ~0x1fffu;
    bits = (uint16_t)(sign | ((r >> 13) - (112u << 10)));
    b = (b & 0x80000000u) | r;
    std::memcpy(&x, &b, 4);
    return x;
  }
  const __half h = __float2half(x);
  std::memcpy(&bits, &h, 2);
  return __half2float(h);
}
// The binary16 terms of v's FP32 rounding, and what they miss, |hi| + |lo|, |lo|
struct Terms {
  uint16_t hi, lo;
};
struct Split {
  double error, size, low;
};
Split split_terms(double v, Terms& t) {
  Split s;
  const float f = (float)v, h = round16(f, t.hi), l = round16(f - h, t.lo);
  s.error = std::fabs(v - (double)h - (double)l);
  s.low = std::fabs((double)l);
  s.size = std::fabs((double)h) + s.low;
  return s;
}

}  // namespace

// Coefficients of the filter's bound (mlp_filter.cuh).
// `terms`: those of the weights of layers 2 to 5 (layer 5 scaled), filled in.
static void build_filter_kappa(const NetF64& net, FilterKappa& out, Terms* terms) {
  constexpr int W[6] = {6, 64, 32, 16, 8, 4};
  constexpr int off[5] = {0, 448, 2528, 3056, 3192};
  const double u = 1.0 / 16777216.0, tiny = std::ldexp(1.0, -125), gap = std::ldexp(1.0, -25);
  auto aw = [&](int l, int o, int i) { return std::fmax(std::fabs(net.p[off[l] + o * W[l] + i]), tiny); };
  auto ab = [&](int l, int o) { return std::fmax(std::fabs(net.p[off[l] + W[l] * W[l + 1] + o]), tiny); };
  // static bound per logit over |x| <= 1: the logits' relative scales
  double M[64], e[64], Mn[64], en[64];
  for (int i = 0; i < 6; ++i) {
    M[i] = 1.0;
    e[i] = 8.0 * u;
  }
  for (int l = 0; l < 5; ++l) {
    for (int o = 0; o < W[l + 1]; ++o) {
      double s = ab(l, o), d = 0.0;
      for (int i = 0; i < W[l]; ++i) {
        s += aw(l, o, i) * M[i];
        d += aw(l, o, i) * e[i];
      }
      Mn[o] = s;
      en[o] = d + (W[l] + 2) * u * s;
    }
    for (int o = 0; o < W[l + 1]; ++o) {
      M[o] = Mn[o];
      e[o] = en[o];
    }
  }
  double G[4][64], Gn[4][64];
  for (int k = 0; k < 4; ++k) {
    const double s = e[0] / e[k];
    out.scale[k] = s > 1e-30 && s < 1e30 ? s : 1.0;
    for (int o = 0; o < 4; ++o) G[k][o] = k == o ? out.scale[k] : 0.0;
  }
  auto up = [](double x) { return std::nextafter((float)(1.01 * x), INFINITY); };
  double k0[4] = {0.0, 0.0, 0.0, 0.0};
  float* dst[5] = {out.in, out.h1, out.h2, out.h3, out.h4};
  for (int l = 4; l >= 0; --l) {
    const int n = W[l], m = W[l + 1];
    const int blocks = (n + 15) / 16;  // of inputs (layers 2-5)
    const double c = 2.5 * (n < 16 ? n : 16);  // units u an instruction may lose
    double own[4][64] = {};  // coefficients of the layer's inputs, per logit
    for (int k = 0; k < 4; ++k)
      for (int i = 0; i < n; ++i) Gn[k][i] = 0.0;
    for (int o = 0; o < m; ++o) {
      double gs[4];  // G, and layer 5's terms, hold the scale already
      for (int k = 0; k < 4; ++k) {
        gs[k] = l == 4 ? G[k][o] / out.scale[k] : G[k][o];
        k0[k] += (l == 0 ? n + 1 : blocks + 1) * u * G[k][o] * ab(l, o);
        if (l > 0) k0[k] += gs[k] * 4 * blocks * tiny;
      }
      for (int i = 0; i < n; ++i) {
        const double a = aw(l, o, i);
        for (int k = 0; k < 4; ++k) Gn[k][i] += G[k][o] * a;
        if (l == 0) continue;
        const double v = net.p[off[l] + o * n + i];
        const Split w = split_terms(l == 4 ? v * out.scale[o] : v, terms[off[l] + o * n + i]);
        // the block's instruction, the additions from it on and the input's
        // split, the weight's split, the dropped product
        const double e = (c + blocks - i / 16 + 2) * u * w.size + w.error + w.low / 2048.0;
        const double abs = gap * (w.size + w.low);
        for (int k = 0; k < 4; ++k) {
          own[k][i] += gs[k] * e;
          k0[k] += gs[k] * abs;
        }
      }
    }
    for (int i = 0; i < n; ++i) {
      double worst = 0.0;
      for (int k = 0; k < 4; ++k) {
        double e = own[k][i];
        if (l == 0) {  // the i-th FMA of the chain and those after it, the weight's and the input's rounding
          e = (n - i + 1 + 8) * u * Gn[k][i];
          k0[k] += Gn[k][i] * tiny;
        }
        worst = std::fmax(worst, e == e ? e : INFINITY);  // a NaN weight: nothing is certified
      }
      dst[l][i] = up(worst);
    }
    for (int k = 0; k < 4; ++k)
      for (int i = 0; i < n; ++i) G[k][i] = Gn[k][i];
  }
  double worst = 0.0;
  for (int k = 0; k < 4; ++k) worst = std::fmax(worst, k0[k] == k0[k] ? k0[k] : INFINITY);
  out.k0 = up(worst);
}

// No heap: the allocation-free step calls it.
void build_net_blob(const NetF64& net, void* blob) {
  constexpr int W[6] = {6, 64, 32, 16, 8, 4};
  constexpr int kW[5] = {0, kFiltW2, kFiltW3, kFiltW4, kFiltW5}, kB[5] = {0, kFiltB2, kFiltB3, kFiltB4, kFiltB5};
  FilterKappa k;
  Terms terms[kNetParams];
  build_filter_kappa(net, k, terms);
  double* Wt = static_cast<double*>(blob);
  float* T = reinterpret_cast<float*>(Wt + kNetParams);
  for (int i = 0; i < kFiltFloats; ++i) T[i] = 0.0f;
  int p = 0;
  for (int l = 0; l < 5; ++l) {
    const int nin = W[l], nout = W[l + 1];
    for (int o = 0; o < nout; ++o) {
      const double scale = l == 4 ? k.scale[o] : 1.0;
      for (int i = 0; i < nin; ++i) {
        const double w = net.p[p + o * nin + i];
        Wt[p + i * nout + o] = w;
        if (l == 0) {
          T[kFiltW1 + 8 * o + i] = (float)w;
          continue;
        }
        // input i of its block: pair (i % 8) / 2 of lane 4 (o % 8) + pair, word
        // i / 8 of hi and of lo
        const int tiles = (nout + 7) / 8, in = i % 16;
        uint16_t* at = reinterpret_cast<uint16_t*>(T + kW[l] + 128 * ((i / 16) * tiles + o / 8) +
                                                   4 * (4 * (o % 8) + in % 8 / 2) + in / 8) + in % 2;
        at[0] = terms[p + o * nin + i].hi;
        at[4] = terms[p + o * nin + i].lo;
      }
      const double b = net.p[p + nin * nout + o];
      Wt[p + nin * nout + o] = b;
      T[l == 0 ? kFiltW1 + 8 * o + 6 : kB[l] + o] = (float)(b * scale);
    }
    p += nin * nout + nout;
  }
  T[kFiltIn] = k.k0;
  for (int i = 0; i < 6; ++i) T[kFiltIn + 1 + i] = k.in[i];
  for (int i = 0; i < 64; ++i) T[kFiltW1 + 8 * i + 7] = k.h1[i];
  for (int i = 0; i < 32; ++i) T[kFiltK2 + i] = k.h2[i];
  for (int i = 0; i < 16; ++i) T[kFiltK3 + i] = k.h3[i];
  for (int i = 0; i < 8; ++i) T[kFiltK4 + i] = k.h4[i];
}

namespace {

template <class G>
cudaError_t launch_tiles(const RhsArgs& a, cudaStream_t s) {
  cudaError_t e =
      cudaFuncSetAttribute(rhs_fp64_kernel<G>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)G::SMEM);
  if (e != cudaSuccess) return e;
  const long long tiles = (long long)((a.nx + G::TX - 1) / G::TX) * ((a.ny + G::TY - 1) / G::TY);
  return dependent_launch(rhs_fp64_kernel<G>, (unsigned)tiles, G::NT, G::SMEM, s, a);
}

// 1/d when d is a power of two whose reciprocal is normal, else 0.
double exact_reciprocal(double d) {
  int e;
  return std::frexp(d, &e) == 0.5 && e > -1000 && e < 1000 ? 1.0 / d : 0.0;
}

}  // namespace

cudaError_t launch_rhs_fp64(int ndim, RhsArgs& a, cudaStream_t s) {
  a.inv_dx = exact_reciprocal(a.dx);
  a.inv_dy = ndim == 2 ? exact_reciprocal(a.dy) : 0.0;
  // Tiles whose (TX + 1) TY x faces and (TY + 1) TX y faces fill whole runs of
  // 32 (the FP64 pipe takes 64 clocks per warp instruction and SM quarter
  // however few lanes are active): 2.13 face slots per cell for 15 x 16, 2.29
  // for 7 x 16.  The smaller the grid, the smaller the tile, so that every SM
  // has warps; the smallest grids give a warp a single field.  Measured in us
  // per RHS, periodic quadrants (threads x CTAs per SM; * taken; tiles dealt out
  // beforehand and the filter's sums one per layer.  Handed out, and a sum per block,
  // the starred ones take 327 at 300^2, 545 at 400^2, 824 at 512^2, 1474 at 700^2,
  // 3018 at 1024^2 and 11670 at 2048^2):
  //                        24x16 64x64 100x100 200x136 300x300 400x400 512^2 700^2 1024^2 2048^2
  //   15 x 16       256x2   209   135    140     142     350     551    822* 1467*  3034*  11696*
  //   15 x 16       192x2   236   154            161                    848         3107   12058
  //   7 x 16        256x2   110    70     74*    114*    330*    547*   842  1606   3229   12769
  //   7 x 8         128x4    99    52     77     118     324     541    831  1569   3201   12611
  //   7 x 3 SPLIT   256x2    68*   44*    84     200     573    1012   1555  3030   6166   24579
  // 1D, n =                       400   4096  16384  65536  131072  1048576
  //   31 SPLIT      96x4           18*    17*    33*   111     197     1411
  //   127           128x4          38     36     39     85*    163*    1030*
  //   127           128x3          36     35     37     97     163     1077
  const auto tiles = [&](int tx, int ty) {
    return (long long)((a.nx + tx - 1) / tx) * ((a.ny + ty - 1) / ty);
  };
  if (ndim == 1) {
    if (tiles(31, 1) <= 152 * 4) return launch_tiles<Tile<1, 31, 1, 96, 4, true>>(a, s);
    return launch_tiles<Tile<1, 127, 1, 128, 4, false>>(a, s);
  }
  if (tiles(7, 3) <= 152 * 2) return launch_tiles<Tile<2, 7, 3, 256, 2, true>>(a, s);
  if (tiles(15, 16) < 152 * 2 * 3) return launch_tiles<Tile<2, 7, 16, 256, 2, false>>(a, s);
  return launch_tiles<Tile<2, 15, 16, 256, 2, false>>(a, s);
}

cudaError_t launch_classify_fp64(const ClassifyParamsF64& p, bool narrow, cudaStream_t s) {
  if (p.n == 0) return cudaSuccess;
  const long long blocks = (p.n + 255) / 256;
  if (narrow)
    classify_fp64_narrow_kernel<<<(unsigned)blocks, 256, 0, s>>>(p);
  else
    classify_fp64_kernel<<<(unsigned)blocks, 256, 0, s>>>(p);
  return cudaGetLastError();
}

cudaError_t launch_cfl_reduce(int ndim, const double* U, int nx, int ny, double gamma,
                              unsigned long long* smax, int* nsmax, int* status, cudaStream_t s) {
  const size_t cells = (size_t)nx * ny;
  const size_t most = (cells + kCflThreads - 1) / kCflThreads;
  const unsigned blocks = most < kCflBlocks ? (unsigned)most : (unsigned)kCflBlocks;
  *nsmax = (int)blocks;
  if (ndim == 2)
    return dependent_launch(cfl_reduce_kernel<2>, blocks, kCflThreads, 0, s, U, nx, ny, gamma, smax, status);
  return dependent_launch(cfl_reduce_kernel<1>, blocks, kCflThreads, 0, s, U, nx, ny, gamma, smax, status);
}

}  // namespace neno6
