// Frozen-mask adjoint of the FP64 NENO6 right-hand side: grad_U = J^T lambda,
// J = dL(U)/dU with the classifier bits and the LLF alpha argmax held at
// their values for U (the mask is piecewise constant in U, so this is the
// derivative of the scheme wherever it exists).
//
// dU_i/dt = -(F_{i+1/2} - F_{i-1/2})/dx - (G_{j+1/2} - G_{j-1/2})/dy, so the
// cotangent of face f (between cells f-1 and f) is (lambda_f - lambda_{f-1})/d
// (lambda of a cell outside the grid taken as 0).  Each face flux depends on
// its six stencil cells.  Two kernels:
//  * vjp_face_kernel, one thread per face: recomputes the face from U (halo
//    recomputation; the forward pass stores nothing), runs reverse mode
//    through it and writes the face's contribution to each of its six cells;
//  * vjp_gather_kernel, one thread per cell: adds the contributions of every
//    face whose stencil holds the cell (six per direction, more where
//    periodic images or zero-gradient ghost cells alias it) in a fixed order.
// Every output is written once; there are no atomics and the result is
// deterministic.
//
// The work is binary64 and bound by the FP64 pipe (two lanes per clock and
// SM), so the derivative is written out in closed form, ~760 FP64 operations
// per face, and everything of a cell that its faces share is formed once per
// tile in shared memory.  1024^2: 3.28 ms (2.9 ms of a full FP64 pipe),
// against 17.4 ms with forward-mode dual numbers over each cell's conserved
// variables and the Roe state (~5000 operations per face).  The velocities, sound speeds and wave speeds keep the
// forward path's order of operations: where cells tie up to rounding, as in
// regions of constant velocity, the first maximum has to be the same one.
#include "fp64_ops.cuh"
#include "internal.h"

namespace neno6 {
namespace {

using namespace f64ops;

// Tile of TX x TY cells: it owns the x faces left of its cells and the y
// faces below them (faces N of a line fall to a further tile).
template <int NDIM_, int TX_, int TY_, int NT_, int OCC_>
struct VTile {
  static constexpr int NDIM = NDIM_, TX = TX_, TY = TY_, NT = NT_, OCC = OCC_;
  static constexpr int NV = NDIM == 2 ? 4 : 3;
  static constexpr int HY = NDIM == 2 ? 3 : 0;
  static constexpr int SX = TX + 5, SY = NDIM == 2 ? TY + 5 : 1, NC = SX * SY;
  static constexpr int NCELLS = TY * SX + (NDIM == 2 ? 5 * TX : 0);  // no corners
  static constexpr int RUNS = TX * TY / 32;                          // of 32 faces, per direction
  // planes: U[NV], u, (v,) c, H, sqrt(rho), 1/rho, gamma/(2 c rho), fluxes but
  // the mass flux: x, then y
  static constexpr int P_U = 0, P_u = NV, P_c = NV + NDIM, P_H = P_c + 1, P_s = P_c + 2, P_r = P_c + 3;
  static constexpr int P_k = P_c + 4, P_F = P_c + 5;
  static constexpr int NPLANES = P_F + NDIM * (NV - 1);
  static constexpr int O_T = (NPLANES * NC + 1) / 2 * 2;  // coefficient pairs of the 256 mask bytes
  static constexpr int O_S = O_T + 256 * 12;   // coefficients of the 16 one-sided masks
  static constexpr size_t SMEM = sizeof(double) * (O_S + 16 * 6);
  static_assert(TX * TY % 32 == 0 && OCC * (SMEM + 1024) <= 228 * 1024, "tile");
};

// With the mask frozen, one side's reconstruction is linear in its six split
// fluxes: g_hat = sum_j c_j s_j, c_j = sum over kept stencils k of
// w_k(eta) times S_k's candidate coefficient on point j (Eqs. (convex),
// (TENOweight_renormalize)); all stencils discarded: c = e_2 (first-order
// fallback, Algorithm 2).
__device__ __forceinline__ double side_coeff(unsigned e, int j, const RhsArgs& a) {
  if (e == 15u) return j == 2 ? 1.0 : 0.0;
  double c = 0.0;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    // S_0 = {i-1, i, i+1}, S_1 = {i, i+1, i+2}, S_2 = {i-2, i-1, i},
    // S_3 = {i, ..., i+3}; stencil point j = 0..5 is cell i-2+j
    const int start = k == 0 ? 1 : (k == 2 ? 0 : 2), len = k == 3 ? 4 : 3;
    if (!((e >> k) & 1u) && j >= start && j < start + len) c = __fma_rn(a.wtab[e][k], a.cand[k][j - start], c);
  }
  return c;
}

// A linear functional of the left eigenvectors: with S = |u|^2/2 w_0 - u_n w_1
// - u_t w_2 + w_E and T = u_n w_0 - w_1 of a vector w (components density,
// normal and tangential momentum, energy), the rows of L applied to w are
//   (b1 S + T/c)/2,  w_0 - b1 S,  w_2 - u_t w_0,  (b1 S - T/c)/2.
struct ST {
  double S, T;
};
template <int NV>
__device__ __forceinline__ ST functional(const double (&w)[4], double a, double b, double hq) {
  ST r;
  double s = __fma_rn(hq, w[0], w[NV - 1]);
  s = __fma_rn(-a, w[1], s);
  if (NV == 4) s = __fma_rn(-b, w[2], s);
  r.S = s;
  r.T = __fma_rn(a, w[0], -w[1]);
  return r;
}

// Reverse mode over one face.  With the mask frozen the face flux is
//   F_hat = sum_m R_m (L_m . W_m) / 2,  W_m = P_m + alpha_m Q_m,
//   P_m = sum_j A_mj F_j,  Q_m = sum_j B_mj U_j,
// A_mj = c+_j + c-_{5-j}, B_mj = c+_j - c-_{5-j} (c- the mirrored "-" side's
// coefficients), alpha_m = |lambda_m| of the first stencil cell holding the
// maximum.  Given the face cotangent f, with z_m = R_m . f and L_m rows of L:
//  - cell j receives (sum_m A_mj z_m L_m / 2) through its flux Jacobian and
//    sum_m alpha_m B_mj z_m L_m / 2 directly;
//  - the argmax cell of field m receives z_m (L_m . Q_m) / 2 through
//    d|lambda_m|/dU;
//  - cells i, i+1 receive the derivative of sum_m z_m (L_m . W_m) / 2 with
//    respect to the Roe state (u_n, u_t, H), W held fixed.
// Vectors are in the face's frame: density, normal and (2D) tangential
// momentum, energy.
template <class G>
__global__ void __launch_bounds__(G::NT, G::OCC) vjp_face_kernel(const __grid_constant__ RhsArgs a,
                                                                 const double* __restrict__ lam,
                                                                 double* __restrict__ contrib) {
  constexpr int NDIM = G::NDIM, NV = G::NV, TX = G::TX, TY = G::TY, SX = G::SX, NC = G::NC, NT = G::NT;
  constexpr int E_ = NV - 1;  // the energy component, and the last field
  extern __shared__ double vsm[];
  double* C = vsm;
  double* pairs = vsm + G::O_T;
  double* sides = vsm + G::O_S;
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  const int nx = a.nx, ny = a.ny;
  const size_t plane = (size_t)nx * ny;
  const double gm1 = a.gm1, gamma = a.gamma;
  // (A_j, B_j) of every mask byte: row of twelve doubles per byte
  for (int i = t; i < 16 * 6; i += NT) sides[i] = side_coeff((unsigned)(i / 6), i % 6, a);
  __syncthreads();
  for (int i = t; i < 256 * 6; i += NT) {
    const int e = i / 6, j = i % 6;
    const double cp = sides[(e & 15) * 6 + j], cm = sides[(e >> 4) * 6 + 5 - j];
    pairs[e * 12 + 2 * j] = __dadd_rn(cp, cm);
    pairs[e * 12 + 2 * j + 1] = __dsub_rn(cp, cm);
  }
  const int ntx = (nx + 1 + TX - 1) / TX;
  const long long ntiles = (long long)ntx * (NDIM == 2 ? (ny + 1 + TY - 1) / TY : 1);
  for (long long tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
    const int i0 = (int)(tile % ntx) * TX, j0 = (int)(tile / ntx) * TY;
    __syncthreads();  // the last tile's faces are done with the planes
    for (int k = t; k < G::NCELLS; k += NT) {
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
      }
      const double rho = U[0], E = U[E_];
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
      const double ri = __drcp_rn(rho);
      C[G::P_u * NC + e] = u;
      C[G::P_c * NC + e] = c;
      C[G::P_H * NC + e] = __dmul_rn(Ep, ri);
      C[G::P_s * NC + e] = __dsqrt_rn(rho);
      C[G::P_r * NC + e] = ri;
      C[G::P_k * NC + e] = __dmul_rn(__dmul_rn(0.5 * gamma, ri), __drcp_rn(c));
      double* F = C + G::P_F * NC + e;
      if (NDIM == 2) {
        C[(G::P_u + 1) * NC + e] = v;
        F[0] = __fma_rn(U[1], u, p);
        F[NC] = __dmul_rn(U[2], u);
        F[2 * NC] = __dmul_rn(Ep, u);
        F[3 * NC] = __dmul_rn(U[1], v);
        F[4 * NC] = __fma_rn(U[2], v, p);
        F[5 * NC] = __dmul_rn(Ep, v);
      } else {
        F[0] = __fma_rn(U[1], u, p);
        F[NC] = __dmul_rn(Ep, u);
      }
    }
    __syncthreads();

#pragma unroll 1
    for (int it = warp; it < NDIM * G::RUNS; it += NT / 32) {
      const int dir = it >= G::RUNS ? 1 : 0;  // warp-uniform
      const int fc = (it - dir * G::RUNS) * 32 + lane;
      const int c0 = fc % TX, r0 = fc / TX;  // the cell right of / above the face
      const int f = dir == 0 ? i0 + c0 : j0 + r0, line = dir == 0 ? j0 + r0 : i0 + c0;
      const int N = dir == 0 ? nx : ny, nl = dir == 0 ? ny : nx;
      const bool valid = f <= N && line < nl;
      if (__ballot_sync(0xffffffffu, valid) == 0u) continue;
      if (!valid) continue;
      const int stride = dir == 0 ? 1 : SX;
      const int cb0 = dir == 0 ? (G::HY + r0) * SX + c0 : r0 * SX + 3 + c0;
      const long long nfaces = (long long)(N + 1) * nl;
      const long long id = dir == 0 ? (long long)line * (nx + 1) + f : (long long)f * nx + line;
      double* out = contrib + (dir == 0 ? 0 : (size_t)6 * NV * (nx + 1) * ny);  // the y faces' follow the x faces'
      auto cell = [&](int i) -> size_t { return dir == 0 ? (size_t)line * nx + i : (size_t)i * nx + line; };
      // component n of the face's frame is conserved variable comp(n)
      const int c1 = 1 + dir, c2_ = 2 - dir;
      auto comp = [&](int n) { return NDIM == 1 ? n : (n == 1 ? c1 : n == 2 ? c2_ : n); };
      const double* pU[4] = {C + G::P_U * NC, C + (G::P_U + c1) * NC, NV == 4 ? C + (G::P_U + c2_) * NC : nullptr,
                             C + (G::P_U + E_) * NC};
      const double* pF[4] = {pU[1], C + (G::P_F + (NDIM == 2 ? 4 * dir : 0)) * NC,
                             NV == 4 ? C + (G::P_F + 1 + 2 * dir) * NC : nullptr,
                             C + (G::P_F + dir * (NV - 1) + NV - 2) * NC};
      const double* pN = C + (G::P_u + dir) * NC;      // normal velocity
      const double* pT = C + (G::P_u + 1 - dir) * NC;  // tangential velocity (2D)
      double fb[4] = {0.0, 0.0, 0.0, 0.0};
      {
        const double invd = dir == 0 ? a.inv_dx : a.inv_dy;
#pragma unroll
        for (int n = 0; n < NV; ++n) {
          const double* l = lam + comp(n) * plane;
          const double lr = f < N ? l[cell(f)] : 0.0, ll = f > 0 ? l[cell(f - 1)] : 0.0;
          fb[n] = __dmul_rn(__dsub_rn(lr, ll), invd);
        }
      }
      const double fE = fb[E_];
      const double* tab[NV];  // coefficient pairs of field m
#pragma unroll
      for (int m = 0; m < NV; ++m) {
        const size_t idx = dir == 0 ? ((size_t)m * ny + line) * (nx + 1) + f
                                    : (size_t)NV * ny * (nx + 1) + ((size_t)m * (ny + 1) + f) * nx + line;
        tab[m] = pairs + 12 * a.mask_in[idx];
      }
      // Roe state
      const int ca = cb0 + 2 * stride, cb = cb0 + 3 * stride;
      const double rden = __drcp_rn(__dadd_rn(C[G::P_s * NC + ca], C[G::P_s * NC + cb]));
      const double wB = __dmul_rn(C[G::P_s * NC + cb], rden), wA = __dmul_rn(C[G::P_s * NC + ca], rden);
      const double un = __fma_rn(wB, __dsub_rn(pN[cb], pN[ca]), pN[ca]);
      const double ut = NV == 4 ? __fma_rn(wB, __dsub_rn(pT[cb], pT[ca]), pT[ca]) : 0.0;
      const double Ht = __fma_rn(wB, __dsub_rn(C[G::P_H * NC + cb], C[G::P_H * NC + ca]), C[G::P_H * NC + ca]);
      double hq = __dmul_rn(0.5 * un, un);
      if (NV == 4) hq = __fma_rn(0.5 * ut, ut, hq);
      const double cc = __dsqrt_rn(__dmul_rn(gm1, __dsub_rn(Ht, hq)));
      const double ic = __drcp_rn(cc), ic2 = __dmul_rn(ic, ic), b1 = __dmul_rn(gm1, ic2);
      // z_m = R_m . f
      double z[NV];
      const double fa = __fma_rn(un, fE, fb[1]);   // f_1 + u_n f_E
      {
        double base = __fma_rn(Ht, fE, __fma_rn(un, fb[1], fb[0]));
        if (NV == 4) base = __fma_rn(ut, fb[2], base);
        z[0] = __fma_rn(-cc, fa, base);
        z[E_] = __fma_rn(cc, fa, base);
        z[1] = __fma_rn(__dsub_rn(hq, Ht), fE, base);
        if (NV == 4) z[2] = __fma_rn(ut, fE, fb[2]);
      }
      // fields: alpha_m and its cell, L_m . W_m, L_m . Q_m, and the gradient
      // of Phi = sum_m z_m (L_m . W_m) / 2 with respect to the Roe quantities
      double alpha[NV], wabs[NV];  // z_m (L_m . Q_m) / 2 times the sign of lambda_m
      int js[NV];
      double ga = 0.0, gb = 0.0, gH = 0.0, gc = 0.0, gB = 0.0, gI = 0.0, yacu = 0.0;
#pragma unroll
      for (int m = 0; m < NV; ++m) {
        if (NV == 4 && m == 2) {
          alpha[m] = alpha[1];  // the same wave speed as the entropy field
          js[m] = js[1];
        } else {
          double al = 0.0, lj = 0.0;
          int jm = 0;
#pragma unroll
          for (int j = 0; j < 6; ++j) {
            const int cj = cb0 + j * stride;
            double l = pN[cj];
            if (m == 0) l = __dsub_rn(l, C[G::P_c * NC + cj]);
            else if (m == E_) l = __dadd_rn(l, C[G::P_c * NC + cj]);
            // the first index of the maximum wins (bit patterns of
            // non-negative values order like the values)
            if (j == 0 || dbits(dabs(l)) > dbits(al)) {
              al = dabs(l);
              lj = l;
              jm = j;
            }
          }
          alpha[m] = al;
          js[m] = jm;
          wabs[m] = lj < 0.0 ? -0.5 : 0.5;
        }
        const double sg = NV == 4 && m == 2 ? 0.0 : wabs[m];
        double P[4] = {0.0, 0.0, 0.0, 0.0}, Q[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll
        for (int j = 0; j < 6; ++j) {
          const int cj = cb0 + j * stride;
          const double2 ab = *reinterpret_cast<const double2*>(tab[m] + 2 * j);
#pragma unroll
          for (int n = 0; n < NV; ++n) {
            if (NV == 4 && m == 2 && (n == 1 || n == 3)) continue;  // row (-u_t, 0, 1, 0)
            P[n] = __fma_rn(ab.x, pF[n == E_ ? 3 : n][cj], P[n]);
            Q[n] = __fma_rn(ab.y, pU[n == E_ ? 3 : n][cj], Q[n]);
          }
        }
        double W[4];
#pragma unroll
        for (int n = 0; n < 4; ++n) W[n] = n < NV ? __fma_rn(alpha[m], Q[n], P[n]) : 0.0;
        const double hz = __dmul_rn(0.5, z[m]);
        if (NV == 4 && m == 2) {
          const double y = __fma_rn(-ut, W[0], W[2]), LQ = __fma_rn(-ut, Q[0], Q[2]);
          // the entropy and shear fields share their wave speed's cell
          wabs[2] = __dmul_rn(hz, LQ);
          gb = __fma_rn(-hz, W[0], gb);
          gb = __fma_rn(__dmul_rn(0.5, y), fE, gb);
          continue;
        }
        const ST w = functional<NV>(W, un, ut, hq), s = functional<NV>(Q, un, ut, hq);
        const double V = NV == 4 ? __fma_rn(ut, W[0], -W[2]) : 0.0;
        if (m == 1) {
          const double hy = __dmul_rn(0.5, __fma_rn(-b1, w.S, W[0]));
          wabs[m] = __dmul_rn(__dmul_rn(sg, z[m]), __fma_rn(-b1, s.S, Q[0]));
          gB = __fma_rn(-hz, w.S, gB);
          const double hb = __dmul_rn(hz, b1);
          ga = __fma_rn(-hb, w.T, ga);
          ga = __fma_rn(hy, fa, ga);
          if (NV == 4) {
            gb = __fma_rn(-hb, V, gb);
            gb = __fma_rn(hy, __fma_rn(ut, fE, fb[2]), gb);
          }
        } else {
          const double si = m == 0 ? ic : -ic;  // row (b1 S +- T/c) / 2
          const double hz2 = __dmul_rn(0.5, hz);
          const double hy = __dmul_rn(0.25, __fma_rn(si, w.T, __dmul_rn(b1, w.S)));
          wabs[m] = __dmul_rn(__dmul_rn(__dmul_rn(0.5, sg), z[m]), __fma_rn(si, s.T, __dmul_rn(b1, s.S)));
          gB = __fma_rn(hz2, w.S, gB);
          gI = __fma_rn(m == 0 ? hz2 : -hz2, w.T, gI);
          ga = __fma_rn(hz2, __fma_rn(si, W[0], __dmul_rn(b1, w.T)), ga);
          const double cs = m == 0 ? -cc : cc;
          ga = __fma_rn(hy, __fma_rn(cs, fE, fb[1]), ga);
          gc = __fma_rn(m == 0 ? -hy : hy, fa, gc);
          yacu = __dadd_rn(yacu, hy);
          if (NV == 4) {
            gb = __fma_rn(__dmul_rn(hz2, b1), V, gb);
            gb = __fma_rn(hy, fb[2], gb);
          }
        }
      }
      if (NV == 4) {
        // both |u_n| fields: one weight at their common cell
        wabs[1] = __fma_rn(pN[cb0 + js[1] * stride] < 0.0 ? -1.0 : 1.0, wabs[2], wabs[1]);
      }
      gH = __dmul_rn(yacu, fE);
      {
        // b1 = gm1/c^2, 1/c and c in terms of c^2 = gm1 (H - |u|^2/2)
        double g2 = __dmul_rn(__dmul_rn(0.5, ic), __fma_rn(-gI, ic2, gc));
        g2 = __fma_rn(-__dmul_rn(b1, ic2), gB, g2);
        g2 = __dmul_rn(gm1, g2);
        gH = __dadd_rn(gH, g2);
        ga = __fma_rn(-g2, un, ga);
        gb = __fma_rn(-g2, ut, gb);
      }
      // the six cells
      double hz[NV], hza[NV];
#pragma unroll
      for (int m = 0; m < NV; ++m) {
        hz[m] = __dmul_rn(0.5, z[m]);
        hza[m] = __dmul_rn(hz[m], alpha[m]);
      }
#pragma unroll 1
      for (int j = 0; j < 6; ++j) {
        const int cj = cb0 + j * stride;
        double A[NV], B[NV];
#pragma unroll
        for (int m = 0; m < NV; ++m) {
          const double2 ab = *reinterpret_cast<const double2*>(tab[m] + 2 * j);
          A[m] = __dmul_rn(hz[m], ab.x);
          B[m] = __dmul_rn(hza[m], ab.y);
        }
        // sum_m x_m L_m
        auto rows = [&](const double (&x)[NV], double (&o)[4]) {
          const double beta = __dmul_rn(b1, __fma_rn(0.5, __dadd_rn(x[0], x[E_]), -x[1]));
          const double del = __dmul_rn(__dmul_rn(0.5, ic), __dsub_rn(x[0], x[E_]));
          o[0] = __fma_rn(hq, beta, __fma_rn(un, del, x[1]));
          o[1] = -__fma_rn(un, beta, del);
          o[2] = 0.0;
          if (NV == 4) {
            o[0] = __fma_rn(-ut, x[2], o[0]);
            o[2] = __fma_rn(-ut, beta, x[2]);
          }
          o[3] = beta;
        };
        double y[4], o[4];
        rows(A, y);
        rows(B, o);
        const double u = pN[cj], v = NV == 4 ? pT[cj] : 0.0, H = C[G::P_H * NC + cj], ri = C[G::P_r * NC + cj];
        // wave-speed terms of the fields whose maximum this cell holds
        const double w0 = js[0] == j ? wabs[0] : 0.0, w3 = js[E_] == j ? wabs[E_] : 0.0;
        const double wu = __dadd_rn(js[1] == j ? wabs[1] : 0.0, __dadd_rn(w0, w3)), wc = __dsub_rn(w3, w0);
        const double k = __dmul_rn(wc, C[G::P_k * NC + cj]);  // through c: k dp - k (p/rho) drho
        // flux Jacobian transposed: s multiplies dp = gm1 (dE - u.dm + |u|^2/2 drho)
        const double s = __dmul_rn(gm1, __dadd_rn(k, __fma_rn(u, y[3], y[1])));
        double hqc = __dmul_rn(0.5 * u, u);
        if (NV == 4) hqc = __fma_rn(0.5 * v, v, hqc);
        const double hy = __fma_rn(H, y[3], __fma_rn(u, y[1], NV == 4 ? __dmul_rn(v, y[2]) : 0.0));  // (u, v, H) . (y1, y2, y3)
        const double wr = __dmul_rn(wu, ri);
        o[0] = __fma_rn(hqc, s, o[0]);
        o[0] = __fma_rn(-u, __dadd_rn(hy, wr), o[0]);
        // p/rho = (gm1/gamma) (H - |u|^2/2)
        o[0] = __fma_rn(-__dmul_rn(k, gm1 / gamma), __dsub_rn(H, hqc), o[0]);
        o[1] = __dadd_rn(o[1], __dadd_rn(__fma_rn(u, y[1], y[0]), __dadd_rn(hy, wr)));
        o[1] = __fma_rn(-u, s, o[1]);
        if (NV == 4) o[2] = __fma_rn(-v, s, __fma_rn(u, y[2], o[2]));
        o[3] = __fma_rn(u, y[3], __dadd_rn(o[3], s));
        if (j == 2 || j == 3) {
          // Roe averages: weights of this side, and the weights' own
          // derivative through sqrt(rho)
          const double wS = j == 2 ? wA : wB;
          double gs = __fma_rn(gH, __dsub_rn(H, Ht), __dmul_rn(ga, __dsub_rn(u, un)));
          if (NV == 4) gs = __fma_rn(gb, __dsub_rn(v, ut), gs);
          const double wr2 = __dmul_rn(wS, ri);
          const double gu = __dmul_rn(wr2, ga), gv = NV == 4 ? __dmul_rn(wr2, gb) : 0.0, gh = __dmul_rn(wr2, gH);
          // d sqrt(rho) / sum = wS / (2 rho) drho
          o[0] = __fma_rn(__dmul_rn(0.5, wr2), gs, o[0]);
          o[0] = __fma_rn(-u, gu, o[0]);
          const double gg = __dmul_rn(gm1, gh);
          o[0] = __fma_rn(gg, hqc, __fma_rn(-H, gh, o[0]));
          o[1] = __dadd_rn(o[1], __fma_rn(-u, gg, gu));
          if (NV == 4) {
            o[0] = __fma_rn(-v, gv, o[0]);
            o[2] = __dadd_rn(o[2], __fma_rn(-v, gg, gv));
          }
          o[3] = __dadd_rn(o[3], __dadd_rn(gh, gg));
        }
#pragma unroll
        for (int n = 0; n < NV; ++n)
          out[(size_t)(j * NV + comp(n)) * nfaces + id] = o[n == E_ ? 3 : n];
      }
    }
  }
}

// One output cell: sum, in a fixed order, the contributions of every face
// whose stencil holds the cell (six per direction; more where periodic images
// or zero-gradient ghost cells alias it).  No atomics: deterministic.
// Memory-bound: it reads the 12 NV contributions of a cell once.
template <int NDIM>
__global__ void __launch_bounds__(256) vjp_gather_kernel(const __grid_constant__ RhsArgs a,
                                                         const double* __restrict__ contrib,
                                                         double* __restrict__ grad) {
  constexpr int NV = NDIM == 2 ? 4 : 3;
  const int nx = a.nx, ny = a.ny;
  const size_t plane = (size_t)nx * ny;
  const size_t cell = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (cell >= plane) return;
  const int ci = (int)(cell % nx), cj = (int)(cell / nx);
  double acc[NV];
#pragma unroll
  for (int n = 0; n < NV; ++n) acc[n] = 0.0;
  const double* base = contrib;
#pragma unroll 1
  for (int dir = 0; dir < NDIM; ++dir) {
    const int N = dir == 0 ? nx : ny;
    const int nl = dir == 0 ? ny : nx;
    const int bc = dir == 0 ? a.bcx : a.bcy;
    const int me = dir == 0 ? ci : cj;
    const int line = dir == 0 ? cj : ci;
    const long long nfaces = (long long)(N + 1) * nl;
    if (me >= 3 && me + 3 < N) {
      // away from the ends of the line: faces me-2 .. me+3, no aliases
      const long long id0 = dir == 0 ? (long long)line * (N + 1) + me - 2 : (long long)(me - 2) * nl + line;
      const long long step = dir == 0 ? 1 : nl;
#pragma unroll
      for (int q = 0; q < 6; ++q)
#pragma unroll
        for (int n = 0; n < NV; ++n) acc[n] += base[(size_t)((5 - q) * NV + n) * nfaces + id0 + q * step];
      base += (size_t)6 * NV * nfaces;
      continue;
    }
    int lo[3], hi[3], nwin = 0;
    if (N <= 16) {
      lo[0] = 0; hi[0] = N; nwin = 1;
    } else {
      lo[nwin] = max(me - 2, 0); hi[nwin] = min(me + 3, N); ++nwin;
      if (bc == 0) {
        if (me + 3 - N >= 0) { lo[nwin] = 0; hi[nwin] = me + 3 - N; ++nwin; }
        if (me - 2 + N <= N) { lo[nwin] = max(me - 2 + N, 0); hi[nwin] = N; ++nwin; }
      }
      // zero-gradient ghost cells alias the edge cells only from faces
      // 0..3 and N-3..N, which the direct window of an edge cell covers
    }
#pragma unroll 1
    for (int w = 0; w < nwin; ++w) {
#pragma unroll 1
      for (int f = lo[w]; f <= hi[w]; ++f) {
        const long long id = dir == 0 ? (long long)line * (N + 1) + f : (long long)f * nl + line;
#pragma unroll
        for (int k = 0; k < 6; ++k) {
          if (wrap_index(f - 3 + k, N, bc) != me) continue;
#pragma unroll
          for (int n = 0; n < NV; ++n) acc[n] += base[(size_t)(k * NV + n) * nfaces + id];
        }
      }
    }
    base += (size_t)6 * NV * nfaces;
  }
#pragma unroll
  for (int n = 0; n < NV; ++n) grad[n * plane + cell] = acc[n];
}

template <class G>
cudaError_t launch_faces(const RhsArgs& a, const double* lam, double* contrib, cudaStream_t s) {
  cudaError_t e =
      cudaFuncSetAttribute(vjp_face_kernel<G>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)G::SMEM);
  if (e != cudaSuccess) return e;
  const long long tiles =
      (long long)(a.nx / G::TX + 1) * (G::NDIM == 2 ? a.ny / G::TY + 1 : 1);  // N + 1 faces per line
  const long long most = 152ll * G::OCC;
  vjp_face_kernel<G><<<(unsigned)(tiles < most ? tiles : most), G::NT, G::SMEM, s>>>(a, lam, contrib);
  return cudaGetLastError();
}

}  // namespace

size_t vjp_scratch_bytes(int ndim, int nx, int ny) {
  const int nv = ndim == 2 ? 4 : 3;
  size_t faces = (size_t)(nx + 1) * ny;
  if (ndim == 2) faces += (size_t)(ny + 1) * nx;
  return faces * 6 * nv * sizeof(double);
}

cudaError_t launch_rhs_vjp(int ndim, const RhsArgs& args, const double* lam, double* grad, double* scratch,
                           cudaStream_t s) {
  RhsArgs a = args;
  a.inv_dx = 1.0 / a.dx;
  a.inv_dy = 1.0 / a.dy;
  // The small tile keeps every SM's quarters in use on small grids: 64^2 in
  // 59 us (87 with two warps a tile instead of four), 200 x 136 in 150; from
  // four waves of the large one on, the halo (13 runs of cells per 16 of faces,
  // against 5 per 4) and the pairs table (24 KB per CTA) decide.
  cudaError_t e;
  if (ndim == 1) e = launch_faces<VTile<1, 32, 1, 32, 4>>(a, lam, scratch, s);
  else if ((long long)(a.nx / 16 + 1) * (a.ny / 16 + 1) < 152 * 2 * 2)
    e = launch_faces<VTile<2, 8, 8, 128, 2>>(a, lam, scratch, s);
  else
    e = launch_faces<VTile<2, 16, 16, 128, 2>>(a, lam, scratch, s);
  if (e != cudaSuccess) return e;
  const size_t cells = (size_t)a.nx * a.ny;
  const unsigned gblocks = (unsigned)((cells + 255) / 256);
  if (ndim == 2) vjp_gather_kernel<2><<<gblocks, 256, 0, s>>>(a, scratch, grad);
  else vjp_gather_kernel<1><<<gblocks, 256, 0, s>>>(a, scratch, grad);
  return cudaGetLastError();
}

}  // namespace neno6
