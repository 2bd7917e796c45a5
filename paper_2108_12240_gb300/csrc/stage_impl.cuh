// The fused RK-stage kernel: reconstruction, HLL/TVDLF face fluxes, geometric
// and GLM sources, the SSP-RK2 stage combination, the Newton conserved-to-
// primitive inversion with its backup and floors, and (stage 2) the per-cell
// CFL rate reduced into one device word.  Included by stage_fp64.cu and
// stage_mixed.cu, which instantiate it for FP64 and FP32 flux arithmetic.
//
// Work decomposition: one CTA owns a column of tx x ty cells of one block and
// marches through its nz planes.  Per plane it reconstructs each cell's edges
// once per direction into shared memory, computes every x-, y- and (top)
// z-face flux of the column once from them, then updates each cell; the
// z-face flux at the top of a plane is carried over as the bottom of the
// next, so no interior face flux is evaluated twice.
#pragma once

#include "amr.h"
#include "bhac_device.cuh"
#include "launch.h"

namespace bhac {

// Largest of the warp's values (none negative, as rates are): their bits order
// like the values, so the FP64 unit is left out.
__device__ __forceinline__ double warp_max_d(double v) {
  unsigned long long b = (unsigned long long)__double_as_longlong(v);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long x = __shfl_xor_sync(0xffffffffu, b, o);
    b = x > b ? x : b;
  }
  return __longlong_as_double((long long)b);
}

// ----------------------------------------------------------------------------
// Geometric + GLM sources for a stationary, phi-independent metric of
// Kerr-Schild structure (derivatives along x1 and x2 only):
//   S(S_j) = 1/2 alpha W^ik d_j gamma_ik + S_i d_j beta^i - E d_j alpha
//   S(tau) = 1/2 W^ik beta^j d_j gamma_ik + W^j_i d_j beta^i - S^j d_j alpha
//   S(psi) = -alpha kappa psi - psi d_i beta^i + ch^2 B^i d_i alpha
// ----------------------------------------------------------------------------
template <typename T, typename R>
BHAC_HD void sources_of(const Met<T>& m, const R* __restrict__ rec, const T* P,
                                           const Derived<T>& s, const T* U, T kappa, T ch2, T* S) {
  const T dal1 = T(rec[C_DAL1]), dal2 = T(rec[C_DAL2]);
  const T db11 = T(rec[C_DBE1_1]), db12 = T(rec[C_DBE1_2]);
  const T Su1 = m.gi11 * U[CS1] + m.gi13 * U[CS3];
  const T Su2 = m.gi22 * U[CS2];
  const T Su3 = m.gi13 * U[CS1] + m.gi33 * U[CS3];
  const T B1_ = P[B1], B2_ = P[B2], B3_ = P[B3];
  const T BvB1 = s.Bv * B1_, BvB2 = s.Bv * B2_, BvB3 = s.Bv * B3_;
  const T W11 = Su1 * s.v1 + s.ptot * m.gi11 - B1_ * B1_ * s.iW2 - BvB1 * s.v1;
  const T W13 = Su3 * s.v1 + s.ptot * m.gi13 - B1_ * B3_ * s.iW2 - BvB1 * s.v3;
  const T W22 = Su2 * s.v2 + s.ptot * m.gi22 - B2_ * B2_ * s.iW2 - BvB2 * s.v2;
  const T W33 = Su3 * s.v3 + s.ptot * m.gi33 - B3_ * B3_ * s.iW2 - BvB3 * s.v3;
  const T G1 = W11 * T(rec[C_DG11_1]) + T(2) * W13 * T(rec[C_DG13_1]) + W22 * T(rec[C_DG22_1]) +
               W33 * T(rec[C_DG33_1]);
  const T G2 = W11 * T(rec[C_DG11_2]) + T(2) * W13 * T(rec[C_DG13_2]) + W22 * T(rec[C_DG22_2]) +
               W33 * T(rec[C_DG33_2]);
  const T E = U[CTAU] + U[CD];
  S[CD] = T(0);
  S[CS1] = T(0.5) * m.al * G1 + U[CS1] * db11 - E * dal1;
  S[CS2] = T(0.5) * m.al * G2 + U[CS1] * db12 - E * dal2;
  S[CS3] = T(0);
  const T Wm11 = U[CS1] * s.v1 + s.ptot - B1_ * s.Bl1 * s.iW2 - BvB1 * s.vl1;  // W^1_1
  const T Wm21 = U[CS1] * s.v2 - B2_ * s.Bl1 * s.iW2 - BvB2 * s.vl1;           // W^2_1
  S[CTAU] = T(0.5) * m.be1 * G1 + Wm11 * db11 + Wm21 * db12 - (Su1 * dal1 + Su2 * dal2);
  S[B1] = T(0); S[B2] = T(0); S[B3] = T(0);
  S[PSI] = -m.al * kappa * P[PSI] - P[PSI] * db11 + ch2 * (B1_ * dal1 + B2_ * dal2);
}

// The same sources from the primitives in one pass (FP64): with X^i = S^i =
// E v^i - (B.v) B^i and Y^i = (B.v) v^i + B^i / W^2 the stress is W^ij = X^i v^j
// - Y^i B^j + p_tot gamma^ij, and tau + D = E - p_tot.  S: the four non-zero
// sources (S_1, S_2, tau, psi); about 95 FP64 instructions where derive,
// cons_of and sources_of take about 125.
template <typename T, typename R>
BHAC_HD void sources_direct(const Met<T>& m, const R* __restrict__ rec, const T* P, T gam_fac, T kappa, T ch2, T* S) {
  const T u1 = P[U1], u2 = P[U2], u3 = P[U3], B1_ = P[B1], B2_ = P[B2], B3_ = P[B3];
  const T ul1 = fma_t(m.g11, u1, m.g13 * u3), ul2 = m.g22 * u2, ul3 = fma_t(m.g13, u1, m.g33 * u3);
  const T Bl1 = fma_t(m.g11, B1_, m.g13 * B3_), Bl2 = m.g22 * B2_, Bl3 = fma_t(m.g13, B1_, m.g33 * B3_);
  const T W2 = fma_t(u1, ul1, fma_t(u2, ul2, fma_t(u3, ul3, T(1))));
  const T iW = rsqrt_t(W2), iW2 = iW * iW;
  const T Bsq = fma_t(B1_, Bl1, fma_t(B2_, Bl2, B3_ * Bl3));
  const T Bv = fma_t(B1_, ul1, fma_t(B2_, ul2, B3_ * ul3)) * iW;
  const T ptot = fma_t(T(0.5), fma_t(Bsq, iW2, Bv * Bv), P[PRS]);
  const T E = fma_t(fma_t(gam_fac, P[PRS], P[RHO]), W2, Bsq);
  const T v1 = u1 * iW, v2 = u2 * iW, v3 = u3 * iW, vl1 = ul1 * iW;
  const T X1 = fma_t(E, v1, -(Bv * B1_)), X2 = fma_t(E, v2, -(Bv * B2_)), X3 = fma_t(E, v3, -(Bv * B3_));
  const T Y1 = fma_t(Bv, v1, iW2 * B1_), Y2 = fma_t(Bv, v2, iW2 * B2_), Y3 = fma_t(Bv, v3, iW2 * B3_);
  const T W11 = fma_t(X1, v1, fma_t(-Y1, B1_, ptot * m.gi11));
  const T W13 = fma_t(X3, v1, fma_t(-Y3, B1_, ptot * m.gi13));
  const T W22 = fma_t(X2, v2, fma_t(-Y2, B2_, ptot * m.gi22));
  const T W33 = fma_t(X3, v3, fma_t(-Y3, B3_, ptot * m.gi33));
  const T W13d = W13 + W13;
  const T G1 = fma_t(W11, T(rec[C_DG11_1]), fma_t(W13d, T(rec[C_DG13_1]),
                     fma_t(W22, T(rec[C_DG22_1]), W33 * T(rec[C_DG33_1]))));
  const T G2 = fma_t(W11, T(rec[C_DG11_2]), fma_t(W13d, T(rec[C_DG13_2]),
                     fma_t(W22, T(rec[C_DG22_2]), W33 * T(rec[C_DG33_2]))));
  const T dal1 = T(rec[C_DAL1]), dal2 = T(rec[C_DAL2]), db11 = T(rec[C_DBE1_1]), db12 = T(rec[C_DBE1_2]);
  const T Et = E - ptot, S1 = fma_t(E, vl1, -(Bv * Bl1)), ha = half_t(m.al);
  S[0] = fma_t(ha, G1, fma_t(S1, db11, -(Et * dal1)));
  S[1] = fma_t(ha, G2, fma_t(S1, db12, -(Et * dal2)));
  const T Wm11 = fma_t(X1, vl1, fma_t(-Y1, Bl1, ptot)), Wm21 = fma_t(X2, vl1, -(Y2 * Bl1));
  S[2] = fma_t(half_t(m.be1), G1, fma_t(Wm11, db11, fma_t(Wm21, db12, fma_t(-X1, dal1, -(X2 * dal2)))));
  S[3] = fma_t(-P[PSI], fma_t(m.al, kappa, db11), ch2 * fma_t(B1_, dal1, B2_ * dal2));
}

// ----------------------------------------------------------------------------
// Conserved -> primitive inversion (FP64).  Two-dimensional Newton-Raphson in
// (Z = rho h W^2, v^2) on the momentum and energy equations (Noble et al.
// 2006), started from the previous primitives; converged when the step
// |dZ| <= tol Z (quadratic convergence: that iterate is accurate to
// round-off).  Backup: bisection on Z of the
// one-dimensional energy residual over a bracket grown from the guess.  Last
// resort: previous primitives (status 3).  Then floors (status 2).
// ----------------------------------------------------------------------------
template <typename T>
struct C2PQ {
  T D, E, S2, Bsq, BS;
};

template <typename T>
BHAC_HD T c2p_v2(const C2PQ<T>& q, T Z) {
  const T iZ = T(1.0) / Z;
  const T num = q.S2 + q.BS * q.BS * (T(2.0) * Z + q.Bsq) * iZ * iZ;
  const T ZB = Z + q.Bsq;
  return num / (ZB * ZB);
}

template <typename T>
BHAC_HD T c2p_f1d(const C2PQ<T>& q, T gf, T v2max, T Z) {
  T v2 = c2p_v2(q, Z);
  v2 = v2 > v2max ? v2max : v2;
  v2 = v2 < T(0.0) ? T(0.0) : v2;
  const T pr = gf * (Z * (T(1.0) - v2) - q.D * sqrt_t(T(1.0) - v2));
  return Z - pr + T(0.5) * q.Bsq * (T(1.0) + v2) - T(0.5) * q.BS * q.BS / (Z * Z) - q.E;
}

// Momentum and energy residuals of the two-dimensional system in (Z, v^2):
//   F1 = (Z + B^2)^2 v^2 - (B.S)^2 (2 Z + B^2) / Z^2 - S^2,
//   F2 = Z - p + B^2 (1 + v^2)/2 - (B.S)^2 / (2 Z^2) - E,
// as f1 = F1 / 2 and f2 = F2 with the constants of c2p_newton_step_t.
template <typename T>
BHAC_HD void c2p_residual_t(const C2PQ<T>& q, T gf, T hB, T hS2, T hBS2, T ec, T gD, T Z, T v2, T& f1, T& f2) {
  const T omv = T(1.0) - v2;
  const T sq = omv * rsqrt_t(omv);
  const T iZ = rcp_t(Z);
  const T h = mul_rn(hBS2, iZ * iZ);
  const T ZB = Z + q.Bsq;
  f1 = fma_t(-h, Z + ZB, fma_t(half_t(ZB) * ZB, v2, -hS2));
  f2 = fma_t(gD, sq, fma_t(-mul_rn(gf, Z), omv, fma_t(hB, v2, Z + ec) - h));
}

// One Jacobian-free Newton-Krylov step at (Z, v^2): the system scaled by rows
// 2/(Z + B^2)^2 and 1/Z, unknowns (dZ/Z, dv^2); GMRES, whose Krylov space is
// the plane after two vectors, on products of the Jacobian with unit vectors
// taken as forward differences with step 2^-26 (backward where the forward
// point would leave 0 <= v^2 < 1).  Writes the step (dZ, dv^2); about 150 FP64
// instructions.
//
// The scaled system at a point: its residual G and products with the Jacobian.
template <typename T>
struct NKSystem {
  const C2PQ<T>& q;
  T gf, hB, hS2, hBS2, ec, gD, Z, v2, rs0, rs1, G1, G2;
  BHAC_HD NKSystem(const C2PQ<T>& q_, T gf_, T hB_, T hS2_, T hBS2_, T ec_, T gD_, T Z_, T v2_)
      : q(q_), gf(gf_), hB(hB_), hS2(hS2_), hBS2(hBS2_), ec(ec_), gD(gD_), Z(Z_), v2(v2_) {
    const T ZB = Z + q.Bsq;
    rs0 = rcp_t(half_t(ZB) * ZB);
    rs1 = rcp_t(Z);
    T F1, F2;
    c2p_residual_t(q, gf, hB, hS2, hBS2, ec, gD, Z, v2, F1, F2);
    G1 = mul_rn(rs0, F1);
    G2 = mul_rn(rs1, F2);
  }
  // the scaled Jacobian times the unit vector (w1, w2) by a one-sided difference
  BHAC_HD void product(T w1, T w2, T& j1, T& j2) const {
    const T eps = T(1.4901161193847656e-08), ieps = T(67108864.0);  // 2^-26, 2^26
    const T w = fma_t(eps, w2, v2);
    const bool back = lt0_x(w) || le_x(T(1.0), w);
    const T e = back ? -eps : eps, s = back ? -ieps : ieps;
    T P1, P2;
    c2p_residual_t(q, gf, hB, hS2, hBS2, ec, gD, fma_t(mul_rn(Z, w1), e, Z), back ? fma_t(e, w2, v2) : w, P1, P2);
    j1 = fma_t(rs0, P1, -G1) * s;
    j2 = fma_t(rs1, P2, -G2) * s;
  }
};

template <typename T>
BHAC_HD void c2p_nk_step_t(const C2PQ<T>& q, T gf, T hB, T hS2, T hBS2, T ec, T gD, T Z, T v2, T& dZ, T& dv2) {
  const NKSystem<T> y(q, gf, hB, hS2, hBS2, ec, gD, Z, v2);
  const T beta = sqrt_t(fma_t(y.G1, y.G1, mul_rn(y.G2, y.G2)));
  dZ = T(0.0);
  dv2 = T(0.0);
  if (!gt0_t(beta)) return;
  const T ib = rcp_t(beta);
  const T a1 = -y.G1 * ib, a2 = -y.G2 * ib;  // first basis vector
  T j1, j2;
  y.product(a1, a2, j1, j2);
  const T h11 = fma_t(j1, a1, mul_rn(j2, a2));
  j1 = fma_t(-h11, a1, j1);
  j2 = fma_t(-h11, a2, j2);
  const T h21 = sqrt_t(fma_t(j1, j1, mul_rn(j2, j2)));
  if (!lt_t(T(1e-14) * abs_t(h11), h21)) {  // a spans an invariant direction
    const T y0 = beta * rcp_t(h11);
    dZ = mul_rn(Z, y0 * a1);
    dv2 = mul_rn(y0, a2);
    return;
  }
  const T i21 = rcp_t(h21);
  const T b1 = j1 * i21, b2 = j2 * i21;  // second basis vector
  T k1, k2;
  y.product(b1, b2, k1, k2);
  const T h12 = fma_t(k1, a1, mul_rn(k2, a2));
  k1 = fma_t(-h12, a1, k1);
  k2 = fma_t(-h12, a2, k2);
  const T h22 = fma_t(k1, b1, mul_rn(k2, b2));
  // min |beta e1 - H y| for the 2 x 2 Hessenberg H: a Givens rotation, then
  // back substitution
  const T r = sqrt_t(fma_t(h11, h11, mul_rn(h21, h21)));
  const T ir = rcp_t(r);
  const T c = h11 * ir, sn = h21 * ir;
  const T R12 = fma_t(c, h12, mul_rn(sn, h22));
  const T R22 = fma_t(-sn, h12, mul_rn(c, h22));
  const T y1 = (-sn * beta) * rcp_t(R22);
  const T y0 = fma_t(c, beta, -mul_rn(R12, y1)) * ir;
  dZ = mul_rn(Z, fma_t(y0, a1, mul_rn(y1, b1)));
  dv2 = fma_t(y0, a2, mul_rn(y1, b2));
}

// The same step for steps two to four with about 110 FP64 instructions: the
// second Krylov vector of a plane is the first one's perpendicular, so the basis
// is a unit vector along the residual, rounded to FP32, and its perpendicular,
// and the solution in that basis comes from the two products by Cramer's rule.
// Residuals, products and solution are FP64; that the basis is orthonormal to
// 1e-7 only does not matter.  False, and no step, where the Jacobian is near
// singular (strongly magnetised cells: there the orthogonalised form above loses
// less) or the residual outside the FP32 range.  Mean step counts and largest
// errors are those of the form above (5000 random states each, as in
// c2p_newton_step_t).  Solving the small system itself in FP32 returned pressures
// off by up to 5% with status 0 at B^2/(rho h) = 1e5, by 4e-9 at 1e3.
template <typename T>
BHAC_HD bool c2p_nk_plane_step_t(const C2PQ<T>& q, T gf, T hB, T hS2, T hBS2, T ec, T gD, T Z, T v2, T& dZ, T& dv2) {
  using L = typename LowOf<T>::type;
  const NKSystem<T> y(q, gf, hB, hS2, hBS2, ec, gD, Z, v2);
  const L g1 = low_t(y.G1), g2 = low_t(y.G2);
  const L beta = sqrt_t(fma_t(g1, g1, mul_rn(g2, g2)));
  if (!lt_t(beta, L(1e15f))) return false;
  dZ = T(0.0);
  dv2 = T(0.0);
  if (!gt0_t(beta)) return true;
  const L ib = rcp_low(beta);
  const T a1 = high_t(-(g1 * ib), T(0)), a2 = high_t(-(g2 * ib), T(0));
  T j1, j2, k1, k2;
  y.product(a1, a2, j1, j2);
  y.product(-a2, a1, k1, k2);
  const T det = fma_t(j1, k2, -mul_rn(j2, k1));
  const L n = abs_t(low_t(j1)) + abs_t(low_t(j2)) + abs_t(low_t(k1)) + abs_t(low_t(k2));
  if (!lt_t(n * n * L(0x1p-14f), abs_t(low_t(det)))) return false;
  const T id = rcp_t(det);
  const T y0 = fma_t(y.G2, k1, -mul_rn(y.G1, k2)) * id, y1 = fma_t(y.G1, j2, -mul_rn(y.G2, j1)) * id;
  dZ = mul_rn(Z, fma_t(y0, a1, -mul_rn(y1, a2)));
  dv2 = fma_t(y0, a2, mul_rn(y1, a1));
  return true;
}

// One Newton step at (Z, v^2) of f1 = F1 / 2 and f2 = F2, with the constants
// hB = B^2/2, hS2 = S^2/2, hBS2 = (B.S)^2/2, ec = B^2/2 - E, gD = g D, hgD =
// g D / 2 (g = (Gamma - 1)/Gamma) and h = (B.S)^2 / (2 Z^2):
//   f1 = (Z+B^2)^2/2 v^2 - h (2 Z + B^2) - S^2/2,
//   f2 = Z + ec + hB v^2 - h - g Z (1 - v^2) + gD sqrt(1 - v^2),
//   j11 = (Z+B^2) (v^2 + 2 h/Z), j12 = (Z+B^2)^2/2, j21 = 1 - g (1 - v^2) + 2 h/Z,
//   j22 = g Z + hB - hgD / sqrt(1 - v^2):
// 43 FP64 instructions.  With ``low`` (steps two to four) the residuals stay
// FP64 and the Jacobian, scaled to the unknowns (dZ/Z, dv^2) and the rows 1/j12
// and 1/Z, is first solved in FP32: 24 FP64 instructions.  An FP32 solve is off
// by at most 2^-21 of e, the sums of the magnitudes of each numerator's terms
// over the determinant, times those of the determinant's own terms over it.  Its
// step is taken in two cases only:
//  - e below 2^-32: the step is the FP64 one to 2^-53 of Z and of 1 - v^2, half a
//    unit in their last place, so the accepted root is the FP64 form's;
//  - dZ/Z above twice the stopping tolerance, so another step follows, and e
//    below 8 steps: an error of 2^-18 of a step, which the next one takes out.
// Any other step (cancelling determinants of strongly magnetised cells, NaN)
// takes the FP64 Jacobian.  On 5000 random states each at rho = 1, p/rho = 1e-2,
// u = 1e-3 .. 30, B^2/(rho h) = 0 .. 1e5 and previous states off by 1e-4 .. 0.3
// the largest errors of p, rho and Z are those of the FP64 form and the mean step
// counts within 0.02 of it.  Without the two tests p came out off by 1.7e-7 with
// status 0 at B^2/(rho h) = 1e5, u = 1e-3, where rounding accounts for 4e-13.
// They cost the torus nothing (most of its cells end with a second step below
// 1e-12), the 12x20x9 blocks of random states 2.3% of a step, the shock tube 1%.
template <typename T>
BHAC_HD void c2p_newton_step_t(const C2PQ<T>& q, T gf, T hB, T hS2, T hBS2, T ec, T gD, T hgD, T tol, T Z, T v2,
                               bool low, T& dZ, T& dv2) {
  const T omv = T(1.0) - v2;
  const T isq = rsqrt_t(omv);
  const T sq = omv * isq;
  const T iZ = rcp_t(Z);
  const T h = mul_rn(hBS2, iZ * iZ);
  const T ZB = Z + q.Bsq;
  const T j12 = half_t(ZB) * ZB;
  const T f1 = fma_t(-h, Z + ZB, fma_t(j12, v2, -hS2));
  const T f2 = fma_t(gD, sq, fma_t(-mul_rn(gf, Z), omv, fma_t(hB, v2, Z + ec) - h));
  if (low && low_range_t(Z) && low_range_t(ZB)) {
    using L = typename LowOf<T>::type;
    const L z = low_t(Z), iz = low_t(iZ), om = low_t(omv), g = low_t(gf);
    const L izb = rcp_low(low_t(ZB)), hz2 = mul_rn(L(2.0f) * low_t(h), iz);
    const L r2 = mul_rn(low_t(f2), iz), r1 = mul_rn(L(2.0f) * low_t(f1) * izb, izb);
    const L a11 = mul_rn(L(2.0f) * (low_t(v2) + hz2) * z, izb), a21 = fma_t(-g, om, L(1.0f)) + hz2;
    const L b = mul_rn(low_t(hB), iz), c = mul_rn(low_t(hgD) * low_t(isq), iz);
    const L a22 = g + (b - c), m22 = g + (b + c);
    const L x12 = mul_rn(r1, a22), x21 = mul_rn(r1, a21), x11 = mul_rn(r2, a11);
    const L id = rcp_low(fma_t(a11, a22, -a21));
    const L q = fma_t(a11, m22, a21) * mul_rn(id, id), dz = (r2 - x12) * id, dv = (x21 - x11) * id;
    const L e = fma_t(om, fma_t(abs_t(r1), m22, abs_t(r2)) * q, (abs_t(x21) + abs_t(x11)) * q);
    const L nz = om * abs_t(dz), nv = abs_t(dv);
    if (le_x(e, L(0x1p-32f) * om) || (lt_t(L(2.0f) * low_t(tol), abs_t(dz)) && le_x(e, L(8.0f) * (nz < nv ? nv : nz)))) {
      dZ = mul_rn(Z, high_t(dz, T(0)));
      dv2 = high_t(dv, T(0));
      return;
    }
  }
  const T hz = mul_rn(h, iZ);
  const T j11 = ZB * fma_t(T(2.0), hz, v2);
  const T j21 = fma_t(T(2.0), hz, fma_t(-gf, omv, T(1.0)));
  const T j22 = fma_t(-hgD, isq, fma_t(gf, Z, hB));
  const T idet = rcp_t(fma_t(j11, j22, -mul_rn(j12, j21)));
  dZ = mul_rn(fma_t(f2, j12, -mul_rn(f1, j22)), idet);
  dv2 = mul_rn(fma_t(f1, j21, -mul_rn(f2, j11)), idet);
}

// Newton starting point from the previous primitives Pg: Z = (rho + Gamma/(Gamma - 1) p) W^2
// and v^2 = u^2 / W^2 with W^2 = 1 + u^2.
template <typename T>
BHAC_HD void c2p_guess(const Met<T>& m, const T* Pg, T gam_fac, T& Z0, T& v2) {
  const T gu1 = m.g11 * Pg[U1] + m.g13 * Pg[U3];
  const T gu2 = m.g22 * Pg[U2];
  const T gu3 = m.g13 * Pg[U1] + m.g33 * Pg[U3];
  const T usq = Pg[U1] * gu1 + Pg[U2] * gu2 + Pg[U3] * gu3;
  Z0 = (Pg[RHO] + gam_fac * Pg[PRS]) * (T(1.0) + usq);
  v2 = usq * rcp_t(T(1.0) + usq);
}

// U undensitized; (Z0g, v2g) the starting point (c2p_guess); Pg the previous
// primitives, variable v at Pg[v ps], read only when every solver fails;
// writes P; returns the status.  gf_d = (Gamma - 1)/Gamma and
// v2max_d = 1 - 1/W_max^2 come precomputed.
// NKM: the primary solver, 0 analytic Newton, 1 Newton-Krylov, 2 chosen at run
// time by nk (kernels that pick the solver at compile time carry no code of the
// other one).
template <typename T, int NKM = 2>
BHAC_HD int con2prim_t(const Met<T>& m, const T* U, const T* Pg, size_t ps, T Z0g, T v2g, T rho_fl, T p_fl,
                       double gf_d, double wmax_d, double v2max_d, double v2skip_d, double tol, int maxit, int nk,
                       T* P) {
  const T gf = T(gf_d);
  const T wmax = T(wmax_d);
  const T v2max = T(v2max_d);
  C2PQ<T> q;
  q.D = U[CD];
  q.E = U[CTAU] + U[CD];
  const T Su1 = m.gi11 * U[CS1] + m.gi13 * U[CS3];
  const T Su2 = m.gi22 * U[CS2];
  const T Su3 = m.gi13 * U[CS1] + m.gi33 * U[CS3];
  const T Bl1 = m.g11 * U[B1] + m.g13 * U[B3];
  const T Bl2 = m.g22 * U[B2];
  const T Bl3 = m.g13 * U[B1] + m.g33 * U[B3];
  q.S2 = Su1 * U[CS1] + Su2 * U[CS2] + Su3 * U[CS3];
  q.Bsq = U[B1] * Bl1 + U[B2] * Bl2 + U[B3] * Bl3;
  q.BS = U[B1] * U[CS1] + U[B2] * U[CS2] + U[B3] * U[CS3];
  bool fin = true;
  for (int v = 0; v < NV; ++v) fin = fin && finite_t(U[v]);
  int status = 0;
  bool solved = false;
  T Z = T(0.0), v2 = T(0.0);
  T W = T(0.0), sq = T(0.0);  // 1/sqrt(1 - v^2) and sqrt(1 - v^2) of the accepted solution
  if (fin && gt0_t(q.D) && gt0_t(q.E)) {
    const T Z0 = (gt0_t(Z0g) && finite_t(Z0g)) ? Z0g : q.E;
    Z = Z0;
    v2 = v2g;
    const T hB = half_t(q.Bsq), hS2 = half_t(q.S2), hBS2 = half_t(q.BS * q.BS), ec = hB - q.E;
    const T gD = gf * q.D, hgD = half_t(gD);
    for (int it = 0; it < maxit; ++it) {
      T dZ, dv2;
      if (NKM == 1 || (NKM == 2 && nk)) {
        if (!(it >= 1 && it <= 3 && c2p_nk_plane_step_t(q, gf, hB, hS2, hBS2, ec, gD, Z, v2, dZ, dv2)))
          c2p_nk_step_t(q, gf, hB, hS2, hBS2, ec, gD, Z, v2, dZ, dv2);
      } else {
        c2p_newton_step_t(q, gf, hB, hS2, hBS2, ec, gD, hgD, T(tol), Z, v2, it >= 1 && it <= 3, dZ, dv2);
      }
      T Zn = Z + dZ, v2n = v2 + dv2;
      if (!gt0_t(Zn)) Zn = half_t(Z);
      if (lt0_x(v2n)) v2n = half_t(v2);
      if (le_x(T(1.0), v2n)) v2n = half_t(v2 + T(1.0));
      const bool conv = le_x(abs_t(Zn - Z), T(tol) * Zn);
      Z = Zn;
      v2 = v2n;
      if (!finite_t(Z) || !finite_t(v2)) break;
      if (conv) {
        solved = true;
        break;
      }
    }
    if (solved && !(le_x(T(0.0), v2) && lt_t(v2, T(1.0)) && gt0_t(Z))) solved = false;
    // the recovered density D sqrt(1 - v^2) must be positive; sqrt(1 - v^2)
    // is formed as (1 - v^2) / sqrt(1 - v^2), the factor the recovery uses
    if (solved) {
      W = rsqrt_t(T(1.0) - v2);
      sq = (T(1.0) - v2) * W;
      if (!gt0_t(q.D * sq)) solved = false;
    }
    if (!solved) {
      T lo = Z0, hi = Z0;
      int k = 0;
      while (c2p_f1d(q, gf, v2max, lo) > T(0.0) && k < 200) {
        lo = lo * T(0.5);
        ++k;
      }
      k = 0;
      while (c2p_f1d(q, gf, v2max, hi) < T(0.0) && k < 200) {
        hi = hi * T(2.0);
        ++k;
      }
      if (c2p_f1d(q, gf, v2max, lo) <= T(0.0) && c2p_f1d(q, gf, v2max, hi) >= T(0.0)) {
        for (int it = 0; it < 200 && hi - lo > T(4e-16) * hi; ++it) {
          const T mid = T(0.5) * (lo + hi);
          if (c2p_f1d(q, gf, v2max, mid) > T(0.0))
            hi = mid;
          else
            lo = mid;
        }
        Z = T(0.5) * (lo + hi);
        v2 = c2p_v2(q, Z);
        v2 = v2 > v2max ? v2max : v2;
        v2 = v2 < T(0.0) ? T(0.0) : v2;
        if (finite_t(Z) && Z > T(0.0)) {
          solved = true;
          status = 1;
          W = rsqrt_t(T(1.0) - v2);
          sq = (T(1.0) - v2) * W;
        }
      }
    }
  }
  if (solved) {
    // W = 1/sqrt(1 - v^2) and sqrt(1 - v^2) came from one reciprocal square
    // root; 1/Z and 1/(Z + B^2) from one reciprocal of their product
    const T omv = T(1.0) - v2;
    const T ZB = Z + q.Bsq;
    const T r = rcp_t(Z * ZB);
    P[RHO] = q.D * sq;
    P[PRS] = gf * (Z * omv - q.D * sq);
    const T c = W * Z * r;
    const T bz = q.BS * ZB * r;
    P[U1] = c * (Su1 + bz * U[B1]);
    P[U2] = c * (Su2 + bz * U[B2]);
    P[U3] = c * (Su3 + bz * U[B3]);
  } else {
    status = 3;
    P[RHO] = Pg[RHO * ps];
    P[PRS] = Pg[PRS * ps];
    P[U1] = Pg[U1 * ps];
    P[U2] = Pg[U2 * ps];
    P[U3] = Pg[U3 * ps];
  }
  P[B1] = U[B1];
  P[B2] = U[B2];
  P[B3] = U[B3];
  P[PSI] = U[PSI];
  bool fl = false;
  if (!le_x(rho_fl, P[RHO])) {
    P[RHO] = rho_fl;
    fl = true;
  }
  if (!le_x(p_fl, P[PRS])) {
    P[PRS] = p_fl;
    fl = true;
  }
  // a Newton root's v^2 is the primitives' 1 - 1/W^2 to within its tolerance,
  // so 2% below the limit the ceiling needs no second look
  if (status != 0 || !lt_t(v2, T(v2skip_d))) {
    const T gu1 = m.g11 * P[U1] + m.g13 * P[U3];
    const T gu2 = m.g22 * P[U2];
    const T gu3 = m.g13 * P[U1] + m.g33 * P[U3];
    const T usq = P[U1] * gu1 + P[U2] * gu2 + P[U3] * gu3;
    if (lt_t(wmax * wmax, T(1.0) + usq)) {
      const T sc = sqrt_t((wmax * wmax - T(1.0)) / usq);
      P[U1] = P[U1] * sc;
      P[U2] = P[U2] * sc;
      P[U3] = P[U3] * sc;
      fl = true;
    }
  }
  if (status == 3) return 3;
  return fl ? 2 : status;
}

template <int NKM>
static __device__ __forceinline__ int con2prim(const Met<double>& m, const double* U, const double* Pg, size_t ps,
                                            double Z0, double v20, double rho_fl, double p_fl, const StageArgs& a,
                                            double* P) {
  return con2prim_t<double, NKM>(m, U, Pg, ps, Z0, v20, rho_fl, p_fl, a.c2p_gf, a.wmax, a.c2p_v2max, a.c2p_v2skip, a.c2p_tol,
                                 a.c2p_maxit, a.c2p_nk, P);
}

// CFL rate of one cell: sum over active d of c_d / dx_d, where c_d is the
// largest of |lambda+-| and ch alpha sqrt(gamma^dd) + |beta^d|.
template <typename T, int DIM>
BHAC_HD T cfl_rate_t(const Met<T>& m, const T* acg, const T* P, double gam, double gam_fac, double ch,
                     const double* idx) {
  if (ch >= 1.0) {
    // The fast-magnetosonic bound boosts a comoving speed a < 1 and so never
    // leaves the light cone: with ch >= 1 the cleaning speed is the largest.
    T rate = T(0.0);
    for (int d = 0; d < DIM; ++d) rate = rate + (T(ch) * acg[d] + (d == 0 ? abs_t(m.be1) : T(0.0))) * T(idx[d]);
    return rate;
  }
  Derived<T> s;
  derive(m, P, T(gam_fac), s);
  T rate = T(0.0);
  for (int d = 0; d < DIM; ++d) {
    T lm, lp;
    speeds_of(m, P, s, d, T(gam), lm, lp);
    const T alp = abs_t(lp), alm = abs_t(lm);
    T c = alp > alm ? alp : alm;
    const T cg = T(ch) * acg[d] + (d == 0 ? abs_t(m.be1) : T(0.0));
    c = cg > c ? cg : c;
    rate = rate + c * T(idx[d]);
  }
  return rate;
}

// The largest CFL rate so far and a cell's: with ch >= 1 the rate depends on the
// metric only and is tabulated (C_RATE; flat: one constant per level).  SCREEN
// (constrained transport, loads, the stand-alone reduction): the signal speeds
// stay inside the light cone for a physical state and Gamma <= 2, so a cell
// whose light-cone rate (FP32 records, 1e-5 added for their rounding) is below
// the largest rate found so far cannot change the maximum, and its three wave
// speeds (125 FP64 instructions) are not formed.  ``seen``: the bits of a rate
// already in the result.  Loading, face loading and two mixed steps of
// constrained transport on 192x96x96 cells went from 8.97 to 7.96 ms with this
// and cons_direct.  (In the stage kernel the test's registers cost more in
// spills than it saves: 2.5% of the mixed step.)
template <int DIM, bool FLAT, bool SCREEN>
__device__ __forceinline__ void cfl_max(const StageArgs& a, const LevelGeo& geo, const Met<double>& m,
                                        const double* crec, const float* crec32, const double* P,
                                        unsigned long long seen, double& rate_max) {
  double rate;
  if (a.ch >= 1.0) {
    rate = FLAT ? geo.rate : crec[C_RATE];
  } else {
    if (SCREEN && !FLAT && a.gam <= 2.0 && gt0_t(P[RHO]) && !lt0_x(P[PRS])) {
      float b = (crec32[C_ACG1] + fabsf(crec32[C_BE1])) * geo.idx_f[0] + crec32[C_ACG2] * geo.idx_f[1];
      if (DIM == 3) b += crec32[C_ACG3] * geo.idx_f[2];
      const double s = __longlong_as_double((long long)seen);
      if (b * 1.00001f < low_t(lt_t(rate_max, s) ? s : rate_max)) return;
    }
    double acg[3] = {1.0, 1.0, 1.0};
    if (!FLAT) {
      acg[0] = crec[C_ACG1];
      acg[1] = crec[C_ACG2];
      acg[2] = crec[C_ACG3];
    }
    rate = cfl_rate_t<double, DIM>(m, acg, P, a.gam, a.gam_fac, a.ch, geo.idx);
  }
  rate_max = lt_t(rate_max, rate) ? rate : rate_max;
}
// the rate already in the result (0 where none is wanted)
__device__ __forceinline__ unsigned long long cfl_seen(const StageArgs& a) {
  return a.ch < 1.0 && a.smax_out ? *reinterpret_cast<volatile unsigned long long*>(a.smax_out) : 0ull;
}

// ----------------------------------------------------------------------------
// Riemann solve at one face: states PL, PR (already reconstructed), face
// metric m, GLM speed factor acg = alpha sqrt(gamma^dd).  HLL or TVDLF; the
// GLM pair (normal B, psi) uses signal speeds no smaller than
// +-ch alpha sqrt(gamma^dd) - beta^d.  Writes the flux densitized by sqrt(gamma).
// ----------------------------------------------------------------------------
//
// Two evaluations.  The plain one forms U and F of both states and combines
// them.  FP64 (ShiftedFlux) uses that HLL and TVDLF need each state only
// through G = F - s U with s the signal speed of the other side:
//   HLL:    sg (s+ G_L(s-) - s- G_R(s+)) / (s+ - s-),
//   TVDLF:  sg (G_L(-c) + G_R(c)) / 2,
// and that with V = alpha v^d - beta^d - s, b = alpha B^d, E' = rho h W^2 + B^2
// and E' - D = tau + p_tot, neither S_j, tau nor their fluxes are needed:
//   G(S_j)  = v_j (V E' - b B.v) - B_j (V B.v + b / W^2) + alpha p_tot delta^d_j,
//   G(tau)  = (E' - D) V - b B.v + (beta^d + s) p_tot,   G(D) = D V,
//   G(B^j)  = V B^j - b v^j + beta^j B^d + alpha gamma^dj psi  (j != d),
//   G(B^d)  = alpha gamma^dd psi - s_g B^d,   G(psi) = ch^2 b - (beta^d + s_g) psi.
// About 210 FP64 instructions per face against about 310: the FP64 unit
// (two lanes per clock and SM) bounds the FP64 form, and its faces are more
// than half of its instructions (192x96x96 torus: step 14.5 -> 11.5 ms;
// constrained transport on 128x64x64 cells: 5.4 -> 4.3 ms).
template <typename T>
struct ShiftedFlux {
  static constexpr bool value = false;
};
template <>
struct ShiftedFlux<double> {
  static constexpr bool value = true;
};

// What the face solve needs of one state (FP64 form).  Products that are later
// added are rounded on their own (mul_rn), so every kernel forms the same bits.
template <typename T>
struct FaceState {
  T ul1, ul2, ul3, Bl1, Bl2, Bl3, iW, iW2, Bv, ptot, D, ZB, Vd, lm, lp;
};

template <typename T>
BHAC_HD void face_state(const Met<T>& m, const T* P, int d, T gam, T gam_fac, FaceState<T>& s) {
  const T u1 = P[U1], u2 = P[U2], u3 = P[U3], B1_ = P[B1], B2_ = P[B2], B3_ = P[B3];
  s.ul1 = fma_t(m.g11, u1, m.g13 * u3);
  s.ul2 = m.g22 * u2;
  s.ul3 = fma_t(m.g13, u1, m.g33 * u3);
  s.Bl1 = fma_t(m.g11, B1_, m.g13 * B3_);
  s.Bl2 = m.g22 * B2_;
  s.Bl3 = fma_t(m.g13, B1_, m.g33 * B3_);
  const T W2 = fma_t(u1, s.ul1, fma_t(u2, s.ul2, fma_t(u3, s.ul3, T(1))));
  s.iW = rsqrt_t(W2);
  s.iW2 = s.iW * s.iW;
  const T Bsq = fma_t(B1_, s.Bl1, fma_t(B2_, s.Bl2, B3_ * s.Bl3));
  s.Bv = fma_t(B1_, s.ul1, fma_t(B2_, s.ul2, B3_ * s.ul3)) * s.iW;
  const T b2 = fma_t(Bsq, s.iW2, s.Bv * s.Bv);
  const T rhoh = fma_t(gam_fac, P[PRS], P[RHO]);
  s.ptot = fma_t(T(0.5), b2, P[PRS]);
  s.D = mul_rn(P[RHO], W2 * s.iW);
  s.ZB = fma_t(rhoh, W2, Bsq);
  // wave speeds (speeds_of): with E - G = rho h - Gamma p and R = E - v^2 G =
  // (E - G) + G / W^2
  const T G = fma_t(gam, P[PRS], b2);
  const T EG = fma_t(-gam, P[PRS], rhoh);
  const T R = fma_t(s.iW2, G, EG);
  const T vd = sel3(d, u1, u2, u3) * s.iW;
  const T c = mul_rn(vd, EG);
  const T gidd = sel3(d, m.gi11, m.gi22, m.gi33);
  T disc = (G * s.iW2) * fma_t(-vd, c, gidd * R);
  disc = gt0_t(disc) ? disc : T(0);
  const T sq = sqrt_t(disc);
  const T ir = m.al * rcp_t(R);
  if (d == 0) {
    s.Vd = fma_t(m.al, vd, -m.be1);
    s.lp = fma_t(c + sq, ir, -m.be1);
    s.lm = fma_t(c - sq, ir, -m.be1);
  } else {
    s.Vd = mul_rn(m.al, vd);
    s.lp = mul_rn(c + sq, ir);
    s.lm = mul_rn(c - sq, ir);
  }
}

// G = F - s U of a state (s_g for B^d and psi).
template <typename T>
BHAC_HD void shifted_flux(const Met<T>& m, const T* P, const FaceState<T>& f, int d, T ch2, T s, T s_g, T* G) {
  const T Bd = sel3(d, P[B1], P[B2], P[B3]);
  const T gidd = sel3(d, m.gi11, m.gi22, m.gi33);
  const T V = f.Vd - s;
  const T b = m.al * Bd, bBv = b * f.Bv, alpsi = m.al * P[PSI];
  const T A = fma_t(V, f.ZB, -bBv) * f.iW, C = fma_t(V, f.Bv, b * f.iW2);
  G[CD] = f.D * V;
  G[CS1] = fma_t(f.ul1, A, -(f.Bl1 * C));
  G[CS2] = fma_t(f.ul2, A, -(f.Bl2 * C));
  G[CS3] = fma_t(f.ul3, A, -(f.Bl3 * C));
  if (d == 0) G[CS1] = fma_t(m.al, f.ptot, G[CS1]);
  if (d == 1) G[CS2] = fma_t(m.al, f.ptot, G[CS2]);
  if (d == 2) G[CS3] = fma_t(m.al, f.ptot, G[CS3]);
  G[CTAU] = fma_t(d == 0 ? m.be1 + s : s, f.ptot, fma_t(f.ZB - f.D, V, -bBv));
  const T k = b * f.iW;
  const T gB = fma_t(-s_g, Bd, alpsi * gidd);
  if (d == 0) {
    G[B1] = gB;
    G[B2] = fma_t(V, P[B2], -(k * P[U2]));
    G[B3] = fma_t(alpsi, m.gi13, fma_t(V, P[B3], -(k * P[U3])));
  } else {
    G[B1] = fma_t(m.be1, Bd, fma_t(V, P[B1], -(k * P[U1])));
    if (d == 1) {
      G[B2] = gB;
      G[B3] = fma_t(V, P[B3], -(k * P[U3]));
    } else {
      G[B1] = fma_t(alpsi, m.gi13, G[B1]);
      G[B2] = fma_t(V, P[B2], -(k * P[U2]));
      G[B3] = gB;
    }
  }
  G[PSI] = fma_t(-(d == 0 ? m.be1 + s_g : s_g), P[PSI], ch2 * b);
}

template <typename T>
BHAC_HD void riemann_shifted(const Met<T>& m, T acg, const T* PL, const T* PR, int d, int riemann, T gam, T gam_fac,
                             T ch, T* out) {
  const T ch2 = ch * ch;
  FaceState<T> sL, sR;
  face_state(m, PL, d, gam, gam_fac, sL);
  face_state(m, PR, d, gam, gam_fac, sR);
  const T bed = d == 0 ? m.be1 : T(0);
  const T lgp = fma_t(acg, ch, -bed), lgm = fma_t(-acg, ch, -bed);
  T G[NV];
  if (riemann == 0) {
    T lp = T(0), lm = T(0);
    lp = lt_t(lp, sL.lp) ? sL.lp : lp;
    lp = lt_t(lp, sR.lp) ? sR.lp : lp;
    lm = lt_t(sL.lm, lm) ? sL.lm : lm;
    lm = lt_t(sR.lm, lm) ? sR.lm : lm;
    const T lpg = lt_t(lp, lgp) ? lgp : lp, lmg = lt_t(lgm, lm) ? lgm : lm;
    const T wh = lp - lm, wg = lpg - lmg;
    const bool okh = gt0_t(wh), okg = gt0_t(wg);
    // both fan widths' reciprocals from one; a degenerate fan (no signal speed
    // at all) falls back to the mean flux
    const T r = okh && okg ? rcp_t(wh * wg) * m.sg : T(0);
    const T ih = okh ? (okg ? wg * r : rcp_t(wh) * m.sg) : T(0);
    const T ihg = okg ? (okh ? wh * r : rcp_t(wg) * m.sg) : T(0);
    const T hs = T(0.5) * m.sg;
    const T aL = okh ? ih * lp : hs, aR = okh ? ih * lm : -hs;
    const T gL = okg ? ihg * lpg : hs, gR = okg ? ihg * lmg : -hs;
    shifted_flux(m, PL, sL, d, ch2, lm, lmg, G);
    for (int v = 0; v < NV; ++v) out[v] = ((v == PSI) || (v == B1 + d) ? gL : aL) * G[v];
    shifted_flux(m, PR, sR, d, ch2, lp, lpg, G);
    for (int v = 0; v < NV; ++v) out[v] = fma_t(-((v == PSI) || (v == B1 + d) ? gR : aR), G[v], out[v]);
  } else {
    T c = abs_t(sL.lp);
    const T almL = abs_t(sL.lm), alpR = abs_t(sR.lp), almR = abs_t(sR.lm);
    c = lt_t(c, almL) ? almL : c;
    c = lt_t(c, alpR) ? alpR : c;
    c = lt_t(c, almR) ? almR : c;
    const T agp = abs_t(lgp), agm = abs_t(lgm);
    T cg = c;
    cg = lt_t(cg, agp) ? agp : cg;
    cg = lt_t(cg, agm) ? agm : cg;
    const T hs = T(0.5) * m.sg;
    shifted_flux(m, PL, sL, d, ch2, -c, -cg, out);
    shifted_flux(m, PR, sR, d, ch2, c, cg, G);
    for (int v = 0; v < NV; ++v) out[v] = hs * (out[v] + G[v]);
  }
}

template <typename T>
BHAC_HD void riemann_flux(const Met<T>& m, T acg, const T* PL, const T* PR, int d, int riemann, T gam, T gam_fac,
                          T ch, T* out) {
  if constexpr (ShiftedFlux<T>::value) {
    riemann_shifted(m, acg, PL, PR, d, riemann, gam, gam_fac, ch, out);
    return;
  }
  const T ch2 = ch * ch;
  Derived<T> sL, sR;
  derive(m, PL, gam_fac, sL);
  derive(m, PR, gam_fac, sR);
  T lmL, lpL, lmR, lpR;
  speeds_of(m, PL, sL, d, gam, lmL, lpL);
  speeds_of(m, PR, sR, d, gam, lmR, lpR);
  const T bed = d == 0 ? m.be1 : T(0);
  const T lgp = acg * ch - bed, lgm = -acg * ch - bed;
  T acc[NV];
  T U[NV], F[NV];
  if (riemann == 0) {
    T lp = T(0), lm = T(0);
    lp = lt_t(lp, lpL) ? lpL : lp;
    lp = lt_t(lp, lpR) ? lpR : lp;
    lm = lt_t(lmL, lm) ? lmL : lm;
    lm = lt_t(lmR, lm) ? lmR : lm;
    const T lpg = lt_t(lp, lgp) ? lgp : lp, lmg = lt_t(lgm, lm) ? lgm : lm;
    const T wh = lp - lm, wg = lpg - lmg;
    const bool okh = gt0_t(wh), okg = gt0_t(wg);
    // both fan widths' reciprocals from one division
    const T r = okh && okg ? rcp_t(wh * wg) : T(0);
    const T ih = okh ? (okg ? wg * r : rcp_t(wh)) : T(0);
    const T ihg = okg ? (okh ? wh * r : rcp_t(wg)) : T(0);
    cons_of(PL, sL, U);
    flux_of(m, PL, sL, U, d, ch2, F);
    T FL[NV];
    for (int v = 0; v < NV; ++v) {
      const bool g = (v == PSI) || (v == B1 + d);
      const T p = g ? lpg : lp, q = g ? lmg : lm;
      acc[v] = p * (F[v] - q * U[v]);
      FL[v] = F[v];
    }
    cons_of(PR, sR, U);
    flux_of(m, PR, sR, U, d, ch2, F);
    for (int v = 0; v < NV; ++v) {
      const bool g = (v == PSI) || (v == B1 + d);
      const T p = g ? lpg : lp, q = g ? lmg : lm, ihv = g ? ihg : ih;
      // a degenerate fan (no signal speed at all) falls back to the mean flux
      out[v] = m.sg * ((g ? okg : okh) ? (acc[v] - q * (F[v] - p * U[v])) * ihv : T(0.5) * (FL[v] + F[v]));
    }
  } else {
    const T alpL = abs_t(lpL), almL = abs_t(lmL), alpR = abs_t(lpR), almR = abs_t(lmR);
    T c = alpL;
    c = lt_t(c, almL) ? almL : c;
    c = lt_t(c, alpR) ? alpR : c;
    c = lt_t(c, almR) ? almR : c;
    const T agp = abs_t(lgp), agm = abs_t(lgm);
    T cg = c;
    cg = lt_t(cg, agp) ? agp : cg;
    cg = lt_t(cg, agm) ? agm : cg;
    cons_of(PL, sL, U);
    flux_of(m, PL, sL, U, d, ch2, F);
    for (int v = 0; v < NV; ++v) {
      const bool g = (v == PSI) || (v == B1 + d);
      acc[v] = F[v] + (g ? cg : c) * U[v];
    }
    cons_of(PR, sR, U);
    flux_of(m, PR, sR, U, d, ch2, F);
    for (int v = 0; v < NV; ++v) {
      const bool g = (v == PSI) || (v == B1 + d);
      out[v] = m.sg * (T(0.5) * (acc[v] + F[v]) - T(0.5) * (g ? cg : c) * U[v]);
    }
  }
}

// ----------------------------------------------------------------------------
// Face fluxes, densitized by the face sqrt(gamma).  (ig, jg, kg): ghosted
// coordinates of the cell on the high side of the face; (I1, I2): level-global
// table indices of the face.
// ----------------------------------------------------------------------------
// Axis faces carry no flux (sqrt(gamma) = 0 there).
template <bool FLAT>
__device__ __forceinline__ bool axis_face(const StageArgs& a, const LevelGeo& geo, int d, int I2) {
  return !FLAT && d == 1 && ((I2 == 0 && a.axis_lo1) || (I2 == geo.N2 && a.axis_hi1));
}

// Reconstructed states with a non-positive density or pressure fall back to
// the two adjacent cell values (first order).  c0: ghosted index of the high cell.
template <typename T>
__device__ __forceinline__ void positivity_fallback(const StageArgs& a, const T* __restrict__ Pb, int sd, int c0,
                                                    T PL[NV], T PR[NV]) {
  if (!gt0_t(PL[RHO]) || !gt0_t(PL[PRS]) || !gt0_t(PR[RHO]) || !gt0_t(PR[PRS])) {
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      const T* p = Pb + (size_t)v * a.ncell + c0;
      PL[v] = p[-sd];
      PR[v] = p[0];
    }
  }
}

// Face metric and Riemann solve of the states PL, PR.
template <typename T, bool FLAT>
__device__ __forceinline__ void face_solve(const StageArgs& a, const LevelGeo& geo, int d, int I1, int I2,
                                           const T PL[NV], const T PR[NV], T* out, int ostride) {
  Met<T> m;
  T acg;
  if (FLAT) {
    m = flat_metric<T>();
    acg = T(1);
  } else if (sizeof(T) == 8) {
    const double* rec = d == 0 ? geo.tf1 + (size_t)(I2 * (geo.N1 + 1) + I1) * FREC
                               : (d == 1 ? geo.tf2 + (size_t)(I2 * geo.N1 + I1) * FREC
                                         : geo.tc + (size_t)(I2 * geo.N1 + I1) * CREC);
    m = load_face_metric<T>(rec);
    acg = T(d == 2 ? rec[C_ACG3] : rec[F_ACG]);
  } else {
    const float* rec = d == 0 ? geo.tf1_32 + (size_t)(I2 * (geo.N1 + 1) + I1) * FREC
                              : (d == 1 ? geo.tf2_32 + (size_t)(I2 * geo.N1 + I1) * FREC
                                        : geo.tc32 + (size_t)(I2 * geo.N1 + I1) * CREC);
    m = load_face_metric<T>(rec);
    acg = T(d == 2 ? rec[C_ACG3] : rec[F_ACG]);
  }
  T F[NV];
  riemann_flux(m, acg, PL, PR, d, a.riemann, pick<T>(a.gam, a.gam_f), pick<T>(a.gam_fac, a.gam_fac_f),
               pick<T>(a.ch, a.ch_f), F);
#pragma unroll
  for (int v = 0; v < NV; ++v) out[v * ostride] = F[v];
}

// One face flux from the six-point stencil across the face (the
// warp-specialised kernel's per-face form).
template <typename T, bool FLAT>
__device__ __forceinline__ void face_flux(const StageArgs& a, const LevelGeo& geo, const T* __restrict__ Pb, int d,
                                          int ig, int jg, int kg, int I1, int I2, T* out, int ostride) {
  const int sd = d == 0 ? 1 : (d == 1 ? a.Nx : a.Nx * a.Ny);
  const int c0 = (kg * a.Ny + jg) * a.Nx + ig;
  if (axis_face<FLAT>(a, geo, d, I2)) {
#pragma unroll
    for (int v = 0; v < NV; ++v) out[v * ostride] = T(0);
    return;
  }
  T PL[NV], PR[NV];
#pragma unroll
  for (int v = 0; v < NV; ++v) {
    const T* p = Pb + (size_t)v * a.ncell + c0;
    const T s0 = p[-3 * sd], s1 = p[-2 * sd], s2 = p[-sd], s3 = p[0], s4 = p[sd], s5 = p[2 * sd];
    recon_var(a.recon, s0, s1, s2, s3, s4, s5, PL[v], PR[v]);
  }
  positivity_fallback(a, Pb, sd, c0, PL, PR);
  face_solve<T, FLAT>(a, geo, d, I1, I2, PL, PR, out, ostride);
}

// Unsigned division by a run-time constant d: floor(n / d) = umulhi(n, m) with
// m = ceil(2^32 / d), exact while n (m d - 2^32) < 2^32 (tile indices: n < 2^20,
// d < 2^12).
struct FastDiv {
  unsigned d, m;
  __device__ __forceinline__ explicit FastDiv(unsigned d_) : d(d_), m(0xFFFFFFFFu / d_ + 1u) {}
  __device__ __forceinline__ void split(int n, int& q, int& r) const {
    q = d == 1u ? n : (int)__umulhi((unsigned)n, m);
    r = n - q * (int)d;
  }
};

// Both reconstructed edges along d of the cell at ghosted index c, all
// variables: aL (low face) to L[v * sl], aR (high face) to R[v * sr].  Every
// load is issued before the first store: the compiler cannot move a load
// above a shared-memory store, and one exposed L2 latency per variable cost
// more than the arithmetic.
template <typename T>
__device__ __forceinline__ void cell_edges(const StageArgs& a, const T* __restrict__ Pb, int sd, int c, T* L, int sl,
                                           T* R, int sr) {
  T q[NV][5];
#pragma unroll
  for (int v = 0; v < NV; ++v)
#pragma unroll
    for (int m = 0; m < 5; ++m) q[v][m] = Pb[(size_t)v * a.ncell + c + (m - 2) * sd];
#pragma unroll
  for (int v = 0; v < NV; ++v) {
    T l, r;
    recon_edges(a.recon, q[v][0], q[v][1], q[v][2], q[v][3], q[v][4], l, r);
    L[v * sl] = l;
    R[v * sr] = r;
  }
}

// Cells per strip of strip_edges.
constexpr int kStrip = 6;

// Both edges along one direction of n <= S consecutive cells of one variable:
// p points at the first cell, sd is the cell stride, so the stride of the
// outputs.  A PPM interface value belongs to the two cells beside it and is
// formed once per strip instead of once per cell, and a strip of S cells loads
// S + 4 values instead of 5 S.  One (strip, variable) pair is one thread's
// task, so a thread holds one load batch in flight and the tasks of a plane
// (864 for a 16x16 tile) fill the CTA evenly.  Against one thread per cell
// looping over the variables, whose loads waited for the stores before them,
// the reconstruction of a plane of a 16x16 mixed tile fell from 28.7k to 9.5k
// cycles (flat 12x20x9 blocks) and the mixed step on 192x96x96 cells from
// 2.99 to 2.59 ms; FP64, bound by its arithmetic, 16.8 to 15.9 ms.
template <typename T, int S>
__device__ __forceinline__ void strip_edges(int recon, const T* __restrict__ p, int sd, int n, T* L, T* R, int so) {
  T q[S + 4];
#pragma unroll
  for (int m = 0; m < S + 4; ++m) q[m] = m < n + 4 ? p[(m - 2) * sd] : T(0);
  if (PpmByDifferences<T>::value && recon == 0) {
    T d[S + 3];
#pragma unroll
    for (int m = 0; m < S + 3; ++m) d[m] = q[m + 1] - q[m];
    T w = ppm_dev(d[0], d[1], d[2]);
#pragma unroll
    for (int m = 0; m < S; ++m) {
      const T wn = ppm_dev(d[m + 1], d[m + 2], d[m + 3]);
      T l = w - d[m + 1], r = wn;
      limit_dev(l, r);
      if (m < n) {
        L[m * so] = low_edge(q[m + 2], l, d[m + 1], q[m + 1]);
        R[m * so] = high_edge(q[m + 2], r, d[m + 2], q[m + 3]);
      }
      w = wn;
    }
  } else if (recon == 0) {
    T f[S + 1];
#pragma unroll
    for (int m = 0; m <= S; ++m) f[m] = ppm_iface(q[m], q[m + 1], q[m + 2], q[m + 3]);
#pragma unroll
    for (int m = 0; m < S; ++m) {
      T l = f[m], r = f[m + 1];
      ppm_limit(q[m + 2], l, r);
      if (m < n) {
        L[m * so] = l;
        R[m * so] = r;
      }
    }
  } else {
#pragma unroll
    for (int m = 0; m < S; ++m) {
      T l, r;
      recon_edges(1, q[m], q[m + 1], q[m + 2], q[m + 3], q[m + 4], l, r);
      if (m < n) {
        L[m * so] = l;
        R[m * so] = r;
      }
    }
  }
}

// A face flux from the two adjacent cells' edges: the low cell's aR (eL,
// stride es) and the high cell's aL (eR).
template <typename T, bool FLAT>
__device__ __forceinline__ void edge_face(const StageArgs& a, const LevelGeo& geo, const T* __restrict__ Pb, int d,
                                          int ig, int jg, int kg, int I1, int I2, const T* eL, const T* eR, int es,
                                          T* out, int ostride) {
  if (axis_face<FLAT>(a, geo, d, I2)) {
#pragma unroll
    for (int v = 0; v < NV; ++v) out[v * ostride] = T(0);
    return;
  }
  const int sd = d == 0 ? 1 : (d == 1 ? a.Nx : a.Nx * a.Ny);
  const int c0 = (kg * a.Ny + jg) * a.Nx + ig;
  T PL[NV], PR[NV];
#pragma unroll
  for (int v = 0; v < NV; ++v) {
    PL[v] = eL[v * es];
    PR[v] = eR[v * es];
  }
  positivity_fallback(a, Pb, sd, c0, PL, PR);
  face_solve<T, FLAT>(a, geo, d, I1, I2, PL, PR, out, ostride);
}

// Copies a block-boundary face flux into the face's register (faces between
// refinement levels only).  fc: index of the face cell in the register, over
// the two transverse dimensions in ascending order.
template <typename T>
__device__ __forceinline__ void to_register(const StageArgs& a, int b, int d, int side, int fc, const T* F,
                                            int stride) {
  const long long off = a.regoff[b * 6 + 2 * d + side];
  if (off < 0) return;
  const int ncf = d == 0 ? a.ny * a.nz : (d == 1 ? a.nx * a.nz : a.nx * a.ny);
#pragma unroll
  for (int v = 0; v < NV; ++v) a.reg[off + (long long)v * ncf + fc] = to_double(F[v * stride]);
}

// Inversion, floors, outputs, counters and (stage 2) the CFL rate of a cell
// whose stage conserved state U (densitized) is final.  The Newton iteration,
// floors and CFL rate are FP64 in both forms.  In the mixed form (T = float)
// the Newton starting point comes from the FP32 previous primitives (G32;
// callers that hold their own FP64 starting point pass G32 = false) and a
// floored cell's D, S_i, tau are rebuilt in FP32.
template <typename T, int DIM, bool FLAT, bool G32 = (sizeof(T) == 4), int NKM = 2, bool SCREEN = false>
__device__ __forceinline__ void finish_cell(const StageArgs& a, const LevelGeo& geo, int b, int ci, int cg, int I1,
                                            int I2, double U[NV], unsigned cnt[4], double& rate_max) {
  const double* crec = FLAT ? nullptr : geo.tc + (size_t)(I2 * geo.N1 + I1) * CREC;
  const float* crec32 = (FLAT || sizeof(T) == 8) ? nullptr : geo.tc32 + (size_t)(I2 * geo.N1 + I1) * CREC;
  const double sg = FLAT ? 1.0 : crec[C_SG];
  const double isg = FLAT ? 1.0 : crec[C_ISG];
  const double rho_fl = FLAT ? a.rho_fl_c : crec[C_RHOFL];
  const double p_fl = FLAT ? a.p_fl_c : crec[C_PFL];
  Met<double> md = FLAT ? flat_metric<double>() : load_centre_metric<double>(crec);
  Met<float> m32;
  if (sizeof(T) == 4) m32 = FLAT ? flat_metric<float>() : load_centre_metric<float>(crec32);
  double Uu[NV], Pn[NV];
  const double* Pd = a.P_in + (size_t)b * NV * a.ncell + cg;
#pragma unroll
  for (int v = 0; v < NV; ++v) Uu[v] = U[v] * isg;
  int st;
  if (G32) {
    // mixed form: the Newton starting point from the FP32 previous primitives
    // (a starting point needs no FP64); the FP64 ones are read only if every
    // solver fails
    const float* P3 = a.P32_in + (size_t)b * NV * a.ncell + cg;
    float Pg32[NV];
#pragma unroll
    for (int v = 0; v < NV; ++v)
      Pg32[v] = (v == RHO || v == PRS || v == U1 || v == U2 || v == U3) ? P3[(size_t)v * a.ncell] : 0.0f;
    float z0, w0;
    c2p_guess<float>(m32, Pg32, a.gam_fac_f, z0, w0);
    st = con2prim<NKM>(md, Uu, Pd, (size_t)a.ncell, widen_f32(z0), widen_f32(w0), rho_fl, p_fl, a, Pn);
  } else {
    double Pg[NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) Pg[v] = Pd[(size_t)v * a.ncell];
    double z0, w0;
    c2p_guess<double>(md, Pg, a.gam_fac, z0, w0);
    st = con2prim<NKM>(md, Uu, Pg, 1, z0, w0, rho_fl, p_fl, a, Pn);
  }
  cnt[st] += 1u;
  a.status[(size_t)b * a.nint + ci] = (unsigned char)st;
  float P32[NV];
  if (sizeof(T) == 4) {
#pragma unroll
    for (int v = 0; v < NV; ++v) P32[v] = narrow_f64(Pn[v]);
  }
  if (st >= 2) {
    if (sizeof(T) == 4) {
      // mixed form: the floored state's D, S_i, tau in FP32 (the field and psi
      // are left as they are); FP64 form: every conserved variable in FP64
      Derived<float> s;
      derive(m32, P32, a.gam_fac_f, s);
      float Uc[NV];
      cons_of(P32, s, Uc);
      const float sg32 = FLAT ? 1.0f : crec32[C_SG];
#pragma unroll
      for (int v = CD; v <= CTAU; ++v) U[v] = widen_f32(sg32 * Uc[v]);
    } else {
      cons_direct(md, Pn, a.gam_fac, Uu);
#pragma unroll
      for (int v = 0; v < NV; ++v) U[v] = sg * Uu[v];
    }
  }
  const size_t ub = (size_t)b * NV * a.nint + ci;
  double* Po = a.P_out + (size_t)b * NV * a.ncell + cg;
#pragma unroll
  for (int v = 0; v < NV; ++v) {
    a.Uout[ub + (size_t)v * a.nint] = U[v];
    Po[(size_t)v * a.ncell] = Pn[v];
  }
  if (sizeof(T) == 4) {
    float* P3o = a.P32_out + (size_t)b * NV * a.ncell + cg;
#pragma unroll
    for (int v = 0; v < NV; ++v) P3o[(size_t)v * a.ncell] = P32[v];
  }
  if (a.stage == 2) {
    const float* r32 = FLAT ? nullptr : geo.tc32 + (size_t)(I2 * geo.N1 + I1) * CREC;
    cfl_max<DIM, FLAT, SCREEN>(a, geo, md, crec, r32, Pn, SCREEN ? cfl_seen(a) : 0ull, rate_max);
  }
}

__device__ __forceinline__ double stage_dt(const StageArgs& a) {
  if (a.dt_host > 0.0) return a.dt_host;
  if (a.stage == 1) return a.cfl / __longlong_as_double((long long)*a.smax_in);
  return *a.dt_dev;
}

// The same for a whole CTA, the division done once: a thread's own would cost
// as many FP64 instructions as a tenth of a cell's inversion.
__device__ __forceinline__ double block_dt(const StageArgs& a) {
  __shared__ double s_dt;
  if (threadIdx.x == 0) s_dt = stage_dt(a);
  __syncthreads();
  return s_dt;
}

__device__ __forceinline__ void reduce_outputs(const StageArgs& a, const unsigned cnt[4], double rate_max) {
  const unsigned lane = threadIdx.x & 31u;
#pragma unroll
  for (int s = 0; s < 4; ++s) {
    const unsigned tot = __reduce_add_sync(0xffffffffu, cnt[s]);
    if (lane == 0 && tot) atomicAdd(a.counts + s, (unsigned long long)tot);
  }
  if (a.stage == 2) {
    const double w = warp_max_d(rate_max);
    if (lane == 0) atomicMax(a.smax_out, (unsigned long long)__double_as_longlong(w));
  }
}

template <typename T, int DIM, bool FLAT, int NKM = 2>
__device__ __forceinline__ void rk_finish(const StageArgs& a, const LevelGeo& geo, int b, int ci, int cg, int I1, int I2,
                                          int bi, int bj, int k, const double rhs[NV], double dt, unsigned cfb,
                                          unsigned cnt[4], double& rate_max);

// Divergence of the face fluxes staged in shared memory, sources, RK stage
// combination and (unless the reflux pass owns the cell) the inversion of cell
// c of plane k in the tile at (x0, y0) of block b.
template <typename T, int DIM, bool FLAT, bool SPLIT, int NKM = 2>
__device__ __forceinline__ void cell_update(const StageArgs& a, const LevelGeo& geo, const T* __restrict__ Pb, int b,
                                            int x0, int y0, int k, int c, const T* Fx, const T* Fy, const T* Fz0,
                                            const T* Fz1, double dt, unsigned cfb, unsigned cnt[4],
                                            double& rate_max) {
  const int tx = a.tx, ty = a.ty;
  const int sFx = ty * (tx + 1), sFy = (ty + 1) * tx, sFz = tx * ty;
  const int kg = k + a.gz;
  const int I1b = a.blk[4 * b + 1] * a.nx + x0, I2b = a.blk[4 * b + 2] * a.ny + y0;
  const int i = c % tx, j = c / tx;
  const int ig = i + x0 + a.gx, jg = j + y0 + a.gy;
  const int cg = (kg * a.Ny + jg) * a.Nx + ig;
  const int ci = (k * a.ny + (j + y0)) * a.nx + (i + x0);
  const int I1 = I1b + i, I2 = I2b + j;
  // flux divergence in the flux arithmetic T (FP32 in the mixed form, whose
  // face fluxes carry FP32 rounding already), then widened once per variable
  T rdiv[NV];
  const T ix = pick<T>(geo.idx[0], geo.idx_f[0]), iy = pick<T>(geo.idx[1], geo.idx_f[1]),
          iz = pick<T>(geo.idx[2], geo.idx_f[2]);
#pragma unroll
  for (int v = 0; v < NV; ++v) {
    T r = -(Fx[v * sFx + j * (tx + 1) + i + 1] - Fx[v * sFx + j * (tx + 1) + i]) * ix;
    r = r - (Fy[v * sFy + (j + 1) * tx + i] - Fy[v * sFy + j * tx + i]) * iy;
    if (DIM == 3) r = r - (Fz1[v * sFz + c] - Fz0[v * sFz + c]) * iz;
    rdiv[v] = r;
  }
  double rhs[NV];
  // explicit damping rate of the cleaning source (with IMEX it is implicit)
  const double kap_x = a.imex ? 0.0 : a.kappa;
  const float kap_xf = a.imex ? 0.f : a.kappa_f;
  // sources from the cell's primitives
  {
    T Pc[NV], Uc[NV], S[NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) Pc[v] = Pb[(size_t)v * a.ncell + cg];
    if (FLAT) {
      rdiv[PSI] = rdiv[PSI] - pick<T>(kap_x, kap_xf) * Pc[PSI];
#pragma unroll
      for (int v = 0; v < NV; ++v) rhs[v] = to_double(rdiv[v]);
    } else {
      const double* crec = geo.tc + (size_t)(I2 * geo.N1 + I1) * CREC;
      Met<T> m;
      if (sizeof(T) == 8) {
        m = load_centre_metric<T>(crec);
      } else {
        m = load_centre_metric<T>(geo.tc32 + (size_t)(I2 * geo.N1 + I1) * CREC);
      }
      if constexpr (sizeof(T) == 8) {
        sources_direct(m, crec, Pc, a.gam_fac, kap_x, a.ch * a.ch, S);
        const double sg = crec[C_SG];
#pragma unroll
        for (int v = 0; v < NV; ++v) rhs[v] = rdiv[v];
        rhs[CS1] = fma_t(sg, S[0], rhs[CS1]);
        rhs[CS2] = fma_t(sg, S[1], rhs[CS2]);
        rhs[CTAU] = fma_t(sg, S[2], rhs[CTAU]);
        rhs[PSI] = fma_t(sg, S[3], rhs[PSI]);
      } else {
        Derived<T> s;
        derive(m, Pc, pick<T>(a.gam_fac, a.gam_fac_f), s);
        cons_of(Pc, s, Uc);
        sources_of(m, geo.tc32 + (size_t)(I2 * geo.N1 + I1) * CREC, Pc, s, Uc, pick<T>(kap_x, kap_xf),
                   pick<T>(a.ch * a.ch, a.ch2_f),
                   S);
        const T sg = T(geo.tc32[(size_t)(I2 * geo.N1 + I1) * CREC + C_SG]);
#pragma unroll
        for (int v = 0; v < NV; ++v) rhs[v] = to_double(rdiv[v] + sg * S[v]);
      }
    }
  }
  if (SPLIT) {  // the cell kernel completes the stage from the stored right-hand side
    T* R = reinterpret_cast<T*>(a.R) + (size_t)b * NV * a.nint + ci;
#pragma unroll
    for (int v = 0; v < NV; ++v) R[(size_t)v * a.nint] = sizeof(T) == 4 ? (T)narrow_f64(rhs[v]) : (T)rhs[v];
    return;
  }
  rk_finish<T, DIM, FLAT, NKM>(a, geo, b, ci, cg, I1, I2, x0 + i, y0 + j, k, rhs, dt, cfb, cnt, rate_max);
}

// RK combination (and the IMEX damping), then the inversion, floors, outputs
// and CFL rate of cell (bi, bj, k) of block b, given the stage right-hand side.
template <typename T, int DIM, bool FLAT, int NKM>
__device__ __forceinline__ void rk_finish(const StageArgs& a, const LevelGeo& geo, int b, int ci, int cg, int I1, int I2,
                                          int bi, int bj, int k, const double rhs[NV], double dt, unsigned cfb,
                                          unsigned cnt[4], double& rate_max) {
  const size_t ub = (size_t)b * NV * a.nint + ci;
  double U[NV];
#pragma unroll
  for (int v = 0; v < NV; ++v) {
    const double un = a.Un[ub + (size_t)v * a.nint];
    if (a.stage == 1)
      U[v] = fma_t(dt, rhs[v], un);
    else
      U[v] = half_t(un + fma_t(dt, rhs[v], a.U1[ub + (size_t)v * a.nint]));
  }
  if (a.imex) {
    // IMEX-SSP2(2,2,2) for the damping -lam psi (lam = alpha kappa, z = lam dt):
    // Y1 = psi_n/(1 + g z); stage 1: Y2 = (psi_n + dt F(Y1) - (1 - 2g) z Y1)/(1 + g z);
    // stage 2: psi = psi_n/2 + (Y2 + dt F(Y2))/2 - z (1 - g) Y2 / 2 - g z Y1
    const double al = FLAT ? 1.0 : geo.tc[(size_t)(I2 * geo.N1 + I1) * CREC + C_AL];
    const double z = al * a.kappa * dt, g = a.imex_g;
    const double un = a.Un[ub + (size_t)PSI * a.nint];
    const double y1 = un / (1.0 + g * z);
    if (a.stage == 1) {
      U[PSI] = (un + dt * rhs[PSI] - (1.0 - 2.0 * g) * z * y1) / (1.0 + g * z);
    } else {
      const double u1 = a.U1[ub + (size_t)PSI * a.nint];
      U[PSI] = 0.5 * un + 0.5 * (u1 + dt * rhs[PSI]) - 0.5 * z * (1.0 - g) * u1 - g * z * y1;
    }
  }
  // cells next to a face bordering finer blocks are finished by the reflux pass
  const bool later = cfb && (((cfb & 1u) && bi == 0) || ((cfb & 2u) && bi == a.nx - 1) ||
                             ((cfb & 4u) && bj == 0) || ((cfb & 8u) && bj == a.ny - 1) ||
                             ((cfb & 16u) && k == 0) || ((cfb & 32u) && k == a.nz - 1));
  if (later) {
#pragma unroll
    for (int v = 0; v < NV; ++v) a.Uout[ub + (size_t)v * a.nint] = U[v];
  } else {
    finish_cell<T, DIM, FLAT, (sizeof(T) == 4), NKM>(a, geo, b, ci, cg, I1, I2, U, cnt, rate_max);
  }
}

// ----------------------------------------------------------------------------
// The stage kernel.  T: flux arithmetic (double: FP64 form; float: mixed form).
// Every block of every level is an item of the same launch.
//
// Per plane k of the CTA's column, three phases, with CTA barriers before and
// after F:
//  R  every cell's two reconstructed edges along x (the tile plus one cell on
//     each x side) and along y (plus one cell on each y side) into shared
//     memory, by strips of cells of one variable; in 3-D each z column also reconstructs its cell of plane k+1,
//     solves the z face between planes k and k+1 from that cell's low edge
//     and plane k's high edge (kept in shared memory from the previous
//     plane), and keeps plane k+1's high edge for the next plane;
//  F  the x and y face fluxes from the edges of the two adjacent cells;
//  C  the cell updates.
// R's tasks (a warp's worth of z cells or of strips) come from a queue, and
// with three z-face planes in shared memory no barrier separates C from the
// next plane's R: a warp that has no cells, or has inverted its own, starts
// reconstructing while the others still occupy the FP64 unit.  Without the
// queue and with a barrier there the step of the 192x96x96 torus took 2.29 ms
// (mixed) against 1.97 with it and the helper warps (launch.h), FP64 11.1
// against 9.8 ms.
//
// Each cell's edges are reconstructed once per direction (up to the one-cell
// tile halo) instead of once for each of its two faces; the face states are
// the same numbers as a per-face reconstruction's.
//
// Shared memory (T): Fx, Fy, [three z-face planes and EzR in 3-D], ExL, ExR, EyL, EyR.
//
// MINB: the register bound (resident CTAs per SM) in its last digit; + 10: the
// face kernel of the split form (no inversion code); + 100: the Newton-Krylov
// inversion in place of the analytic Newton step.
// ----------------------------------------------------------------------------
template <typename T, int DIM, bool FLAT, int MINB>
__global__ void __launch_bounds__(stage_threads_max(sizeof(T) == 8, MINB), MINB % 10) stage_kernel(StageArgs a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int tx = a.tx, ty = a.ty;
  const int sFx = ty * (tx + 1), sFy = (ty + 1) * tx, sFz = tx * ty;
  const int nex = (tx + 2) * ty, ney = tx * (ty + 2);
  T* Fx = reinterpret_cast<T*>(smem_raw);
  T* Fy = Fx + NV * sFx;
  T* Fz = Fy + NV * sFy;  // a.zbuf planes of z faces
  T* EzR = Fz + (DIM == 3 ? a.zbuf * NV * sFz : 0);
  T* ExL = EzR + (DIM == 3 ? NV * sFz : 0);
  T* ExR = ExL + NV * nex;
  T* EyL = ExR + NV * nex;
  T* EyR = EyL + NV * ney;
  __shared__ int s_item;
  // next reconstruction task, alternating over the planes this CTA runs: F of
  // one plane resets the counter of the next
  __shared__ int s_task[2];
  if (threadIdx.x < 2) s_task[threadIdx.x] = 0;
  int par = 0;
  const int lane = threadIdx.x & 31;

  const double dt = block_dt(a);
  if (a.stage == 1 && blockIdx.x == 0 && threadIdx.x == 0) *a.dt_dev = dt;

  const T* Pb_all = sizeof(T) == 8 ? reinterpret_cast<const T*>(a.P_in) : reinterpret_cast<const T*>(a.P32_in);
  unsigned cnt[4] = {0u, 0u, 0u, 0u};
  double rate_max = 0.0;
  const int ntile = a.ntx * a.nty;
  const int sy = a.Nx, sz = a.Nx * a.Ny;
  const int nzc = DIM == 3 ? sFz : 0;
  // reconstruction strips: per variable, nsx strips in each of the tile's ty
  // rows and nsy in each of its tx columns
  const int nsx = (tx + 2 + kStrip - 1) / kStrip, nsy = (ty + 2 + kStrip - 1) / kStrip;
  const int nlx = NV * nsx * ty, nly = NV * nsy * tx;
  const FastDiv dtx(tx), dtx1(tx + 1), dsx(nsx), dlx(nsx * ty), dly(nsy * tx);

  int item = a.persistent ? -1 : (int)blockIdx.x + a.item0;
  for (;;) {
    if (a.persistent) {
      __syncthreads();
      if (threadIdx.x == 0) s_item = a.item0 + (int)atomicAdd(a.work, 1u);
      __syncthreads();
      item = s_item;
    }
    if (item >= a.item1) break;
    // item = (visiting-order block, tile, z part); a part runs planes [kbeg, kend)
    const int zp = item % a.nzp, it2 = item / a.nzp;
    const int ord = it2 / ntile;
    const int b = a.order[ord];
    const int tile = it2 - ord * ntile;
    const int kbeg = zp * (a.nz / a.nzp), kend = kbeg + a.nz / a.nzp;
    const int x0 = (tile % a.ntx) * tx, y0 = (tile / a.ntx) * ty;
    const int L = a.blk[4 * b];
    const LevelGeo geo = level_geo(a, L);
    const int bx = a.blk[4 * b + 1], by = a.blk[4 * b + 2];
    const int I1b = bx * a.nx + x0, I2b = by * a.ny + y0;
    const T* Pb = Pb_all + (size_t)b * NV * a.ncell;
    const unsigned cfb = a.nlev > 1 ? a.cf[b] : 0u;
    const bool regs = a.nlev > 1;
    T* Fz0 = Fz;
    T* Fz1 = DIM == 3 ? Fz + NV * sFz : Fz;
    T* Fz2 = DIM == 3 && a.zbuf == 3 ? Fz1 + NV * sFz : Fz;
    __syncthreads();
    if (DIM == 3) {
      // bottom face of plane kbeg from the high edge of plane kbeg - 1 and the
      // low edge of plane kbeg; plane kbeg's high edge is kept for the face
      // above it (the same arithmetic as the face carried up from below)
      for (int t = threadIdx.x; t < sFz; t += blockDim.x) {
        const int i = t % tx, j = t / tx;
        const int ig = i + x0 + a.gx, jg = j + y0 + a.gy;
        const int c0 = ((kbeg + a.gz) * a.Ny + jg) * a.Nx + ig;
        T PL[NV], PR[NV], tmp[NV];
        if (axis_face<FLAT>(a, geo, 2, I2b + j)) {
#pragma unroll
          for (int v = 0; v < NV; ++v) Fz0[v * sFz + t] = T(0);
        } else {
          cell_edges(a, Pb, sz, c0 - sz, tmp, 1, PL, 1);
          cell_edges(a, Pb, sz, c0, PR, 1, EzR + t, sFz);
          positivity_fallback(a, Pb, sz, c0, PL, PR);
          face_solve<T, FLAT>(a, geo, 2, I1b + i, I2b + j, PL, PR, Fz0 + t, sFz);
        }
        if (regs && kbeg == 0) to_register(a, b, 2, 0, (j + y0) * a.nx + i + x0, Fz0 + t, sFz);
      }
      __syncthreads();
    }
    for (int k = kbeg; k < kend; ++k) {
      const int kg = k + a.gz;
      // R: edges (and the z face above plane k), taken by whole warps from a
      // queue: warps that have no cell of plane k - 1, or are done with it,
      // are here while the others still invert theirs
      for (;;) {
        int t = 0;
        if (lane == 0) t = atomicAdd(&s_task[par], 32);
        t = __shfl_sync(0xffffffffu, t, 0);
        if (t >= nzc + nlx + nly) break;
        t += lane;
        if (t >= nzc + nlx + nly) continue;
        if (t < nzc) {
          int i, j;
          dtx.split(t, j, i);
          const int ig = i + x0 + a.gx, jg = j + y0 + a.gy;
          const int c1 = ((kg + 1) * a.Ny + jg) * a.Nx + ig;
          T PL[NV], PR[NV];
#pragma unroll
          for (int v = 0; v < NV; ++v) PL[v] = EzR[v * sFz + t];
          cell_edges(a, Pb, sz, c1, PR, 1, EzR + t, sFz);
          positivity_fallback(a, Pb, sz, c1, PL, PR);
          face_solve<T, FLAT>(a, geo, 2, I1b + i, I2b + j, PL, PR, Fz1 + t, sFz);
          if (regs && k + 1 == a.nz) to_register(a, b, 2, 1, (j + y0) * a.nx + i + x0, Fz1 + t, sFz);
        } else if (t < nzc + nlx) {
          int v, u, j, q;
          dlx.split(t - nzc, v, u);
          dsx.split(u, j, q);
          const int i = q * kStrip - 1;  // the strip's first cell
          const int c = (kg * a.Ny + j + y0 + a.gy) * a.Nx + i + x0 + a.gx;
          const int e = v * nex + j * (tx + 2) + i + 1;
          strip_edges<T, kStrip>(a.recon, Pb + (size_t)v * a.ncell + c, 1, tx + 1 - i, ExL + e, ExR + e, 1);
        } else {
          int v, u, i, q;
          dly.split(t - nzc - nlx, v, u);
          dtx.split(u, q, i);
          const int j = q * kStrip - 1;
          const int c = (kg * a.Ny + j + y0 + a.gy) * a.Nx + i + x0 + a.gx;
          const int e = v * ney + (j + 1) * tx + i;
          strip_edges<T, kStrip>(a.recon, Pb + (size_t)v * a.ncell + c, sy, ty + 1 - j, EyL + e, EyR + e, tx);
        }
      }
      __syncthreads();
      // F: x and y faces
      par ^= 1;
      if (threadIdx.x == 0) s_task[par] = 0;
      for (int t = threadIdx.x; t < sFx + sFy; t += blockDim.x) {
        if (t < sFx) {
          int i, j;
          dtx1.split(t, j, i);
          const int e = j * (tx + 2) + i;  // edge slot of the low cell
          edge_face<T, FLAT>(a, geo, Pb, 0, i + x0 + a.gx, j + y0 + a.gy, kg, I1b + i, I2b + j, ExR + e, ExL + e + 1,
                             nex, Fx + t, sFx);
          if (regs && (x0 + i == 0 || x0 + i == a.nx))
            to_register(a, b, 0, x0 + i == 0 ? 0 : 1, k * a.ny + j + y0, Fx + t, sFx);
        } else {
          const int u = t - sFx;
          int i, j;
          dtx.split(u, j, i);
          edge_face<T, FLAT>(a, geo, Pb, 1, i + x0 + a.gx, j + y0 + a.gy, kg, I1b + i, I2b + j, EyR + u,
                             EyL + u + tx, ney, Fy + u, sFy);
          if (regs && (y0 + j == 0 || y0 + j == a.ny))
            to_register(a, b, 1, y0 + j == 0 ? 0 : 1, k * a.nx + i + x0, Fy + u, sFy);
        }
      }
      __syncthreads();
      // C: cell updates
      for (int c = threadIdx.x; c < sFz; c += blockDim.x)
        cell_update<T, DIM, FLAT, (MINB % 100 >= 10), (MINB >= 100 ? 1 : 0)>(a, geo, Pb, b, x0, y0, k, c, Fx, Fy, Fz0,
                                                                          Fz1, dt, cfb, cnt, rate_max);
      // with three z planes no barrier: the next plane's R touches neither Fx,
      // Fy nor the two z planes C reads, and the barrier after R is behind
      // every warp's C
      if (DIM == 3 && a.zbuf == 2) __syncthreads();
      T* tmp = Fz0;
      Fz0 = Fz1;
      Fz1 = Fz2;
      Fz2 = a.zbuf == 3 ? tmp : Fz0;  // of two planes the third name is the current lower one
    }
    if (!a.persistent) break;
  }
  reduce_outputs(a, cnt, rate_max);
}

// ----------------------------------------------------------------------------
// Warp-specialised form of the 3-D stage kernel.  The first pwarps warps
// (producers) compute the face fluxes of plane k+1 while the other warps
// (consumers) update the cells of plane k, so the FP64 work of the cell
// updates is not interrupted by the face phase.  Face fluxes are double
// buffered (x and y faces per plane parity, z faces in three slots: plane k
// reads faces k and k+1 while plane k+1's producer writes face k+2); named
// barriers FULL[parity] (producers -> consumers) and EMPTY[parity]
// (consumers -> producers) hand the buffers over.  It reconstructs per face
// (recon_var), gives each role only part of the CTA's warps, and measured
// slower than the phased kernel on the tori; it is selected only by an
// explicit producer-warp count in bhac_set_launch.
// ----------------------------------------------------------------------------
// Named barriers (ids 1..4; 0 is __syncthreads).  Producer and consumer roles
// are whole warps; each warp reconverges before the barrier instruction.
__device__ __forceinline__ void named_sync(int id, int n) {
  __syncwarp();
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(n) : "memory");
}
__device__ __forceinline__ void named_arrive(int id, int n) {
  __syncwarp();
  asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(n) : "memory");
}
constexpr int BAR_FULL = 1, BAR_EMPTY = 3;

template <typename T, bool FLAT>
__device__ __forceinline__ void produce_plane(const StageArgs& a, const LevelGeo& geo, const T* __restrict__ Pb, int b,
                                              int x0, int y0, int k, bool bottom, T* Fx, T* Fy, T* Fzlo, T* Fzhi,
                                              int ptid, int nprod) {
  const int tx = a.tx, ty = a.ty;
  const int sFx = ty * (tx + 1), sFy = (ty + 1) * tx, sFz = tx * ty;
  const int I1b = a.blk[4 * b + 1] * a.nx + x0, I2b = a.blk[4 * b + 2] * a.ny + y0;
  const bool regs = a.nlev > 1;
  const int kg = k + a.gz;
  const int nb = bottom ? sFz : 0;
  const int n = nb + sFx + sFy + sFz;
  for (int t = ptid; t < n; t += nprod) {
    if (t < nb) {
      const int i = t % tx, j = t / tx;
      face_flux<T, FLAT>(a, geo, Pb, 2, i + x0 + a.gx, j + y0 + a.gy, kg, I1b + i, I2b + j, Fzlo + t, sFz);
      if (regs) to_register(a, b, 2, 0, (j + y0) * a.nx + i + x0, Fzlo + t, sFz);
      continue;
    }
    const int u0 = t - nb;
    if (u0 < sFx) {
      const int i = u0 % (tx + 1), j = u0 / (tx + 1);
      face_flux<T, FLAT>(a, geo, Pb, 0, i + x0 + a.gx, j + y0 + a.gy, kg, I1b + i, I2b + j, Fx + u0, sFx);
      if (regs && (x0 + i == 0 || x0 + i == a.nx)) to_register(a, b, 0, x0 + i == 0 ? 0 : 1, k * a.ny + j + y0, Fx + u0, sFx);
    } else if (u0 < sFx + sFy) {
      const int u = u0 - sFx;
      const int i = u % tx, j = u / tx;
      face_flux<T, FLAT>(a, geo, Pb, 1, i + x0 + a.gx, j + y0 + a.gy, kg, I1b + i, I2b + j, Fy + u, sFy);
      if (regs && (y0 + j == 0 || y0 + j == a.ny)) to_register(a, b, 1, y0 + j == 0 ? 0 : 1, k * a.nx + i + x0, Fy + u, sFy);
    } else {
      const int u = u0 - sFx - sFy;
      const int i = u % tx, j = u / tx;
      face_flux<T, FLAT>(a, geo, Pb, 2, i + x0 + a.gx, j + y0 + a.gy, kg + 1, I1b + i, I2b + j, Fzhi + u, sFz);
      if (regs && k + 1 == a.nz) to_register(a, b, 2, 1, (j + y0) * a.nx + i + x0, Fzhi + u, sFz);
    }
  }
}

template <typename T, bool FLAT, int MINB>
__global__ void __launch_bounds__(256, MINB) stage_kernel_ws(StageArgs a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int tx = a.tx, ty = a.ty;
  const int sFx = ty * (tx + 1), sFy = (ty + 1) * tx, sFz = tx * ty;
  T* base = reinterpret_cast<T*>(smem_raw);
  T* FxB[2] = {base, base + NV * sFx};
  T* FyB[2] = {base + 2 * NV * sFx, base + 2 * NV * sFx + NV * sFy};
  T* FzB[3];
  for (int q = 0; q < 3; ++q) FzB[q] = base + 2 * NV * (sFx + sFy) + q * NV * sFz;
  __shared__ int s_item;

  const double dt = block_dt(a);
  if (a.stage == 1 && blockIdx.x == 0 && threadIdx.x == 0) *a.dt_dev = dt;
  const T* Pb_all = sizeof(T) == 8 ? reinterpret_cast<const T*>(a.P_in) : reinterpret_cast<const T*>(a.P32_in);
  const int nthr = blockDim.x, nprod = a.pwarps * 32, ncons = nthr - nprod;
  const bool producer = (int)threadIdx.x < nprod;
  unsigned cnt[4] = {0u, 0u, 0u, 0u};
  double rate_max = 0.0;
  const int ntile = a.ntx * a.nty;
  int item = a.persistent ? -1 : (int)blockIdx.x;
  for (;;) {
    if (a.persistent) {
      __syncthreads();
      if (threadIdx.x == 0) s_item = (int)atomicAdd(a.work, 1u);
      __syncthreads();
      item = s_item;
    }
    if (item >= a.nitems) break;
    const int ord = item / ntile;
    const int b = a.order[ord];
    const int tile = item - ord * ntile;
    const int x0 = (tile % a.ntx) * tx, y0 = (tile / a.ntx) * ty;
    const LevelGeo geo = level_geo(a, a.blk[4 * b]);
    const T* Pb = Pb_all + (size_t)b * NV * a.ncell;
    const unsigned cfb = a.nlev > 1 ? a.cf[b] : 0u;
    if (producer) {
      for (int k = 0; k < a.nz; ++k) {
        const int par = k & 1;
        if (k >= 2) named_sync(BAR_EMPTY + par, nthr);
        produce_plane<T, FLAT>(a, geo, Pb, b, x0, y0, k, k == 0, FxB[par], FyB[par], FzB[k % 3], FzB[(k + 1) % 3],
                               threadIdx.x, nprod);
        __threadfence_block();
        named_arrive(BAR_FULL + par, nthr);
      }
      // take the consumers' last releases so every barrier starts the next item clean
      for (int k = a.nz - 2 < 0 ? 0 : a.nz - 2; k < a.nz; ++k) named_sync(BAR_EMPTY + (k & 1), nthr);
    } else {
      for (int k = 0; k < a.nz; ++k) {
        const int par = k & 1;
        named_sync(BAR_FULL + par, nthr);
        for (int c = threadIdx.x - nprod; c < sFz; c += ncons)
          cell_update<T, 3, FLAT, false>(a, geo, Pb, b, x0, y0, k, c, FxB[par], FyB[par], FzB[k % 3], FzB[(k + 1) % 3], dt,
                                  cfb, cnt, rate_max);
        __threadfence_block();
        named_arrive(BAR_EMPTY + par, nthr);
      }
    }
    if (!a.persistent) break;
  }
  reduce_outputs(a, cnt, rate_max);
}

// Split form, second kernel: one thread per interior cell of the items
// [item0, item1): the stage right-hand side the face kernel stored, then
// rk_finish (the same arithmetic as the fused kernel).
template <typename T, int DIM, bool FLAT>
__global__ void __launch_bounds__(256) cell_kernel(StageArgs a) {
  const double dt = block_dt(a);
  unsigned cnt[4] = {0u, 0u, 0u, 0u};
  double rate_max = 0.0;
  const int tx = a.tx, ty = a.ty, ntile = a.ntx * a.nty;
  const long long per = (long long)tx * ty * a.nz;
  const long long n = (long long)(a.item1 - a.item0) * per;
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < n; t += (long long)gridDim.x * blockDim.x) {
    const int item = a.item0 + (int)(t / per);
    const int rem = (int)(t - (long long)(item - a.item0) * per);
    const int k = rem / (tx * ty), c = rem - k * tx * ty;
    const int i = c % tx, j = c / tx;
    const int ord = item / ntile;
    const int b = a.order[ord];
    const int tile = item - ord * ntile;
    const int bi = (tile % a.ntx) * tx + i, bj = (tile / a.ntx) * ty + j;
    const int ci = (k * a.ny + bj) * a.nx + bi;
    const int cg = ((k + a.gz) * a.Ny + (bj + a.gy)) * a.Nx + (bi + a.gx);
    const LevelGeo geo = level_geo(a, a.blk[4 * b]);
    const int I1 = a.blk[4 * b + 1] * a.nx + bi, I2 = a.blk[4 * b + 2] * a.ny + bj;
    const unsigned cfb = a.nlev > 1 ? a.cf[b] : 0u;
    const T* R = reinterpret_cast<const T*>(a.R) + (size_t)b * NV * a.nint + ci;
    double rhs[NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) rhs[v] = to_double(R[(size_t)v * a.nint]);
    rk_finish<T, DIM, FLAT>(a, geo, b, ci, cg, I1, I2, bi, bj, k, rhs, dt, cfb, cnt, rate_max);
  }
  reduce_outputs(a, cnt, rate_max);
}

template <typename T, int DIM, bool FLAT>
static cudaError_t launch_cells_t(const StageArgs& a, int grid, cudaStream_t st) {
  cell_kernel<T, DIM, FLAT><<<grid, 256, 0, st>>>(a);
  return cudaGetLastError();
}

template <typename T>
static cudaError_t launch_cells_any(const StageArgs& a, int grid, cudaStream_t st) {
  if (a.ndim == 3) return a.flat ? launch_cells_t<T, 3, true>(a, grid, st) : launch_cells_t<T, 3, false>(a, grid, st);
  return a.flat ? launch_cells_t<T, 2, true>(a, grid, st) : launch_cells_t<T, 2, false>(a, grid, st);
}

// Coarse-fine flux correction: each listed coarse cell trades the coarse flux
// through a face bordering finer blocks for the mean of the fine fluxes that
// cover it (U += f dt (F_fine - F_coarse) / dx, sign by side, f = 1 in stage 1
// and 1/2 in stage 2), then is inverted like every other cell.
template <typename T, int DIM, bool FLAT>
__global__ void __launch_bounds__(128) reflux_kernel(StageArgs a) {
  const double dt = block_dt(a);
  const double f = a.stage == 1 ? 1.0 : 0.5;
  unsigned cnt[4] = {0u, 0u, 0u, 0u};
  double rate_max = 0.0;
  const int n = a.nrcells;
  const int nthreads = gridDim.x * blockDim.x;
  const int rounds = (n + nthreads - 1) / nthreads;
  for (int r = 0; r < rounds; ++r) {
    const int t = r * nthreads + blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= n) continue;
    const RefluxCell rc = a.rcells[t];
    const LevelGeo geo = level_geo(a, rc.level);
    const size_t ub = (size_t)rc.b * NV * a.nint + rc.ci;
    double U[NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) U[v] = a.Uout[ub + (size_t)v * a.nint];
    for (int q = 0; q < rc.nterm; ++q) {
      const RefluxTerm T_ = a.rterms[rc.term0 + q];
      const double w = f * dt * geo.idx[T_.d] * (double)T_.sign;
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        double acc = 0.0;
        for (int m = 0; m < T_.nfine; ++m) acc += a.reg[T_.fine[m] + (long long)v * T_.fstride];
        const double Ff = acc / T_.nfine;
        const double Fc = a.reg[T_.coarse + (long long)v * T_.cstride];
        // the IMEX first stage divides the explicit increment of psi by 1 + g z
        const double wv = (v == PSI && a.imex && a.stage == 1)
                              ? w / (1.0 + a.imex_g * geo.tc[(size_t)(rc.I2 * geo.N1 + rc.I1) * CREC + C_AL] * a.kappa * dt)
                              : w;
        U[v] += wv * (Ff - Fc);
      }
    }
    finish_cell<T, DIM, FLAT>(a, geo, rc.b, rc.ci, rc.cg, rc.I1, rc.I2, U, cnt, rate_max);
  }
  reduce_outputs(a, cnt, rate_max);
}

// Stand-alone CFL rate reduction over interior cells (FP64 primitives); a
// grid-stride loop over (block, cell) with 32-bit index arithmetic (the
// library's grids hold fewer than 2^31 interior cells).
template <int DIM, bool FLAT>
__global__ void __launch_bounds__(256) cfl_kernel(StageArgs a) {
  double rate_max = 0.0;
  const unsigned n = (unsigned)a.nblocks * (unsigned)a.nint;
  for (unsigned t = blockIdx.x * blockDim.x + threadIdx.x; t < n; t += gridDim.x * blockDim.x) {
    const int b = (int)(t / (unsigned)a.nint);
    const int ci = (int)(t - (unsigned)b * (unsigned)a.nint);
    const int i = ci % a.nx, j = (ci / a.nx) % a.ny, k = ci / (a.nx * a.ny);
    const int cg = ((k + a.gz) * a.Ny + (j + a.gy)) * a.Nx + (i + a.gx);
    const LevelGeo geo = level_geo(a, a.blk[4 * b]);
    const unsigned long long seen = cfl_seen(a);
    double P[NV];
    const double* Pd = a.P_in + (size_t)b * NV * a.ncell + cg;
#pragma unroll
    for (int v = 0; v < NV; ++v) P[v] = Pd[(size_t)v * a.ncell];
    Met<double> m = flat_metric<double>();
    const double* crec = nullptr;
    const float* crec32 = nullptr;
    if (!FLAT) {
      const int I1 = a.blk[4 * b + 1] * a.nx + i, I2 = a.blk[4 * b + 2] * a.ny + j;
      crec = geo.tc + (size_t)(I2 * geo.N1 + I1) * CREC;
      crec32 = geo.tc32 + (size_t)(I2 * geo.N1 + I1) * CREC;
      m = load_centre_metric<double>(crec);
    }
    cfl_max<DIM, FLAT, true>(a, geo, m, crec, crec32, P, seen, rate_max);
  }
  const double w = warp_max_d(rate_max);
  if ((threadIdx.x & 31u) == 0) atomicMax(a.smax_out, (unsigned long long)__double_as_longlong(w));
}

// Loading a state in one pass: the interior primitives src ([block][var][cell],
// FP64) go to the ghosted FP64 array P and (mixed form) its FP32 copy P32; the
// densitized conserved state U follows from them, and the CFL rate of the
// loaded primitives is reduced into smax_out unless that is null (the same
// per-cell rate as cfl_kernel's).  Same loop as cfl_kernel; four CTAs per SM as
// the register bound, so that enough loads are in flight beside the FP64 work
// (mixed, 1.8 M cells: 267 us without the bound, 251 with three, 230 with four).
template <int DIM, bool FLAT>
__global__ void __launch_bounds__(256, 4) load_kernel(StageArgs a, const double* __restrict__ src, double* P, float* P32,
                                                   double* U) {
  double rate_max = 0.0;
  const unsigned n = (unsigned)a.nblocks * (unsigned)a.nint;
  for (unsigned t = blockIdx.x * blockDim.x + threadIdx.x; t < n; t += gridDim.x * blockDim.x) {
    const int b = (int)(t / (unsigned)a.nint);
    const int ci = (int)(t - (unsigned)b * (unsigned)a.nint);
    const int i = ci % a.nx, j = (ci / a.nx) % a.ny, k = ci / (a.nx * a.ny);
    const int cg = ((k + a.gz) * a.Ny + (j + a.gy)) * a.Nx + (i + a.gx);
    const LevelGeo geo = level_geo(a, a.blk[4 * b]);
    const unsigned long long seen = cfl_seen(a);
    double Pc[NV], Uc[NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      Pc[v] = src[((size_t)b * NV + v) * a.nint + ci];
      P[((size_t)b * NV + v) * a.ncell + cg] = Pc[v];
      if (P32) P32[((size_t)b * NV + v) * a.ncell + cg] = narrow_f64(Pc[v]);
    }
    Met<double> m = flat_metric<double>();
    double sg = 1.0;
    const double* rec = nullptr;
    const float* rec32 = nullptr;
    if (!FLAT) {
      const int I1 = a.blk[4 * b + 1] * a.nx + i, I2 = a.blk[4 * b + 2] * a.ny + j;
      rec = geo.tc + (size_t)(I2 * geo.N1 + I1) * CREC;
      rec32 = geo.tc32 + (size_t)(I2 * geo.N1 + I1) * CREC;
      m = load_centre_metric<double>(rec);
      sg = rec[C_SG];
    }
    cons_direct(m, Pc, a.gam_fac, Uc);
#pragma unroll
    for (int v = 0; v < NV; ++v) U[((size_t)b * NV + v) * a.nint + ci] = FLAT ? Uc[v] : sg * Uc[v];
    if (a.smax_out) cfl_max<DIM, FLAT, true>(a, geo, m, rec, rec32, Pc, seen, rate_max);
  }
  if (!a.smax_out) return;
  const double w = warp_max_d(rate_max);
  if ((threadIdx.x & 31u) == 0) atomicMax(a.smax_out, (unsigned long long)__double_as_longlong(w));
}

// Raises a kernel's dynamic shared-memory limit to kMaxDynSmem, or to what
// the device's opt-in limit leaves beside the kernel's static shared memory
// if that is less.
template <typename K>
static cudaError_t raise_smem_limit(K kernel) {
  cudaFuncAttributes fa;
  cudaError_t e = cudaFuncGetAttributes(&fa, kernel);
  if (e != cudaSuccess) return e;
  int dev = 0, optin = 0;
  e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  if (e != cudaSuccess) return e;
  int lim = optin - (int)fa.sharedSizeBytes;
  lim = lim < kMaxDynSmem ? lim : kMaxDynSmem;
  return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, lim);
}

template <typename T, int DIM, bool FLAT, int MINB>
static cudaError_t configure_stage_t() {
  static bool configured = false;
  if (!configured) {
    cudaError_t e = raise_smem_limit(stage_kernel<T, DIM, FLAT, MINB>);
    if (e != cudaSuccess) return e;
    configured = true;
  }
  return cudaSuccess;
}

template <typename T, bool FLAT, int MINB>
static cudaError_t configure_ws_t() {
  static bool configured = false;
  if (!configured) {
    cudaError_t e = raise_smem_limit(stage_kernel_ws<T, FLAT, MINB>);
    if (e != cudaSuccess) return e;
    configured = true;
  }
  return cudaSuccess;
}

template <typename T>
static cudaError_t configure_all_t() {
  cudaError_t e = cudaSuccess;
  if (e == cudaSuccess) e = configure_stage_t<T, 2, true, 1>();
  if (e == cudaSuccess) e = configure_stage_t<T, 2, false, 1>();
  if constexpr (sizeof(T) == 4) {
    if (e == cudaSuccess) e = configure_stage_t<T, 2, true, 2>();
    if (e == cudaSuccess) e = configure_stage_t<T, 2, false, 2>();
  }
  if (e == cudaSuccess) e = configure_stage_t<T, 3, true, 1>();
  if (e == cudaSuccess) e = configure_stage_t<T, 3, false, 1>();
  if (e == cudaSuccess) e = configure_stage_t<T, 3, true, 2>();
  if (e == cudaSuccess) e = configure_stage_t<T, 3, false, 2>();
  if (e == cudaSuccess) e = configure_ws_t<T, true, 1>();
  if (e == cudaSuccess) e = configure_ws_t<T, false, 1>();
  if (e == cudaSuccess) e = configure_ws_t<T, true, 2>();
  if (e == cudaSuccess) e = configure_ws_t<T, false, 2>();
  return e;
}

template <typename T, int DIM, bool FLAT>
static cudaError_t launch_reflux_t(const StageArgs& a, cudaStream_t st);

template <typename T, int DIM, bool FLAT, int MINB>
static cudaError_t launch_stage_t(const StageArgs& a, int grid, int threads, size_t smem, cudaStream_t st) {
  cudaError_t e;
  if constexpr (DIM == 3 && MINB < 10) {
    if (a.pwarps > 0) {
      e = configure_ws_t<T, FLAT, MINB>();
      if (e != cudaSuccess) return e;
      stage_kernel_ws<T, FLAT, MINB><<<grid, threads, smem, st>>>(a);
      e = cudaGetLastError();
      if (e != cudaSuccess || a.nrcells == 0 || a.split) return e;
      return launch_reflux_t<T, DIM, FLAT>(a, st);
    }
  }
  {
    e = configure_stage_t<T, DIM, FLAT, MINB>();
    if (e != cudaSuccess) return e;
    stage_kernel<T, DIM, FLAT, MINB><<<grid, threads, smem, st>>>(a);
  }
  e = cudaGetLastError();
  if (e != cudaSuccess || a.nrcells == 0 || a.split) return e;
  return launch_reflux_t<T, DIM, FLAT>(a, st);
}

template <typename T, int DIM, bool FLAT>
static cudaError_t launch_reflux_t(const StageArgs& a, cudaStream_t st) {
  int g = (a.nrcells + 127) / 128;
  reflux_kernel<T, DIM, FLAT><<<g, 128, 0, st>>>(a);
  return cudaGetLastError();
}

template <typename T>
static cudaError_t launch_reflux_any(const StageArgs& a, cudaStream_t st) {
  if (a.nrcells == 0) return cudaSuccess;
  if (a.ndim == 3) return a.flat ? launch_reflux_t<T, 3, true>(a, st) : launch_reflux_t<T, 3, false>(a, st);
  return a.flat ? launch_reflux_t<T, 2, true>(a, st) : launch_reflux_t<T, 2, false>(a, st);
}

// Resident CTAs per SM of the phased 3-D kernel that launch_stage_any would
// launch for these arguments (non-split), at this CTA size and shared memory.
template <typename T, bool FLAT, int MINB>
static int occupancy_t(int threads, size_t smem) {
  if (configure_stage_t<T, 3, FLAT, MINB>() != cudaSuccess) return 1;
  int n = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, stage_kernel<T, 3, FLAT, MINB>, threads, smem) != cudaSuccess) {
    cudaGetLastError();
    return 1;
  }
  return n > 0 ? n : 1;
}

template <typename T>
static int stage_occupancy_any(const StageArgs& a, int threads, size_t smem) {
  if (a.c2p_nk)
    return a.minb >= 2 ? (a.flat ? occupancy_t<T, true, 102>(threads, smem) : occupancy_t<T, false, 102>(threads, smem))
                       : (a.flat ? occupancy_t<T, true, 101>(threads, smem) : occupancy_t<T, false, 101>(threads, smem));
  return a.minb >= 2 ? (a.flat ? occupancy_t<T, true, 2>(threads, smem) : occupancy_t<T, false, 2>(threads, smem))
                     : (a.flat ? occupancy_t<T, true, 1>(threads, smem) : occupancy_t<T, false, 1>(threads, smem));
}

// Kernels exist with one or two resident CTAs per SM as the register bound;
// 2-D grids in FP64 use the one-CTA form.
template <typename T>
static cudaError_t launch_stage_any(const StageArgs& a, int grid, int threads, size_t smem, cudaStream_t st) {
  if (a.split) {
    if (a.ndim == 3) {
      if (a.minb == 3)
        return a.flat ? launch_stage_t<T, 3, true, 13>(a, grid, threads, smem, st)
                      : launch_stage_t<T, 3, false, 13>(a, grid, threads, smem, st);
      if (a.minb == 2)
        return a.flat ? launch_stage_t<T, 3, true, 12>(a, grid, threads, smem, st)
                      : launch_stage_t<T, 3, false, 12>(a, grid, threads, smem, st);
      return a.flat ? launch_stage_t<T, 3, true, 11>(a, grid, threads, smem, st)
                    : launch_stage_t<T, 3, false, 11>(a, grid, threads, smem, st);
    }
    return a.flat ? launch_stage_t<T, 2, true, 11>(a, grid, threads, smem, st)
                  : launch_stage_t<T, 2, false, 11>(a, grid, threads, smem, st);
  }
  if (a.c2p_nk && a.pwarps == 0) {  // the Newton-Krylov inversion compiled in
    if (a.ndim == 3) {
      if (a.minb >= 2)
        return a.flat ? launch_stage_t<T, 3, true, 102>(a, grid, threads, smem, st)
                      : launch_stage_t<T, 3, false, 102>(a, grid, threads, smem, st);
      return a.flat ? launch_stage_t<T, 3, true, 101>(a, grid, threads, smem, st)
                    : launch_stage_t<T, 3, false, 101>(a, grid, threads, smem, st);
    }
    if constexpr (sizeof(T) == 4) {
      if (a.minb >= 2)
        return a.flat ? launch_stage_t<T, 2, true, 102>(a, grid, threads, smem, st)
                      : launch_stage_t<T, 2, false, 102>(a, grid, threads, smem, st);
    }
    return a.flat ? launch_stage_t<T, 2, true, 101>(a, grid, threads, smem, st)
                  : launch_stage_t<T, 2, false, 101>(a, grid, threads, smem, st);
  }
  if (a.ndim == 3) {
    if (a.minb >= 2)
      return a.flat ? launch_stage_t<T, 3, true, 2>(a, grid, threads, smem, st)
                    : launch_stage_t<T, 3, false, 2>(a, grid, threads, smem, st);
    return a.flat ? launch_stage_t<T, 3, true, 1>(a, grid, threads, smem, st)
                  : launch_stage_t<T, 3, false, 1>(a, grid, threads, smem, st);
  }
  if constexpr (sizeof(T) == 4) {
    if (a.minb >= 2)
      return a.flat ? launch_stage_t<T, 2, true, 2>(a, grid, threads, smem, st)
                    : launch_stage_t<T, 2, false, 2>(a, grid, threads, smem, st);
  }
  return a.flat ? launch_stage_t<T, 2, true, 1>(a, grid, threads, smem, st)
                : launch_stage_t<T, 2, false, 1>(a, grid, threads, smem, st);
}

}  // namespace bhac
