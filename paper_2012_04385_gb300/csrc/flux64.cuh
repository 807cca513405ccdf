// FP64 face flux of the bit-exact path: reconstruction in characteristic
// variables with the Roe / local Lax-Friedrichs switch per field, the
// standalone LLF and HLLC fluxes (Sec. 2.2 of arXiv:2012.04385) and the
// Navier-Stokes viscous flux.
//
// What bounds it is the FP64 pipe: two lanes per cycle and SM, so one FP64
// warp instruction costs as much as 64 integer or FP32 ones.  Everything here
// keeps the value of every rounded operation of the scheme's fixed evaluation
// order (the comments below write it out) and takes work off that pipe:
//   * cell quantities (velocity, pressure, fluxes, sound speed, enthalpy) are
//     formed once per cell and direction (flux64_cell), not once per face that
//     reads them (six times);
//   * divisions and square roots run on the integer pipe (arith64.cuh);
//   * products by powers of two are exact, so they are folded into the next
//     addition as one fused multiply-add (a - 2b and 0.5 P + 0.5 G round once
//     either way) or done on the exponent field;
//   * the rows of the left eigenvectors share their products (rows of fields
//     0, 1 and 4 differ in sign and factor 1/2 only), and products with their
//     exact zeros and ones are not formed: adding 0 x changes nothing but the
//     sign of a zero, which add_zero reproduces;
//   * the projection of the state is formed only for fields that split;
//   * six equal cells need one projection instead of six, and WENO5-JS on five
//     equal values has constant weights.
#pragma once

#include "arith64.cuh"

namespace mrb {

constexpr int FLUX_ROE = 0, FLUX_LLF = 1, FLUX_HLLC = 2;

// Cell quantities in shared memory, direction frame: conserved state, fluxes
// F1..F4 (F0 is the normal momentum), velocities, sound speed, sqrt(rho),
// enthalpy.
constexpr int CQ_U = 0, CQ_F = 5, CQ_VEL = 9, CQ_C = 12, CQ_SQ = 13, CQ_H = 14, CQ_N = 15;

// The cells of one stencil row: quantity q of cell m.
struct Row64 {
  const double* s;
  int qs, ms;          // strides of quantity and cell
  __host__ __device__ __forceinline__ double operator()(int q, int m) const { return s[q * qs + m * ms]; }
};

__host__ __device__ __forceinline__ double fma64(double a, double b, double c) {
#ifdef __CUDA_ARCH__
  return __fma_rn(a, b, c);
#else
  return std::fma(a, b, c);
#endif
}

// 0.5 x (exact): on the exponent field for normal numbers with room below.
__host__ __device__ __forceinline__ double half64(double x) {
  const uint64_t w = d2bits(x);
  const uint32_t e = (uint32_t)(w >> 52) & 2047u;
  if ((uint32_t)(e - 2u) < 2045u) return bits2d(w - 0x0010000000000000ull);
  return (w << 1) == 0 ? x : 0.5 * x;
}

__host__ __device__ __forceinline__ double neg64(double x) { return bits2d(d2bits(x) ^ 0x8000000000000000ull); }

// s + 0 x for finite x, 0 x being the zero of x's sign (flip: of the other
// sign): s itself, unless s is a zero, and then negative only if both are.
__host__ __device__ __forceinline__ double add_zero(double s, double x) {
  const uint64_t w = d2bits(s);
  return (w << 1) == 0 ? bits2d(w & d2bits(x)) : s;
}

// x > 0 and x < 0 without the FP64 pipe (false for NaN).
__host__ __device__ __forceinline__ bool pos64(double x) { return d2bits(x) - 1u < 0x7FF0000000000000ull; }
__host__ __device__ __forceinline__ bool neg64q(double x) {
  return (d2bits(x) ^ 0x8000000000000000ull) - 1u < 0x7FF0000000000000ull;
}
// plus = 0.5 (G + P), minus = 0.5 (G - P): the halves taken before the sum,
// which is then one rounding (fused), unless both are so small that the halving
// itself could round (tails of transverse momenta do get there).
__host__ __device__ __forceinline__ void half_sums64(double G, double P, double& plus, double& minus) {
  const uint64_t lim = 64ull << 53;                                        // exponent field 64, sign shifted out
  if ((d2bits(G) << 1) < lim && (d2bits(P) << 1) < lim) {
    plus = half64(G + P);
    minus = half64(G - P);
  } else {
    const double h = half64(G);
    plus = fma64(0.5, P, h);
    minus = fma64(-0.5, P, h);
  }
}
// max(|a|, |b|), a NaN giving way to the other operand.
__host__ __device__ __forceinline__ double absmax64(double a, double b) {
  const uint64_t x = d2bits(a) & 0x7FFFFFFFFFFFFFFFull, y = d2bits(b) & 0x7FFFFFFFFFFFFFFFull;
  const bool xn = x > 0x7FF0000000000000ull, yn = y > 0x7FF0000000000000ull;
  return bits2d(xn ? y : (yn ? x : (x > y ? x : y)));
}

// ---------------------------------------------------------------- reconstruction
// Smoothness indicators of the three parabolas (Jiang & Shu 1996),
//   beta0 = 13/12 ((a - 2b) + c)^2 + 1/4 ((a - 4b) + 3c)^2,
//   beta1 = 13/12 ((b - 2c) + d)^2 + 1/4 (b - d)^2,
//   beta2 = 13/12 ((c - 2d) + e)^2 + 1/4 ((3c - 4d) + e)^2
// (each term 13/12 t t and 1/4 t t from the left), and their values
//   q0 = ((2a - 7b) + 11c)/6, q1 = ((-b + 5c) + 2d)/6, q2 = ((2c + 5d) - e)/6.
__host__ __device__ __forceinline__ void betas64(double a, double b, double c, double d, double e, double be[3]) {
  const double k = 13.0 / 12.0, c3 = 3.0 * c;
  double t1 = fma64(-2.0, b, a) + c, t2 = fma64(-4.0, b, a) + c3;
  be[0] = fma64(0.25, t2 * t2, (k * t1) * t1);
  t1 = fma64(-2.0, c, b) + d;
  t2 = b - d;
  be[1] = fma64(0.25, t2 * t2, (k * t1) * t1);
  t1 = fma64(-2.0, d, c) + e;
  t2 = fma64(-4.0, d, c3) + e;
  be[2] = fma64(0.25, t2 * t2, (k * t1) * t1);
}
__host__ __device__ __forceinline__ void parabolas64(double a, double b, double c, double d, double e, double q[3]) {
  q[0] = div64_6(fma64(2.0, a, neg64(7.0 * b)) + 11.0 * c);
  q[1] = div64_6(fma64(2.0, d, 5.0 * c - b));
  q[2] = div64_6(fma64(2.0, c, 5.0 * d) - e);
}

// ((w0 q0 + w1 q1) + w2 q2)
__host__ __device__ __forceinline__ double blend64(const double w[3], const double q[3]) {
  return (w[0] * q[0] + w[1] * q[1]) + w[2] * q[2];
}

// WENO5-JS: epsilon = 1e-6, linear weights (0.1, 0.6, 0.3).
__host__ __device__ __forceinline__ double weno5_64(double a, double b, double c, double d, double e) {
  double s[3], q[3], w[3];
  betas64(a, b, c, d, e, s);
  s[0] = 1e-6 + s[0];
  s[1] = 1e-6 + s[1];
  s[2] = 1e-6 + s[2];
  w[0] = div64(0.1, s[0] * s[0]);
  w[1] = div64(0.6, s[1] * s[1]);
  w[2] = div64(0.3, s[2] * s[2]);
  parabolas64(a, b, c, d, e, q);
  return div64(blend64(w, q), (w[0] + w[1]) + w[2]);
}

// WENO5-JS of five equal values: beta0 and beta1 vanish, and beta2 is a quarter
// of the square of a rounding error of 3c, below half an ulp of epsilon for
// |c| < 1e4; larger values (and NaN) take the general form.
__host__ __device__ __forceinline__ double weno5_64_flat(double c) {
  if (!((d2bits(c) & 0x7FFFFFFFFFFFFFFFull) < 0x40C3880000000000ull)) return weno5_64(c, c, c, c, c);
  const double ee = 1e-6 * 1e-6;
  const double w[3] = {0.1 / ee, 0.6 / ee, 0.3 / ee};
  double q[3];
  parabolas64(c, c, c, c, c, q);
  return div64(blend64(w, q), (w[0] + w[1]) + w[2]);
}

__host__ __device__ __forceinline__ double linear5_64(double a, double b, double c, double d, double e) {
  double q[3];
  parabolas64(a, b, c, d, e, q);
  return (0.1 * q[0] + 0.6 * q[1]) + 0.3 * q[2];
}

// TENO5 (Fu, Hu & Adams 2016): the WENO5 stencils kept or dropped by a sharp
// cutoff C_T = 1e-5 on chi_k = gamma_k / sum gamma, gamma_k = (1 + tau5 /
// (beta_k + eps))^6, tau5 = |beta0 - beta2|, eps = 1e-40; the kept stencils
// combined with the linear weights, renormalised.
__host__ __device__ __forceinline__ double teno5_64(double a, double b, double c, double d, double e) {
  double be[3], q[3], w[3], g[3];
  betas64(a, b, c, d, e, be);
  const double tau = bits2d(d2bits(be[0] - be[2]) & 0x7FFFFFFFFFFFFFFFull);
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    double r = 1.0 + div64(tau, be[k] + 1e-40);
    r = r * r * r;
    g[k] = r * r;
  }
  const Div64 s = div64_prep((g[0] + g[1]) + g[2]);
  const double lin[3] = {0.1, 0.6, 0.3};
#pragma unroll
  for (int k = 0; k < 3; ++k) w[k] = (div64(g[k], s) < 1e-5) ? 0.0 : lin[k];
  parabolas64(a, b, c, d, e, q);
  return div64(blend64(w, q), (w[0] + w[1]) + w[2]);
}

// WENO-AO(5,3) (Balsara, Garain & Shu 2016): the quartic through the five
// cell averages blended with WENO5's three parabolas.  Linear weights from
// gamma_hi = gamma_lo = 0.85 (quartic gamma_hi, middle parabola (1 - gamma_hi)
// gamma_lo, outer parabolas half the rest each); the quartic's smoothness from
// its Legendre coefficients on the middle cell; WENO-Z type weights gamma_k (1
// + (tau / (beta_k + eps))^2), tau the mean of |beta_5 - beta_k|, eps = 1e-12.
__host__ __device__ __forceinline__ double wenoao53_64(double a, double b, double c, double d, double e) {
  const double eps = 1e-12, ghi = 0.85, glo = 0.85;
  double be[3], q[3];
  betas64(a, b, c, d, e, be);
  const double u1 = div64(((11.0 * a - 82.0 * b) + 82.0 * d) - 11.0 * e, div64_of(120));
  const double u2 = div64((((-3.0 * a + 40.0 * b) - 74.0 * c) + 40.0 * d) - 3.0 * e, div64_of(56));
  const double u3 = div64(fma64(-2.0, d, fma64(2.0, b, neg64(a))) + e, div64_of(12));
  const double u4 = div64(fma64(-4.0, d, fma64(-4.0, b, a) + 6.0 * c) + e, div64_of(24));
  const double s1 = u1 + div64(u3, div64_of(10)), s2 = u2 + (123.0 / 455.0) * u4;
  const double beta5 = ((s1 * s1 + (13.0 / 3.0) * (s2 * s2)) + (781.0 / 20.0) * (u3 * u3)) +
                       (1421461.0 / 2275.0) * (u4 * u4);
  const double g5 = ghi, g1 = (1.0 - ghi) * glo, g0 = 0.5 * ((1.0 - ghi) * (1.0 - glo)), g2 = g0;
  const double tau = div64((fabs(beta5 - be[0]) + fabs(beta5 - be[1])) + fabs(beta5 - be[2]), div64_of(3));
  const double r5 = div64(tau, beta5 + eps), r0 = div64(tau, be[0] + eps), r1 = div64(tau, be[1] + eps),
               r2 = div64(tau, be[2] + eps);
  double w5 = g5 * (1.0 + r5 * r5), w0 = g0 * (1.0 + r0 * r0), w1 = g1 * (1.0 + r1 * r1), w2 = g2 * (1.0 + r2 * r2);
  const Div64 s = div64_prep(((w5 + w0) + w1) + w2);
  w5 = div64(w5, s);
  w0 = div64(w0, s);
  w1 = div64(w1, s);
  w2 = div64(w2, s);
  parabolas64(a, b, c, d, e, q);
  const double q5 = div64((((2.0 * a - 13.0 * b) + 47.0 * c) + 27.0 * d) - 3.0 * e, div64_of(60));
  return div64(w5, g5) * (((q5 - g0 * q[0]) - g1 * q[1]) - g2 * q[2]) + ((w0 * q[0] + w1 * q[1]) + w2 * q[2]);
}

// Reconstruction by mode (0 WENO5-JS, 2 linear, 3 TENO5, 4 WENO-AO(5,3)).
// Each is one function call: ten inlined copies would not fit the instruction
// cache, and a call costs next to nothing beside its FP64 work.
#ifdef __CUDACC__
#define MRB_CALL64 static __host__ __device__ __noinline__
#else
#define MRB_CALL64 static inline
#endif
MRB_CALL64 double recon64(int mode, double a, double b, double c, double d, double e) {
  if (mode == 2) return linear5_64(a, b, c, d, e);
  if (mode == 3) return teno5_64(a, b, c, d, e);
  if (mode == 4) return wenoao53_64(a, b, c, d, e);
  return weno5_64(a, b, c, d, e);
}
MRB_CALL64 double recon64_flat(int mode, double c) {
  return (mode == 0 || mode == 1) ? weno5_64_flat(c) : recon64(mode, c, c, c, c, c);
}

// ---------------------------------------------------------------- cells
// Velocity, pressure and sound speed of a conserved state in any axis order:
// p = (gamma - 1)(E - (0.5 rho) q2) - gamma B, q2 = (v0^2 + v1^2) + v2^2,
// c = sqrt(gamma (p + B) / rho).
struct Prim64 {
  double vel[3], p, c;
};
__host__ __device__ __forceinline__ Prim64 prim64(const double U[5], double g, double B, const Div64& rho) {
  Prim64 q;
  q.vel[0] = div64(U[1], rho);
  q.vel[1] = div64(U[2], rho);
  q.vel[2] = div64(U[3], rho);
  const double q2 = (q.vel[0] * q.vel[0] + q.vel[1] * q.vel[1]) + q.vel[2] * q.vel[2];
  q.p = (g - 1.0) * (U[4] - half64(U[0]) * q2) - g * B;
  q.c = sqrt64(div64(g * (q.p + B), rho));
  return q;
}

// Quantities of one cell of direction D at s (quantity stride qs), whose
// conserved state (direction frame) is there already.  The sum of squares of
// the velocity keeps the x, y, z order in every frame.
__host__ __device__ __forceinline__ void flux64_cell(int D, double g, double B, double* s, int qs) {
  const double r = s[0], m0 = s[qs], m1 = s[2 * qs], m2 = s[3 * qs], E = s[4 * qs];
  const Div64 rho = div64_prep(r);
  const double U[5] = {r, D == 0 ? m0 : (D == 1 ? m2 : m1), D == 0 ? m1 : (D == 1 ? m0 : m2),
                       D == 0 ? m2 : (D == 1 ? m1 : m0), E};
  const Prim64 q = prim64(U, g, B, rho);
  const double v0 = D == 0 ? q.vel[0] : (D == 1 ? q.vel[1] : q.vel[2]);
  const double v1 = D == 0 ? q.vel[1] : (D == 1 ? q.vel[2] : q.vel[0]);
  const double v2 = D == 0 ? q.vel[2] : (D == 1 ? q.vel[0] : q.vel[1]);
  const double Ep = E + q.p;
  s[(CQ_F + 0) * qs] = m0 * v0 + q.p;
  s[(CQ_F + 1) * qs] = m0 * v1;
  s[(CQ_F + 2) * qs] = m0 * v2;
  s[(CQ_F + 3) * qs] = v0 * Ep;
  s[(CQ_VEL + 0) * qs] = v0;
  s[(CQ_VEL + 1) * qs] = v1;
  s[(CQ_VEL + 2) * qs] = v2;
  s[CQ_C * qs] = q.c;
  s[CQ_SQ * qs] = sqrt64(r);
  s[CQ_H * qs] = div64(Ep, rho);
}

// ---------------------------------------------------------------- HLLC
// HLLC (Toro, Spruce & Speares 1994) between rotated-frame states UL, UR
// (normal momentum in slot 1): Einfeldt's outer speeds S_L = min(u_L - c_L,
// u~ - c~), S_R = max(u_R + c_R, u~ + c~) from the Roe average of UL and UR;
// contact speed S* from the momentum balance over the outer waves; flux F_L,
// F*_L, F*_R or F_R by the position of x/t = 0, F*_K = F_K + S_K (U*_K - U_K).
__host__ __device__ __forceinline__ void hllc64(const double UL[5], const double UR[5], double g, double B,
                                                double F[5]) {
  const Div64 dL = div64_prep(UL[0]), dR = div64_prep(UR[0]);
  const Prim64 a = prim64(UL, g, B, dL), b = prim64(UR, g, B, dR);
  const double sL = sqrt64(UL[0]), sR = sqrt64(UR[0]);
  const Div64 den = div64_prep(sL + sR);
  const double un = div64(sL * a.vel[0] + sR * b.vel[0], den);
  const double ut1 = div64(sL * a.vel[1] + sR * b.vel[1], den);
  const double ut2 = div64(sL * a.vel[2] + sR * b.vel[2], den);
  const double HL = div64(UL[4] + a.p, dL), HR = div64(UR[4] + b.p, dR);
  const double H = div64(sL * HL + sR * HR, den);
  const double q2 = (un * un + ut1 * ut1) + ut2 * ut2;
  const double c = sqrt64((g - 1.0) * fma64(-0.5, q2, H));
  const double uL = a.vel[0], uR = b.vel[0];
  const double l0 = un - c, l4 = un + c, xL = uL - a.c, xR = uR + b.c;
  const double SL = (l0 < xL) ? l0 : xL;
  const double SR = (xR < l4) ? l4 : xR;
  const double mL = UL[0] * (SL - uL), mR = UR[0] * (SR - uR);
  const double Ss = div64(((b.p - a.p) + uL * mL) - uR * mR, mL - mR);
  const bool all_left = SL >= 0.0, all_right = !all_left && SR <= 0.0;
  const bool left = all_left || (!all_right && Ss >= 0.0);
  const double* U = left ? UL : UR;
  const double v0 = left ? uL : uR, v1 = left ? a.vel[1] : b.vel[1], v2 = left ? a.vel[2] : b.vel[2];
  const double p = left ? a.p : b.p;
  const double U0 = U[0], U1 = U[1], U2 = U[2], U3 = U[3], U4 = U[4];
  F[0] = U1;
  F[1] = U1 * v0 + p;
  F[2] = U1 * v1;
  F[3] = U1 * v2;
  F[4] = v0 * (U4 + p);
  if (!all_left && !all_right) {
    const double SK = left ? SL : SR, mK = left ? mL : mR;
    const double fac = div64(mK, SK - Ss);
    F[0] = F[0] + SK * (fac - U0);
    F[1] = F[1] + SK * (fac * Ss - U1);
    F[2] = F[2] + SK * (fac * v1 - U2);
    F[3] = F[3] + SK * (fac * v2 - U3);
    F[4] = F[4] + SK * (fac * (div64(U4, left ? dL : dR) + (Ss - v0) * (Ss + div64(p, mK))) - U4);
  }
}

// A reconstructed face state usable by HLLC: rho > 0 and p + B > 0.
__host__ __device__ __forceinline__ bool admissible64(const double U[5], double g, double B) {
  if (!pos64(U[0])) return false;
  const double q2 = div64((U[1] * U[1] + U[2] * U[2]) + U[3] * U[3], U[0]);
  const double p = (g - 1.0) * fma64(-0.5, q2, U[4]) - g * B;
  return pos64(p + B);
}

// ---------------------------------------------------------------- face flux
// One value of the characteristic projections: row (l0, l1, l2, l3, l4) with
// the shared products applied by the caller.
struct Eig64 {
  double un, ut1, ut2, H, c, hq2;          // Roe state, 0.5 q2
  double b1, b2, uic, ic, b1u, b1t1, b1t2; // b2 = 0.5 b1 q2, uic = un / c
};

// Rows of fields 0, 1, 4 applied to X (X0 the mass component): with
// L0 = b2 + un/c, L1 = -(b1 un) - 1/c (field 0; field 4 the other signs of the
// 1/c terms), value = 0.5 ((((L0 X0 + L1 X1) - b1 ut1 X2) - b1 ut2 X3) + b1 X4),
// the factor 0.5 of every element of those rows taken out of the sum (exact);
// field 1: (((1 - b2) X0 + b1 un X1) + b1 ut1 X2) + b1 ut2 X3 - b1 X4.
__host__ __device__ __forceinline__ void rows014(const Eig64& e, double X0, double X1, double X2, double X3, double X4,
                                                 double& x0, double& x1, double& x4) {
  const double P2 = e.b1t1 * X2, P3 = e.b1t2 * X3, P4 = e.b1 * X4;
  x0 = half64((((e.b2 + e.uic) * X0 - (e.b1u + e.ic) * X1) - P2) - P3 + P4);
  x4 = half64((((e.b2 - e.uic) * X0 + (e.ic - e.b1u) * X1) - P2) - P3 + P4);
  x1 = ((((1.0 - e.b2) * X0 + e.b1u * X1) + P2) + P3) - P4;
}
// One of them alone.
__host__ __device__ __forceinline__ double row014(const Eig64& e, int k, double X0, double X1, double X2, double X3,
                                                  double X4) {
  const double P2 = e.b1t1 * X2, P3 = e.b1t2 * X3, P4 = e.b1 * X4;
  if (k == 1) return ((((1.0 - e.b2) * X0 + e.b1u * X1) + P2) + P3) - P4;
  const double L0 = (k == 0) ? e.b2 + e.uic : e.b2 - e.uic;
  const double L1 = (k == 0) ? neg64(e.b1u + e.ic) : e.ic - e.b1u;
  return half64(((L0 * X0 + L1 * X1) - P2) - P3 + P4);
}
// Fields 2 (t = X2, ut = ut1) and 3: -ut X0 + 0 X1 + X2 + 0 X3 + 0 X4 (field 2),
// -ut X0 + 0 X1 + 0 X2 + X3 + 0 X4 (field 3).
__host__ __device__ __forceinline__ double row2(double ut1, double X0, double X1, double X2, double X3, double X4) {
  return add_zero(add_zero(add_zero(neg64(ut1 * X0), X1) + X2, X3), X4);
}
__host__ __device__ __forceinline__ double row3(double ut2, double X0, double X1, double X2, double X3, double X4) {
  return add_zero(add_zero(add_zero(neg64(ut2 * X0), X1), X2) + X3, X4);
}

// Characteristic value of the state, field k, cell m.
__host__ __device__ __forceinline__ double state_row(const Row64& r, const Eig64& e, int k, int m) {
  const double X0 = r(0, m), X1 = r(1, m), X2 = r(2, m), X3 = r(3, m), X4 = r(4, m);
  if (k == 2) return row2(e.ut1, X0, X1, X2, X3, X4);
  if (k == 3) return row3(e.ut2, X0, X1, X2, X3, X4);
  return row014(e, k, X0, X1, X2, X3, X4);
}

// Reconstructed characteristic flux of field k from the six values G: upwind
// where the two face cells' and the Roe eigenvalue share a strict sign, else
// (always with LLF) from 0.5 (G + a v) and 0.5 (G - a v), a = max |lam|.
// FLAT: all six cells equal, G[0] alone given.
template <bool FLAT>
__host__ __device__ __forceinline__ double field64(const Row64& r, const Eig64& e, int k, int mode, int flux,
                                                   const double (&G)[6], double lL, double lR, double lt) {
  if (flux == FLUX_ROE) {
    const bool up = pos64(lL) && pos64(lR) && pos64(lt), dn = neg64q(lL) && neg64q(lR) && neg64q(lt);
    if (FLAT) {
      if (up || dn) return recon64_flat(mode, G[0]);
    } else if (up || dn) {
      return recon64(mode, up ? G[0] : G[5], up ? G[1] : G[4], up ? G[2] : G[3], up ? G[3] : G[2], up ? G[4] : G[1]);
    }
  }
  const double alpha = absmax64(lL, lR);
  if (FLAT) {
    double fp, fm;
    half_sums64(G[0], alpha * state_row(r, e, k, 0), fp, fm);
    return recon64_flat(mode, fp) + recon64_flat(mode, fm);
  }
  double fp[6], fm[6];
#pragma unroll
  for (int m = 0; m < 6; ++m) half_sums64(G[m], alpha * state_row(r, e, k, m), fp[m], fm[m]);
  return recon64(mode, fp[0], fp[1], fp[2], fp[3], fp[4]) + recon64(mode, fm[5], fm[4], fm[3], fm[2], fm[1]);
}

// Numerical flux between cells 2 and 3 of the row (direction frame).  Roe
// averages (sL x_L + sR x_R) / (sL + sR) with s = sqrt(rho); FLAT as above.
template <bool FLAT>
__host__ __device__ __forceinline__ void face_flux64(const Row64& r, double g, double B, int mode, int flux,
                                                     double F[5]) {
  constexpr int mL = FLAT ? 0 : 2, mR = FLAT ? 0 : 3;
  Eig64 e;
  {
    const double sL = r(CQ_SQ, mL), sR = r(CQ_SQ, mR);
    const Div64 den = div64_prep(sL + sR);
    e.un = div64(sL * r(CQ_VEL, mL) + sR * r(CQ_VEL, mR), den);
    e.ut1 = div64(sL * r(CQ_VEL + 1, mL) + sR * r(CQ_VEL + 1, mR), den);
    e.ut2 = div64(sL * r(CQ_VEL + 2, mL) + sR * r(CQ_VEL + 2, mR), den);
    e.H = div64(sL * r(CQ_H, mL) + sR * r(CQ_H, mR), den);
    const double q2 = (e.un * e.un + e.ut1 * e.ut1) + e.ut2 * e.ut2;
    e.hq2 = half64(q2);
    const double c2 = (g - 1.0) * (e.H - e.hq2);
    e.c = sqrt64(c2);
    e.ic = div64(1.0, e.c);
    e.b1 = div64(g - 1.0, c2);
    e.b2 = half64(e.b1 * q2);
    e.uic = e.un * e.ic;
    e.b1u = e.b1 * e.un;
    e.b1t1 = e.b1 * e.ut1;
    e.b1t2 = e.b1 * e.ut2;
  }
  const double uc = e.un * e.c;
  if (flux == FLUX_HLLC) {
    // characteristic variables reconstructed from both sides, mapped back with R
    double UL[5], UR[5];
#pragma unroll 1
    for (int k = 0; k < 5; ++k) {
      double v[6];
#pragma unroll
      for (int m = 0; m < (FLAT ? 1 : 6); ++m) v[m] = state_row(r, e, k, m);
      double x, y;
      if (FLAT) {
        x = y = recon64_flat(mode, v[0]);
      } else {
        x = recon64(mode, v[0], v[1], v[2], v[3], v[4]);
        y = recon64(mode, v[5], v[4], v[3], v[2], v[1]);
      }
#pragma unroll
      for (int sd = 0; sd < 2; ++sd) {
        double* X = sd ? UR : UL;
        const double z = sd ? y : x;
        if (k == 0) {
          X[0] = z;
          X[1] = (e.un - e.c) * z;
          X[2] = e.ut1 * z;
          X[3] = e.ut2 * z;
          X[4] = (e.H - uc) * z;
        } else if (k == 1 || k == 4) {
          X[0] = X[0] + z;
          X[1] = X[1] + ((k == 1) ? e.un : e.un + e.c) * z;
          X[2] = X[2] + e.ut1 * z;
          X[3] = X[3] + e.ut2 * z;
          X[4] = X[4] + ((k == 1) ? e.hq2 : e.H + uc) * z;
        } else {
          X[0] = add_zero(X[0], z);
          X[1] = add_zero(X[1], z);
          X[2] = (k == 2) ? X[2] + z : add_zero(X[2], z);
          X[3] = (k == 3) ? X[3] + z : add_zero(X[3], z);
          X[4] = X[4] + ((k == 2) ? e.ut1 : e.ut2) * z;
        }
      }
    }
    if (!admissible64(UL, g, B) || !admissible64(UR, g, B)) {
#pragma unroll
      for (int j = 0; j < 5; ++j) {
        UL[j] = r(j, mL);
        UR[j] = r(j, mR);
      }
    }
    hllc64(UL, UR, g, B, F);
    return;
  }
  const double unL = r(CQ_VEL, mL), unR = r(CQ_VEL, mR), cL = r(CQ_C, mL), cR = r(CQ_C, mR);
  double gh0, gh1, gh4;
  {
    double G0[6], G1[6], G4[6];
#pragma unroll
    for (int m = 0; m < (FLAT ? 1 : 6); ++m)
      rows014(e, r(1, m), r(CQ_F, m), r(CQ_F + 1, m), r(CQ_F + 2, m), r(CQ_F + 3, m), G0[m], G1[m], G4[m]);
    gh0 = field64<FLAT>(r, e, 0, mode, flux, G0, unL - cL, unR - cR, e.un - e.c);
    gh1 = field64<FLAT>(r, e, 1, mode, flux, G1, unL, unR, e.un);
    gh4 = field64<FLAT>(r, e, 4, mode, flux, G4, unL + cL, unR + cR, e.un + e.c);
  }
  F[0] = gh0 + gh1;
  F[1] = (e.un - e.c) * gh0 + e.un * gh1;
  F[2] = e.ut1 * gh0 + e.ut1 * gh1;
  F[3] = e.ut2 * gh0 + e.ut2 * gh1;
  F[4] = (e.H - uc) * gh0 + e.hq2 * gh1;
  {
    double G[6];
#pragma unroll
    for (int m = 0; m < (FLAT ? 1 : 6); ++m)
      G[m] = row2(e.ut1, r(1, m), r(CQ_F, m), r(CQ_F + 1, m), r(CQ_F + 2, m), r(CQ_F + 3, m));
    const double z = field64<FLAT>(r, e, 2, mode, flux, G, unL, unR, e.un);
    F[0] = add_zero(F[0], z);
    F[1] = add_zero(F[1], z);
    F[2] = F[2] + z;
    F[3] = add_zero(F[3], z);
    F[4] = F[4] + e.ut1 * z;
  }
  {
    double G[6];
#pragma unroll
    for (int m = 0; m < (FLAT ? 1 : 6); ++m)
      G[m] = row3(e.ut2, r(1, m), r(CQ_F, m), r(CQ_F + 1, m), r(CQ_F + 2, m), r(CQ_F + 3, m));
    const double z = field64<FLAT>(r, e, 3, mode, flux, G, unL, unR, e.un);
    F[0] = add_zero(F[0], z);
    F[1] = add_zero(F[1], z);
    F[2] = add_zero(F[2], z);
    F[3] = F[3] + z;
    F[4] = F[4] + e.ut2 * z;
  }
  F[0] = F[0] + gh4;
  F[1] = F[1] + (e.un + e.c) * gh4;
  F[2] = F[2] + e.ut1 * gh4;
  F[3] = F[3] + e.ut2 * gh4;
  F[4] = F[4] + (e.H + uc) * gh4;
}

}  // namespace mrb
