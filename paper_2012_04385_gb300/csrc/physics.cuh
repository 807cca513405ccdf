// Layout constants, the Roe / LLF census rule and the Navier-Stokes viscous flux
// of the block-based MR Euler method (arXiv:2012.04385).  The FP64 face flux
// (EOS, Roe eigensystem, reconstructions, flux schemes) lives in flux64.cuh,
// the mixed-precision one in stage_f32.cuh, the prediction of Eq. (Prediction)
// in mr.cuh.
//
// Every FP64 formula is written in one fixed evaluation order; the FP64 kernels
// are compiled without FMA contraction (-fmad=false), so each double result is
// the correctly rounded value of that exact sequence of operations.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

#include "flux64.cuh"

namespace mrb {

constexpr int NB = 16;                 // internal cells per block edge
constexpr int HW = 4;                  // halo width
constexpr int NS = NB + 2 * HW;        // 24 stored cells per edge
constexpr int NCELL = NS * NS * NS;    // 13824
constexpr int NINT = NB * NB * NB;     // 4096
constexpr int NV = 5;
constexpr int NFACE = NB * NB;         // 256
constexpr int SLOT_U = NV * NCELL;     // doubles per stage buffer
constexpr int SLOT_N = NV * NINT;      // doubles per u^n buffer
constexpr int SLOT_F = 6 * NV * NFACE; // doubles per face-flux set
constexpr int SLOT_SEL = 4 * (34 + 34 + 40);  // uint32 selector decision bits per block (4 z-slabs x 3 directions)
constexpr int SLOT_SH = 6 * NINT;      // floats per FP32 record set (mixed-precision path)

__host__ __device__ __forceinline__ int sidx(int i, int j, int k) { return ((k + HW) * NS + (j + HW)) * NS + (i + HW); }
__host__ __device__ __forceinline__ int iidx(int i, int j, int k) { return (k * NB + j) * NB + i; }

// ---------------------------------------------------------------- viscous flux
// Navier-Stokes viscous flux (Stokes' hypothesis, constant mu, no heat
// conduction) at the face between the stored cells sL and sL + step_d of a
// block (FP64 state with halos), lab frame: (0, tau_xd, tau_yd, tau_zd,
// u . tau_d), tau_ij = mu (du_i/dx_j + du_j/dx_i) - 2/3 mu (div u) delta_ij.
// Second-order compact face gradients: normal derivative from the two face
// cells, tangential derivative as the mean of their central differences;
// face velocity the mean of the two cells'.
__device__ __forceinline__ void cell_vel(const double* __restrict__ u, int s, double w[3]) {
  const Div64 rho = div64_prep(u[s]);
  w[0] = div64(u[NCELL + s], rho);
  w[1] = div64(u[2 * NCELL + s], rho);
  w[2] = div64(u[3 * NCELL + s], rho);
}

// (dx and 4 dx as prepared divisors)
static __device__ __noinline__ void viscous_flux(const double* __restrict__ u, int d, int sL, double mu, const Div64& dx,
                                                 const Div64& dx4, double Fv[5]) {
  const int stepd = (d == 0) ? 1 : (d == 1 ? NS : NS * NS);
  const int sR = sL + stepd;
  double uL[3], uR[3];
  cell_vel(u, sL, uL);
  cell_vel(u, sR, uR);
  // gradients of the normal velocity (Gd) and of every component along d (Gn)
  double Gn[3], Gd[3], Gt[3];          // du_i/dx_d, du_d/dx_i, du_i/dx_i
#pragma unroll
  for (int i = 0; i < 3; ++i) Gn[i] = div64(uR[i] - uL[i], dx);
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    if (j == d) {
      Gd[j] = Gn[j];
      Gt[j] = Gn[j];
      continue;
    }
    const int st = (j == 0) ? 1 : (j == 1 ? NS : NS * NS);
    double a[3], b[3], c[3], e[3];
    cell_vel(u, sL + st, a);
    cell_vel(u, sL - st, b);
    cell_vel(u, sR + st, c);
    cell_vel(u, sR - st, e);
    const double ad = d == 0 ? a[0] : (d == 1 ? a[1] : a[2]), bd = d == 0 ? b[0] : (d == 1 ? b[1] : b[2]);
    const double cd = d == 0 ? c[0] : (d == 1 ? c[1] : c[2]), ed = d == 0 ? e[0] : (d == 1 ? e[1] : e[2]);
    Gd[j] = div64((ad - bd) + (cd - ed), dx4);
    Gt[j] = div64((a[j] - b[j]) + (c[j] - e[j]), dx4);
  }
  const double div = (Gt[0] + Gt[1]) + Gt[2];
  double ub[3], tau[3];
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    ub[i] = half64(uL[i] + uR[i]);
    tau[i] = mu * (Gn[i] + Gd[i]);
    if (i == d) tau[i] = tau[i] - ((2.0 / 3.0) * mu) * div;
  }
  Fv[0] = 0.0;
  Fv[1] = tau[0];
  Fv[2] = tau[1];
  Fv[3] = tau[2];
  Fv[4] = (ub[0] * tau[0] + ub[1] * tau[1]) + ub[2] * tau[2];
}

// Fields (bit k) that take the LLF split at the face between the lab-frame
// states UL, UR along d under the Roe / LLF rule of face_flux64: the same
// primitive variables, Roe average and eigenvalue tests.
__device__ __forceinline__ unsigned split_fields(const double UL[5], const double UR[5], int d, double g, double B) {
  double s[2][CQ_N];
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    const double* U = q ? UR : UL;
    s[q][0] = U[0];
    s[q][1] = U[1 + d];
    s[q][2] = U[1 + (d + 1) % 3];
    s[q][3] = U[1 + (d + 2) % 3];
    s[q][4] = U[4];
    flux64_cell(d, g, B, s[q], 1);
  }
  const double sL = s[0][CQ_SQ], sR = s[1][CQ_SQ];
  const Div64 den = div64_prep(sL + sR);
  const double un = div64(sL * s[0][CQ_VEL] + sR * s[1][CQ_VEL], den);
  const double ut1 = div64(sL * s[0][CQ_VEL + 1] + sR * s[1][CQ_VEL + 1], den);
  const double ut2 = div64(sL * s[0][CQ_VEL + 2] + sR * s[1][CQ_VEL + 2], den);
  const double H = div64(sL * s[0][CQ_H] + sR * s[1][CQ_H], den);
  const double q2 = (un * un + ut1 * ut1) + ut2 * ut2;
  const double c = sqrt64((g - 1.0) * (H - half64(q2)));
  unsigned mask = 0;
#pragma unroll
  for (int k = 0; k < 5; ++k) {
    double lL = s[0][CQ_VEL], lR = s[1][CQ_VEL], lt = un;
    if (k == 0) { lL = lL - s[0][CQ_C]; lR = lR - s[1][CQ_C]; lt = un - c; }
    if (k == 4) { lL = lL + s[0][CQ_C]; lR = lR + s[1][CQ_C]; lt = un + c; }
    const bool up = (pos64(lL) && pos64(lR) && pos64(lt)) || (neg64q(lL) && neg64q(lR) && neg64q(lt));
    if (!up) mask |= 1u << k;
  }
  return mask;
}

}  // namespace mrb
