// Right-hand side and Runge-Kutta stage of the FP64 path (Sec. 2.2 and Alg.
// ComputeLoop of arXiv:2012.04385, with the Shu-Osher TVD-RK3 or TVD-RK2
// stages); every reconstruction, flux scheme and the viscous terms are run-time
// choices here.
//
// Two kernels.  k_flux_f64 works on items of 32 pencils (rows of 16 cells of one
// leaf along one direction, with three cells of halo at each end): the cell
// quantities of the 22 x 32 cells go to shared memory, one warp computes the 32
// fluxes of one face plane, and the flux differences of the 16 x 32 cells go to
// global memory (boundary-face fluxes also to the block's face buffers for the
// jump correction).  k_update_f64 adds the three directions' differences in the
// order x, y, z and forms the stage.
//
// The path is bound by the FP64 pipe, at less than 1% of its memory traffic's
// time, so the split follows the FP64 work: no face and no cell quantity of a
// direction is computed twice (z-slabs shared 17 planes per 16 in x and y but
// five per four in z, and formed every cell's primitives for each of the six
// faces that read it), and 24 or 48 items per leaf occupy the GPU from eight
// leaves on, where four slabs per leaf left 120 of 152 SMs idle.
//
// Uniform data.  A warp whose 32 stencils hold six equal cells takes the flat
// form of the flux (one projection instead of six, constant WENO weights), and
// in an item of constant pencils one face plane stands for all 17.  Both give
// the same bits as the general form; cells are compared bit for bit.
//
// Measured (GB300; flux and update kernels together, before: one kernel per
// z-slab with compiler divisions): shock-bubble on levels 0..2, 316 leaves,
// 27.1 ms -> 7.6 ms per stage; TENO5 and LLF on 60 periodic leaves without
// uniform data 5.34 ms -> 2.17 ms; Sod tube on 8 leaves 2.78 ms -> 0.23 ms.  With
// nine warps a CTA the FP64 pipe is 83% busy (eight: 77%), with 15% of the issue
// slots used.
//
// Scratch.  The differences live in the stage buffer that the stage is about to
// write: those of x at the cells themselves, those of y and z in its halo, which
// no call reads before a fill rewrites it (the right-hand side alone leaves all
// three there).
#pragma once

#include "kernels.cuh"

namespace mrb {

constexpr int F64_P = 32;                     // pencils per item (16 on small trees)
constexpr int F64_L = NB + 6;                 // cells per pencil
// 17 face planes are two rounds of nine warps (of eight: three, the last with one
// warp), which outweighs the 96 registers a thread that two such CTAs leave (128).
// Flux kernel with 8 -> 9 warps: 60 smooth blocks 2.33 -> 2.16 ms, Sod tube 231 -> 218
// us, shock-bubble 7.54 -> 7.48 ms; 6 warps and 168 registers 2.18, 234, 7.76; 11 warps
// and 88 registers 2.21, 217, 7.66.
constexpr int F64_WARPS = 9;
constexpr int F64_THREADS = 32 * F64_WARPS;
constexpr size_t F64_SMEM = sizeof(double) * (CQ_N * F64_L * F64_P + NV * (NB + 1) * F64_P);

// Place of the differences of direction d at cell c (x fastest) in a stage
// buffer, for every variable: x at the cell, y in the 8 x 576 cells of the z
// halo planes, z in the x and y halo of the plane z (192 cells of the eight
// y-halo rows and 64 of the x halo).
__device__ __forceinline__ int diff_place(int d, int c) {
  const int k = c >> 8, q = c & 255;
  if (d == 0) return sidx(q & 15, q >> 4, k);
  if (d == 1) return c < 2048 ? c : (NS - HW) * NS * NS + c - 2048;
  const int in = q < 96 ? q : (q < 192 ? NS * (NS - HW) + q - 96 : (HW + ((q - 192) >> 2)) * NS + (q & 3));
  return (k + HW) * NS * NS + in;
}

// Lane p of plane i along direction d, pencil number pp of the block.
__device__ __forceinline__ void pencil_cell(int d, int pp, int i, int& x, int& y, int& z) {
  const int a = pp & 15, b = pp >> 4;
  x = d == 0 ? i : a;
  y = d == 0 ? a : (d == 1 ? i : b);
  z = d == 2 ? i : b;
}

// Items are (leaf, direction, P pencils); a warp takes 32/P face planes at a
// time.  P = 32, or 16 while the items of 32 pencils would not give every SM
// two (Sod tube of eight leaves: the 64 items along x carry nearly all of the
// work).
static __global__ void __launch_bounds__(F64_THREADS, 2)
    k_flux_f64(Topo t, Phys p, Pool pool, int cur, int level) {
  extern __shared__ __align__(16) double f64_smem[];
  double* cq = f64_smem;
  double* fl = cq + CQ_N * F64_L * F64_P;
  __shared__ unsigned eqm[F64_L - 1];         // bit l: cells i and i + 1 of pencil l are equal
  const int nodes = stage_nodes(t, level);
  const int lp = (nodes * (3 * NFACE / F64_P) < (int)gridDim.x) ? 4 : 5;
  const int P = 1 << lp, per_dir = NFACE >> lp, per_leaf = 3 * per_dir, QS = F64_L << lp;
  const double* __restrict__ src = pool.bufp(cur);
  double* __restrict__ dst = pool.bufp(cur ^ 1);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int pl = lane & (P - 1), sub = lane >> lp, nsub = 32 >> lp;      // pencil, and which of the warp's planes
  const unsigned full = P == 32 ? 0xffffffffu : 0xffffu;
  const ItemRange IR = item_range(nodes * per_leaf, p.blocked);
  for (int w = IR.first; w < IR.end; w += IR.step) {
    const int node = stage_node(t, level, w / per_leaf);
    const int D = (w % per_leaf) / per_dir, pp = ((w % per_dir) << lp) + pl;
    const int4 own = *reinterpret_cast<const int4*>(t.side + (size_t)node * 8 + 4);
    const int slot = own.z;
    const double* __restrict__ u = src + (size_t)slot * SLOT_U;
    for (int i = warp * nsub + sub; i < F64_L; i += F64_WARPS * nsub) {
      // beyond the block: the face neighbour's internal cells, the block's own
      // cells mapped back at a boundary, or its stored (predicted) halo
      int c = i - 3;
      const double* __restrict__ cells = u;
      bool flip = false;
      if (c < 0 || c >= NB) {
        const int hi = c >= NB, nb = t.side[(size_t)node * 8 + 2 * D + hi];
        if (nb >= 0) {
          cells = src + (size_t)nb * SLOT_U;
          c += hi ? -NB : NB;
        } else if (nb == -2) {
          const bool mirror = p.bc[2 * D + hi] == 2;
          c = mirror ? (hi ? 2 * NB - 1 - c : -1 - c) : (hi ? NB - 1 : 0);
          flip = mirror;
        }
      }
      int x, y, z;
      pencil_cell(D, pp, c, x, y, z);
      const int s = sidx(x, y, z);
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        const int q = (v == 0 || v == 4) ? v : 1 + (v + 2 - D) % 3;      // lab component v - 1 in the direction frame
        const double a = cells[v * NCELL + s];
        cq[q * QS + (i << lp) + pl] = (flip && q == 1) ? neg64(a) : a;
      }
    }
    __syncthreads();
    for (int i = warp; i < F64_L - 1; i += F64_WARPS) {
      bool eq = true;
#pragma unroll
      for (int v = 0; v < NV; ++v)
        eq = eq && d2bits(cq[v * QS + (i << lp) + pl]) == d2bits(cq[v * QS + ((i + 1) << lp) + pl]);
      const unsigned m = __ballot_sync(0xffffffffu, eq);
      if (lane == 0) eqm[i] = m & full;
    }
    __syncthreads();
    unsigned all = full;
#pragma unroll
    for (int i = 0; i < F64_L - 1; ++i) all &= eqm[i];
    // every pencil constant: its first face stands for all (not with viscous
    // terms, whose gradients read other pencils)
    const bool uniform = all == full && !(p.mu > 0.0);
    for (int i = warp * nsub + sub; i < (uniform ? 1 : F64_L); i += F64_WARPS * nsub)
      flux64_cell(D, p.gamma, p.B, cq + (i << lp) + pl, QS);
    __syncthreads();
    const int nplane = uniform ? 1 : NB + 1;
    for (int f0 = warp * nsub; f0 < nplane; f0 += F64_WARPS * nsub) {
      const int fa = f0 + sub < nplane ? f0 + sub : f0;                  // (the last warp's spare lanes repeat its first plane)
      const Row64 r{cq + (fa << lp) + pl, QS, P};
      const unsigned m = eqm[fa] & eqm[fa + 1] & eqm[fa + 2] & eqm[fa + 3] & eqm[fa + 4];
      double F[5];
      if (__all_sync(0xffffffffu, (m >> pl) & 1u)) face_flux64<true>(r, p.gamma, p.B, p.recon, p.flux, F);
      else face_flux64<false>(r, p.gamma, p.B, p.recon, p.flux, F);
      if (p.mu > 0.0) {
        // Navier-Stokes: F(U) - F_v at the face between stencil cells 2 and 3
        int x, y, z;
        pencil_cell(D, pp, fa - 1, x, y, z);
        const double dx = ldexp(p.dx0, -t.level[node]);
        double Fv[5];
        viscous_flux(u, D, sidx(x, y, z), p.mu, div64_prep(dx), div64_prep(4.0 * dx), Fv);
        F[0] = F[0] - Fv[0];
        F[1] = F[1] - (D == 0 ? Fv[1] : (D == 1 ? Fv[2] : Fv[3]));
        F[2] = F[2] - (D == 0 ? Fv[2] : (D == 1 ? Fv[3] : Fv[1]));
        F[3] = F[3] - (D == 0 ? Fv[3] : (D == 1 ? Fv[1] : Fv[2]));
        F[4] = F[4] - Fv[4];
      }
#pragma unroll
      for (int v = 0; v < NV; ++v) fl[((v * (NB + 1) + fa) << lp) + pl] = F[v];
    }
    __syncthreads();
    // flux differences and boundary-face fluxes, lab frame (component j of the
    // direction frame is axis (D + j) mod 3)
    double* __restrict__ o = dst + (size_t)slot * SLOT_U;
    double* __restrict__ fb = pool.face + (size_t)slot * SLOT_F;
    const unsigned fm = (unsigned)own.w & 63u;  // sides whose fluxes something reads
    for (int e = warp * nsub + sub; e < NV * (NB + 2); e += F64_WARPS * nsub) {
      const int v = e / (NB + 2), i = e % (NB + 2);
      const int vl = (v == 0 || v == 4) ? v : 1 + (D + v - 1) % 3;
      const double* f = fl + ((v * (NB + 1)) << lp) + pl;
      if (i < NB) {
        int x, y, z;
        pencil_cell(D, pp, i, x, y, z);
        o[vl * NCELL + diff_place(D, iidx(x, y, z))] = f[uniform ? 0 : i << lp] - f[uniform ? 0 : (i + 1) << lp];
      } else {
        const int hi = i - NB;
        if ((fm >> (2 * D + hi)) & 1u) fb[((2 * D + hi) * NV + vl) * NFACE + pp] = f[(uniform || !hi) ? 0 : NB << lp];
      }
    }
    __syncthreads();
  }
}

// L = ((dF_x + dF_y) + dF_z) / dx + S and the stage out = a u^n + b (u + dt L)
// (or L itself), one CTA per four planes of a block.  Elementwise: it reads and
// writes each cell of dst in the same thread, the halo only as scratch.
static __global__ void __launch_bounds__(256) k_update_f64(Topo t, Phys p, Pool pool, int cur, int stage,
                                                           const double* __restrict__ dt, double* __restrict__ rhs_out,
                                                           int level) {
  const int nitems = stage_nodes(t, level) * 4;
  const double* __restrict__ src = pool.bufp(cur);
  double* __restrict__ dst = pool.bufp(cur ^ 1);
  const double ka = kRkA[rk_row(p)][stage], kb = kRkB[rk_row(p)][stage];
  for (int w = blockIdx.x; w < nitems; w += gridDim.x) {
    const int li = w >> 2, node = stage_node(t, level, li), slot = t.slot[node];
    const double* __restrict__ u = src + (size_t)slot * SLOT_U;
    double* __restrict__ unb = pool.un + (size_t)slot * SLOT_N;
    double* __restrict__ o = dst + (size_t)slot * SLOT_U;
    const Div64 dx = div64_prep(ldexp(p.dx0, -t.level[node]));
    const double h = dt ? node_dt(t, p, dt, node, level) : 0.0;
#pragma unroll 1
    for (int q = 0; q < 4; ++q) {
      const int c = (w & 3) * 1024 + q * 256 + threadIdx.x;
      const int s = diff_place(0, c), s1 = diff_place(1, c), s2 = diff_place(2, c);
      double us[NV], d0[NV], d1[NV], d2[NV], un[NV];
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        us[v] = u[v * NCELL + s];
        d0[v] = o[v * NCELL + s];
        d1[v] = o[v * NCELL + s1];
        d2[v] = o[v * NCELL + s2];
        un[v] = (stage != 0 && !rhs_out) ? unb[v * NINT + c] : us[v];
      }
      double L[NV];
#pragma unroll
      for (int v = 0; v < NV; ++v) L[v] = div64((d0[v] + d1[v]) + d2[v], dx);
      if (p.has_grav) {
        L[1] = L[1] + us[0] * p.grav[0];
        L[2] = L[2] + us[0] * p.grav[1];
        L[3] = L[3] + us[0] * p.grav[2];
        L[4] = L[4] + ((us[1] * p.grav[0] + us[2] * p.grav[1]) + us[3] * p.grav[2]);
      }
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        if (rhs_out) {
          rhs_out[((size_t)li * NV + v) * NINT + c] = L[v];
        } else {
          if (stage == 0) unb[v * NINT + c] = us[v];
          const double tt = us[v] + h * L[v];
          o[v * NCELL + s] = (stage == 0) ? tt : ka * un[v] + kb * tt;
        }
      }
    }
  }
}

static void launch_rhs_rk_impl(const Topo& t, const Phys& p, const Pool& pool, int cur, int stage, const double* dt,
                               double* rhs_out, cudaStream_t st, int level) {
  static int resident = 0;
  if (resident == 0) {
    cudaFuncSetAttribute(k_flux_f64, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)F64_SMEM);
    int per_sm = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_flux_f64, F64_THREADS, F64_SMEM);
    resident = sm_count() * (per_sm < 1 ? 1 : per_sm);
  }
  const int grid = resident * (g_tune.stage_waves < 1 ? 1 : g_tune.stage_waves);
  k_flux_f64<<<grid, F64_THREADS, F64_SMEM, st>>>(t, p, pool, cur, level);
  k_update_f64<<<sm_count() * 8, 256, 0, st>>>(t, p, pool, cur, stage, dt, rhs_out, level);
  g_kernel_launches += 2;
}

}  // namespace mrb
