// FP64 kernels of the block-based MR Euler hot path (arXiv:2012.04385): halo
// fill, fused RHS + TVD-RK3 stage, face-flux averaging and jump correction,
// averaging (projection), CFL reduction, MR details and tags, refinement
// prediction, neighbour table, conservation sums, state import/export.
//
// Built with -fmad=false: every double is the correctly rounded result of the
// operation order written here.
#include "mr.cuh"
#include "rhs.cuh"

namespace mrb {

long long g_kernel_launches = 0;

Tune g_tune = {1, 8, 4, 8};

int sm_count() {
  static int n = 0;
  if (n == 0) {
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
    if (n <= 0) n = 1;
  }
  return n;
}

// ---------------------------------------------------------------- state in/out
__global__ void k_set_state(Topo t, Phys p, Pool pool, int cur, const int32_t* __restrict__ nodes, int n,
                            const double* __restrict__ prim) {
  const double g = p.gamma, B = p.B;
  const size_t total = (size_t)n * NINT;
  for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < total; e += (size_t)gridDim.x * blockDim.x) {
    const int b = (int)(e / NINT), c = (int)(e % NINT);
    const int i = c % 16, j = (c / 16) % 16, k = c / 256;
    const double* P = prim + (size_t)b * NV * NINT;
    double rho = P[c], u = P[NINT + c], v = P[2 * NINT + c], w = P[3 * NINT + c], pr = P[4 * NINT + c];
    double q2 = (u * u + v * v) + w * w;
    double* U = pool.bufp(cur) + (size_t)t.slot[nodes[b]] * SLOT_U;
    const int s = sidx(i, j, k);
    U[s] = rho;
    U[NCELL + s] = rho * u;
    U[2 * NCELL + s] = rho * v;
    U[3 * NCELL + s] = rho * w;
    U[4 * NCELL + s] = (pr + g * B) / (g - 1.0) + 0.5 * rho * q2;
  }
}

void launch_set_state(const Topo& t, const Phys& p, const Pool& pool, int cur, const int32_t* nodes, int n,
                      const double* prim, cudaStream_t st) {
  if (n <= 0) return;
  k_set_state<<<sm_count() * 4, 256, 0, st>>>(t, p, pool, cur, nodes, n, prim);
  ++g_kernel_launches;
}

// Conserved states in and out: plain copies, bound by memory.  A CTA moves 16-byte
// pairs of one variable of one block, eight per thread in flight (rows of 16
// cells start on 32-byte boundaries of the stored array); buffers of the caller
// that are not 16-byte aligned go through single doubles.  Before, a thread
// moved one double at a time with four divisions for its index: 5,776 blocks
// (0.95 GB) out in 625 us.
template <bool VEC>
__device__ __forceinline__ double2 load_pair(const double* __restrict__ p) {
  if (VEC) return *reinterpret_cast<const double2*>(p);
  return make_double2(p[0], p[1]);
}
template <bool VEC>
__device__ __forceinline__ void store_pair(double* __restrict__ p, double2 x) {
  if (VEC) {
    *reinterpret_cast<double2*>(p) = x;
  } else {
    p[0] = x.x;
    p[1] = x.y;
  }
}
// stored offset of the pair e (0 .. 2047) of a variable's internal cells
__device__ __forceinline__ int pair_sidx(int e) { return sidx(2 * (e & 7), (e >> 3) & 15, e >> 7); }

template <bool VEC>
__global__ void __launch_bounds__(256) k_set_cons(Topo t, Pool pool, int cur, const int32_t* __restrict__ nodes, int n,
                                                  const double* __restrict__ cons) {
  for (int w = blockIdx.x; w < n * NV; w += gridDim.x) {
    const double* __restrict__ src = cons + (size_t)w * NINT;
    double* __restrict__ U = pool.bufp(cur) + (size_t)t.slot[nodes[w / NV]] * SLOT_U + (size_t)(w % NV) * NCELL;
    double2 x[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) x[q] = load_pair<VEC>(src + 2 * (threadIdx.x + 256 * q));
#pragma unroll
    for (int q = 0; q < 8; ++q) store_pair<true>(U + pair_sidx(threadIdx.x + 256 * q), x[q]);
  }
}

void launch_set_cons(const Topo& t, const Phys& p, const Pool& pool, int cur, const int32_t* nodes, int n,
                     const double* cons, cudaStream_t st) {
  if (n <= 0) return;
  if (p.precision == 1) {
    launch_set_cons_f32(t, p, pool, cur, nodes, n, cons, st);
    return;
  }
  const int grid = item_grid((int64_t)n * NV);
  if (((uintptr_t)cons & 15) == 0) k_set_cons<true><<<grid, 256, 0, st>>>(t, pool, cur, nodes, n, cons);
  else k_set_cons<false><<<grid, 256, 0, st>>>(t, pool, cur, nodes, n, cons);
  ++g_kernel_launches;
}

constexpr int GET_PARTS = 27;     // of a block with its halo
template <bool VEC>
__global__ void __launch_bounds__(256) k_get_state(Topo t, Pool pool, int cur, const int32_t* __restrict__ nodes, int n,
                                                   double* __restrict__ out, int with_halo) {
  if (with_halo) {        // a block's stored cells are contiguous
    constexpr int PARTS = GET_PARTS, PER = SLOT_U / 2 / PARTS;       // 27 x 1280 pairs
    static_assert(PARTS * PER * 2 == SLOT_U && PER == 5 * 256, "whole parts");
    for (int w = blockIdx.x; w < n * PARTS; w += gridDim.x) {
      const size_t off = (size_t)(w % PARTS) * 2 * PER + 2 * threadIdx.x;
      const double* __restrict__ U = pool.bufp(cur) + (size_t)t.slot[nodes[w / PARTS]] * SLOT_U + off;
      double* __restrict__ o = out + (size_t)(w / PARTS) * SLOT_U + off;
      double2 x[5];
#pragma unroll
      for (int q = 0; q < 5; ++q) x[q] = load_pair<true>(U + 512 * q);
#pragma unroll
      for (int q = 0; q < 5; ++q) store_pair<VEC>(o + 512 * q, x[q]);
    }
    return;
  }
  for (int w = blockIdx.x; w < n * NV; w += gridDim.x) {
    const double* __restrict__ U = pool.bufp(cur) + (size_t)t.slot[nodes[w / NV]] * SLOT_U + (size_t)(w % NV) * NCELL;
    double* __restrict__ o = out + (size_t)w * NINT;
    double2 x[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) x[q] = load_pair<true>(U + pair_sidx(threadIdx.x + 256 * q));
#pragma unroll
    for (int q = 0; q < 8; ++q) store_pair<VEC>(o + 2 * (threadIdx.x + 256 * q), x[q]);
  }
}

void launch_get_state(const Topo& t, const Pool& pool, int cur, const int32_t* nodes, int n, double* out,
                      int with_halo, cudaStream_t st) {
  if (n <= 0) return;
  const int grid = item_grid((int64_t)n * (with_halo ? GET_PARTS : NV));
  if (((uintptr_t)out & 15) == 0) k_get_state<true><<<grid, 256, 0, st>>>(t, pool, cur, nodes, n, out, with_halo);
  else k_get_state<false><<<grid, 256, 0, st>>>(t, pool, cur, nodes, n, out, with_halo);
  ++g_kernel_launches;
}

// ---------------------------------------------------------------- halo fill (mr.cuh)
void launch_fill_copies(const Topo& t, const Pool& pool, int cur, int n_nodes, cudaStream_t st) {
  const int64_t need = ((int64_t)n_nodes * 26 + 7) / 8;         // a warp per region
  k_fill_regions<<<(int)std::min<int64_t>(need, 4 * sm_count() * g_tune.fill_copy), 256, 0, st>>>(t, pool, cur, NodeSet{nullptr, 0});
  ++g_kernel_launches;
}

void launch_fill_bc(const Topo& t, const Phys& p, const Pool& pool, int cur, cudaStream_t st) {
  k_fill_bc<<<sm_count() * 4, 256, 0, st>>>(t, p, pool, cur, NodeSet{nullptr, 0});
  ++g_kernel_launches;
}

void launch_predict(const Topo& t, const Phys& p, const Pool& pool, int cur, int level, int n_nodes, int mode,
                    cudaStream_t st) {
  if (p.precision == 1) {
    launch_predict_f32(t, p, pool, cur, level, n_nodes, mode, st);
    return;
  }
  const bool stage = mode == FILL_STAGE;
  k_predict_t<double><<<predict_grid(n_nodes), 256, 0, st>>>(t, p, pool, cur, stage ? t.pst : t.pall, t.cnt, level,
                                                             stage ? t.smask : t.miss, mode);
  ++g_kernel_launches;
}

void launch_predict_lts(const Topo& t, const Phys& p, const Pool& pool, int cur, int dst, int level, int n_nodes,
                        double th, cudaStream_t st) {
  if (p.precision == 1) {
    launch_predict_lts_f32(t, p, pool, cur, dst, level, n_nodes, th, st);
    return;
  }
  k_predict_t<double, true><<<predict_grid(n_nodes), 256, 0, st>>>(t, p, pool, cur, t.pst, t.cnt, level, t.smask,
                                                                   FILL_STAGE, dst, th);
  ++g_kernel_launches;
}

void launch_fill_list(const Topo& t, const Phys& p, const Pool& pool, int cur, const int32_t* list, int n,
                      cudaStream_t st) {
  if (n <= 0) return;
  if (p.precision == 1) {
    launch_fill_list_f32(t, p, pool, cur, list, n, st);
    return;
  }
  const NodeSet ns{list, n};
  k_fill_regions<<<sm_count() * 8, 256, 0, st>>>(t, pool, cur, ns);
  k_predict_t<double><<<sm_count() * 4, 256, 0, st>>>(t, p, pool, cur, list, nullptr, n, t.miss, FILL_FULL);
  k_fill_bc<<<sm_count() * 4, 256, 0, st>>>(t, p, pool, cur, ns);
  g_kernel_launches += 3;
}

// ---------------------------------------------------------------- RHS + RK (FP64)
void launch_rhs_rk_f64(const Topo& t, const Phys& p, const Pool& pool, int cur, int stage, const double* dt,
                       double* rhs_out, cudaStream_t st, int level) {
  launch_rhs_rk_impl(t, p, pool, cur, stage, dt, rhs_out, st, level);
}

// ---------------------------------------------------------------- fine side of a jump
// Child of an internal node that covers quarter (ct1, ct2) of its side s.
__device__ __forceinline__ int side_child(const Topo& t, int node, int s, int ct1, int ct2) {
  const int d = s / 2, b1 = (d == 0) ? 2 : 1, b2 = (d == 2) ? 2 : 4, bd = (d == 0) ? 1 : (d == 1 ? 2 : 4);
  return t.child0[node] + ((s & 1) ? bd : 0) + (ct1 ? b1 : 0) + (ct2 ? b2 : 0);
}
// Mean of two face cells and the two above them.
__device__ __forceinline__ double mean4(const double* cf) {
  const double2 lo = *reinterpret_cast<const double2*>(cf), up = *reinterpret_cast<const double2*>(cf + NB);
  return 0.25 * ((lo.x + lo.y) + (up.x + up.y));
}
// Flux of an internal node's face cell (side s, position aa, bb): the mean of
// the 2 x 2 covering child face cells.  Formed where a jump reads it; averaging
// every face of every internal node level by level took a launch per level and
// 135 us per stage on the shock-bubble, for the few per cent of faces that a jump
// reads.
__device__ __forceinline__ double fine_flux(const Topo& t, const double* faces, int node, int s, int v, int aa, int bb) {
  const int ct1 = aa / 8, ct2 = bb / 8;
  const double* cf = faces + (size_t)t.slot[side_child(t, node, s, ct1, ct2)] * SLOT_F + (s * NV + v) * NFACE +
                     2 * (bb - 8 * ct2) * NB + 2 * (aa - 8 * ct1);
  return mean4(cf);
}
// (children of `node` on its side s are refined)
__device__ __forceinline__ bool deep_side(const Topo& t, int node, int s) {
  bool deep = false;
#pragma unroll
  for (int q = 0; q < 4; ++q) deep |= t.child0[side_child(t, node, s, q & 1, q >> 1)] >= 0;
  return deep;
}
// Side s of the refined neighbour `top` where leaves two or more levels finer
// meet the jump (rare: the details of neighbours differ little): the refined
// children on that side, deepest first, get the means of their own children's
// fluxes, in their own face buffers, which nothing else uses.  All threads of the
// CTA; the (up to four) refined children of a node together, as the chain of loads
// is what a pass lasts.  Only one coarse leaf meets any of these sides.  (One thread
// per face cell of `top` descending by itself left most threads without work:
// beside a corner refined six levels deep a right-hand side took 1275 us, now 105;
// beside a whole side four levels finer 760, now 630.)
static __device__ __noinline__ void average_side(const Topo& t, double* faces, int top, int s) {
  int node[MAXL + 1], depth = 0;
  unsigned todo[MAXL + 1];       // children on the side still to descend into: those with refined children there
  const int lane = threadIdx.x & 31, g = lane & 15;
  auto enter = [&](int n) {      // (lanes 4 q .. 4 q + 3 ask the children of child q)
    const int ch = side_child(t, n, s, (g >> 2) & 1, g >> 3);
    const bool deep = t.child0[ch] >= 0 && t.child0[side_child(t, ch, s, g & 1, (g >> 1) & 1)] >= 0;
    const unsigned m = __ballot_sync(0xffffffffu, deep);
    node[depth] = n;
    todo[depth] = ((m & 15u) != 0u) | ((m & 0xf0u) ? 2u : 0u) | ((m & 0xf00u) ? 4u : 0u) | ((m & 0xf000u) ? 8u : 0u);
  };
  enter(top);
  while (depth >= 0) {
    const int n = node[depth];
    if (todo[depth] != 0u) {
      const int q = __ffs(todo[depth]) - 1;
      todo[depth] &= todo[depth] - 1u;
      ++depth;
      enter(side_child(t, n, s, q & 1, q >> 1));
      continue;
    }
    // child q by 64 threads, rows of 16 cells 4 i + 0 .. 3 at a time: the lower ones from its
    // lower children, the upper ones from its upper children
    const int q = threadIdx.x >> 6, ch = side_child(t, n, s, q & 1, q >> 1);     // (256 threads)
    if (t.child0[ch] >= 0) {
      const int a = threadIdx.x & 15, r = (threadIdx.x >> 4) & 3;
      double* F = faces + (size_t)t.slot[ch] * SLOT_F + s * NV * NFACE + (threadIdx.x & 63);
      const int in = s * NV * NFACE + 2 * r * NB + 2 * (a & 7);
      const double* C[2];
#pragma unroll
      for (int up = 0; up < 2; ++up) C[up] = faces + (size_t)t.slot[side_child(t, ch, s, a >> 3, up)] * SLOT_F + in;
#pragma unroll
      for (int up = 0; up < 2; ++up) {
        double x[2][NV];
#pragma unroll
        for (int k = 0; k < 2; ++k)
#pragma unroll
          for (int v = 0; v < NV; ++v) x[k][v] = mean4(C[up] + v * NFACE + 8 * k * NB);
#pragma unroll
        for (int k = 0; k < 2; ++k)
#pragma unroll
          for (int v = 0; v < NV; ++v) F[v * NFACE + 64 * (2 * up + k)] = x[k][v];
      }
    }
    __syncthreads();
    --depth;
  }
}

// ---------------------------------------------------------------- local time stepping
// (Eq. LtsTimestep; the reading: a level's step advances all its nodes, the
// halo fill of each stage sees coarser levels interpolated in time, levels are
// averaged from their children when their step ends, and the boundary-face
// fluxes integrated over the macro step are exchanged at its end.)

// Nodes of levels 0 .. below-1: their internal cells become (1 - theta) u^n +
// theta u, the end state u kept in the other stage buffer (restore = 0), or are
// put back from there (restore = 1).
__global__ void k_lts_interp(Topo t, Pool pool, int cur, int below, LevelTheta th, int restore) {
  const int end = t.cnt[CNT_LVL + below];
  for (int w = t.cnt[CNT_LVL + 0] + blockIdx.x; w < end; w += gridDim.x) {
    const int node = t.lvl_nodes[w];
    const size_t slot = (size_t)t.slot[node];
    double* U = pool.bufp(cur) + slot * SLOT_U;
    double* K = pool.bufp(cur ^ 1) + slot * SLOT_U;
    const double* N = pool.un + slot * SLOT_N;
    const double q = th.th[t.level[node]];
    for (int e = threadIdx.x; e < NV * NINT; e += blockDim.x) {
      const int v = e / NINT, ii = e % NINT;
      const int s = v * NCELL + sidx(ii % 16, (ii / 16) % 16, ii / 256);
      if (restore) {
        U[s] = K[s];
      } else {
        const double u = U[s];
        K[s] = u;
        U[s] = (1.0 - q) * N[e] + q * u;
      }
    }
  }
}

void launch_lts_interp(const Topo& t, const Pool& pool, int cur, int below, const LevelTheta& th, int restore,
                       cudaStream_t st) {
  if (below <= 0) return;
  k_lts_interp<<<sm_count() * 4, 256, 0, st>>>(t, pool, cur, below, th, restore);
  ++g_kernel_launches;
}

// Internal cells (and FP32 records) of the nodes of `level`: cur^1 -> cur.  Items
// are 2048 16-byte words of a node (a variable, or a third of the records), every
// thread with its eight in flight: a level has few nodes, and with one CTA per node
// and a word per pass each took 74 us on the shock-bubble with levels 1 and 2 (360
// nodes), so 18 us.
__global__ void __launch_bounds__(256) k_lts_copyback(Topo t, Pool pool, int cur, int level) {
  const int beg = t.cnt[CNT_LVL + level], end = t.cnt[CNT_LVL + level + 1];
  const int parts = pool.shp(0) ? 8 : NV;
  for (int w = blockIdx.x; w < (end - beg) * parts; w += gridDim.x) {
    const size_t slot = (size_t)t.slot[t.lvl_nodes[beg + w / parts]];
    const int part = w % parts;
    double2 x[8];
    double* O;
    const double* I;
    int at, step;
    if (part < NV) {
      // pair (8 per row) p of the variable: rows of a plane 32 apart per pass
      const int row = threadIdx.x >> 3;
      at = part * NCELL + sidx(2 * (threadIdx.x & 7), row & 15, row >> 4);
      step = 2 * NS * NS;
      O = pool.bufp(cur) + slot * SLOT_U;
      I = pool.bufp(cur ^ 1) + slot * SLOT_U;
    } else {
      at = ((part - NV) * 2048 + threadIdx.x) * 2;
      step = 512;
      O = reinterpret_cast<double*>(pool.shp(cur) + slot * SLOT_SH);
      I = reinterpret_cast<const double*>(pool.shp(cur ^ 1) + slot * SLOT_SH);
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) x[i] = load_now(I + at + i * step);
#pragma unroll
    for (int i = 0; i < 8; ++i) *reinterpret_cast<double2*>(O + at + i * step) = x[i];
  }
}
static_assert(SLOT_SH * sizeof(float) == 3 * 2048 * sizeof(double2) && NINT * sizeof(double) == 2048 * sizeof(double2),
              "parts of k_lts_copyback");

void launch_lts_copyback(const Topo& t, const Pool& pool, int cur, int level, cudaStream_t st) {
  k_lts_copyback<<<sm_count() * 6, 256, 0, st>>>(t, pool, cur, level);
  ++g_kernel_launches;
}

// Integrated boundary-face fluxes of leaves: zero all (zero = 1) or, for the
// leaves of `level`, add (w_stage x dt 2^(lmax - level)) x the stage's face fluxes.
// Items are (leaf, side) pairs: NV * NFACE values, in 16-byte words.
__global__ void __launch_bounds__(256) k_lts_fmac(Topo t, Phys p, Pool pool, int level, int stage,
                                                  const double* __restrict__ dt, int zero) {
  const int beg = zero ? 0 : t.cnt[CNT_LVL + level];
  const int end = zero ? t.cnt[CNT_NLEAVES] : t.cnt[CNT_LVL + level + 1];
  constexpr int NP = NV * NFACE / 2;
  for (int w = blockIdx.x; w < (end - beg) * 6; w += gridDim.x) {
    const int node = zero ? t.leaves[beg + w / 6] : t.lvl_nodes[beg + w / 6], sd = w % 6;
    if (t.child0[node] >= 0) continue;
    const size_t at = (size_t)t.slot[node] * SLOT_F + sd * NV * NFACE;
    double2* M = reinterpret_cast<double2*>(pool.fmac + at);
    if (zero) {
      for (int e = threadIdx.x; e < NP; e += blockDim.x) M[e] = make_double2(0.0, 0.0);
      continue;
    }
    if (!((t.fmask[node] >> sd) & 1u)) continue;                   // (the sides that the reflux reads)
    const double2* F = reinterpret_cast<const double2*>(pool.face + at);
    const double wgt = kRkW[rk_row(p)][stage] * ldexp(dt[t.inst[node]], p.lmax[t.inst[node]] - level);
    for (int e = threadIdx.x; e < NP; e += blockDim.x) {
      const double2 m = M[e], x = F[e];
      M[e] = make_double2(m.x + wgt * x.x, m.y + wgt * x.y);
    }
  }
}

void launch_lts_fmac(const Topo& t, const Phys& p, const Pool& pool, int level, int stage, const double* dt,
                     int zero, cudaStream_t st) {
  k_lts_fmac<<<sm_count() * 8, 256, 0, st>>>(t, p, pool, level, stage, dt, zero);
  ++g_kernel_launches;
}

// u += (F_c - F_f)/dx on an upper face, (F_f - F_c)/dx on a lower one, with the
// integrated fluxes of the leaf and of its refined same-level neighbour.
__global__ void __launch_bounds__(256, 4) k_lts_reflux(Topo t, Phys p, Pool pool, int cur) {
  const int nitems = t.cnt[CNT_JUMP];
  for (int w = blockIdx.x; w < nitems; w += gridDim.x) {
    const int li = t.jump[w] >> 6, mask = t.jump[w] & 63;
    const int node = t.leaves[li];
    const double* Fc_all = pool.fmac + (size_t)t.slot[node] * SLOT_F;
    const Div64 dx = div64_prep(ldexp(p.dx0, -t.level[node]));
    double* U = pool.bufp(cur) + (size_t)t.slot[node] * SLOT_U;
#pragma unroll 1
    for (int s = 0; s < 6; ++s) {
      const int d = s / 2, hi = s & 1;
      int sv[3] = {0, 0, 0};
      sv[d] = hi ? 1 : -1;
      const int r = (sv[2] + 1) * 9 + (sv[1] + 1) * 3 + (sv[0] + 1);
      if (!((mask >> s) & 1)) continue;
      const int nb = t.nbr[(size_t)node * 27 + r];
      const int so = s ^ 1;
      if (deep_side(t, nb, so)) average_side(t, pool.fmac, nb, so);
      const int t1 = (d == 0) ? 1 : 0, t2 = (d == 2) ? 1 : 2;
      for (int e = threadIdx.x; e < NFACE; e += blockDim.x) {
        const int aa = e % 16, bb = e / 16;
        int c[3];
        c[d] = hi ? NB - 1 : 0;
        c[t1] = aa;
        c[t2] = bb;
#pragma unroll
        for (int v = 0; v < NV; ++v) {
          const double Fc = Fc_all[(s * NV + v) * NFACE + e];
          const double Ff = fine_flux(t, pool.fmac, nb, so, v, aa, bb);
          const double dU = div64(hi ? Fc - Ff : Ff - Fc, dx);
          double& ur = U[v * NCELL + sidx(c[0], c[1], c[2])];
          ur = ur + dU;
        }
      }
      __syncthreads();
    }
  }
}

void launch_lts_reflux(const Topo& t, const Phys& p, const Pool& pool, int cur, cudaStream_t st) {
  k_lts_reflux<<<sm_count() * 4, 256, 0, st>>>(t, p, pool, cur);
  ++g_kernel_launches;
}

// ---------------------------------------------------------------- jump correction
// A leaf face whose same-level neighbour is refined takes the averaged fine
// flux: dL = (F_c - F_f)/dx on an upper face, (F_f - F_c)/dx on a lower one,
// applied to the stage result as u += b_s (dt dL) (or added to L in the
// inspection form), sides x-, x+, y-, y+, z-, z+ in order.
__global__ void __launch_bounds__(256, 4) k_jump(Topo t, Phys p, Pool pool, int target, int stage,
                                                 const double* __restrict__ dt, double* __restrict__ rhs_out) {
  const int nitems = t.cnt[CNT_JUMP];
  for (int w = blockIdx.x; w < nitems; w += gridDim.x) {
    const int li = t.jump[w] >> 6, mask = t.jump[w] & 63;
    const int node = t.leaves[li];
    const double* Fc_all = pool.face + (size_t)t.slot[node] * SLOT_F;
    const Div64 dx = div64_prep(ldexp(p.dx0, -t.level[node]));
    const double h = dt ? dt[t.inst[node]] : 0.0;
    const double bs = kRkB[rk_row(p)][stage];
    double* U = pool.bufp(target) + (size_t)t.slot[node] * SLOT_U;
#pragma unroll 1
    for (int s = 0; s < 6; ++s) {
      const int d = s / 2, hi = s & 1;
      int sv[3] = {0, 0, 0};
      sv[d] = hi ? 1 : -1;
      const int r = (sv[2] + 1) * 9 + (sv[1] + 1) * 3 + (sv[0] + 1);
      if (!((mask >> s) & 1)) continue;      // the side's neighbour is not refined
      const int nb = t.nbr[(size_t)node * 27 + r];
      const int so = s ^ 1;
      if (deep_side(t, nb, so)) average_side(t, pool.face, nb, so);
      const int t1 = (d == 0) ? 1 : 0, t2 = (d == 2) ? 1 : 2;
      for (int e = threadIdx.x; e < NFACE; e += blockDim.x) {
        const int aa = e % 16, bb = e / 16;
        int c[3];
        c[d] = hi ? NB - 1 : 0;
        c[t1] = aa;
        c[t2] = bb;
#pragma unroll
        for (int v = 0; v < NV; ++v) {
          const double Fc = Fc_all[(s * NV + v) * NFACE + e];
          const double Ff = fine_flux(t, pool.face, nb, so, v, aa, bb);
          const double dL = div64(hi ? Fc - Ff : Ff - Fc, dx);
          if (rhs_out) {
            double& Lr = rhs_out[((size_t)li * NV + v) * NINT + iidx(c[0], c[1], c[2])];
            Lr = Lr + dL;
          } else {
            double& ur = U[v * NCELL + sidx(c[0], c[1], c[2])];
            ur = ur + bs * (h * dL);
            // the mixed-precision path's FP32 stage increment follows the correction
            if (pool.dl) pool.dl[(size_t)t.slot[node] * SLOT_N + v * NINT + iidx(c[0], c[1], c[2])] += (float)(bs * (h * dL));
          }
        }
      }
      __syncthreads();
    }
  }
}

void launch_jump(const Topo& t, const Phys& p, const Pool& pool, int target, int stage, const double* dt,
                 double* rhs_out, cudaStream_t st) {
  k_jump<<<sm_count() * 8, 256, 0, st>>>(t, p, pool, target, stage, dt, rhs_out);
  ++g_kernel_launches;
}

// ---------------------------------------------------------------- averaging (mr.cuh)
static __global__ void __launch_bounds__(256) k_project(Topo t, Pool pool, int buf, int level) {
  project_level(t, pool, buf, level, NoRecord{});
}

void launch_project_level(const Topo& t, const Phys& p, const Pool& pool, int buf, int level, cudaStream_t st) {
  if (p.precision == 1) {
    launch_project_level_f32(t, p, pool, buf, level, st);
    return;
  }
  k_project<<<sm_count() * g_tune.project, 256, 0, st>>>(t, pool, buf, level);
  ++g_kernel_launches;
}

// ---------------------------------------------------------------- CFL
// Block-wide maxima of N values per thread (sh: [N][8] for 256 threads); the
// result is valid in the first warp.
template <int N>
__device__ __forceinline__ void block_max(double v[N], double* sh) {
  for (int q = 0; q < N; ++q)
    for (int o = 16; o > 0; o >>= 1) v[q] = fmax(v[q], __shfl_xor_sync(0xffffffffu, v[q], o));
  const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (lane == 0)
    for (int q = 0; q < N; ++q) sh[q * 8 + wid] = v[q];
  __syncthreads();
  if (threadIdx.x < 32) {
    for (int q = 0; q < N; ++q) {
      double x = (lane < 8) ? sh[q * 8 + lane] : 0.0;
      for (int o = 4; o > 0; o >>= 1) x = fmax(x, __shfl_xor_sync(0xffffffffu, x, o));
      v[q] = x;
    }
  }
  __syncthreads();
}

// Items are quarters of a leaf (FP64-pipe work, so that few leaves spread over the
// SMs: Sod tube's 8 blocks 38 -> 16 us).
__global__ void __launch_bounds__(256) k_cfl(Topo t, Phys p, Pool pool, int cur, unsigned long long* __restrict__ smax,
                                             int* __restrict__ status, double* __restrict__ dt, double** hist) {
  __shared__ double sh[32];
  const int nitems = t.cnt[CNT_NLEAVES] * 4;
  for (int w = blockIdx.x; w < nitems; w += gridDim.x) {
    const int node = t.leaves[w >> 2];
    const double* U = pool.bufp(cur) + (size_t)t.slot[node] * SLOT_U;
    double m[4] = {0.0, 0.0, 0.0, 0.0};   // max |u_d| + c per direction, max 1/rho
    bool bad = false;
    for (int e = (w & 3) * (NINT / 4) + threadIdx.x; e < ((w & 3) + 1) * (NINT / 4); e += blockDim.x) {
      const int s = sidx(e % 16, (e / 16) % 16, e / 256);
      double Uc[5];
#pragma unroll
      for (int v = 0; v < 5; ++v) Uc[v] = U[v * NCELL + s];
      const Div64 rho = div64_prep(Uc[0]);
      const Prim64 q = prim64(Uc, p.gamma, p.B, rho);
      if (!pos64(Uc[0]) || !pos64(q.p + p.B)) bad = true;
#pragma unroll
      for (int d = 0; d < 3; ++d) m[d] = fmax(m[d], fabs(q.vel[d]) + q.c);
      if (p.mu > 0.0) m[3] = fmax(m[3], div64(1.0, rho));
    }
    if (bad) atomicExch(status, (int)ST_NONPHYS);
    block_max<4>(m, sh);
    if (threadIdx.x == 0) {
      const int inst = t.inst[node];
      for (int d = 0; d < 4; ++d) atomicMax(&smax[inst * 4 + d], (unsigned long long)__double_as_longlong(m[d]));
    }
  }
  cfl_finish(p, smax, dt, hist);
}

void launch_cfl(const Topo& t, const Phys& p, const Pool& pool, int cur, int n_leaves, unsigned long long* smax,
                double* dt, double** hist, int* status, cudaStream_t st) {
  if (p.precision == 1) {
    launch_cfl_f32(t, p, pool, cur, n_leaves, smax, dt, hist, status, st);
    return;
  }
  k_cfl<<<std::min(4 * n_leaves, 4 * sm_count()), 256, 0, st>>>(t, p, pool, cur, smax, status, dt, hist);
  ++g_kernel_launches;
}

static __global__ void k_set_hist(double** hist, double* row) { *hist = row; }
void launch_set_hist(double** hist, double* row, cudaStream_t st) {
  k_set_hist<<<1, 1, 0, st>>>(hist, row);
  ++g_kernel_launches;
}

// ---------------------------------------------------------------- MR details (mr.cuh) and tags
__global__ void k_tags(Topo t, Phys p, const double* __restrict__ delta_node, int allow_refine,
                       int8_t* __restrict__ tags, double* __restrict__ delta_leaf) {
  const int nleaves = t.cnt[CNT_NLEAVES];
  for (int li = blockIdx.x * blockDim.x + threadIdx.x; li < nleaves; li += gridDim.x * blockDim.x) {
    const int node = t.leaves[li];
    const int lvl = t.level[node];
    const double dl = (lvl >= 1) ? delta_node[node] : 0.0;
    int8_t tag = 0;
    if (lvl >= 1) {
      const int lmx = p.lmax[t.inst[node]];
      const double el = ldexp(p.eps, -3 * (lmx - lvl));
      if (allow_refine && dl > el && lvl < lmx) {
        tag = 1;
      } else if (lvl >= 2) {
        const int c0 = t.child0[t.parent[node]];
        bool all = true;
        for (int c = 0; c < 8; ++c) {
          const int sn = c0 + c;
          if (t.child0[sn] >= 0 || !(delta_node[sn] < el)) {
            all = false;
            break;
          }
        }
        // between time steps a group stays while its parent's own detail asks
        // for it (the parent would be refined again at once)
        if (all && allow_refine && delta_node[t.parent[node]] > ldexp(p.eps, -3 * (lmx - (lvl - 1)))) all = false;
        if (all) tag = -1;
      }
    }
    tags[li] = tag;
    if (delta_leaf) delta_leaf[li] = dl;
  }
}

void launch_delta_tags(const Topo& t, const Phys& p, const Pool& pool, int cur, double* delta_node,
                       int allow_refine, int8_t* tags, double* delta_leaf, int n_leaves_cap, int n_nodes, cudaStream_t st) {
  if (p.precision == 1) launch_delta_f32(t, p, pool, cur, delta_node, allow_refine, allow_refine ? n_nodes : n_leaves_cap, st);
  else {
    cudaMemsetAsync(delta_node, 0, (size_t)n_nodes * sizeof(double), st);
    k_delta_f64<<<item_grid((int64_t)(allow_refine ? n_nodes : n_leaves_cap) * 4), 256, 0, st>>>(t, p, pool, cur, delta_node, allow_refine);
    ++g_kernel_launches;
  }
  k_tags<<<(n_leaves_cap + 255) / 256, 256, 0, st>>>(t, p, delta_node, allow_refine, tags, delta_leaf);
  ++g_kernel_launches;
}

// ---------------------------------------------------------------- Roe / LLF census
// counts[k] += faces (of every leaf, 17 x 16 x 16 per direction) where field k
// takes the LLF split; counts[5] += faces.  Per-thread counts, warp sums, one
// atomic per warp and counter.
__global__ void __launch_bounds__(256) k_flux_census(Topo t, Phys p, Pool pool, int cur,
                                                     unsigned long long* __restrict__ counts) {
  const long long nfaces = (long long)t.cnt[CNT_NLEAVES] * 3 * 17 * NFACE;
  unsigned c[6] = {0, 0, 0, 0, 0, 0};
  for (long long it = (long long)blockIdx.x * blockDim.x + threadIdx.x; it < nfaces;
       it += (long long)gridDim.x * blockDim.x) {
    const int li = (int)(it / (3 * 17 * NFACE));
    const int r = (int)(it % (3 * 17 * NFACE));
    const int d = r / (17 * NFACE), f = (r % (17 * NFACE)) / NFACE, ab = r % NFACE;
    const int a = ab % NB, b = ab / NB;
    int cl[3];
    cl[d] = f - 1;
    cl[(d == 0) ? 1 : 0] = a;
    cl[(d == 2) ? 1 : 2] = b;
    const int step[3] = {1, NS, NS * NS};
    const int sL = sidx(cl[0], cl[1], cl[2]), sR = sL + step[d];
    const double* U = pool.bufp(cur) + (size_t)t.slot[t.leaves[li]] * SLOT_U;
    double UL[5], UR[5];
#pragma unroll
    for (int v = 0; v < 5; ++v) {
      UL[v] = U[v * NCELL + sL];
      UR[v] = U[v * NCELL + sR];
    }
    const unsigned m = split_fields(UL, UR, d, p.gamma, p.B);
#pragma unroll
    for (int k = 0; k < 5; ++k) c[k] += (m >> k) & 1u;
    c[5] += 1;
  }
#pragma unroll
  for (int k = 0; k < 6; ++k) {
    unsigned x = c[k];
    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    if ((threadIdx.x & 31) == 0 && x) atomicAdd(&counts[k], (unsigned long long)x);
  }
}

void launch_flux_census(const Topo& t, const Phys& p, const Pool& pool, int cur, unsigned long long* counts,
                        cudaStream_t st) {
  cudaMemsetAsync(counts, 0, 6 * sizeof(unsigned long long), st);
  k_flux_census<<<sm_count() * 8, 256, 0, st>>>(t, p, pool, cur, counts);
  ++g_kernel_launches;
}

// ---------------------------------------------------------------- refinement (mr.cuh)
void launch_refine_fill(const Topo& t, const Phys& p, const Pool& pool, int cur, const int32_t* pairs, int n,
                        cudaStream_t st) {
  if (n <= 0) return;
  if (p.precision == 1) k_refine_fill_t<float><<<item_grid((int64_t)n * NV), 256, 0, st>>>(t, pool, cur, pairs, n);
  else k_refine_fill_t<double><<<item_grid((int64_t)n * NV), 256, 0, st>>>(t, pool, cur, pairs, n);
  ++g_kernel_launches;
}

// ---------------------------------------------------------------- neighbour table
// Same-level neighbour of every node in the 26 directions from block
// coordinates: outside a non-periodic boundary -> -2; otherwise the id of the
// (wrapped) neighbour position is looked up by binary search in the sorted ids
// (-1 when no node of that level exists there).
__device__ __forceinline__ uint64_t make_key_dev(int inst, int level, const int X[3]) {
  const int ng = 7 + level;
  uint64_t m = 0;
  for (int b = 0; b < ng; ++b)
    for (int d = 0; d < 3; ++d) m |= (uint64_t)((X[d] >> b) & 1) << (3 * b + d);
  return ((uint64_t)inst << 56) | (1ull << (3 * ng)) | m;
}

__global__ void k_nbr(Topo t, Phys p, int32_t* __restrict__ nbr_out) {
  const int nn = t.cnt[CNT_NNODES];
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < nn * 27; e += gridDim.x * blockDim.x) {
    const int node = e / 27, r = e % 27;
    if (r == 13) {
      nbr_out[e] = node;
      continue;
    }
    const int s[3] = {r % 3 - 1, (r / 3) % 3 - 1, r / 9 - 1};
    const int lvl = t.level[node];
    int X[3];
    bool outside = false;
    for (int d = 0; d < 3; ++d) {
      const int nl = p.nb[d] << lvl;
      int x = t.X[(size_t)node * 3 + d] + s[d];
      if (x < 0 || x >= nl) {
        if (p.bc[2 * d] == 1) x = (x + nl) % nl;
        else outside = true;
      }
      X[d] = x;
    }
    if (outside) {
      nbr_out[e] = -2;
      continue;
    }
    const uint64_t key = make_key_dev(t.inst[node], lvl, X);
    int lo = 0, hi = nn - 1, found = -1;
    while (lo <= hi) {
      const int mid = (lo + hi) >> 1;
      const uint64_t km = t.keys[mid];
      if (km == key) { found = mid; break; }
      if (km < key) lo = mid + 1;
      else hi = mid - 1;
    }
    nbr_out[e] = found;
  }
}

// Predicted regions.  miss: every region without a same-level node (nor beyond the
// boundary).  smask: those a stage needs -- of a leaf (and with local time
// stepping of every node) the face regions; of an internal node what the wanted
// regions of its children read: a region s of the child in octant cb reads the
// parent's cells within two of it, which lie beyond the parent on axis d (on the
// octant's side) when s_d is 0 or points out of the parent.
constexpr uint32_t FACE_REGIONS = (1u << 12) | (1u << 14) | (1u << 10) | (1u << 16) | (1u << 4) | (1u << 22);
__global__ void k_masks(Topo t, Phys p, uint32_t* __restrict__ miss, uint32_t* __restrict__ smask,
                        uint32_t* __restrict__ fmask, int32_t* __restrict__ side, int32_t* __restrict__ pst,
                        int32_t* __restrict__ pall, int32_t* __restrict__ cnt, int level) {
  const int beg = t.cnt[CNT_LVL + level], end = t.cnt[CNT_LVL + level + 1];
  for (int w = beg + blockIdx.x * blockDim.x + threadIdx.x; w < end; w += gridDim.x * blockDim.x) {
    const int node = t.lvl_nodes[w];
    uint32_t ms = 0;
    for (int r = 0; r < 27; ++r)
      if (t.nbr[(size_t)node * 27 + r] == -1) ms |= 1u << r;
    const int c0 = t.child0[node];
    uint32_t need = (c0 < 0 || p.lts) ? FACE_REGIONS : 0u;
    for (int ch = 0; c0 >= 0 && ch < 8; ++ch) {
      uint32_t m = smask[c0 + ch];
      while (m) {
        const int r = __ffs(m) - 1;
        m &= m - 1;
        const int s[3] = {r % 3 - 1, (r / 3) % 3 - 1, r / 9 - 1};
        int beyond = 0;
        for (int d = 0; d < 3; ++d)
          if (s[d] == 0 || s[d] == (((ch >> d) & 1) ? 1 : -1)) beyond |= 1 << d;
        for (int q = 1; q < 8; ++q) {
          if (q & ~beyond) continue;
          int rr = 13;
          for (int d = 0; d < 3; ++d)
            if ((q >> d) & 1) rr += (((ch >> d) & 1) ? 1 : -1) * (d == 0 ? 1 : (d == 1 ? 3 : 9));
          need |= 1u << rr;
        }
      }
    }
    uint32_t fm = 0;
    const int rn[6] = {12, 14, 10, 16, 4, 22};
    for (int sd = 0; sd < 6; ++sd) {
      const int nb = t.nbr[(size_t)node * 27 + rn[sd]];
      if (nb == -1 || (nb >= 0 && t.child0[nb] >= 0)) fm |= 1u << sd;
      side[(size_t)node * 8 + sd] = nb >= 0 ? t.slot[nb] : nb;
    }
    if (c0 >= 0) fm = 0u;
    fmask[node] = fm;
    side[(size_t)node * 8 + 6] = t.slot[node];
    side[(size_t)node * 8 + 7] = (int32_t)(fm | ((uint32_t)level << 8));
    miss[node] = ms;
    smask[node] = need & ms;
    if (need & ms) pst[beg + atomicAdd(&cnt[CNT_PST + level], 1)] = node;
    if (ms) pall[beg + atomicAdd(&cnt[CNT_PALL + level], 1)] = node;
  }
}

void launch_masks(const Topo& t, const Phys& p, uint32_t* miss, uint32_t* smask, uint32_t* fmask, int32_t* side,
                  int32_t* pst, int32_t* pall, int32_t* cnt, int max_level, cudaStream_t st) {
  for (int l = max_level; l >= 0; --l) {
    k_masks<<<sm_count(), 128, 0, st>>>(t, p, miss, smask, fmask, side, pst, pall, cnt, l);
    ++g_kernel_launches;
  }
}

__global__ void k_jump_list(Topo t, int32_t* __restrict__ jump, int32_t* __restrict__ cnt) {
  const int nleaves = t.cnt[CNT_NLEAVES];
  for (int li = blockIdx.x * blockDim.x + threadIdx.x; li < nleaves; li += gridDim.x * blockDim.x) {
    const int node = t.leaves[li];
    int mask = 0;
#pragma unroll
    for (int s = 0; s < 6; ++s) {
      const int d = s / 2, hi = s & 1;
      const int r = 13 + (hi ? 1 : -1) * (d == 0 ? 1 : (d == 1 ? 3 : 9));
      const int nb = t.nbr[(size_t)node * 27 + r];
      if (nb >= 0 && t.child0[nb] >= 0) mask |= 1 << s;
    }
    if (mask) jump[atomicAdd(&cnt[CNT_JUMP], 1)] = 64 * li + mask;
  }
}

void launch_jump_list(const Topo& t, int32_t* jump, int32_t* cnt, int n_leaves_cap, cudaStream_t st) {
  k_jump_list<<<(n_leaves_cap + 255) / 256 + 1, 256, 0, st>>>(t, jump, cnt);
  ++g_kernel_launches;
}

void launch_nbr(const Topo& t, const Phys& p, int32_t* nbr_out, int nnodes_cap, cudaStream_t st) {
  const int n = nnodes_cap * 27;
  k_nbr<<<(n + 255) / 256, 256, 0, st>>>(t, p, nbr_out);
  ++g_kernel_launches;
}

// ---------------------------------------------------------------- conservation sums
__global__ void __launch_bounds__(256) k_sums_partial(Topo t, Phys p, Pool pool, int cur, double* __restrict__ partial) {
  __shared__ double sh[5][8];
  const int nleaves = t.cnt[CNT_NLEAVES];
  for (int li = blockIdx.x; li < nleaves; li += gridDim.x) {
    const int node = t.leaves[li];
    const double* U = pool.bufp(cur) + (size_t)t.slot[node] * SLOT_U;
    double s[5] = {0, 0, 0, 0, 0};
    for (int e0 = threadIdx.x; e0 < NINT; e0 += 4 * blockDim.x) {      // twenty loads in flight, added in order
      double x[4][5];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int e = e0 + q * 256, c = sidx(e % 16, (e / 16) % 16, e / 256);
#pragma unroll
        for (int v = 0; v < 5; ++v) x[q][v] = U[v * NCELL + c];
      }
#pragma unroll
      for (int q = 0; q < 4; ++q)
#pragma unroll
        for (int v = 0; v < 5; ++v) s[v] += x[q][v];
    }
#pragma unroll
    for (int v = 0; v < 5; ++v)
      for (int o = 16; o > 0; o >>= 1) s[v] += __shfl_xor_sync(0xffffffffu, s[v], o);
    if ((threadIdx.x & 31) == 0)
      for (int v = 0; v < 5; ++v) sh[v][threadIdx.x >> 5] = s[v];
    __syncthreads();
    if (threadIdx.x < 5) {
      double x = 0.0;
      for (int q = 0; q < 8; ++q) x += sh[threadIdx.x][q];
      const double dx = ldexp(p.dx0, -t.level[node]);
      partial[(size_t)li * 5 + threadIdx.x] = x * (dx * dx * dx);
    }
    __syncthreads();
  }
}

// One CTA per instance, whose leaves are consecutive; a warp per variable.  (One
// thread per variable adding in leaf order was a chain of FP64 additions 49 ns apart:
// 149 us for 3,056 leaves, so 14.)
__global__ void __launch_bounds__(32 * NV) k_sums_finish(Topo t, Phys p, const double* __restrict__ partial,
                                                         double* __restrict__ out) {
  const int inst = blockIdx.x, nleaves = t.cnt[CNT_NLEAVES], v = threadIdx.x >> 5;
  int below = 0, mine = nleaves;
  if (p.n_inst > 1) {
    __shared__ int cnt[2];
    if (threadIdx.x < 2) cnt[threadIdx.x] = 0;
    __syncthreads();
    int c0 = 0, c1 = 0;
    for (int li = threadIdx.x; li < nleaves; li += blockDim.x) {
      const int i = t.inst[t.leaves[li]];
      c0 += i < inst;
      c1 += i == inst;
    }
    atomicAdd(&cnt[0], c0);
    atomicAdd(&cnt[1], c1);
    __syncthreads();
    below = cnt[0];
    mine = cnt[1];
  }
  const double total = block_total(partial + (size_t)below * NV, mine, v);
  if ((threadIdx.x & 31) == 0) out[inst * NV + v] = total;
}

void launch_sums(const Topo& t, const Phys& p, const Pool& pool, int cur, double* partial, double* out,
                 int nleaves_cap, cudaStream_t st) {
  (void)nleaves_cap;
  k_sums_partial<<<sm_count() * 16, 256, 0, st>>>(t, p, pool, cur, partial);
  ++g_kernel_launches;
  k_sums_finish<<<p.n_inst, 32 * NV, 0, st>>>(t, p, partial, out);
  ++g_kernel_launches;
}

}  // namespace mrb
