// Kernels of the block-based MR Euler hot path (arXiv:2012.04385) and their
// launch interface.  Work lists, node arrays and counts live in device memory,
// so every kernel runs a grid-stride loop over a count it reads on the device;
// the same launch stays valid when remeshing changes the tree (which is what
// lets the stage sequence be replayed from a CUDA graph).
#pragma once

#include <algorithm>
#include "physics.cuh"

namespace mrb {

constexpr int MAXL = 11;              // deepest level
constexpr int CNT_NNODES = 0, CNT_NLEAVES = 1, CNT_LVL = 2;   // lvl offsets at CNT_LVL + l, l = 0..MAXL+1
constexpr int CNT_BC = CNT_LVL + MAXL + 2;                     // bc item offsets at CNT_BC + l, l = 0..MAXL+1
constexpr int CNT_JUMP = CNT_BC + MAXL + 2;                    // number of jump items
constexpr int CNT_PST = CNT_JUMP + 1;                          // nodes with stage predictions per level, l = 0..MAXL
constexpr int CNT_PALL = CNT_PST + MAXL + 1;                   // nodes with any predicted region per level
constexpr int CNT_SIZE = CNT_PALL + MAXL + 1;

enum : int { ST_OK = 0, ST_NONPHYS = 6 };

// Halo fill modes.  A halo cell facing a same-level node is that node's internal
// cell, and one beyond a non-periodic boundary is a mapped cell, so the kernels
// of a step read those where they are (mr.cuh, region_base and bc_map) and only predicted
// regions, which exist nowhere else, are ever computed for them:
//   FILL_FULL       every region of every node in its stored halo (mrb_fill_halos,
//                   and the stages with viscous terms, which read edges);
//   FILL_STAGE      the predicted regions that a stage reads: face regions of the
//                   leaves, and what their predictions read of internal nodes;
//   FILL_DETAIL     every predicted region, of leaves rho and E only (the detail
//                   norm's inputs).
// Measured per step: shock-bubble (levels 0..4, 6,600 nodes) 3.12 -> 0.86 ms of fills
// and 60 -> 16 launches, ensemble of five 2.56 -> 0.49 ms, explosion 1.22 -> 0.18 ms.
enum : int { FILL_FULL = 0, FILL_STAGE = 1, FILL_DETAIL = 2 };

// Node arrays, in ascending id order (instance, level, Morton).
struct Topo {
  const uint64_t* keys;
  const int32_t* slot;     // pool slot of the node
  const int32_t* level;
  const int32_t* inst;
  const int32_t* X;        // [n][3] block coordinates on the node's level
  const int32_t* parent;   // node index or -1
  const int32_t* child0;   // first of 8 consecutive children, or -1 for a leaf
  const int32_t* nbr;      // [n][27] same-level neighbour node, -1 none, -2 beyond the boundary
  const int32_t* leaves;   // leaf node indices, ascending id
  const int32_t* lvl_nodes;// node indices grouped by level
  const int32_t* bc_items; // 8 * node + side of every non-periodic domain-boundary side, grouped by level
  const int32_t* jump;     // 64 * leaf index + mask of the sides whose same-level neighbour is refined
  const uint32_t* miss;    // 27-bit mask of a node's predicted halo regions (nbr == -1)
  const uint32_t* smask;   // those that a stage needs (see k_masks)
  const int32_t* pst;      // nodes with smask != 0, grouped by level like lvl_nodes (count CNT_PST + l)
  const int32_t* pall;     // nodes with miss != 0, likewise (count CNT_PALL + l)
  const int32_t* side;     // [8] per node: slots of the face neighbours (x-, x+, y-, y+, z-, z+; -1 none, -2
                           // beyond the boundary), own slot, fmask | level << 8: what a stage item asks first
  const uint32_t* fmask;   // 6-bit mask of a leaf's sides whose face fluxes something reads: next to a refined
                           // neighbour (the jump correction's coarse side) or to none (its fine side)
  const int32_t* cnt;      // counts, see CNT_*
};

struct Phys {
  double gamma, B, cfl, dx0, eps;
  double mu;               // dynamic viscosity of the Navier-Stokes terms; 0 = Euler
  double inv_dx0;          // 1 / dx0 (1 / dx of level l is its exact 2^l multiple)
  double grav[3];
  int bc[6];
  int nb[3];
  int n_inst;
  int recon;
  int has_grav;
  int precision;           // 0 FP64, 1 FP32 bulk (MRB_FP64 / MRB_FP32_ACC64)
  int rk;                  // Runge-Kutta stages per step: 3 (TVD-RK3) or 2 (TVD-RK2)
  int flux;                // MRB_FLUX_*: Roe with LLF fallback, LLF, HLLC
  float mlp_tau;           // learned selector: linear reconstruction when logit < mlp_tau
  const float* mlp;        // learned selector parameters (device, FP32), or null
  unsigned long long* lin_count;   // [0] faces sent to linear, [1] faces evaluated
  const int32_t* lmax;     // device [n_inst]
  int blocked;             // stage kernels: 1 = a contiguous run of work items per CTA, 0 = strided by the grid
  int lts;                 // local time stepping (Eq. LtsTimestep)
};

// Launch shapes of the scheduling-only tunables (mrb_autotune): every choice
// gives bit-identical results.  Set from the calling context before its
// launches.
struct Tune {
  int stage_waves;         // stage-kernel CTAs = SMs x resident CTAs per SM x stage_waves
  int fill_copy;           // region-copy fill CTAs per SM
  int fill_pred;           // prediction fill CTAs per SM
  int project;             // averaging CTAs per SM
};
extern Tune g_tune;

// This CTA's work items: strided by the grid, or one contiguous run.
struct ItemRange {
  int first, step, end;
};
__device__ __forceinline__ ItemRange item_range(int nitems, int blocked) {
  if (!blocked) return ItemRange{(int)blockIdx.x, (int)gridDim.x, nitems};
  const int per = (nitems + (int)gridDim.x - 1) / (int)gridDim.x;
  const int a = (int)blockIdx.x * per;
  return ItemRange{a, 1, a + per < nitems ? a + per : nitems};
}

// Shu-Osher coefficients of stage s: out = a u^n + b (u + dt L); row 0 TVD-RK3,
// row 1 TVD-RK2.
__device__ __constant__ static const double kRkA[2][3] = {{0.0, 0.75, 1.0 / 3.0}, {0.0, 0.5, 0.0}};
__device__ __constant__ static const double kRkB[2][3] = {{1.0, 0.25, 2.0 / 3.0}, {1.0, 0.5, 0.0}};
__device__ __forceinline__ int rk_row(const Phys& p) { return p.rk == 2 ? 1 : 0; }
// Weights of the stage right-hand sides in the step (u^(n+1) = u^n + dt sum_s
// w_s L(u^(s))): TVD-RK3 1/6, 1/6, 2/3; TVD-RK2 1/2, 1/2.
__device__ __constant__ static const double kRkW[2][3] = {{1.0 / 6.0, 1.0 / 6.0, 2.0 / 3.0}, {0.5, 0.5, 0.0}};

// Work items of a stage launch: every leaf (level < 0) or every node of one
// level (local time stepping); the node of item k and the item count.
__device__ __forceinline__ int stage_nodes(const Topo& t, int level) {
  return level < 0 ? t.cnt[CNT_NLEAVES] : t.cnt[CNT_LVL + level + 1] - t.cnt[CNT_LVL + level];
}
__device__ __forceinline__ int stage_node(const Topo& t, int level, int k) {
  return level < 0 ? t.leaves[k] : t.lvl_nodes[t.cnt[CNT_LVL + level] + k];
}
// The time step of a node: dt of its instance, times 2^(lmax - level) under
// local time stepping.
__device__ __forceinline__ double node_dt(const Topo& t, const Phys& p, const double* dt, int node, int level) {
  const int inst = t.inst[node];
  return level < 0 ? dt[inst] : ldexp(dt[inst], p.lmax[inst] - level);
}

struct Pool {
  double* buf[2];          // stage buffers, [slot][5][24^3]
  double* un;              // u^n, [slot][5][16^3]
  double* face;            // face fluxes, [slot][6][5][16][16]
  uint32_t* sel;           // learned selector decisions of the current step, [slot][SLOT_SEL]
  // FP32 primitive records (rho, vx, vy, vz, p, E) of the internal cells of
  // buf[b], [slot][6][16^3]; kept by the mixed-precision path only (null
  // otherwise), rewritten by every kernel that writes internal cells
  float* sh[2];
  // boundary-face fluxes integrated over a macro time step (local time
  // stepping only), [slot][6][5][16][16]
  double* fmac;
  // FP32 increments u^(s) - u^n of the stage (mixed-precision path only, null
  // otherwise), [slot][5][16^3]
  float* dl;
  // The arrays of stage buffer b, chosen by selection: indexing the arrays
  // above with a run-time b would make the compiler copy the whole kernel
  // parameter into local memory and read the pointers back from there.
  __host__ __device__ __forceinline__ double* bufp(int b) const { return b ? buf[1] : buf[0]; }
  __host__ __device__ __forceinline__ float* shp(int b) const { return b ? sh[1] : sh[0]; }
};

__device__ __forceinline__ double ldexp_(double x, int e) { return ldexp(x, e); }

// ---------------------------------------------------------------- launches
// (defined in kern_f64.cu / kern_f32.cu; all asynchronous on `st`)
void launch_set_state(const Topo& t, const Phys& p, const Pool& pool, int cur, const int32_t* nodes, int n,
                      const double* prim, cudaStream_t st);
// (with the FP32 records of the cells, mixed precision)
void launch_set_cons(const Topo& t, const Phys& p, const Pool& pool, int cur, const int32_t* nodes, int n,
                     const double* cons, cudaStream_t st);
void launch_set_cons_f32(const Topo& t, const Phys& p, const Pool& pool, int cur, const int32_t* nodes, int n,
                         const double* cons, cudaStream_t st);
void launch_get_state(const Topo& t, const Pool& pool, int cur, const int32_t* nodes, int n, double* out,
                      int with_halo, cudaStream_t st);
// stored halos facing same-level nodes, and ghost cells beyond the boundary, of every node
void launch_fill_copies(const Topo& t, const Pool& pool, int cur, int n_nodes, cudaStream_t st);
void launch_fill_bc(const Topo& t, const Phys& p, const Pool& pool, int cur, cudaStream_t st);
// predicted regions of the nodes of `level` (after those of the coarser levels)
void launch_predict(const Topo& t, const Phys& p, const Pool& pool, int cur, int level, int n_nodes, int mode,
                    cudaStream_t st);
// The stage's predictions of `level` into buffer dst, the coarser level taken at
// fraction th of its step (local time stepping).
void launch_predict_lts(const Topo& t, const Phys& p, const Pool& pool, int cur, int dst, int level, int n_nodes,
                        double th, cudaStream_t st);
// every halo region of the listed nodes (device list of n node indices), all variables
void launch_fill_list(const Topo& t, const Phys& p, const Pool& pool, int cur, const int32_t* list, int n,
                      cudaStream_t st);
// level < 0: every leaf with dt; level >= 0 (local time stepping): every node
// of that level, leaves and internal nodes, with dt 2^(lmax - level)
void launch_rhs_rk_f64(const Topo& t, const Phys& p, const Pool& pool, int cur, int stage, const double* dt,
                       double* rhs_out, cudaStream_t st, int level = -1);
void launch_rhs_rk_f32(const Topo& t, const Phys& p, const Pool& pool, int cur, int stage, const double* dt,
                       double* rhs_out, cudaStream_t st, int n_nodes, int level = -1);
// The same on slabs of two planes (n_nodes: the leaves, or the nodes of `level`).
// Taken while all their slabs are resident at two CTAs per SM: the stage then lasts as
// long as one item, 15 us instead of 23 on the Sod tube's 8 blocks.  Beyond that the
// two forms differ by how their last rounds fill.  Microseconds of a single-level step
// of 38 / 39 / 48 / 56 / 76 / 90 / 114 / 152 leaves that vary everywhere: thin 95 / 140
// / 141 / 170 / 174 / 213 / 255 / 336, slabs of four 152 / 152 / 154 / 154 / 155 / 233 /
// 292 / 303; that vary along one direction: thin 65 / 98 / 86 / 110 / 111 / 141 / 159 /
// 211, slabs of four 96 / 96 / 82 / 97 / 98 / 148 / 180 / 192.
void launch_rhs_rk_f32_thin(const Topo& t, const Phys& p, const Pool& pool, int cur, int stage, const double* dt,
                            double* rhs_out, cudaStream_t st, int level = -1);
// FP32 stage kernels of the flux variants (separate translation units):
// LLF on every field, and HLLC, each with every non-learned reconstruction.
void launch_rhs_rk_f32_llf(const Topo& t, const Phys& p, const Pool& pool, int cur, int stage, const double* dt,
                           double* rhs_out, cudaStream_t st, int level = -1);
void launch_rhs_rk_f32_hllc(const Topo& t, const Phys& p, const Pool& pool, int cur, int stage, const double* dt,
                            double* rhs_out, cudaStream_t st, int level = -1);
// ---- local time stepping
// Interpolation in time of the nodes of levels < below (factor theta[m] per
// level m; the end state kept in the other stage buffer), or its undoing.
struct LevelTheta {
  double th[MAXL + 1];
};
void launch_lts_interp(const Topo& t, const Pool& pool, int cur, int below, const LevelTheta& th, int restore,
                       cudaStream_t st);
// Internal cells (and FP32 records) of the nodes of `level`: buffer cur^1 -> cur.
void launch_lts_copyback(const Topo& t, const Pool& pool, int cur, int level, cudaStream_t st);
// Integrated fluxes: zero those of every leaf, or add weight x face fluxes to
// those of the leaves of `level` (weight = kRkW[stage] x dt 2^(lmax - level)).
void launch_lts_fmac(const Topo& t, const Phys& p, const Pool& pool, int level, int stage, const double* dt,
                     int zero, cudaStream_t st);
// End of the macro step: leaf faces next to refined neighbours take the finer
// side's integrated flux.
void launch_lts_reflux(const Topo& t, const Phys& p, const Pool& pool, int cur, cudaStream_t st);
void launch_jump(const Topo& t, const Phys& p, const Pool& pool, int target, int stage, const double* dt,
                 double* rhs_out, cudaStream_t st);
// averaging of the internal nodes of `level`, with their FP32 records (mixed precision)
void launch_project_level(const Topo& t, const Phys& p, const Pool& pool, int buf, int level, cudaStream_t st);
void launch_project_level_f32(const Topo& t, const Phys& p, const Pool& pool, int buf, int level, cudaStream_t st);
// smax: 4 maxima per instance and a count, all zero between launches.  hist (nullable): device pointer to where the
// next row of time steps also goes.
void launch_cfl(const Topo& t, const Phys& p, const Pool& pool, int cur, int n_leaves, unsigned long long* smax,
                double* dt, double** hist, int* status, cudaStream_t st);
void launch_set_hist(double** hist, double* row, cudaStream_t st);
void launch_delta_tags(const Topo& t, const Phys& p, const Pool& pool, int cur, double* delta_node,
                       int allow_refine, int8_t* tags, double* delta_leaf, int n_leaves_cap, int n_nodes,
                       cudaStream_t st);
void launch_refine_fill(const Topo& t, const Phys& p, const Pool& pool, int cur, const int32_t* pairs, int n,
                        cudaStream_t st);
// Leaves with resolution jumps (a same-level face neighbour that is refined):
// jump[] = 64 * leaf index + side mask, counted into cnt[CNT_JUMP] (item
// order unspecified; every item is independent).
void launch_jump_list(const Topo& t, int32_t* jump, int32_t* cnt, int n_leaves_cap, cudaStream_t st);
void launch_nbr(const Topo& t, const Phys& p, int32_t* nbr_out, int nnodes_cap, cudaStream_t st);
// Masks of predicted regions and the lists of the nodes that have any, levels
// fine to coarse (max_level .. 0).
void launch_masks(const Topo& t, const Phys& p, uint32_t* miss, uint32_t* smask, uint32_t* fmask, int32_t* side, int32_t* pst,
                  int32_t* pall, int32_t* cnt, int max_level, cudaStream_t st);
void launch_sums(const Topo& t, const Phys& p, const Pool& pool, int cur, double* partial, double* out,
                 int nleaves_cap, cudaStream_t st);
// mixed-precision variants (kern_f32.cu)
void launch_predict_lts_f32(const Topo& t, const Phys& p, const Pool& pool, int cur, int dst, int level, int n_nodes,
                            double th, cudaStream_t st);
void launch_predict_f32(const Topo& t, const Phys& p, const Pool& pool, int cur, int level, int n_nodes, int mode,
                        cudaStream_t st);
void launch_fill_list_f32(const Topo& t, const Phys& p, const Pool& pool, int cur, const int32_t* list, int n,
                          cudaStream_t st);
// Roe / LLF census of every leaf face (FP64 decisions on the stage buffer):
// counts[k] faces where field k takes the LLF split, counts[5] faces.
void launch_flux_census(const Topo& t, const Phys& p, const Pool& pool, int cur, unsigned long long* counts,
                        cudaStream_t st);
void launch_delta_f32(const Topo& t, const Phys& p, const Pool& pool, int cur, double* delta_node, int all_nodes,
                      int n_nodes, cudaStream_t st);
void launch_cfl_f32(const Topo& t, const Phys& p, const Pool& pool, int cur, int n_leaves, unsigned long long* smax,
                    double* dt, double** hist, int* status, cudaStream_t st);
// FP32 records of stage buffer b from its FP64 internal cells (mixed-precision
// path): SH_JUMP the boundary planes that the jump correction changed, SH_LIST
// the nodes of a device list of n entries (every `stride`-th entry is a node
// index).  The stage kernel and the averaging write the records of their cells.
enum : int { SH_JUMP = 1, SH_LIST = 2 };
void launch_shadow(const Topo& t, const Phys& p, const Pool& pool, int b, int mode, const int32_t* list, int n,
                   int stride, cudaStream_t st);
// Records of the listed nodes (kept, or converted afresh from the FP64 state).
void launch_get_records(const Topo& t, const Phys& p, const Pool& pool, int cur, const int32_t* nodes, int n,
                        float* out, int fresh, cudaStream_t st);
void launch_face_samples(const Topo& t, const Phys& p, const Pool& pool, int cur, float tau_lab, int64_t stride,
                         float* feats, uint8_t* labels, int64_t* where, int64_t cap, cudaStream_t st);
int sm_count();
inline bool thin_slabs(int n_nodes) { return n_nodes * 8 <= 2 * sm_count(); }
// Grids of kernels whose items differ in length (a detail box of one value, a copy
// that meets the cache): a CTA per item up to 32 per SM, handed out as CTAs end.
// With four per SM, of which the registers admit three, the fourth ran alone
// afterwards: details of the shock-bubble (levels 0..4) 679 -> 474 us, get_state 344
// -> 326, set_cons 464 -> 416.
inline int item_grid(int64_t items) { return (int)std::min<int64_t>(items, 32 * (int64_t)sm_count()); }
// The counts that shape a launch are those at its capture where a graph replays it;
// the kernels take every item on any grid.
//
// Predictions: a CTA per node (up to four items of one), between fill_pred and four
// times that per SM.  Shock-bubble, 16 launches: 840 us with 4 per SM, 709 with 16;
// on a few hundred nodes 16 per SM cost a microsecond a launch more than 4.
inline int predict_grid(int n_nodes) {
  const int per = g_tune.fill_pred * sm_count();
  return std::min(std::max(n_nodes, per), 4 * per);
}
// kernel launches issued by this process (host-side counter, bumped by every launch_* wrapper)
extern long long g_kernel_launches;

// Total of the per-block sums src[b][NV], b < n, of variable v: lane l adds blocks l,
// l + 32, ... in turn, then the lanes' sums pairwise -- the fixed order of every
// total (one warp per variable; the result is in every lane).
__device__ __forceinline__ double block_total(const double* __restrict__ src, int64_t n, int v) {
  double acc = 0.0;
  int64_t b = threadIdx.x & 31;
  for (; b + 96 < n; b += 128) {                 // (four loads in flight)
    const double x0 = src[b * NV + v], x1 = src[(b + 32) * NV + v], x2 = src[(b + 64) * NV + v], x3 = src[(b + 96) * NV + v];
    acc = ((((acc + x0) + x1) + x2) + x3);
  }
  for (; b < n; b += 32) acc += src[b * NV + v];
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  return acc;
}

}  // namespace mrb
