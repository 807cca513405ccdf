// Mixed-precision stage kernel (MRB_FP32_ACC64): reconstruction, fluxes and
// flux differences in FP32 from the FP64 state; the TVD-RK3 update of the FP64
// state in FP64.  Built with FMA contraction and the fast FP32 reciprocal and
// square-root approximations.
#include "mr.cuh"
#include "stage_f32.cuh"

namespace mrb {

void launch_rhs_rk_f32(const Topo& t, const Phys& p, const Pool& pool, int cur, int stage, const double* dt,
                       double* rhs_out, cudaStream_t st, int n_nodes, int level) {
  if (thin_slabs(n_nodes) && !(p.recon == 1 && p.mlp)) launch_rhs_rk_f32_thin(t, p, pool, cur, stage, dt, rhs_out, st, level);
  else if (p.mu > 0.0) launch_stage_f32<32>(t, p, pool, cur, stage, dt, rhs_out, st, level);   // WENO5, Roe, viscous
  else if (p.flux == 1) launch_rhs_rk_f32_llf(t, p, pool, cur, stage, dt, rhs_out, st, level);
  else if (p.flux == 2) launch_rhs_rk_f32_hllc(t, p, pool, cur, stage, dt, rhs_out, st, level);
  else if (p.recon == 2) launch_stage_f32<2>(t, p, pool, cur, stage, dt, rhs_out, st, level);
  else if (p.recon == 3) launch_stage_f32<4>(t, p, pool, cur, stage, dt, rhs_out, st, level);
  else if (p.recon == 4) launch_stage_f32<5>(t, p, pool, cur, stage, dt, rhs_out, st, level);
  else if (p.recon == 1 && p.mlp) {
    // the selector is evaluated on the stage-0 state; stages 1 and 2 use its decisions
    if (stage == 0 || rhs_out) launch_stage_f32<1>(t, p, pool, cur, stage, dt, rhs_out, st, level);
    else launch_stage_f32<3>(t, p, pool, cur, stage, dt, rhs_out, st, level);
  } else launch_stage_f32<0>(t, p, pool, cur, stage, dt, rhs_out, st, level);
}

void launch_predict_f32(const Topo& t, const Phys& p, const Pool& pool, int cur, int level, int n_nodes, int mode,
                        cudaStream_t st) {
  const bool stage = mode == FILL_STAGE;
  k_predict_t<float><<<predict_grid(n_nodes), 256, 0, st>>>(t, p, pool, cur, stage ? t.pst : t.pall, t.cnt, level,
                                                            stage ? t.smask : t.miss, mode);
  ++g_kernel_launches;
}

void launch_predict_lts_f32(const Topo& t, const Phys& p, const Pool& pool, int cur, int dst, int level, int n_nodes,
                            double th, cudaStream_t st) {
  k_predict_t<float, true><<<predict_grid(n_nodes), 256, 0, st>>>(t, p, pool, cur, t.pst, t.cnt, level, t.smask,
                                                                  FILL_STAGE, dst, th);
  ++g_kernel_launches;
}

void launch_fill_list_f32(const Topo& t, const Phys& p, const Pool& pool, int cur, const int32_t* list, int n,
                          cudaStream_t st) {
  const NodeSet ns{list, n};
  k_fill_regions<<<sm_count() * 8, 256, 0, st>>>(t, pool, cur, ns);
  k_predict_t<float><<<sm_count() * 4, 256, 0, st>>>(t, p, pool, cur, list, nullptr, n, t.miss, FILL_FULL);
  k_fill_bc<<<sm_count() * 4, 256, 0, st>>>(t, p, pool, cur, ns);
  g_kernel_launches += 3;
}

// Averaging with the FP32 records of the averaged cells.
struct PutRecord {
  float* R;
  float g, B, gm1;
  __device__ __forceinline__ void operator()(int slot, int ii, const double* U) const {
    float rec[6];
    make_record(U[0], U[1], U[2], U[3], U[4], g, B, gm1, rec);
    float* __restrict__ o = R + (size_t)slot * SLOT_SH + ii;
#pragma unroll
    for (int f = 0; f < 6; ++f) o[f * NINT] = rec[f];
  }
};
__global__ void __launch_bounds__(256) k_project_f32(Topo t, Phys p, Pool pool, int buf, int level) {
  project_level(t, pool, buf, level,
                PutRecord{pool.shp(buf), (float)p.gamma, (float)p.B, (float)(p.gamma - 1.0)});
}

// Conserved states in, with their records (k_set_cons of the FP64 unit, then a
// pass that read everything back, before): one CTA per quarter of a block, a
// thread moves two cells' five pairs and six record pairs.
template <bool VEC>
__global__ void __launch_bounds__(256) k_set_cons_f32(Topo t, Phys p, Pool pool, int cur, const int32_t* __restrict__ nodes,
                                                      int n, const double* __restrict__ cons) {
  const float g = (float)p.gamma, B = (float)p.B, gm1 = (float)(p.gamma - 1.0);
  for (int w = blockIdx.x; w < n * 4; w += gridDim.x) {
    const int slot = t.slot[nodes[w >> 2]];
    const double* __restrict__ src = cons + (size_t)(w >> 2) * SLOT_N;
    double* __restrict__ U = pool.bufp(cur) + (size_t)slot * SLOT_U;
    float* __restrict__ R = pool.shp(cur) + (size_t)slot * SLOT_SH;
    double2 x[2][NV];
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const int e = (w & 3) * 512 + q * 256 + threadIdx.x;
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        const double* c = src + v * NINT + 2 * e;
        x[q][v] = VEC ? *reinterpret_cast<const double2*>(c) : make_double2(c[0], c[1]);
      }
    }
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const int e = (w & 3) * 512 + q * 256 + threadIdx.x, s = sidx(2 * (e & 7), (e >> 3) & 15, e >> 7);
#pragma unroll
      for (int v = 0; v < NV; ++v) *reinterpret_cast<double2*>(U + v * NCELL + s) = x[q][v];
      float a[6], b[6];
      make_record(x[q][0].x, x[q][1].x, x[q][2].x, x[q][3].x, x[q][4].x, g, B, gm1, a);
      make_record(x[q][0].y, x[q][1].y, x[q][2].y, x[q][3].y, x[q][4].y, g, B, gm1, b);
#pragma unroll
      for (int f = 0; f < 6; ++f) *reinterpret_cast<float2*>(R + f * NINT + 2 * e) = make_float2(a[f], b[f]);
    }
  }
}

void launch_set_cons_f32(const Topo& t, const Phys& p, const Pool& pool, int cur, const int32_t* nodes, int n,
                         const double* cons, cudaStream_t st) {
  const int grid = item_grid((int64_t)n * 4);
  if (((uintptr_t)cons & 15) == 0) k_set_cons_f32<true><<<grid, 256, 0, st>>>(t, p, pool, cur, nodes, n, cons);
  else k_set_cons_f32<false><<<grid, 256, 0, st>>>(t, p, pool, cur, nodes, n, cons);
  ++g_kernel_launches;
}

void launch_project_level_f32(const Topo& t, const Phys& p, const Pool& pool, int buf, int level, cudaStream_t st) {
  k_project_f32<<<sm_count() * g_tune.project, 256, 0, st>>>(t, p, pool, buf, level);
  ++g_kernel_launches;
}

// FP32 records of stage buffer b: one CTA per item, the records of the item's
// internal cells recomputed from the FP64 values (make_record, the same
// arithmetic as the stage kernel's own conversion).
__global__ void __launch_bounds__(256) k_shadow(Topo t, Phys p, Pool pool, int b, int mode,
                                                const int32_t* __restrict__ list, int n, int stride) {
  const float g = (float)p.gamma, B = (float)p.B, gm1 = (float)(p.gamma - 1.0);
  const int nitems = mode == SH_JUMP ? t.cnt[CNT_JUMP] : n;
  for (int w = blockIdx.x; w < nitems; w += gridDim.x) {
    int node, mask = 0;
    if (mode == SH_JUMP) {
      node = t.leaves[t.jump[w] >> 6];
      mask = t.jump[w] & 63;
    } else {
      node = list[(size_t)w * stride];
    }
    const double* U = pool.bufp(b) + (size_t)t.slot[node] * SLOT_U;
    float* R = pool.shp(b) + (size_t)t.slot[node] * SLOT_SH;
    if (mode == SH_JUMP) {
      // the plane of cells next to each side whose neighbour is refined
      for (int sd = 0; sd < 6; ++sd) {
        if (!((mask >> sd) & 1)) continue;
        const int d = sd / 2, hi = sd & 1;
        const int t1 = (d == 0) ? 1 : 0, t2 = (d == 2) ? 1 : 2;
        for (int e = threadIdx.x; e < NFACE; e += blockDim.x) {
          int c[3];
          c[d] = hi ? NB - 1 : 0;
          c[t1] = e % 16;
          c[t2] = e / 16;
          const int s = sidx(c[0], c[1], c[2]), ii = iidx(c[0], c[1], c[2]);
          float rec[6];
          make_record(U[s], U[NCELL + s], U[2 * NCELL + s], U[3 * NCELL + s], U[4 * NCELL + s], g, B, gm1, rec);
#pragma unroll
          for (int f = 0; f < 6; ++f) R[f * NINT + ii] = rec[f];
        }
      }
    } else {
      for (int e = threadIdx.x; e < NINT; e += blockDim.x) {
        const int s = sidx(e % 16, (e / 16) % 16, e / 256);
        float rec[6];
        make_record(U[s], U[NCELL + s], U[2 * NCELL + s], U[3 * NCELL + s], U[4 * NCELL + s], g, B, gm1, rec);
#pragma unroll
        for (int f = 0; f < 6; ++f) R[f * NINT + e] = rec[f];
      }
    }
  }
}

void launch_shadow(const Topo& t, const Phys& p, const Pool& pool, int b, int mode, const int32_t* list, int n,
                   int stride, cudaStream_t st) {
  if (!pool.shp(0)) return;
  k_shadow<<<sm_count() * 4, 256, 0, st>>>(t, p, pool, b, mode, list, n, stride);
  ++g_kernel_launches;
}

// Records of the listed nodes' internal cells (kept, or converted afresh).
__global__ void __launch_bounds__(256) k_get_records(Topo t, Phys p, Pool pool, int cur,
                                                     const int32_t* __restrict__ nodes, int n, float* __restrict__ out,
                                                     int fresh) {
  const float g = (float)p.gamma, B = (float)p.B, gm1 = (float)(p.gamma - 1.0);
  for (int b = blockIdx.x; b < n; b += gridDim.x) {
    const int slot = t.slot[nodes[b]];
    const double* U = pool.bufp(cur) + (size_t)slot * SLOT_U;
    const float* R = pool.shp(cur) + (size_t)slot * SLOT_SH;
    float* o = out + (size_t)b * SLOT_SH;
    for (int e = threadIdx.x; e < NINT; e += blockDim.x) {
      if (fresh) {
        const int s = sidx(e % 16, (e / 16) % 16, e / 256);
        float rec[6];
        make_record(U[s], U[NCELL + s], U[2 * NCELL + s], U[3 * NCELL + s], U[4 * NCELL + s], g, B, gm1, rec);
#pragma unroll
        for (int f = 0; f < 6; ++f) o[f * NINT + e] = rec[f];
      } else {
#pragma unroll
        for (int f = 0; f < 6; ++f) o[f * NINT + e] = R[f * NINT + e];
      }
    }
  }
}

void launch_get_records(const Topo& t, const Phys& p, const Pool& pool, int cur, const int32_t* nodes, int n,
                        float* out, int fresh, cudaStream_t st) {
  if (n <= 0) return;
  k_get_records<<<sm_count() * 4, 256, 0, st>>>(t, p, pool, cur, nodes, n, out, fresh);
  ++g_kernel_launches;
}

// Details of the mixed-precision path with rho and E in packed FP32 pairs:
// the parent box staged once as (rho, E) pairs, the Q-terms of Eq.
// Prediction and the eight predictions of each parent cell computed two
// variables per instruction.  delta = max over both variables of
// |u - P(u_parent)| / |u|, as k_delta_f64.
// A half-warp takes a 4 x 4 tile of parent cells of one plane: with rows 20 pairs
// apart its 16 eight-byte reads fall into 32 different banks (twelve in a row and
// four of the next one, rows 16 apart, collided: twice the wavefronts of 125 reads per
// cell; shock-bubble levels 0..4: 862 -> 678 us).
constexpr int DP_X = 20, DP_XY = 16 * DP_X;
struct SAcc2 {
  const float2* s;
  int i0, j0, k0;
  __device__ __forceinline__ float2 operator()(int i, int j, int k) const {
    return s[(k - k0) * DP_XY + (j - j0) * DP_X + (i - i0)];
  }
};

__device__ __forceinline__ float2 mix2p(const SAcc2& P, int i, int j, int k, int Ax, int Bx, int p, int q) {
  const int a1 = Ax == 0 ? p : 0, b1 = Ax == 1 ? p : 0, c1 = Ax == 2 ? p : 0;
  const int a2 = Bx == 0 ? q : 0, b2 = Bx == 1 ? q : 0, c2 = Bx == 2 ? q : 0;
  return f2sub(f2add(P(i + a1 + a2, j + b1 + b2, k + c1 + c2), P(i - a1 - a2, j - b1 - b2, k - c1 - c2)),
               f2add(P(i - a1 + a2, j - b1 + b2, k - c1 + c2), P(i + a1 - a2, j + b1 - b2, k + c1 - c2)));
}

__device__ __forceinline__ float2 mix3p(const SAcc2& P, int i, int j, int k, int p, int q, int r) {
  const int sg[4][3] = {{1, 1, 1}, {1, -1, -1}, {-1, -1, 1}, {-1, 1, -1}};
  float2 acc = make_float2(0.f, 0.f);
#pragma unroll
  for (int t = 0; t < 4; ++t) {
    const float2 term = f2sub(P(i + sg[t][0] * p, j + sg[t][1] * q, k + sg[t][2] * r),
                              P(i - sg[t][0] * p, j - sg[t][1] * q, k - sg[t][2] * r));
    acc = (t == 0) ? term : f2add(acc, term);
  }
  return acc;
}

__global__ void __launch_bounds__(256) k_delta_p(Topo t, Phys p, Pool pool, int cur, double* __restrict__ delta_node,
                                                 int all_nodes) {
  __shared__ double sh[8];
  __shared__ float2 box[16 * DP_XY];   // (rho, E) of the parent's cells 8 cb - 4 .. 8 cb + 11 per axis
  __shared__ ParentBox pb;
  __shared__ const double* own[27]; // the node's stored cells by region
  const int nitems = all_nodes ? t.cnt[CNT_NNODES] : t.cnt[CNT_NLEAVES];
  const double* B = pool.bufp(cur);
  const float C0 = -22.f / 128.f, C1 = 3.f / 128.f;
  for (int li = blockIdx.x; li < nitems; li += gridDim.x) {
    const int node = all_nodes ? li : t.leaves[li];
    const int lvl = t.level[node];
    if (lvl == 0) {
      if (threadIdx.x == 0) delta_node[node] = 0.0;
      continue;
    }
    const int par = t.parent[node];
    const int ch = (int)(t.keys[node] & 7ull);
    parent_box(t, p, B, par, ch, pb);
    if (threadIdx.x < 27) own[threadIdx.x] = region_base(t, B, node, threadIdx.x);
    __syncthreads();
    bool gl[3], gh[3];
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      const int nl = p.nb[d] << lvl;
      const int Xd = t.X[(size_t)node * 3 + d];
      gl[d] = (Xd == 0) && (p.bc[2 * d] != 1);
      gh[d] = (Xd == nl - 1) && (p.bc[2 * d + 1] != 1);
    }
    const unsigned w0 = box_word(pb, 0, 0, 0);
    const float2 first = make_float2(d2f_fast(box_value(pb, w0, 0)), d2f_fast(box_value(pb, w0, 4)));
    bool eq = const_safe(first.x) && const_safe(first.y);
    for (int e = threadIdx.x; e < 4096; e += blockDim.x) {
      const unsigned w = box_word(pb, e & 15, (e >> 4) & 15, e >> 8);
      const double* __restrict__ c = pb.p[(w >> 16) & 7u] + (w & 0xffffu);
      const float2 x = make_float2(d2f_fast(c[0]), d2f_fast(c[4 * NCELL]));
      box[(e >> 4) * DP_X + (e & 15)] = x;
      eq = eq && same_bits(x.x, first.x) && same_bits(x.y, first.y);
    }
    const bool constant = __syncthreads_and(eq);      // (a box of one value predicts it)
    const SAcc2 A{box, 0, 0, 0};
    float m = 0.f;
    for (int q = threadIdx.x; q < 1728; q += blockDim.x) {
      const int tile = q >> 4;                            // 3 x 3 tiles in a plane
      const int rx = 4 * (tile % 3) + (q & 3) - 2, ry = 4 * ((tile / 3) % 3) + ((q >> 2) & 3) - 2, rz = q / 144 - 2;
      const bool ghost = (rx < 0 && gl[0]) || (rx >= 8 && gh[0]) || (ry < 0 && gl[1]) || (ry >= 8 && gh[1]) ||
                         (rz < 0 && gl[2]) || (rz >= 8 && gh[2]);
      if (ghost) continue;
      const int i = rx + 4, j = ry + 4, k = rz + 4;
      // the eight fine cells, loaded ahead of the Q-terms in aligned pairs
      const double* __restrict__ U = own[own_region(rx, ry, rz)] + sidx(2 * rx, 2 * ry, 2 * rz);
      double2 fr[4], fe[4];
#pragma unroll
      for (int q2 = 0; q2 < 4; ++q2) {       // rows y + (q2 & 1), z + (q2 >> 1)
        const int o = ((q2 >> 1) * NS + (q2 & 1)) * NS;
        fr[q2] = *reinterpret_cast<const double2*>(U + o);
        fe[q2] = *reinterpret_cast<const double2*>(U + 4 * NCELL + o);
      }
      if (constant) {
        // every prediction is the box's value
#pragma unroll
        for (int q2 = 0; q2 < 4; ++q2) {
#pragma unroll
          for (int a = 0; a < 2; ++a) {
            const float2 uf = make_float2(d2f_fast(a ? fr[q2].y : fr[q2].x), d2f_fast(a ? fe[q2].y : fe[q2].x));
            const float2 dd = f2sub(uf, first);
            m = fmaxf(m, fmaxf(fabsf(dd.x / uf.x), fabsf(dd.y / uf.y)));
          }
        }
        continue;
      }
      const float2 u = A(i, j, k);
      const float2 Qx = f2fma(f2s(C0), f2sub(A(i + 1, j, k), A(i - 1, j, k)), f2mul(f2s(C1), f2sub(A(i + 2, j, k), A(i - 2, j, k))));
      const float2 Qy = f2fma(f2s(C0), f2sub(A(i, j + 1, k), A(i, j - 1, k)), f2mul(f2s(C1), f2sub(A(i, j + 2, k), A(i, j - 2, k))));
      const float2 Qz = f2fma(f2s(C0), f2sub(A(i, j, k + 1), A(i, j, k - 1)), f2mul(f2s(C1), f2sub(A(i, j, k + 2), A(i, j, k - 2))));
      const int pq[4][2] = {{1, 1}, {2, 2}, {1, 2}, {2, 1}};
      float2 Qxy = make_float2(0.f, 0.f), Qxz = Qxy, Qyz = Qxy;
#pragma unroll
      for (int t2 = 0; t2 < 4; ++t2) {
        const int pp = pq[t2][0], qq = pq[t2][1];
        const float cc = (pp == 1 ? C0 : C1) * (qq == 1 ? C0 : C1);
        const float2 a = f2mul(f2s(cc), mix2p(A, i, j, k, 0, 1, pp, qq));
        const float2 b = f2mul(f2s(cc), mix2p(A, i, j, k, 0, 2, pp, qq));
        const float2 c = f2mul(f2s(cc), mix2p(A, i, j, k, 1, 2, pp, qq));
        Qxy = (t2 == 0) ? a : f2add(Qxy, a);
        Qxz = (t2 == 0) ? b : f2add(Qxz, b);
        Qyz = (t2 == 0) ? c : f2add(Qyz, c);
      }
      const int pqr[8][3] = {{1, 1, 1}, {2, 2, 2}, {1, 1, 2}, {2, 2, 1}, {1, 2, 2}, {2, 1, 1}, {1, 2, 1}, {2, 1, 2}};
      float2 Qxyz = make_float2(0.f, 0.f);
#pragma unroll
      for (int t3 = 0; t3 < 8; ++t3) {
        const int pp = pqr[t3][0], qq = pqr[t3][1], rr = pqr[t3][2];
        const float cc = (pp == 1 ? C0 : C1) * (qq == 1 ? C0 : C1) * (rr == 1 ? C0 : C1);
        const float2 a = f2mul(f2s(cc), mix3p(A, i, j, k, pp, qq, rr));
        Qxyz = (t3 == 0) ? a : f2add(Qxyz, a);
      }
#pragma unroll
      for (int sub = 0; sub < 8; ++sub) {
        const int a = sub & 1, b = (sub >> 1) & 1, c = (sub >> 2) & 1;
        // the lower child takes +Q: signs of the seven terms of the prediction
        float2 pr = a ? f2sub(u, Qx) : f2add(u, Qx);
        pr = b ? f2sub(pr, Qy) : f2add(pr, Qy);
        pr = c ? f2sub(pr, Qz) : f2add(pr, Qz);
        pr = (a ^ b) ? f2sub(pr, Qxy) : f2add(pr, Qxy);
        pr = (a ^ c) ? f2sub(pr, Qxz) : f2add(pr, Qxz);
        pr = (b ^ c) ? f2sub(pr, Qyz) : f2add(pr, Qyz);
        pr = (a ^ b ^ c) ? f2sub(pr, Qxyz) : f2add(pr, Qxyz);
        const int q2 = b + 2 * c;
        const float2 uf = make_float2(d2f_fast(a ? fr[q2].y : fr[q2].x), d2f_fast(a ? fe[q2].y : fe[q2].x));
        const float2 dd = f2sub(uf, pr);
        const float r0 = fabsf(dd.x / uf.x), r1 = fabsf(dd.y / uf.y);
        m = fmaxf(m, fmaxf(r0, r1));
      }
    }
    double md = f2d_fast(m);
    for (int o = 16; o > 0; o >>= 1) md = fmax(md, __shfl_xor_sync(0xffffffffu, md, o));
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = md;
    __syncthreads();
    if (threadIdx.x == 0) {
      double x = sh[0];
      for (int q = 1; q < (int)(blockDim.x >> 5); ++q) x = fmax(x, sh[q]);
      delta_node[node] = x;
    }
    __syncthreads();
  }
}

void launch_delta_f32(const Topo& t, const Phys& p, const Pool& pool, int cur, double* delta_node, int all_nodes,
                      int n_nodes, cudaStream_t st) {
  k_delta_p<<<item_grid(n_nodes), 256, 0, st>>>(t, p, pool, cur, delta_node, all_nodes);
  ++g_kernel_launches;
}

// Per-instance maxima of |u_d| + c (and of 1/rho, for the viscous limit) over
// the leaves' internal cells: speeds in FP32 from the records (the FP32
// primitives of the FP64 state, half its bytes and no conversion; shock-bubble
// levels 0..4: 242 -> 115 us), maxima (exact) and the time step of Eq. (Cfl) in
// FP64.
__global__ void __launch_bounds__(256) k_cfl_f32(Topo t, Phys p, Pool pool, int cur,
                                                 unsigned long long* __restrict__ smax, int* __restrict__ status,
                                                 double* __restrict__ dt, double** hist) {
  __shared__ float sh[4][8];
  const int nleaves = t.cnt[CNT_NLEAVES];
  const float g = (float)p.gamma, B = (float)p.B;
  for (int li = blockIdx.x; li < nleaves; li += gridDim.x) {
    const int node = t.leaves[li];
    const float* __restrict__ R = pool.shp(cur) + (size_t)t.slot[node] * SLOT_SH;
    float m0 = 0.f, m1 = 0.f, m2 = 0.f, m3 = 0.f;   // max |u_d| + c, max 1/rho
    bool bad = false;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      float4 f[2][5];                                // rho, vx, vy, vz, p of 2 x 4 cells, loaded together
#pragma unroll
      for (int q = 0; q < 2; ++q)
#pragma unroll
        for (int k = 0; k < 5; ++k)
          f[q][k] = *reinterpret_cast<const float4*>(R + k * NINT + 4 * (threadIdx.x + 256 * (2 * h + q)));
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        const float r4[4] = {f[q][0].x, f[q][0].y, f[q][0].z, f[q][0].w}, x4[4] = {f[q][1].x, f[q][1].y, f[q][1].z, f[q][1].w};
        const float y4[4] = {f[q][2].x, f[q][2].y, f[q][2].z, f[q][2].w}, z4[4] = {f[q][3].x, f[q][3].y, f[q][3].z, f[q][3].w};
        const float p4[4] = {f[q][4].x, f[q][4].y, f[q][4].z, f[q][4].w};
#pragma unroll
        for (int c4 = 0; c4 < 4; ++c4) {
          const float r = r4[c4], ir = frcp(r), pr = p4[c4];
          if (!(r > 0.f) || !(pr + B > 0.f)) bad = true;
          const float c = sqrtf(g * (pr + B) * ir);
          m0 = fmaxf(m0, fabsf(x4[c4]) + c);
          m1 = fmaxf(m1, fabsf(y4[c4]) + c);
          m2 = fmaxf(m2, fabsf(z4[c4]) + c);
          m3 = fmaxf(m3, ir);
        }
      }
    }
    if (bad) atomicExch(status, (int)ST_NONPHYS);
    for (int o = 16; o > 0; o >>= 1) {
      m0 = fmaxf(m0, __shfl_xor_sync(0xffffffffu, m0, o));
      m1 = fmaxf(m1, __shfl_xor_sync(0xffffffffu, m1, o));
      m2 = fmaxf(m2, __shfl_xor_sync(0xffffffffu, m2, o));
      m3 = fmaxf(m3, __shfl_xor_sync(0xffffffffu, m3, o));
    }
    if ((threadIdx.x & 31) == 0) {
      sh[0][threadIdx.x >> 5] = m0;
      sh[1][threadIdx.x >> 5] = m1;
      sh[2][threadIdx.x >> 5] = m2;
      sh[3][threadIdx.x >> 5] = m3;
    }
    __syncthreads();
    if (threadIdx.x < 4) {
      float x = sh[threadIdx.x][0];
      for (int q = 1; q < 8; ++q) x = fmaxf(x, sh[threadIdx.x][q]);
      atomicMax(&smax[t.inst[node] * 4 + threadIdx.x], (unsigned long long)__double_as_longlong(f2d_fast(x)));
    }
    __syncthreads();
  }
  cfl_finish(p, smax, dt, hist);
}

void launch_cfl_f32(const Topo& t, const Phys& p, const Pool& pool, int cur, int n_leaves, unsigned long long* smax,
                    double* dt, double** hist, int* status, cudaStream_t st) {
  k_cfl_f32<<<std::min(n_leaves, 4 * sm_count()), 256, 0, st>>>(t, p, pool, cur, smax, status, dt, hist);
  ++g_kernel_launches;
}

}  // namespace mrb
