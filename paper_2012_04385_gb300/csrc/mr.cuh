// Multiresolution kernels templated on the arithmetic type R: halo fill
// (copy / prediction / boundary condition) and the MR details of the leaves.
// R = double reproduces the FP64 operation order exactly (built with
// -fmad=false); R = float serves the mixed-precision path, where halo values
// are stencil inputs and the details a refinement heuristic.
//
// Prediction (Eq. Prediction with the appendix Q-terms) is evaluated once per
// parent cell: the eight fine cells of a parent cell share its Q-terms and
// differ only in the signs (+ for the lower half along an axis, - for the
// upper).  A halo of four fine cells is two parent cells deep, so the eight
// fine cells of a parent cell always lie in the same halo region.
#pragma once

#include "convert.cuh"
#include "kernels.cuh"

namespace mrb {

template <class R> struct QT {
  R u, Qx, Qy, Qz, Qxy, Qxz, Qyz, Qxyz;
};

template <class R> __device__ __forceinline__ R to_r(double x) { return R(x); }
template <> __device__ __forceinline__ float to_r<float>(double x) { return d2f_fast(x); }
template <class R> __device__ __forceinline__ double from_r(R x) { return double(x); }
template <> __device__ __forceinline__ double from_r<float>(float x) { return f2d_fast(x); }

// Parent values for the Q-terms: a box of R values staged in shared memory
// (origin i0, j0, k0 in stored coordinates, row length nx, plane size nxy).
template <class R> struct SAcc {
  const R* s;
  int i0, j0, k0, nx, nxy;
  __device__ __forceinline__ R operator()(int i, int j, int k) const {
    return s[(k - k0) * nxy + (j - j0) * nx + (i - i0)];
  }
};

template <class R> __device__ __forceinline__ R qc(int off) { return off == 1 ? R(-22.0 / 128.0) : R(3.0 / 128.0); }

template <class R, class A>
__device__ __forceinline__ R mix2t(const A& P, int i, int j, int k, int Ax, int Bx, int p, int q) {
  int o1[3] = {0, 0, 0}, o2[3] = {0, 0, 0}, o3[3] = {0, 0, 0}, o4[3] = {0, 0, 0};
  o1[Ax] = p; o1[Bx] = q;
  o2[Ax] = -p; o2[Bx] = -q;
  o3[Ax] = -p; o3[Bx] = q;
  o4[Ax] = p; o4[Bx] = -q;
  return (P(i + o1[0], j + o1[1], k + o1[2]) + P(i + o2[0], j + o2[1], k + o2[2])) -
         (P(i + o3[0], j + o3[1], k + o3[2]) + P(i + o4[0], j + o4[1], k + o4[2]));
}

template <class R, class A> __device__ __forceinline__ R mix3t(const A& P, int i, int j, int k, int p, int q, int r) {
  const int sg[4][3] = {{1, 1, 1}, {1, -1, -1}, {-1, -1, 1}, {-1, 1, -1}};
  R acc = R(0);
#pragma unroll
  for (int t = 0; t < 4; ++t) {
    R term = P(i + sg[t][0] * p, j + sg[t][1] * q, k + sg[t][2] * r) - P(i - sg[t][0] * p, j - sg[t][1] * q, k - sg[t][2] * r);
    acc = (t == 0) ? term : acc + term;
  }
  return acc;
}

// Q-terms of parent cell (i, j, k) (Eq. Prediction with the appendix
// coefficients c0 = -22/128, c1 = 3/128).
template <class R, class A> __device__ __forceinline__ QT<R> qterms_t(const A& P, int i, int j, int k) {
  const R C0 = R(-22.0 / 128.0), C1 = R(3.0 / 128.0);
  QT<R> t;
  t.u = P(i, j, k);
  t.Qx = C0 * (P(i + 1, j, k) - P(i - 1, j, k)) + C1 * (P(i + 2, j, k) - P(i - 2, j, k));
  t.Qy = C0 * (P(i, j + 1, k) - P(i, j - 1, k)) + C1 * (P(i, j + 2, k) - P(i, j - 2, k));
  t.Qz = C0 * (P(i, j, k + 1) - P(i, j, k - 1)) + C1 * (P(i, j, k + 2) - P(i, j, k - 2));
  const int pq[4][2] = {{1, 1}, {2, 2}, {1, 2}, {2, 1}};
  R qxy = R(0), qxz = R(0), qyz = R(0);
#pragma unroll
  for (int t2 = 0; t2 < 4; ++t2) {
    const int p = pq[t2][0], q = pq[t2][1];
    const R cc = qc<R>(p) * qc<R>(q);
    const R a = cc * mix2t<R>(P, i, j, k, 0, 1, p, q);
    const R b = cc * mix2t<R>(P, i, j, k, 0, 2, p, q);
    const R c = cc * mix2t<R>(P, i, j, k, 1, 2, p, q);
    qxy = (t2 == 0) ? a : qxy + a;
    qxz = (t2 == 0) ? b : qxz + b;
    qyz = (t2 == 0) ? c : qyz + c;
  }
  t.Qxy = qxy;
  t.Qxz = qxz;
  t.Qyz = qyz;
  const int pqr[8][3] = {{1, 1, 1}, {2, 2, 2}, {1, 1, 2}, {2, 2, 1}, {1, 2, 2}, {2, 1, 1}, {1, 2, 1}, {2, 1, 2}};
  R qxyz = R(0);
#pragma unroll
  for (int t3 = 0; t3 < 8; ++t3) {
    const int p = pqr[t3][0], q = pqr[t3][1], r = pqr[t3][2];
    const R cc = qc<R>(p) * qc<R>(q) * qc<R>(r);
    const R a = cc * mix3t<R>(P, i, j, k, p, q, r);
    qxyz = (t3 == 0) ? a : qxyz + a;
  }
  t.Qxyz = qxyz;
  return t;
}

// ---------------------------------------------------------------- stored cells where they are
// Boundary condition of one axis: block coordinate x beyond a non-periodic side
// (condition blo / bhi, -1 for none) mapped back into the block (zero gradient:
// the nearest internal cell; symmetry: the mirror cell, with the normal
// momentum negated: `bit` of flip).
__device__ __forceinline__ int bc_map(int x, int blo, int bhi, int& flip, int bit) {
  if (x < 0 && blo >= 0) {
    flip ^= (blo == 2) ? bit : 0;
    return blo == 0 ? 0 : -1 - x;
  }
  if (x >= NB && bhi >= 0) {
    flip ^= (bhi == 2) ? bit : 0;
    return bhi == 0 ? NB - 1 : 2 * NB - 1 - x;
  }
  return x;
}

// Base of region r (0 .. 26) of a node such that the node's stored index of a
// cell of that region applies: the same-level neighbour's internal cells, or
// the node's own stored halo where there is none (predicted).
__device__ __forceinline__ const double* region_base(const Topo& t, const double* __restrict__ buf, int node, int r) {
  const int nb = t.nbr[(size_t)node * 27 + r];
  if (nb < 0) return buf + (size_t)t.slot[node] * SLOT_U;
  const int sx = r % 3 - 1, sy = (r / 3) % 3 - 1, sz = r / 9 - 1;
  return buf + (size_t)t.slot[nb] * SLOT_U - NB * (sx + NS * (sy + NS * sz));
}

// The 16^3 parent cells that a child in octant ch reads: 8 cb - 4 .. 8 cb + 11 per
// axis, i.e. cells of the parent and of the seven regions on the octant's side
// of it.  Per axis a table of the 16 coordinates: the offset in the stored array
// of the cell that holds the value (bits 0-15; the coordinate itself, or the one
// it maps to beyond a boundary), bit 16 + d when it lies in the region beyond
// axis d, bit 20 + d when the mapping mirrors.  The sum of three entries is the
// cell's offset and its flags, so a staged cell costs two additions and one
// pointer select.
struct ParentBox {
  const double* p[8];      // bases by which axes are beyond the parent (bit d)
  unsigned tab[3][16];
};
// (threads 0 .. 47; the caller synchronises)
__device__ __forceinline__ void parent_box(const Topo& t, const Phys& p, const double* __restrict__ buf, int par, int ch,
                                           ParentBox& b) {
  const int q = threadIdx.x;
  if (q < 8) {
    int r = 13;
#pragma unroll
    for (int d = 0; d < 3; ++d)
      if ((q >> d) & 1) r += (((ch >> d) & 1) ? 1 : -1) * (d == 0 ? 1 : (d == 1 ? 3 : 9));
    b.p[q] = region_base(t, buf, par, r);
  }
  if (q < 48) {
    const int d = q >> 4, hi = (ch >> d) & 1;
    const int nl = (d == 0 ? p.nb[0] : (d == 1 ? p.nb[1] : p.nb[2])) << t.level[par], X = t.X[(size_t)par * 3 + d];
    const int code = d == 0 ? (hi ? p.bc[1] : p.bc[0]) : (d == 1 ? (hi ? p.bc[3] : p.bc[2]) : (hi ? p.bc[5] : p.bc[4]));
    const int bc = (X == (hi ? nl - 1 : 0) && code != 1) ? code : -1;
    int x = 8 * hi - 4 + (q & 15), flip = 0;
    unsigned w = 0;
    if (x < 0 || x >= NB) {
      if (bc >= 0) x = bc_map(x, hi ? -1 : bc, hi ? bc : -1, flip, 1);
      else w = 1u << (16 + d);
    }
    w |= (unsigned)flip << (20 + d);
    b.tab[d][q & 15] = w + (unsigned)((x + HW) * (d == 0 ? 1 : (d == 1 ? NS : NS * NS)));
  }
}
// Flags and offset of box cell (i, j, k) in 0 .. 15; the value of variable v there.
__device__ __forceinline__ unsigned box_word(const ParentBox& b, int i, int j, int k) {
  return b.tab[0][i] + b.tab[1][j] + b.tab[2][k];
}
__device__ __forceinline__ double box_value(const ParentBox& b, unsigned w, int v) {
  const double x = b.p[(w >> 16) & 7u][v * NCELL + (w & 0xffffu)];
  return (v >= 1 && v <= 3 && ((w >> (19 + v)) & 1u)) ? -x : x;
}

// Local time stepping: the box's parent level at time fraction q of its step,
// (1 - q) u^n + q u, blended where it is read (stored halos already hold
// predictions of blended values).  n[]: bases of u^n by region, null where the
// region is a stored halo; tab: offsets in its 16^3 layout.
struct BlendBox {
  const double* n[8];
  int tab[3][16];
};
// (threads 0 .. 47, after parent_box of the same item; the caller synchronises)
__device__ __forceinline__ void blend_box(const Topo& t, const double* __restrict__ un, int par, int ch,
                                          const ParentBox& b, BlendBox& l) {
  const int q = threadIdx.x;
  if (q < 8) {
    int r = 13, shift = 0;
#pragma unroll
    for (int d = 0; d < 3; ++d)
      if ((q >> d) & 1) {
        const int s = ((ch >> d) & 1) ? 1 : -1;
        r += s * (d == 0 ? 1 : (d == 1 ? 3 : 9));
        shift += s * (d == 0 ? NB : (d == 1 ? NB * NB : NB * NB * NB));
      }
    const int nb = q == 0 ? par : t.nbr[(size_t)par * 27 + r];
    l.n[q] = nb < 0 ? nullptr : un + (size_t)t.slot[nb] * SLOT_N - shift;
  }
  if (q < 48) {
    const int d = q >> 4, x = (int)(b.tab[d][q & 15] & 0xffffu) / (d == 0 ? 1 : (d == 1 ? NS : NS * NS)) - HW;
    l.tab[d][q & 15] = x * (d == 0 ? 1 : (d == 1 ? NB : NB * NB));
  }
}
// (rounded alike in every translation unit)
__device__ __forceinline__ double blend(double q, double n, double u) {
  return __dadd_rn(__dmul_rn(1.0 - q, n), __dmul_rn(q, u));
}

// A value c whose box of equal values predicts c: every difference and mixed
// difference is +0, every Q-term +0, and c + (+-0) is c unless c is -0; c + c stays
// finite.
__device__ __forceinline__ bool const_safe(float c) {
  return fabsf(c) < 1e30f && __float_as_uint(c) != 0x80000000u;
}
__device__ __forceinline__ bool const_safe(double c) {
  return fabs(c) < 1e300 && (unsigned long long)__double_as_longlong(c) != 0x8000000000000000ull;
}
__device__ __forceinline__ bool same_bits(float a, float b) { return __float_as_uint(a) == __float_as_uint(b); }
__device__ __forceinline__ bool same_bits(double a, double b) { return __double_as_longlong(a) == __double_as_longlong(b); }

// Stage the cells [i0, i0+nx) x [j0, j0+ny) x [k0, k0+nz) of the box (nx, ny, nz
// 6, 12 or 16) of every variable (or rho and E only) as R, the
// q-th at s + q * nx ny nz; all threads.  A group of 8 or 16 lanes owns a row.
// Returns the variables (bit q) whose cells staged by this thread all equal the
// box's first cell.
template <class R, bool BLEND = false>
__device__ __forceinline__ unsigned stage_box(R* __restrict__ s, const ParentBox& b, bool detail_only, int i0, int j0,
                                          int k0, int nx, int ny, int nz, const BlendBox* l = nullptr, double th = 0.0) {
  const int lg = nx > 8 ? 4 : 3, i = threadIdx.x & ((1 << lg) - 1);
  unsigned eq = 31u;
  if (i >= nx) return eq;
  const int n = nx * ny * nz, inv = ny == 16 ? 4096 : (ny == 12 ? 5462 : 10923);   // row / ny = row inv / 2^16 (rows < 256)
  const unsigned wi = b.tab[0][i0 + i], w0 = box_word(b, i0, j0, k0);
  R first[NV];
#pragma unroll
  for (int q = 0; q < NV; ++q)
    if (!detail_only || q < 2) {
      double y = box_value(b, w0, detail_only ? 4 * q : q);
      if (BLEND) {
        const double* un = l->n[(w0 >> 16) & 7u];
        const bool flip = q >= 1 && q <= 3 && ((w0 >> (19 + q)) & 1u);
        if (un) {
          y = blend(th, un[q * NINT + l->tab[0][i0] + l->tab[1][j0] + l->tab[2][k0]], flip ? -y : y);
          if (flip) y = -y;
        }
      }
      first[q] = to_r<R>(y);
    }
  for (int row = threadIdx.x >> lg; row < ny * nz; row += blockDim.x >> lg) {
    const int k = (row * inv) >> 16, j = row - k * ny;
    const unsigned w = wi + b.tab[1][j0 + j] + b.tab[2][k0 + k];
    const double* __restrict__ c = b.p[(w >> 16) & 7u] + (w & 0xffffu);
    R* o = s + row * nx + i;
    if (detail_only) {
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        const R x = to_r<R>(c[4 * q * NCELL]);
        if (!same_bits(x, first[q])) eq &= ~(1u << q);
        o[q * n] = x;
      }
    } else {
      const double* __restrict__ un = BLEND ? l->n[(w >> 16) & 7u] : nullptr;
      if (BLEND && un) un += l->tab[0][i0 + i] + l->tab[1][j0 + j] + l->tab[2][k0 + k];
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        double y = c[v * NCELL];
        if (BLEND && un) y = blend(th, un[v * NINT], y);
        const R x = to_r<R>((v >= 1 && v <= 3 && ((w >> (19 + v)) & 1u)) ? -y : y);
        if (!same_bits(x, first[v])) eq &= ~(1u << v);
        o[v * n] = x;
      }
    }
  }
  return eq;
}
// The same from the parent's own stored cells (halo filled).
template <class R>
__device__ __forceinline__ void stage_stored(R* __restrict__ s, const double* __restrict__ P, int i0, int j0, int k0,
                                             int nx, int ny, int nz) {
  const int n = nx * ny * nz;
  for (int e = threadIdx.x; e < n; e += blockDim.x) {
    const int i = e % nx, j = (e / nx) % ny, k = e / (nx * ny);
    s[e] = to_r<R>(P[sidx(i0 + i, j0 + j, k0 + k)]);
  }
}

template <class R> __device__ __forceinline__ R predict_t(const QT<R>& t, R sx, R sy, R sz) {
  return t.u + sx * t.Qx + sy * t.Qy + sz * t.Qz + (sx * sy) * t.Qxy + (sx * sz) * t.Qxz + (sy * sz) * t.Qyz +
         (sx * sy * sz) * t.Qxyz;
}


// ---------------------------------------------------------------- halo fill by region
// Sec. 3 (Fig. MrCommunicationMesh): a halo region facing a same-level node
// is a copy of its internal cells, one facing no same-level node is predicted
// from the node's parent (one parent cell, eight fine cells, per step), and
// ghost cells take the boundary conditions.  The stored copies and ghost cells
// are written only for FILL_FULL (and the listed nodes about to be refined):
// copies depend on no halo and run for all levels at once, predictions level by
// level, ghost cells (which may continue a copy or a prediction) at the end.

struct NodeSet {
  const int32_t* list;      // these nodes, or every node when null
  int n;
};

// Variable q of the fill: all five, or rho (q = 0) and E (q = 1) only.
__device__ __forceinline__ int fill_var(bool detail_only, int q) { return detail_only ? 4 * q : q; }

__device__ __forceinline__ int region_start(int s) { return s < 0 ? -HW : (s == 0 ? 0 : NB); }

__device__ __forceinline__ int region_log2(int s) { return s == 0 ? 4 : 2; }   // extents 16 or 4

// One warp per (node, halo region).  Extents are powers of two, so the element
// index splits with shifts; copies move 16-byte pairs of doubles (every
// region row starts on a 32-byte boundary of the 24^3 array).
static __global__ void __launch_bounds__(256) k_fill_regions(Topo t, Pool pool, int cur, NodeSet ns) {
  double* buf = pool.bufp(cur);
  const int nitems = (ns.list ? ns.n : t.cnt[CNT_NNODES]) * 26;
  const int lane = threadIdx.x & 31;
  const int wpb = blockDim.x >> 5;
  for (int w = blockIdx.x * wpb + (threadIdx.x >> 5); w < nitems; w += gridDim.x * wpb) {
    const int node = ns.list ? ns.list[w / 26] : w / 26;
    const int r = w % 26 < 13 ? w % 26 : w % 26 + 1;      // skip the centre
    const int nb = t.nbr[(size_t)node * 27 + r];
    if (nb < 0) continue;
    const int sx = r % 3 - 1, sy = (r / 3) % 3 - 1, sz = r / 9 - 1;
    double* u = buf + (size_t)t.slot[node] * SLOT_U;
    const double* src = buf + (size_t)t.slot[nb] * SLOT_U;
    const int lx = region_log2(sx) - 1, ly = region_log2(sy), lz = region_log2(sz);   // x in pairs
    const int x0 = region_start(sx), y0 = region_start(sy), z0 = region_start(sz);
    const int lxy = lx + ly, ln = lxy + lz;
    const int soff = -NB * (sx + NS * (sy + NS * sz));
    const int ne = NV << ln;                 // a multiple of 32
    // four 16-byte loads in flight per lane before their stores
    for (int e0 = lane; e0 < ne; e0 += 128) {
      double2 val[4];
      int dst[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int e = e0 + 32 * q;
        const int v = e >> ln, c = e & ((1 << ln) - 1);
        const int i = x0 + 2 * (c & ((1 << lx) - 1)), j = y0 + ((c >> lx) & ((1 << ly) - 1)), k = z0 + (c >> lxy);
        dst[q] = v * NCELL + sidx(i, j, k);
        if (e < ne) val[q] = *reinterpret_cast<const double2*>(src + dst[q] + soff);
      }
#pragma unroll
      for (int q = 0; q < 4; ++q)
        if (e0 + 32 * q < ne) *reinterpret_cast<double2*>(u + dst[q]) = val[q];
    }
  }
}

// Predicted halo regions (no same-level node on that side): the regions of a
// node's mask are shared out to PRED_SPLIT CTAs (a leaf at a jump has nine or
// more), each taking one after the other; the parent cells of the region and
// their +-2 stencil (6 or 12 per axis) are staged in shared memory as R for the
// variables filled, then every thread evaluates the Q-terms of parent cells
// and writes their eight fine cells.  Jumps lie where the solution is smooth, so
// most boxes hold one value: it predicts itself (const_safe), without the 125
// shared-memory loads of the Q-terms.
// BLEND (local time stepping): the parent level at fraction th of its step, and
// the halos go to the nodes' places in stage buffer dst, where their level is.
constexpr int PRED_SPLIT = 4;
template <class R, bool BLEND = false>
__global__ void __launch_bounds__(256) k_predict_t(Topo t, Phys p, Pool pool, int cur, const int32_t* __restrict__ list,
                                                   const int32_t* __restrict__ cnt, int n,
                                                   const uint32_t* __restrict__ mask, int mode, int dst = 0,
                                                   double th = 0.0) {
  // the nodes of level n in a list grouped by level (cnt given), or n listed nodes
  __shared__ R box[NV * 864];
  __shared__ ParentBox pb;
  __shared__ BlendBox lb;
  __shared__ unsigned eqs[8];
  double* buf = pool.bufp(cur);
  double* out = BLEND ? pool.bufp(dst) : buf;
  const int nnode = cnt ? cnt[(mode == FILL_STAGE ? CNT_PST : CNT_PALL) + n] : n, nitems = nnode * PRED_SPLIT;
  if (cnt) list += cnt[CNT_LVL + n];
  // (the parts of all nodes one after the other: the first holds most of the
  // work, and must not fall to every fourth CTA only)
  for (int w = blockIdx.x; w < nitems; w += gridDim.x) {
    const int node = list[w % nnode];
    unsigned m = mask[node];
    const int part = w / nnode;
    if (__popc(m) <= part) continue;
    const int par = t.parent[node];
    const int ch = (int)(t.keys[node] & 7ull);
    __syncthreads();                                         // the previous item's box is free
    parent_box(t, p, buf, par, ch, pb);
    __syncthreads();
    if (BLEND) {
      blend_box(t, pool.un, par, ch, pb, lb);
      __syncthreads();
    }
    const bool detail_only = !BLEND && mode == FILL_DETAIL && t.child0[node] < 0;
    const int nvar = detail_only ? 2 : NV;
    double* u = out + (size_t)t.slot[node] * SLOT_U;
    for (int rank = 0; m; ++rank) {
      const int r = __ffs(m) - 1;
      m &= m - 1;
      if (rank % PRED_SPLIT != part) continue;
      const int sx = r % 3 - 1, sy = (r / 3) % 3 - 1, sz = r / 9 - 1;
      // parent cells of the region relative to the child's origin: [q0, q0 + n)
      const int lx = sx == 0 ? 3 : 1, ly = sy == 0 ? 3 : 1, lz = sz == 0 ? 3 : 1;
      const int qx0 = sx < 0 ? -2 : (sx == 0 ? 0 : 8), qy0 = sy < 0 ? -2 : (sy == 0 ? 0 : 8), qz0 = sz < 0 ? -2 : (sz == 0 ? 0 : 8);
      // staged box: those parent cells +-2 (box coordinates: relative to 8 cb - 4)
      const int bx0 = qx0 + 2, by0 = qy0 + 2, bz0 = qz0 + 2;
      const int nx = (1 << lx) + 4, ny = (1 << ly) + 4, nz = (1 << lz) + 4;
      const int nb = nx * ny * nz;
      const unsigned eq = __reduce_and_sync(0xffffffffu, stage_box<R, BLEND>(box, pb, detail_only, bx0, by0, bz0, nx, ny, nz, &lb, th));
      if ((threadIdx.x & 31) == 0) eqs[threadIdx.x >> 5] = eq;
      __syncthreads();
      unsigned constant = eqs[0];
#pragma unroll
      for (int q = 1; q < 8; ++q) constant &= eqs[q];
      const int lxy = lx + ly, ln = lxy + lz;
      for (int e = threadIdx.x; e < (nvar << ln); e += blockDim.x) {
        const int q = e >> ln, c = e & ((1 << ln) - 1);
        const int v = fill_var(detail_only, q);
        const int rx = qx0 + (c & ((1 << lx) - 1)), ry = qy0 + ((c >> lx) & ((1 << ly) - 1)), rz = qz0 + (c >> lxy);
        if (((constant >> q) & 1u) && const_safe(box[q * nb])) {
          const double x = from_r<R>(box[q * nb]);
#pragma unroll
          for (int sub = 0; sub < 4; ++sub)
            *reinterpret_cast<double2*>(u + v * NCELL + sidx(2 * rx, 2 * ry + (sub & 1), 2 * rz + (sub >> 1))) = make_double2(x, x);
          continue;
        }
        const SAcc<R> A{box + q * nb, bx0, by0, bz0, nx, nx * ny};
        const QT<R> qt = qterms_t<R>(A, rx + 4, ry + 4, rz + 4);
        // the two fine cells of a row are one aligned 16-byte store
#pragma unroll
        for (int sub = 0; sub < 8; sub += 2) {
          const int b = (sub >> 1) & 1, cc = (sub >> 2) & 1;
          const R v0 = predict_t<R>(qt, R(1), b ? R(-1) : R(1), cc ? R(-1) : R(1));
          const R v1 = predict_t<R>(qt, R(-1), b ? R(-1) : R(1), cc ? R(-1) : R(1));
          *reinterpret_cast<double2*>(u + v * NCELL + sidx(2 * rx, 2 * ry + b, 2 * rz + cc)) =
              make_double2(from_r<R>(v0), from_r<R>(v1));
        }
      }
      __syncthreads();
    }
  }
}

// Stored ghost cells of the nodes on the domain boundary (after their copies and
// predictions).  The oracle applies the x, y and z passes in turn; their
// composition maps each ghost cell to one source cell (bc_map), so one warp per
// (node, side) item fills the side's 4 x 24 x 24 slab from source cells that this
// kernel never writes; cells in two slabs get the same value twice.  Work
// items are (node, side, chunk of 256 slab cells), one warp each.
static __global__ void __launch_bounds__(256) k_fill_bc(Topo t, Phys p, Pool pool, int cur, NodeSet ns) {
  // sides: every boundary item, or every side of the listed nodes
  int beg, cnt;
  if (ns.list) {
    beg = 0;
    cnt = 6 * ns.n;
  } else {
    beg = t.cnt[CNT_BC];
    cnt = t.cnt[CNT_BC + MAXL + 1] - beg;
  }
  double* buf = pool.bufp(cur);
  constexpr int NCHUNK = 9;                  // 2304 slab cells = 9 chunks of 256
  const int nitems = cnt * NCHUNK;
  const int lane = threadIdx.x & 31;
  const int wpb = blockDim.x >> 5;
  for (int w = blockIdx.x * wpb + (threadIdx.x >> 5); w < nitems; w += gridDim.x * wpb) {
    int node, side;
    if (ns.list) {
      node = ns.list[w / (6 * NCHUNK)];
      side = (w / NCHUNK) % 6;
    } else {
      const int it = t.bc_items[beg + w / NCHUNK];
      node = it >> 3;
      side = it & 7;
    }
    const int d = side >> 1, chunk = w % NCHUNK;
    const int level = t.level[node];
    int blo[3], bhi[3];   // condition of each boundary side of this node, -1 if none (or periodic)
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      const int nl = p.nb[q] << level, Xq = t.X[(size_t)node * 3 + q];
      blo[q] = (Xq == 0 && p.bc[2 * q] != 1) ? p.bc[2 * q] : -1;
      bhi[q] = (Xq == nl - 1 && p.bc[2 * q + 1] != 1) ? p.bc[2 * q + 1] : -1;
    }
    const int bself = (side & 1) ? (d == 0 ? bhi[0] : (d == 1 ? bhi[1] : bhi[2]))
                                 : (d == 0 ? blo[0] : (d == 1 ? blo[1] : blo[2]));
    if (bself < 0) continue;
    double* u = buf + (size_t)t.slot[node] * SLOT_U;
    constexpr int n = HW * NS * NS;           // 2304 = 72 x 32
    for (int e0 = chunk * 256 + lane; e0 < (chunk + 1) * 256; e0 += 4 * 32) {
      double val[4][NV];
      int di[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int e = e0 + 32 * q;
        const int g0 = e % HW, a1 = (e / HW) % NS - HW, a2 = e / (HW * NS) - HW;
        const int a = (side & 1) ? NB + g0 : -1 - g0;
        const int x = (d == 0) ? a : (d == 1 ? a2 : a1);
        const int y = (d == 0) ? a1 : (d == 1 ? a : a2);
        const int z = (d == 0) ? a2 : (d == 1 ? a1 : a);
        int flip = 0;
        const int sx = bc_map(x, blo[0], bhi[0], flip, 1);
        const int sy = bc_map(y, blo[1], bhi[1], flip, 2);
        const int sz = bc_map(z, blo[2], bhi[2], flip, 4);
        di[q] = sidx(x, y, z);
        const int si = sidx(sx, sy, sz);
        if (e < n) {
#pragma unroll
          for (int v = 0; v < NV; ++v) {
            const double s = u[v * NCELL + si];
            val[q][v] = (v >= 1 && v <= 3 && ((flip >> (v - 1)) & 1)) ? -s : s;
          }
        }
      }
#pragma unroll
      for (int q = 0; q < 4; ++q)
        if (e0 + 32 * q < n) {
#pragma unroll
          for (int v = 0; v < NV; ++v)
            u[v * NCELL + di[q]] = val[q][v];
        }
    }
  }
}

// ---------------------------------------------------------------- details
// delta of a node at level >= 1: max over its stored cells that are not ghost
// cells and over rho, E of |u - P(u_parent)| / |u|.  Every leaf, and with
// `all_nodes` every node (the tags then also read the details of the parents
// of leaf groups).  In FP64 the pipe bounds it.  Items are a variable and half of the
// planes of a node, so that a few hundred nodes spread evenly over the SMs; their
// maxima meet in delta_node, which starts at zero.  Shock-bubble with levels 1 and 2:
// 1119 -> 650 us.
// Region of the fine cells of parent cell (rx, ry, rz) (-2 .. 9 relative to the child's origin).
__device__ __forceinline__ int own_region(int rx, int ry, int rz) {
  return (rx < 0 ? 0 : (rx < 8 ? 1 : 2)) + 3 * (ry < 0 ? 0 : (ry < 8 ? 1 : 2)) + 9 * (rz < 0 ? 0 : (rz < 8 ? 1 : 2));
}
static __global__ void __launch_bounds__(256) k_delta_f64(Topo t, Phys p, Pool pool, int cur, double* __restrict__ delta_node,
                                                 int all_nodes) {
  __shared__ double sh[8];
  __shared__ double box[2560];      // the parent's cells 8 cb - 4 .. 8 cb + 11 in x and y, ten planes
  __shared__ ParentBox pb;
  __shared__ const double* own[27]; // the node's stored cells by region

  const int nnode = all_nodes ? t.cnt[CNT_NNODES] : t.cnt[CNT_NLEAVES];
  const double* B = pool.bufp(cur);
  for (int it = blockIdx.x; it < nnode * 4; it += gridDim.x) {
    const int node = all_nodes ? it % nnode : t.leaves[it % nnode];
    const int v = (it / nnode) & 1 ? 4 : 0, rz0 = it / nnode < 2 ? -2 : 4;
    const int lvl = t.level[node];
    if (lvl == 0) continue;
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
    double m = 0.0;
    const double first = box_value(pb, box_word(pb, 0, 0, rz0 + 2), v);
    bool eq = const_safe(first);
    for (int e = threadIdx.x; e < 2560; e += blockDim.x) {
      const double x = box_value(pb, box_word(pb, e & 15, (e >> 4) & 15, rz0 + 2 + (e >> 8)), v);
      box[e] = x;
      eq = eq && same_bits(x, first);
    }
    const bool constant = __syncthreads_and(eq);         // (a box of one value predicts it)
    const SAcc<double> A{box, 0, 0, rz0 + 2, 16, 256};
    // (the warp's lanes stay together: they share their maximum below)
    for (int q0 = threadIdx.x & ~31; q0 < 864; q0 += blockDim.x) {
      const int q = q0 + (threadIdx.x & 31);
      const int rx = q % 12 - 2, ry = (q / 12) % 12 - 2, rz = q / 144 + rz0;
      // all eight fine cells of this parent cell share the ghost status
      const bool ghost = (rx < 0 && gl[0]) || (rx >= 8 && gh[0]) || (ry < 0 && gl[1]) || (ry >= 8 && gh[1]) ||
                         (rz < 0 && gl[2]) || (rz >= 8 && gh[2]);
      const unsigned live = __ballot_sync(0xffffffffu, !ghost);
      if (ghost) continue;
      const double* U = own[own_region(rx, ry, rz)] + v * NCELL + sidx(2 * rx, 2 * ry, 2 * rz);
      double2 uf[4];
#pragma unroll
      for (int q2 = 0; q2 < 4; ++q2)
        uf[q2] = *reinterpret_cast<const double2*>(U + ((q2 >> 1) * NS + (q2 & 1)) * NS);   // rows y + (q2 & 1), z + (q2 >> 1)
      QT<double> qt;
      if (!constant) qt = qterms_t<double>(A, rx + 4, ry + 4, rz + 4);
#pragma unroll
      for (int sub = 0; sub < 8; ++sub) {
        const int a = sub & 1, b = (sub >> 1) & 1, c = (sub >> 2) & 1;
        const double pr = constant ? first : predict_t<double>(qt, a ? -1.0 : 1.0, b ? -1.0 : 1.0, c ? -1.0 : 1.0);
        const double u0 = a ? uf[b + 2 * c].y : uf[b + 2 * c].x, n = fabs(u0 - pr);
        // A quotient |u - P| / |u| no greater than a maximum of the warp is not
        // formed (a division is a dozen FP64 instructions): with x <= the maximum and
        // the product rounded down, |u - P| <= x |u| bounds it.  The comparison is of
        // bit patterns, in which a NaN is large and takes the division.
        const double seen = __hiloint2double((int)__reduce_max_sync(live, (unsigned)__double2hiint(m)), 0);
        if (d2bits(n) <= d2bits(__dmul_rd(seen, fabs(u0)))) continue;
        const double r = n / fabs(u0);
        m = r > m ? r : m;
      }
    }
    for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = m;
    __syncthreads();
    if (threadIdx.x == 0) {
      double x = sh[0];
      for (int q = 1; q < (int)(blockDim.x >> 5); ++q) x = fmax(x, sh[q]);
      // (the parts of a node; bit patterns of non-negative doubles are ordered)
      atomicMax(reinterpret_cast<unsigned long long*>(delta_node + node), (unsigned long long)d2bits(x));
    }
    __syncthreads();
  }
}

}  // namespace mrb

namespace mrb {

// New child: every stored cell predicted from the parent (Eq. Prediction).
// R = double evaluates the prediction in FP64; R = float evaluates the Q-term
// corrections in FP32 and adds them to the FP64 parent value, so that the
// children's mean stays the parent value up to FP64 rounding (the eight
// corrections of a parent cell are sign-symmetric and cancel exactly).
template <class R>
__global__ void __launch_bounds__(256) k_refine_fill_t(Topo t, Pool pool, int cur, const int32_t* __restrict__ pairs,
                                                      int n) {
  __shared__ R box[4096];           // the parent's cells 8 cb - 4 .. 8 cb + 11 per axis, one variable
  double* B = pool.bufp(cur);
  const int nitems = n * NV;
  for (int w = blockIdx.x; w < nitems; w += gridDim.x) {
    const int child = pairs[2 * (w / NV)], par = pairs[2 * (w / NV) + 1];
    const int v = w % NV;
    double* U = B + (size_t)t.slot[child] * SLOT_U + v * NCELL;
    const double* P = B + (size_t)t.slot[par] * SLOT_U + v * NCELL;
    const int ch = (int)(t.keys[child] & 7ull);
    const int cb[3] = {ch & 1, (ch >> 1) & 1, (ch >> 2) & 1};
    const int bx0 = 8 * cb[0] - 4, by0 = 8 * cb[1] - 4, bz0 = 8 * cb[2] - 4;
    stage_stored<R>(box, P, bx0, by0, bz0, 16, 16, 16);
    __syncthreads();
    const SAcc<R> A{box, bx0, by0, bz0, 16, 256};
    for (int r = threadIdx.x; r < 1728; r += blockDim.x) {
      const int pi = 8 * cb[0] - 2 + r % 12, pj = 8 * cb[1] - 2 + (r / 12) % 12, pk = 8 * cb[2] - 2 + r / 144;
      const QT<R> q = qterms_t<R>(A, pi, pj, pk);
      const double base = P[sidx(pi, pj, pk)];
#pragma unroll
      for (int sub = 0; sub < 8; ++sub) {
        const int a = sub & 1, b = (sub >> 1) & 1, c = (sub >> 2) & 1;
        const int fi = 2 * (pi - 8 * cb[0]) + a, fj = 2 * (pj - 8 * cb[1]) + b, fk = 2 * (pk - 8 * cb[2]) + c;
        double val;
        if (sizeof(R) == sizeof(double)) {
          val = from_r<R>(predict_t<R>(q, a ? R(-1) : R(1), b ? R(-1) : R(1), c ? R(-1) : R(1)));
        } else {
          QT<R> q0 = q;
          q0.u = R(0);
          val = base + from_r<R>(predict_t<R>(q0, a ? R(-1) : R(1), b ? R(-1) : R(1), c ? R(-1) : R(1)));
        }
        U[sidx(fi, fj, fk)] = val;
      }
    }
    __syncthreads();
  }
}

// Averaging, Eq. (Averaging), levels fine to coarse; one work item per
// (internal node, octant): the octant's 512 parent cells come from one child.
// A thread forms all five variables of a parent cell (twenty 16-byte loads in
// flight) and, on the mixed-precision path (REC), its FP32 record, which a
// kernel of its own used to read the average back for.  Eight FP64 instructions
// per value bounded it where the children differ; with the means formed by integers
// (mean8) it reads the children at 6.0 TB/s of memory traffic: an internal row is 128
// bytes of 192, and memory is read 128 at a time, so half as much again as the cells
// hold.  Averaging and records per stage: shock-bubble (levels 0..4) 450 -> 301 us
// in one pass; ensemble of five 300 -> 269 us with mean8.
// A 16-byte load that stays where it is written (the compiler moved the loads of
// later variables behind the arithmetic of earlier ones: four in flight).
__device__ __forceinline__ double2 load_now(const double* p) {
  double2 x;
  asm volatile("ld.global.v2.f64 {%0, %1}, [%2];" : "=d"(x.x), "=d"(x.y) : "l"(p));
  return x;
}
struct NoRecord {
  __device__ __forceinline__ void operator()(int, int, const double*) const {}
};
template <class REC>
static __device__ __forceinline__ void project_level(const Topo& t, const Pool& pool, int buf, int level, REC rec) {
  const int beg = t.cnt[CNT_LVL + level], end = t.cnt[CNT_LVL + level + 1];
  double* B = pool.bufp(buf);
  const int nitems = (end - beg) * 8;
  for (int w = blockIdx.x; w < nitems; w += gridDim.x) {
    const int node = t.lvl_nodes[beg + w / 8];
    const int c0 = t.child0[node];
    if (c0 < 0) continue;
    const int o = w % 8, slot = t.slot[node];
    double* __restrict__ Pp = B + (size_t)slot * SLOT_U;
    const double* __restrict__ C = B + (size_t)t.slot[c0 + o] * SLOT_U;
    const int ox = 8 * (o & 1), oy = 8 * ((o >> 1) & 1), oz = 8 * ((o >> 2) & 1);
    for (int c = threadIdx.x; c < 512; c += blockDim.x) {
      const int I = c % 8, J = (c / 8) % 8, K = c / 64;
      double2 a[NV][4];
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        // 2 I is even: each x-pair of children is one aligned 16-byte load
        const double* u = C + v * NCELL + sidx(2 * I, 2 * J, 2 * K);
        a[v][0] = load_now(u);
        a[v][1] = load_now(u + NS);
        a[v][2] = load_now(u + NS * NS);
        a[v][3] = load_now(u + NS * NS + NS);
      }
      double U[NV];
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        const double x[8] = {a[v][0].x, a[v][0].y, a[v][1].x, a[v][1].y, a[v][2].x, a[v][2].y, a[v][3].x, a[v][3].y};
        U[v] = mean8(x);
        Pp[v * NCELL + sidx(ox + I, oy + J, oz + K)] = U[v];
      }
      rec(slot, iidx(ox + I, oy + J, oz + K), U);
    }
  }
}

// ---------------------------------------------------------------- time step
// The end of a CFL kernel: the CTA that finishes last turns the instances' maxima
// into time steps (Eq. (Cfl)), and leaves the maxima and the count of CTAs
// (smax[4 n_inst]) at zero for the next one; with `hist` the steps also go to
// *hist, which moves on by one row.  (A fill before, a kernel and a copy after
// it cost a single-level step three launches of six, and their gaps.)
static __device__ __forceinline__ void cfl_finish(const Phys& p, unsigned long long* __restrict__ smax,
                                                  double* __restrict__ dt, double** hist) {
  __shared__ bool last;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) last = atomicAdd(&smax[4 * p.n_inst], 1ull) == gridDim.x - 1;
  __syncthreads();
  if (!last) return;
  __threadfence();
  double* row = hist ? *hist : nullptr;
  for (int i = threadIdx.x; i < p.n_inst; i += blockDim.x) {
    double s[4];
    for (int d = 0; d < 4; ++d) {
      s[d] = __longlong_as_double((long long)__ldcg(&smax[i * 4 + d]));
      smax[i * 4 + d] = 0ull;
    }
    const double dxl = ldexp(p.dx0, -p.lmax[i]);
    double h = p.cfl * dxl / ((s[0] + s[1]) + s[2]);
    if (p.mu > 0.0) {
      // explicit diffusion limit of the viscous terms: k dx^2 / (6 max(mu / rho))
      const double hv = (p.cfl * (dxl * dxl)) / ((6.0 * p.mu) * s[3]);
      h = (hv < h) ? hv : h;
    }
    dt[i] = h;
    if (row) row[i] = h;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    smax[4 * p.n_inst] = 0ull;
    if (row) *hist = row + p.n_inst;
  }
}

}  // namespace mrb
