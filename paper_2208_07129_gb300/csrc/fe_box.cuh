// Cell kernel of axis-aligned box cells (every structured mesh given without
// vertices, and refined meshes): FP64, FP32 and double-float arithmetic.
//
// A box cell's metric is diagonal and constant, and with sqrt(w) folded into
// the tables the quadrature weights are 1, so the stiffness at the quadrature
// points is separable,
//   D~_x^T g00 D~_x + D~_y^T g11 D~_y + D~_z^T g22 D~_z,   and   D~^T D~ = K
// is one symmetric n_q x n_q matrix: three 1D passes with K take the place of
// the six passes with D~ and D~^T of trilinear cells (fe_general.cuh), and
// nothing but the values t = N u has to be kept besides their image s.  K is
// formed in FP64 on the host; the cell's one factor g22 multiplies at the end
// (g00 / g22 and g11 / g22 are the same for every cell of a mesh and are part
// of the x and y tables).
//
// Each 1D matrix is (skew-)centrosymmetric, so it splits into an even and an
// odd half (see fe_cells.cuh).  Here the halves stay apart between passes:
// a direction's values are kept as (even, odd) parts from N's pass until the
// pass that needs point values, so K works on them without sums before or
// after.  For p = 6, n_q = 8 a cell and vector take 22.5 K operations against
// 36.2 K for the D~ form.
//
// Seven passes over 1D lines, each thread one line (W vectors of it) in
// registers, in place on two shared tiles t and s of n_q^3 values per vector:
//   1 x: gather, N            2 y: N
//   3 z: N, s = K t, both to point values along z
//   4 y: s += K t, both to point values along y
//   5 x: s += K t; c t at the points; + g22 s; N^T
//   6 y: N^T                  7 z: N^T, scatter
// The tiles hold one vector group after the other with constant strides, so
// every access has an immediate offset; rows are padded to an odd length and
// the distance of two groups is chosen so that no pass meets a bank conflict.
//
// What bounds it, and what it measured (32^3 periodic, p = 6, n_q = 8, 64
// vectors; the D~ form before): FP64 148.0 -> 89.9 ms, the FP64 pipe (22.5 K
// operations at 0.595 T/s are 79 ms); double-float 38.9 -> 20.9 ms, the issue
// of FP32 instructions.  FP32, 24^3, 128 vectors: 6.92 -> 2.99 ms, shared
// memory (7.5 K values per cell and vector, 1.2 ms) and the barriers between
// the passes.
#pragma once

#include "fe_cells.cuh"

namespace fe {

// Tables of the box kernel for C coefficients.  N: nodes to points, Nt its
// transpose; K maps
// (even, odd) parts to (even, odd) parts.
template <typename C, int NP, int NQ>
struct BoxTables {
  EOTab<C, NQ, NP> N;
  EOTab<C, NP, NQ> Nt;
  EOTab<C, NQ, NQ> Kx, Ky, Kz;
};

// One cell e and B groups of W vectors: thread (v, ty) of B x nty threads
// works on group vb B + v.  Switches: SC the scaled
// product, MAP the explicit map of refined meshes, LOCAL the per-cell scratch.
// vec: X, Y and n_vec are multiples of W values (set by the launch), so a
// group moves in one access.
template <typename V, int NP, int NQ, bool SC = false, bool MAP = false, bool LOCAL = false>
__device__ __forceinline__ void cell_body_box(const BoxTables<typename Arith<V>::C, NP, NQ>& tab, const MeshDev& m,
                                              const Geom<typename Arith<V>::G>& geo, int e, int vb, int B, int v,
                                              int ty, int nty, int n_vec, bool vec,
                                              const typename Arith<V>::D* __restrict__ X,
                                              typename Arith<V>::D* __restrict__ Y, V* smem,
                                              const Scale<typename Arith<V>::D>& sc,
                                              const int* __restrict__ map = nullptr) {
  using A = Arith<V>;
  using G = typename A::G;
  using D = typename A::D;
  using TS = BoxTile<NQ>;
  constexpr int P = NP - 1, RP = TS::RP, PP = TS::PP, W = A::W;
  constexpr int HQ = (NQ + 1) / 2, OQ = NQ / 2 > 0 ? NQ / 2 : 1, HP = (NP + 1) / 2, OP = NP / 2 > 0 ? NP / 2 : 1;
  const int pitch = TS::pitch(B, (int)sizeof(V));
  V* T = smem + v * pitch;
  V* S = T + B * pitch;
  const int vg = (vb * B + v) * W;
  const int have = n_vec - vg;   // vectors from this group on (<= 0: none)
  const BoxDir dx(e % m.nx, m.nx, m.Nx, P, m.periodic, m.last_odd_x);
  const BoxDir dy((e / m.nx) % m.ny, m.ny, m.Ny, P, m.periodic, m.last_odd_y);
  const BoxDir dz(e / (m.nx * m.ny), m.nz, m.Nz, P, m.periodic, m.last_odd_z);

  // ---- 1: extraction and x pass of N ----
  for (int l = ty; l < NP * NP; l += nty) {
    const int i2 = l % NP, i3 = l / NP;
    V u[NP], a[NQ], ue[HP], uo[OP];
    gather_line<A, NP, SC>(node_line<A, NP, 0, MAP>(m, dx, dy, dz, i2, i3, e, map), X, n_vec, vg, have, vec, sc, u);
    eo_split<A, NP>(u, ue, uo);
    eo_parts<A, NQ, NP>(tab.N, ue, uo, a);
    V* dst = T + i3 * PP + i2 * RP;
#pragma unroll
    for (int q = 0; q < NQ; ++q) dst[q] = a[q];
  }
  __syncthreads();
  // ---- 2: y pass of N ----
  for (int l = ty; l < NQ * NP; l += nty) {
    V* line = T + (l / NQ) * PP + l % NQ;
    V u[NP], a[NQ], ue[HP], uo[OP];
#pragma unroll
    for (int i = 0; i < NP; ++i) u[i] = line[i * RP];
    eo_split<A, NP>(u, ue, uo);
    eo_parts<A, NQ, NP>(tab.N, ue, uo, a);
#pragma unroll
    for (int q = 0; q < NQ; ++q) line[q * RP] = a[q];
  }
  __syncthreads();
  // ---- 3: z pass of N, z stiffness, to point values along z ----
  for (int l = ty; l < NQ * NQ; l += nty) {
    const int at = (l / NQ) * RP + l % NQ;
    V u[NP], t[NQ], s[NQ], ue[HP], uo[OP];
#pragma unroll
    for (int i = 0; i < NP; ++i) u[i] = T[i * PP + at];
    eo_split<A, NP>(u, ue, uo);
    eo_parts<A, NQ, NP>(tab.N, ue, uo, t);
    eo_parts<A, NQ, NQ>(tab.Kz, t, t + HQ, s);
    eo_join<A, NQ>(t);
    eo_join<A, NQ>(s);
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
      T[q * PP + at] = t[q];
      S[q * PP + at] = s[q];
    }
  }
  __syncthreads();
  // ---- 4: y stiffness, to point values along y ----
  for (int l = ty; l < NQ * NQ; l += nty) {
    const int at = (l / NQ) * PP + l % NQ;
    V t[NQ], s[NQ];
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
      t[q] = T[q * RP + at];
      s[q] = S[q * RP + at];
    }
    eo_parts<A, NQ, NQ, true>(tab.Ky, t, t + HQ, s);
    eo_join<A, NQ>(t);
    eo_join<A, NQ>(s);
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
      T[q * RP + at] = t[q];
      S[q * RP + at] = s[q];
    }
  }
  __syncthreads();
  // ---- 5: x stiffness, potential at the points, x pass of N^T ----
  const G g = geo.cellG[(size_t)e * 6 + 5], g2 = A::twice(g);
  const G* ptC = geo.ptC + (size_t)e * NQ * NQ * NQ;
  for (int l = ty; l < NQ * NQ; l += nty) {
    V* line = T + l * RP;
    V t[NQ], s[NQ], he[HQ], ho[OQ], o[NP];
    G c[NQ];
    load_row<G, NQ>(ptC + l * NQ, c);
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
      t[q] = line[q];
      s[q] = S[l * RP + q];
    }
    eo_parts<A, NQ, NQ, true>(tab.Kx, t, t + HQ, s);
    eo_join<A, NQ>(t);
    // the mirrored sums and differences N^T needs; those of s's values are
    // twice its parts (once at the middle point)
#pragma unroll
    for (int q = 0; q < NQ / 2; ++q)
      A::point_pair(c[q], t[q], c[NQ - 1 - q], t[NQ - 1 - q], g2, s[q], s[HQ + q], he[q], ho[q]);
    if constexpr (NQ & 1) he[NQ / 2] = A::point(c[NQ / 2], t[NQ / 2], g, s[NQ / 2]);
    eo_parts<A, NP, NQ>(tab.Nt, he, ho, o);
    eo_join<A, NP>(o);
#pragma unroll
    for (int i = 0; i < NP; ++i) line[i] = o[i];
  }
  __syncthreads();
  // ---- 6: y pass of N^T ----
  for (int l = ty; l < NQ * NP; l += nty) {
    V* line = T + (l / NP) * PP + l % NP;
    V h[NQ], he[HQ], ho[OQ], o[NP];
#pragma unroll
    for (int q = 0; q < NQ; ++q) h[q] = line[q * RP];
    eo_split<A, NQ>(h, he, ho);
    eo_parts<A, NP, NQ>(tab.Nt, he, ho, o);
    eo_join<A, NP>(o);
#pragma unroll
    for (int i = 0; i < NP; ++i) line[i * RP] = o[i];
  }
  __syncthreads();
  // ---- 7: z pass of N^T and assembly ----
  if constexpr (!LOCAL) wait_for_earlier_launch();
  if (have <= 0) return;
  for (int l = ty; l < NP * NP; l += nty) {
    const int i1 = l % NP, i2 = l / NP;
    const NodeLine<A, NP> nodes = node_line<A, NP, 2, MAP>(m, dx, dy, dz, i1, i2, e, map);
    Pack<D, W> old[NP];
    if constexpr (!LOCAL) read_old<A, NP, SC>(nodes, Y, n_vec, vg, have, vec, sc, old);
    V h[NQ], he[HQ], ho[OQ], o[NP];
#pragma unroll
    for (int q = 0; q < NQ; ++q) h[q] = T[q * PP + i2 * RP + i1];
    eo_split<A, NQ>(h, he, ho);
    eo_parts<A, NP, NQ>(tab.Nt, he, ho, o);
    eo_join<A, NP>(o);
    if constexpr (LOCAL) {
      D* w = Y + ((size_t)e * NP * NP * NP + l) * n_vec + vg;
#pragma unroll
      for (int i = 0; i < NP; ++i) store_pack<D, W>(w + (size_t)i * NP * NP * n_vec, A::to(o[i]), have, vec);
    } else {
      scatter_line<A, NP, SC>(nodes, o, old, X, Y, n_vec, vg, have, vec, sc);
    }
  }
}

template <typename V, int NP, int NQ, bool SC, bool MAP>
__global__ void __launch_bounds__(256) cell_apply_box_kernel(
    const BoxTables<typename Arith<V>::C, NP, NQ> tab, const MeshDev m, const Geom<typename Arith<V>::G> geo,
    const int* __restrict__ cells, int n_vec, int n_vb, bool vec, const typename Arith<V>::D* __restrict__ X,
    typename Arith<V>::D* __restrict__ Y, const Scale<typename Arith<V>::D> sc, const int* __restrict__ map) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  let_next_launch_start();
  cell_body_box<V, NP, NQ, SC, MAP>(tab, m, geo, cells[blockIdx.x / n_vb], blockIdx.x % n_vb, blockDim.x,
                                    threadIdx.x, threadIdx.y, blockDim.y, n_vec, vec, X, Y,
                                    reinterpret_cast<V*>(smem_raw),
                                    sc, map);
}

// Small meshes: every cell in one launch, results to the per-cell scratch.
template <typename V, int NP, int NQ>
__global__ void __launch_bounds__(256) cell_apply_box_local_kernel(
    const BoxTables<typename Arith<V>::C, NP, NQ> tab, const MeshDev m, const Geom<typename Arith<V>::G> geo,
    int n_vec, int n_vb, bool vec, const typename Arith<V>::D* __restrict__ X, typename Arith<V>::D* __restrict__ Wk) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  let_next_launch_start();
  cell_body_box<V, NP, NQ, false, false, true>(tab, m, geo, blockIdx.x / n_vb, blockIdx.x % n_vb, blockDim.x,
                                               threadIdx.x, threadIdx.y, blockDim.y, n_vec, vec, X, Wk,
                                               reinterpret_cast<V*>(smem_raw), Scale<typename Arith<V>::D>{});
}

// Host: (even, odd)-part table of f K (see fe_ctx::Ks).
template <typename C, int NQ>
void make_stiffness(EOTab<C, NQ, NQ>& t, const fe_ctx* c, double f) {
  constexpr int H = NQ / 2, HE = (NQ + 1) / 2;
  for (int o = 0; o < HE; ++o) {
    for (int i = 0; i < HE; ++i) t.E[o][i] = (C)(f * c->Ks[o * HE + i]);
    for (int i = 0; i < H; ++i) t.O[o][i] = (C)(f * c->Kd[o * HE + i]);
  }
}

template <typename C, int NP, int NQ>
BoxTables<C, NP, NQ> make_boxtables(const fe_ctx* c) {
  BoxTables<C, NP, NQ> t;
  double Nt[NP * NQ];
  for (int q = 0; q < NQ; ++q)
    for (int i = 0; i < NP; ++i) Nt[i * NQ + q] = c->Nf[q * NP + i];
  make_eotab(t.N, c->Nf.data());
  make_eotab(t.Nt, Nt);
  // g_dd = mu det J (2 / h_d)^2
  const double* h = c->box_h;
  make_stiffness(t.Kx, c, (h[2] / h[0]) * (h[2] / h[0]));
  make_stiffness(t.Ky, c, (h[2] / h[1]) * (h[2] / h[1]));
  make_stiffness(t.Kz, c, 1.0);
  return t;
}

template <typename V, int NP, int NQ, bool SC = false, bool MAP = false>
cudaError_t launch_box(const fe_ctx* c, const typename Arith<V>::D* X, typename Arith<V>::D* Y, int n_vec,
                       cudaStream_t s, LineTile want, const Geom<typename Arith<V>::G>& geo,
                       const Scale<typename Arith<V>::D>& sc = Scale<typename Arith<V>::D>{}) {
  using D = typename Arith<V>::D;
  constexpr int W = Arith<V>::W;
  const bool vec = vec_ok<V>(X, Y, n_vec);
  const BoxTables<typename Arith<V>::C, NP, NQ> tab = make_boxtables<typename Arith<V>::C, NP, NQ>(c);
  if constexpr (!SC && !MAP) {
    // Small meshes (scratch allocated at setup): one launch over all cells
    // writing each cell's result to the scratch, then one gather in colour order.
    const bool fits = (size_t)n_vec * NP * NP * NP * c->n_cells * sizeof(D) <= c->small.bytes();
    if (void* scratch = fits ? c->small.block(s) : nullptr) {
      auto lk = cell_apply_box_local_kernel<V, NP, NQ>;
      int lanes = 1;
      size_t lsm = 0;
      cudaError_t e = small_shape<V, NQ, 2>(c->n_cells, n_vec, &lanes, &lsm);
      if (e == cudaSuccess) e = ensure_dyn_smem(reinterpret_cast<const void*>(lk), lsm);
      if (e != cudaSuccess) return e;
      D* Wk = static_cast<D*>(scratch);
      const int blocks = (n_vec + lanes * W - 1) / (lanes * W);
      e = launch_kernel(lk, c->n_cells * (size_t)blocks, dim3(lanes, NQ * NQ), lsm, s, false, tab, c->mdev, geo, n_vec,
                        blocks, vec, X, Wk);
      if (e == cudaSuccess) {
        const size_t tot = c->n_dofs * (size_t)n_vec;
        e = launch_kernel(assemble_local_kernel<D, NP>, std::min<size_t>((tot + 255) / 256, 152 * 8), dim3(256), 0, s,
                          true, c->mdev, Wk, Y, c->n_dofs, n_vec);
      }
      const cudaError_t e2 = c->small.enqueued(s);
      return e != cudaSuccess ? e : e2;
    }
  }
  auto kern = cell_apply_box_kernel<V, NP, NQ, SC, MAP>;
  const BoxShape sh = box_shape<V, NQ, 2>(want, Arith<V>::box_tile(NQ), n_vec);
  cudaError_t e = ensure_dyn_smem(reinterpret_cast<const void*>(kern), sh.smem);
  if (e != cudaSuccess) return e;
  const int n_vb = (n_vec + sh.lanes * W - 1) / (sh.lanes * W);
  bool overlap = false;
  for (int k = 0; k < c->colors.n_colors; ++k) {
    const int n = c->colors.offset[k + 1] - c->colors.offset[k];
    if (n == 0) continue;
    e = launch_kernel(kern, (size_t)n * n_vb, dim3(sh.lanes, sh.lines), sh.smem, s, overlap, tab, c->mdev, geo,
                      c->d_cells + c->colors.offset[k], n_vec, n_vb, vec, X, Y, sc, MAP ? c->d_map : nullptr);
    if (e != cudaSuccess) return e;
    overlap = true;
  }
  return cudaSuccess;
}

}  // namespace fe
