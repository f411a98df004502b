// Cell kernel of axis-aligned box cells (every structured mesh given without
// vertices, and refined meshes): FP64, FP32 and double-float arithmetic.
//
// A box cell's metric is diagonal and constant, and with sqrt(w) folded into
// the tables the quadrature weights are 1, so the stiffness at the quadrature
// points is separable,
//   D~_x^T g00 D~_x + D~_y^T g11 D~_y + D~_z^T g22 D~_z,   and   D~^T D~ = K
// is one symmetric n_q x n_q matrix: three 1D passes with K take the place of
// the six passes with D~ and D~^T of trilinear cells (fe_general.cuh), and
// nothing but the values t = N u has to be kept besides their image s.  The
// cell's one factor g22 multiplies at the end (g00 / g22 and g11 / g22 are the
// same for every cell of a mesh and are part of the tables).
//
// Each 1D matrix is (skew-)centrosymmetric, so it splits into an even and an
// odd half (see fe_cells.cuh).  Here the halves stay apart between passes:
// a direction's values are kept as (even, odd) parts from N's pass until the
// pass that needs point values, so K works on them without sums before or
// after.
//
// K is applied in factors.  As one rounded matrix it would no longer annihilate
// the constant, and the energy x.(A x) that a solver or a filter takes from the
// product would have a first-order error of eps |K| there (FP32, 12^3 cells, p =
// 6: 4e-4 of the energy of a constant, 6e-6 of one period's); with D~ the energy
// is |D~ t|^2 and the rounding of a table enters it squared.  So each half is
// kept as L^T d L, L unit lower triangular, with the rank the half has: the
// energy is a sum of products of (L t)_k with d_k (L t)_k, both of which are
// small where t is smooth.  Rows start at the centre of the rule and go out, and
// the centre itself has none.  FP32 energies are then as accurate as the D~
// form's (1.2e-7 and 1.1e-7).  L and d L^T take R (R + 1) / 2 products each, less
// L's unit diagonal: one operation less than the matrix.  For p = 6, n_q = 8 a
// cell and vector take 22.1 K operations against 36.2 K for the D~ form.
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
// vectors; the D~ form before): FP64 148.0 -> 89.3 ms, the FP64 pipe (22.1 K
// operations at 0.595 T/s are 78 ms); double-float 38.9 -> 21.9 ms, the issue
// of FP32 instructions.  FP32, 24^3, 128 vectors: 6.92 -> 3.03 ms, shared
// memory (7.5 K values per cell and vector, 1.2 ms) and the barriers between
// the passes.  With K as one matrix the three were 89.9, 21.4 and 3.00 ms; the
// 12^3 p = 6 solve with FP32 inner iterations took 156 ms with it and takes 148.
#pragma once

#include "fe_cells.cuh"

namespace fe {

// K = L^T d L by halves of R rows: R = RE for the even half, which has one part
// more, the centre; R = RO for the odd half.  L, the same for every direction:
// row k has e[k (k-1)/2 + i] for the parts i < k and c[k] for the centre.
template <typename C, int NQ>
struct StiffTab {
  static constexpr int H = NQ / 2, HE = (NQ + 1) / 2, RE = HE - 1, RO = H;
  C e[RE > 1 ? RE * (RE - 1) / 2 : 1];
  C c[RE > 0 ? RE : 1];
  C o[RO > 1 ? RO * (RO - 1) / 2 : 1];
};

// d L^T of one direction, its metric factor included: e[k (k+1)/2 + i] for the
// parts i <= k, c[k] for the centre.
template <typename C, int NQ>
struct StiffBack {
  using T = StiffTab<C, NQ>;
  C e[T::RE > 0 ? T::RE * (T::RE + 1) / 2 : 1];
  C c[T::RE > 0 ? T::RE : 1];
  C o[T::RO * (T::RO + 1) / 2];
};

// Tables of the box kernel for C coefficients.  N: nodes to points, Nt its
// transpose; K maps (even, odd) parts to (even, odd) parts.
template <typename C, int NP, int NQ>
struct BoxTables {
  EOTab<C, NQ, NP> N;
  EOTab<C, NP, NQ> Nt;
  StiffTab<C, NQ> K;
  StiffBack<C, NQ> kx, ky, kz;
};

// One half of s (+)= L^T d L t over R rows; CENTRE: the even half, with its
// centre t[R] and s[R].  (ADD: see eo_row.)
template <typename A, int R, bool CENTRE, bool ADD, typename TC>
__device__ __forceinline__ void stiff_half(const TC* l, const TC* lc, const TC* b, const TC* bc,
                                           const typename A::V* t, typename A::V* s) {
  if constexpr (R > 0) {
    typename A::V y[R];
#pragma unroll
    for (int k = 0; k < R; ++k) {
      typename A::Acc a = A::init(t[k]);
#pragma unroll
      for (int i = 0; i < k; ++i) A::fma(a, l[k * (k - 1) / 2 + i], t[i]);
      if constexpr (CENTRE) A::fma(a, lc[k], t[R]);
      y[k] = CENTRE || k > 0 ? A::value(a) : t[k];
    }
    constexpr bool kFromSum = ADD && !A::kSumApart;
#pragma unroll
    for (int i = 0; i < R; ++i) {
      typename A::Acc a = kFromSum ? A::init(s[i]) : A::first(b[i * (i + 1) / 2 + i], y[i]);
#pragma unroll
      for (int k = kFromSum ? i : i + 1; k < R; ++k) A::fma(a, b[k * (k + 1) / 2 + i], y[k]);
      s[i] = ADD && !kFromSum ? A::add(s[i], A::value(a)) : A::value(a);
    }
    if constexpr (CENTRE) eo_row<A, R, ADD>(bc, y, s[R]);
  } else if constexpr (CENTRE && !ADD) {
    s[0] = A::zero();
  }
}

// s (+)= K t on (even, odd) parts, b of one direction.
template <typename A, int NQ, bool ADD = false>
__device__ __forceinline__ void stiff_parts(const StiffTab<typename A::C, NQ>& K,
                                            const StiffBack<typename A::C, NQ>& b, const typename A::V* t,
                                            typename A::V* s) {
  using T = StiffTab<typename A::C, NQ>;
  stiff_half<A, T::RE, true, ADD>(K.e, K.c, b.e, b.c, t, s);
  stiff_half<A, T::RO, false, ADD>(K.o, K.o, b.o, b.o, t + T::HE, s + T::HE);
}

// One cell e and B groups of W vectors: thread (v, ty) of B x nty threads
// works on group vb B + v.  kx, ky: tab's, or those of another mesh of the degree.  Switches: SC the scaled
// product, MAP the explicit map of refined meshes, LOCAL the per-cell scratch.
// vec: X, Y and n_vec are multiples of W values (set by the launch), so a
// group moves in one access.
template <typename V, int NP, int NQ, bool SC = false, bool MAP = false, bool LOCAL = false>
__device__ __forceinline__ void cell_body_box(const BoxTables<typename Arith<V>::C, NP, NQ>& tab,
                                              const StiffBack<typename Arith<V>::C, NQ>& kx,
                                              const StiffBack<typename Arith<V>::C, NQ>& ky, const MeshDev& m,
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
    stiff_parts<A, NQ>(tab.K, tab.kz, t, s);
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
    stiff_parts<A, NQ, true>(tab.K, ky, t, s);
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
    stiff_parts<A, NQ, true>(tab.K, kx, t, s);
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
  cell_body_box<V, NP, NQ, SC, MAP>(tab, tab.kx, tab.ky, m, geo, cells[blockIdx.x / n_vb], blockIdx.x % n_vb, blockDim.x,
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
  cell_body_box<V, NP, NQ, false, false, true>(tab, tab.kx, tab.ky, m, geo, blockIdx.x / n_vb, blockIdx.x % n_vb, blockDim.x,
                                               threadIdx.x, threadIdx.y, blockDim.y, n_vec, vec, X, Wk,
                                               reinterpret_cast<V*>(smem_raw), Scale<typename Arith<V>::D>{});
}

// Host: L, and f d L^T (see fe_ctx::KLe; a middle point stands once where a
// pair stands twice).
template <typename C, int NQ>
void make_stiffness(StiffTab<C, NQ>& t, const fe_ctx* c) {
  for (size_t i = 0; i < c->KLe.size(); ++i) t.e[i] = (C)c->KLe[i];
  for (size_t i = 0; i < c->KLc.size(); ++i) t.c[i] = (C)c->KLc[i];
  for (size_t i = 0; i < c->KLo.size(); ++i) t.o[i] = (C)c->KLo[i];
}

template <typename C, int NQ>
void make_stiffness_back(StiffBack<C, NQ>& t, const fe_ctx* c, double f) {
  auto half = [f](C* b, const std::vector<double>& L, const std::vector<double>& d) {
    const int R = (int)d.size();
    for (int k = 0; k < R; ++k)
      for (int i = 0; i <= k; ++i)
        b[k * (k + 1) / 2 + i] = (C)(f * d[k] * (i == k ? 1.0 : L[k * (k - 1) / 2 + i]));
  };
  half(t.e, c->KLe, c->KDe);
  half(t.o, c->KLo, c->KDo);
  for (size_t k = 0; k < c->KDe.size(); ++k) t.c[k] = (C)((NQ & 1 ? 2.0 : 1.0) * f * c->KDe[k] * c->KLc[k]);
}

template <typename C, int NP, int NQ>
BoxTables<C, NP, NQ> make_boxtables(const fe_ctx* c) {
  BoxTables<C, NP, NQ> t{};
  double Nt[NP * NQ];
  for (int q = 0; q < NQ; ++q)
    for (int i = 0; i < NP; ++i) Nt[i * NQ + q] = c->Nf[q * NP + i];
  make_eotab(t.N, c->Nf.data());
  make_eotab(t.Nt, Nt);
  // g_dd = mu det J (2 / h_d)^2
  const double* h = c->box_h;
  make_stiffness(t.K, c);
  make_stiffness_back(t.kx, c, (h[2] / h[0]) * (h[2] / h[0]));
  make_stiffness_back(t.ky, c, (h[2] / h[1]) * (h[2] / h[1]));
  make_stiffness_back(t.kz, c, 1.0);
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
