// Cell kernel of axis-aligned box cells (every structured mesh given without
// vertices, and refined meshes): FP64, FP32 and double-float arithmetic.
//
// A box cell's metric is diagonal and constant, and with sqrt(w) folded into
// the tables the quadrature weights are 1, so the stiffness at the quadrature
// points is separable,
//   D~_x^T g00 D~_x + D~_y^T g11 D~_y + D~_z^T g22 D~_z,   and   D~^T D~ = K
// is one symmetric n_q x n_q matrix: three 1D passes with K take the place of
// the six passes with D~ and D~^T of trilinear cells (fe_evenodd.cuh), and
// nothing but the values t = N u has to be kept besides their image s.  K is
// formed in FP64 on the host; the cell's one factor g22 multiplies at the end
// (g00 / g22 and g11 / g22 are the same for every cell of a mesh and are part
// of the x and y tables).
//
// Each 1D matrix is (skew-)centrosymmetric, so it splits into an even and an
// odd half (see fe_evenodd.cuh).  Here the halves stay apart between passes:
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
#pragma once

#include <algorithm>

#include "fe_arith.cuh"
#include "fe_evenodd.cuh"

namespace fe {

// Tables of the box kernel for C coefficients.  N, Nt as in EOTables; K maps
// (even, odd) parts to (even, odd) parts.
template <typename C, int NP, int NQ>
struct BoxTables {
  EOTab<C, NQ, NP> N;
  EOTab<C, NP, NQ> Nt;
  EOTab<C, NQ, NQ> Kx, Ky, Kz;
};

// Sums and differences of mirrored values: in -> (even, odd).
template <typename A, int N>
__device__ __forceinline__ void eo_split(const typename A::V* in, typename A::V* e, typename A::V* o) {
#pragma unroll
  for (int i = 0; i < N / 2; ++i) {
    e[i] = A::add(in[i], in[N - 1 - i]);
    o[i] = A::sub(in[i], in[N - 1 - i]);
  }
  if constexpr (N & 1) e[N / 2] = in[N / 2];
}

// Values from their (even, odd) parts; part k is stored at index k of x
// (even parts first), the values replace them.
template <typename A, int N>
__device__ __forceinline__ void eo_join(typename A::V* x) {
  constexpr int H = N / 2, HE = (N + 1) / 2;
  typename A::V t[N];
#pragma unroll
  for (int i = 0; i < H; ++i) {
    t[i] = A::add(x[i], x[HE + i]);
    t[N - 1 - i] = A::sub(x[i], x[HE + i]);
  }
  if constexpr (N & 1) t[H] = x[H];
#pragma unroll
  for (int i = 0; i < N; ++i) x[i] = t[i];
}

// out parts = tables times in parts (even parts first in out); with ADD the
// products are added to what out holds.  Double-float and FP32 sum the products
// first and add the sum: what out holds is larger than one direction's share,
// and every term added to it would be rounded at its scale (the double-float
// error of a p = 6 product is 1.2e-14 this way, 1.4e-14 the other).  FP64
// starts its sum from it: one operation less on the pipe that bounds it.
template <typename A, int NI, typename TC, typename TV>
__device__ __forceinline__ typename A::V eo_dot(const TC* c, const TV* x) {
  typename A::Acc a = A::first(c[0], x[0]);
#pragma unroll
  for (int i = 1; i < NI; ++i) A::fma(a, c[i], x[i]);
  return A::value(a);
}

template <typename A, int NI, bool ADD, typename TC>
__device__ __forceinline__ void eo_row(const TC* c, const typename A::V* x, typename A::V& out) {
  if constexpr (!ADD) {
    out = eo_dot<A, NI>(c, x);
  } else if constexpr (A::kSumApart) {
    out = A::add(out, eo_dot<A, NI>(c, x));
  } else {
    typename A::Acc a = A::init(out);
#pragma unroll
    for (int i = 0; i < NI; ++i) A::fma(a, c[i], x[i]);
    out = A::value(a);
  }
}

template <typename A, int NO, int NI, bool ADD = false>
__device__ __forceinline__ void eo_parts(const EOTab<typename A::C, NO, NI>& t, const typename A::V* e,
                                         const typename A::V* o, typename A::V* out) {
  constexpr int HI = NI / 2, HE = (NI + 1) / 2, HO = (NO + 1) / 2;
#pragma unroll
  for (int k = 0; k < HO; ++k) eo_row<A, HE, ADD>(t.E[k], e, out[k]);
#pragma unroll
  for (int k = 0; k < NO / 2; ++k) {
    if constexpr (HI > 0) eo_row<A, HI, ADD>(t.O[k], o, out[HO + k]);
    else if (!ADD) out[HO + k] = A::zero();
  }
}

// Shared-memory shape: rows of RP values, planes of NQ rows.
template <int NQ>
struct BoxTile {
  static constexpr int RP = NQ | 1;        // row, padded to an odd length
  static constexpr int PP = NQ * RP;       // plane
  // distance of the tiles of two vector groups when B of them share a CTA,
  // values of `bytes` bytes: the U values that one 128-byte wavefront serves
  // come from B groups x U / B lines, so groups lie U / B (mod U) apart
  static __host__ __device__ constexpr int pitch(int B, int bytes) {
    const int U = 128 / bytes, want = B >= U ? 1 : U / B, size = NQ * PP;
    return size + ((want - size) % U + U) % U;
  }
};

// A cell along one direction: only its first and last nodes can be shared,
// wrapped or constrained.
struct BoxDir {
  int g0, gP;                    // global coordinates of its nodes 0 and P
  bool con0, conP, first0, firstP;
  __device__ __forceinline__ BoxDir(int c, int n, int N, int P, int periodic, int last_odd)
      : g0(c * P), gP(node_coord(c, P, P, N, periodic)), con0(!periodic && c == 0), conP(!periodic && c == n - 1),
        first0(first_along(c, n, 0, P, periodic, last_odd)), firstP(first_along(c, n, P, P, periodic, last_odd)) {}
  __device__ __forceinline__ int at(int i, int P) const { return i == P ? gP : g0 + i; }
  __device__ __forceinline__ bool con(int i, int P) const { return (i == 0 && con0) || (i == P && conP); }
  __device__ __forceinline__ bool first(int i, int P) const { return (i != 0 || first0) && (i != P || firstP); }
};

// N consecutive coefficients, as wide as their alignment (rows of N from an
// aligned base) allows.
template <typename G, int N>
__device__ __forceinline__ void load_row(const G* __restrict__ p, G* c) {
  constexpr int VW = sizeof(G) == 4 && N % 4 == 0 ? 4 : N % 2 == 0 ? 2 : 1;
#pragma unroll
  for (int k = 0; k < N; k += VW) {
    const Pack<G, VW> v = *reinterpret_cast<const Pack<G, VW>*>(p + k);
#pragma unroll
    for (int j = 0; j < VW; ++j) c[k + j] = v.a[j];
  }
}

// One cell e and B groups of W vectors: thread (v, ty) of B x nty threads
// works on group vb B + v.  Switches as in cell_body_eo: SC the scaled
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
  using PK = Pack<D, W>;
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
    if constexpr (MAP) {
#pragma unroll
      for (int i1 = 0; i1 < NP; ++i1) {
        const int code = __ldg(map + (size_t)e * NP * NP * NP + l * NP + i1);
        const bool use = have > 0 && (code & kMapConstrained) == 0;
        u[i1] = use ? A::from(load_pack<D, W>(X + (size_t)(code & kMapIndex) * n_vec + vg, have, vec)) : A::zero();
      }
    } else {
      const bool use = have > 0 && !dy.con(i2, P) && !dz.con(i3, P);
      const size_t row = (dy.at(i2, P) + (size_t)m.Ny * dz.at(i3, P)) * m.Nx;
#pragma unroll
      for (int i1 = 0; i1 < NP; ++i1) {
        const size_t node = row + dx.at(i1, P);
        if (use && !dx.con(i1, P)) {
          PK x = load_pack<D, W>(X + node * n_vec + vg, have, vec);
          if constexpr (SC) {
            const D ms = __ldg(sc.msq + node);
#pragma unroll
            for (int k = 0; k < W; ++k) x.a[k] *= ms;
          }
          u[i1] = A::from(x);
        } else {
          u[i1] = A::zero();
        }
      }
    }
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
    // nodes of the line; the values that a later colour adds to are read
    // before the contraction, and all of them before the first store
    size_t node[NP];
    bool con[NP], first[NP];
    PK old[NP];
    if constexpr (MAP) {
#pragma unroll
      for (int i = 0; i < NP; ++i) {
        const int code = __ldg(map + (size_t)e * NP * NP * NP + (i * NP + i2) * NP + i1);
        node[i] = (size_t)(code & kMapIndex);
        con[i] = (code & kMapConstrained) != 0;
        first[i] = (code & kMapFirst) != 0;
      }
    } else if constexpr (!LOCAL) {
      const size_t col = dx.at(i1, P) + (size_t)m.Nx * dy.at(i2, P), plane = (size_t)m.Nx * m.Ny;
      const bool con_xy = dx.con(i1, P) || dy.con(i2, P), first_xy = dx.first(i1, P) && dy.first(i2, P);
#pragma unroll
      for (int i = 0; i < NP; ++i) {
        node[i] = col + plane * dz.at(i, P);
        con[i] = con_xy || dz.con(i, P);
        first[i] = first_xy && dz.first(i, P);
      }
    }
    if constexpr (!LOCAL) {
#pragma unroll
      for (int i = 0; i < NP; ++i)
        if (!con[i] && (!first[i] || (SC && sc.c != D(0)))) old[i] = load_pack<D, W>(Y + node[i] * n_vec + vg, have, vec);
    }
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
#pragma unroll
      for (int i = 0; i < NP; ++i) {
        PK r = A::to(o[i]);
        if constexpr (SC) {
          // first writer: a M^-1/2 (cell sum) + b X + c Y_old; later ones add
          const D ams = sc.a * __ldg(sc.msq + node[i]);
          PK x;
          if (first[i] && !con[i] && sc.b != D(0)) x = load_pack<D, W>(X + node[i] * n_vec + vg, have, vec);
#pragma unroll
          for (int k = 0; k < W; ++k) {
            r.a[k] *= ams;
            if (first[i] && !con[i] && sc.b != D(0)) r.a[k] += sc.b * x.a[k];
            if (first[i] && !con[i] && sc.c != D(0)) r.a[k] += sc.c * old[i].a[k];
          }
        }
        if (first[i]) {
          if (con[i]) {
#pragma unroll
            for (int k = 0; k < W; ++k) r.a[k] = D(0);
          }
          store_pack<D, W>(Y + node[i] * n_vec + vg, r, have, vec);
        } else if (!con[i]) {
#pragma unroll
          for (int k = 0; k < W; ++k) r.a[k] = old[i].a[k] + r.a[k];
          store_pack<D, W>(Y + node[i] * n_vec + vg, r, have, vec);
        }
      }
    }
  }
}

// Whether a group of W vectors of X and Y can move in one access.
template <typename V>
__host__ __device__ inline bool vec_ok(const void* X, const void* Y, int n_vec) {
  constexpr size_t bytes = sizeof(typename Arith<V>::D) * Arith<V>::W;
  return n_vec % Arith<V>::W == 0 && reinterpret_cast<size_t>(X) % bytes == 0 && reinterpret_cast<size_t>(Y) % bytes == 0;
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

// Lanes (vector groups) x lines of a CTA, and its shared memory: the tile set
// with fe_set_tile, or (want.vb = 0) the default one, whose threads a narrow
// block keeps by taking more lines.
struct BoxShape {
  int lanes, lines;
  size_t smem;
};

template <typename V, int NQ>
BoxShape box_shape(LineTile want, int n_vec) {
  constexpr int W = Arith<V>::W;
  const LineTile t = want.vb > 0 ? want : Arith<V>::box_tile(NQ);
  const int groups = (n_vec + W - 1) / W;
  int b = 1;
  while (b * 2 * W <= t.vb) b *= 2;
  const int lanes0 = b;
  auto bytes = [](int k) { return (size_t)2 * k * BoxTile<NQ>::pitch(k, sizeof(V)) * sizeof(V); };
  while (b > 1 && bytes(b) > 200 * 1024) b /= 2;
  while (b > 1 && b / 2 >= groups) b /= 2;
  int lines = t.lines;
  if (want.vb <= 0 && b < lanes0) lines = std::min(lines * (lanes0 / b), NQ * NQ);
  if (b * lines > 256) lines = 256 / b;
  while ((b * lines) % 32 != 0 && b * lines < 256) ++lines;
  return BoxShape{b, lines, bytes(b)};
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
    // (one vector group per CTA, so even a few cells fill the GPU) writing
    // each cell's result to the scratch, then one gather in colour order.
    if (c->d_small && (size_t)n_vec * NP * NP * NP * c->n_cells * sizeof(D) <= c->small_bytes) {
      auto lk = cell_apply_box_local_kernel<V, NP, NQ>;
      constexpr int lines = NQ * NQ < 64 ? 32 : 64;
      const size_t lsm = (size_t)2 * BoxTile<NQ>::pitch(1, sizeof(V)) * sizeof(V);
      cudaError_t e = ensure_dyn_smem(reinterpret_cast<const void*>(lk), lsm);
      if (e != cudaSuccess) return e;
      D* Wk = static_cast<D*>(c->d_small);
      const int groups = (n_vec + W - 1) / W;
      e = launch_kernel(lk, c->n_cells * (size_t)groups, dim3(1, lines), lsm, s, false, tab, c->mdev, geo, n_vec, groups,
                        vec, X, Wk);
      if (e != cudaSuccess) return e;
      const size_t tot = c->n_dofs * (size_t)n_vec;
      return launch_kernel(assemble_local_kernel<D, NP>, std::min<size_t>((tot + 255) / 256, 152 * 8), dim3(256), 0, s,
                           true, c->mdev, Wk, Y, c->n_dofs, n_vec);
    }
  }
  auto kern = cell_apply_box_kernel<V, NP, NQ, SC, MAP>;
  const BoxShape sh = box_shape<V, NQ>(want, n_vec);
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
