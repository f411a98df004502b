// Cell kernel of trilinear cells (a symmetric 3 x 3 metric at every point) in
// FP64, FP32 and double-float arithmetic; the other arithmetic and the shared
// pieces are those of the box kernel (fe_arith.cuh, fe_cells.cuh).
//
// Algorithm 2 with the collocation derivative D~: gradients of t = N u along
// the three directions, the metric, the transposed derivatives, N^T.  Each
// direction's values stay apart as (even, odd) parts until the pass that takes
// them to point values, so N is not joined and D~ not split again, and D~ is
// applied in the pass that already holds the line:
//   1 x: N                      2 y: N
//   3 z: N, d2 = D~ t           4 y: d1 = D~ t
//   5 x: d0 = D~ t, metric, c t + D~^T h0
//   6 y: + D~^T h1              7 z: + D~^T h2, N^T
//   8 y: N^T                    9 x: N^T, scatter
// Nine passes on three shared tiles; the quadrature-point operation runs on
// the x-lines, whose metric rows are contiguous in memory.  Before, every
// contraction split and joined its line: ten passes, 89 K operations per cell
// and vector at n_q = 10 against 86.7 K.
//
// Measured, before -> now: FP64 16^3 p = 8, n_q = 10, 256 vectors 190.6 ->
// 184.5 ms (the FP64 pipe: 153 ms at 0.595 T operations/s), 13^3 p = 6, 64
// vectors 11.5 -> 10.2 ms; FP32 (two vectors per thread on packed
// instructions) 13 x 9 x 11 p = 5, 50 vectors 263 -> 169 us; double-float 12^3
// p = 7, 64 vectors 5.2 -> 3.3 ms.
#pragma once

#include "fe_cells.cuh"

namespace fe {

// Tables of the skew matrix D~ for (even, odd) parts: E gives the even parts
// from odd ones, O the odd parts from even ones.
template <typename C, int NQ>
struct SkewTab {
  static constexpr int H = NQ / 2 > 0 ? NQ / 2 : 1, HE = (NQ + 1) / 2;
  C E[HE][H];
  C O[H][HE];
};

template <typename C, int NP, int NQ>
struct GeneralTables {
  EOTab<C, NQ, NP> N;
  EOTab<C, NP, NQ> Nt;
  SkewTab<C, NQ> D;     // parts of values -> parts of values
  SkewTab<C, NQ> Dt;    // D~^T: mirrored sums and differences -> parts of values
  SkewTab<C, NQ> Dtd;   // D~^T: mirrored sums and differences -> the same of the result
};

// out = parts of the skew product of the parts (e, o); with ADD added to out.
template <typename A, int NQ, bool ADD = false>
__device__ __forceinline__ void skew_parts(const SkewTab<typename A::C, NQ>& t, const typename A::V* e,
                                           const typename A::V* o, typename A::V* oe, typename A::V* oo) {
  constexpr int H = NQ / 2, HE = (NQ + 1) / 2;
#pragma unroll
  for (int k = 0; k < HE; ++k) eo_row<A, H, ADD>(t.E[k], o, oe[k]);
#pragma unroll
  for (int k = 0; k < H; ++k) eo_row<A, HE, ADD>(t.O[k], e, oo[k]);
}

template <typename V, int NP, int NQ, bool SC = false, bool LOCAL = false>
__device__ __forceinline__ void cell_body_general(const GeneralTables<typename Arith<V>::C, NP, NQ>& tab,
                                                  const MeshDev& m, const Geom<typename Arith<V>::G>& geo, int e,
                                                  int vb, int B, int v, int ty, int nty, int n_vec, bool vec,
                                                  const typename Arith<V>::D* __restrict__ X,
                                                  typename Arith<V>::D* __restrict__ Y, V* smem,
                                                  const Scale<typename Arith<V>::D>& sc) {
  using A = Arith<V>;
  using G = typename A::G;
  using D = typename A::D;
  using TS = BoxTile<NQ>;
  constexpr int P = NP - 1, RP = TS::RP, PP = TS::PP, W = A::W, NQ3 = NQ * NQ * NQ;
  constexpr int HQ = (NQ + 1) / 2, OQ = NQ / 2, HP = (NP + 1) / 2, OP = NP / 2;
  const int pitch = TS::pitch(B, (int)sizeof(V));
  V* T = smem + v * pitch;
  V* S1 = T + B * pitch;
  V* S2 = S1 + B * pitch;
  const int vg = (vb * B + v) * W;
  const int have = n_vec - vg;   // vectors from this group on (<= 0: none)
  const BoxDir dx(e % m.nx, m.nx, m.Nx, P, m.periodic, m.last_odd_x);
  const BoxDir dy((e / m.nx) % m.ny, m.ny, m.Ny, P, m.periodic, m.last_odd_y);
  const BoxDir dz(e / (m.nx * m.ny), m.nz, m.Nz, P, m.periodic, m.last_odd_z);

  // ---- 1: extraction and x pass of N ----
  for (int l = ty; l < NP * NP; l += nty) {
    const int i2 = l % NP, i3 = l / NP;
    V u[NP], a[NQ], ue[HP], uo[OP];
    gather_line<A, NP, SC>(node_line<A, NP, 0, false>(m, dx, dy, dz, i2, i3, e, nullptr), X, n_vec, vg, have, vec, sc,
                           u);
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
  // ---- 3: z pass of N, gradient along z ----
  for (int l = ty; l < NQ * NQ; l += nty) {
    const int at = (l / NQ) * RP + l % NQ;
    V u[NP], t[NQ], d[NQ], ue[HP], uo[OP];
#pragma unroll
    for (int i = 0; i < NP; ++i) u[i] = T[i * PP + at];
    eo_split<A, NP>(u, ue, uo);
    eo_parts<A, NQ, NP>(tab.N, ue, uo, t);
    skew_parts<A, NQ>(tab.D, t, t + HQ, d, d + HQ);
    eo_join<A, NQ>(t);
    eo_join<A, NQ>(d);
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
      T[q * PP + at] = t[q];
      S2[q * PP + at] = d[q];
    }
  }
  __syncthreads();
  // ---- 4: gradient along y ----
  for (int l = ty; l < NQ * NQ; l += nty) {
    const int at = (l / NQ) * PP + l % NQ;
    V t[NQ], d[NQ];
#pragma unroll
    for (int q = 0; q < NQ; ++q) t[q] = T[q * RP + at];
    skew_parts<A, NQ>(tab.D, t, t + HQ, d, d + HQ);
    eo_join<A, NQ>(t);
    eo_join<A, NQ>(d);
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
      T[q * RP + at] = t[q];
      S1[q * RP + at] = d[q];
    }
#pragma unroll
    for (int q = 0; q < NQ; ++q) d[q] = S2[q * RP + at];
    eo_join<A, NQ>(d);
#pragma unroll
    for (int q = 0; q < NQ; ++q) S2[q * RP + at] = d[q];
  }
  __syncthreads();
  // ---- 5: gradient along x, quadrature-point operation, transposed gradient along x ----
  const G* ptG = geo.ptG + (size_t)e * 6 * NQ3;
  const G* ptC = geo.ptC + (size_t)e * NQ3;
  for (int l = ty; l < NQ * NQ; l += nty) {
    const int at = l * RP;
    V t[NQ], d0[NQ], d1[NQ], d2[NQ], he[HQ], ho[OQ];
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
      t[q] = T[at + q];
      d1[q] = S1[at + q];
      d2[q] = S2[at + q];
    }
    skew_parts<A, NQ>(tab.D, t, t + HQ, d0, d0 + HQ);
    eo_join<A, NQ>(t);
    eo_join<A, NQ>(d0);
    eo_join<A, NQ>(d1);
    eo_join<A, NQ>(d2);
    const G* pg = ptG + l * NQ;
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
      const G g00 = pg[q], g01 = pg[NQ3 + q], g02 = pg[2 * NQ3 + q], g11 = pg[3 * NQ3 + q], g12 = pg[4 * NQ3 + q],
              g22 = pg[5 * NQ3 + q];
      typename A::Acc a0 = A::first(g00, d0[q]), a1 = A::first(g01, d0[q]), a2 = A::first(g02, d0[q]);
      A::fma(a0, g01, d1[q]);
      A::fma(a1, g11, d1[q]);
      A::fma(a2, g12, d1[q]);
      A::fma(a0, g02, d2[q]);
      A::fma(a1, g12, d2[q]);
      A::fma(a2, g22, d2[q]);
      d0[q] = A::value(a0);
      S1[at + q] = A::value(a1);
      S2[at + q] = A::value(a2);
    }
    eo_split<A, NQ>(d0, he, ho);
    skew_parts<A, NQ>(tab.Dt, he, ho, d1, d1 + HQ);
    eo_join<A, NQ>(d1);
    G c[NQ];
    load_row<G, NQ>(ptC + l * NQ, c);
#pragma unroll
    for (int q = 0; q < NQ; ++q) T[at + q] = A::muladd(c[q], t[q], d1[q]);
  }
  __syncthreads();
  // ---- 6: transposed gradient along y ----
  for (int l = ty; l < NQ * NQ; l += nty) {
    const int at = (l / NQ) * PP + l % NQ;
    V h[NQ], he[HQ], ho[OQ], o[NQ];
#pragma unroll
    for (int q = 0; q < NQ; ++q) h[q] = S1[q * RP + at];
    eo_split<A, NQ>(h, he, ho);
    skew_parts<A, NQ>(tab.Dt, he, ho, o, o + HQ);
    eo_join<A, NQ>(o);
#pragma unroll
    for (int q = 0; q < NQ; ++q) T[q * RP + at] = A::add(T[q * RP + at], o[q]);
  }
  __syncthreads();
  // ---- 7: transposed gradient along z, z pass of N^T ----
  for (int l = ty; l < NQ * NQ; l += nty) {
    const int at = (l / NQ) * RP + l % NQ;
    V h[NQ], he[HQ], ho[OQ], te[HQ], to[OQ], o[NP];
#pragma unroll
    for (int q = 0; q < NQ; ++q) h[q] = T[q * PP + at];
    eo_split<A, NQ>(h, te, to);
#pragma unroll
    for (int q = 0; q < NQ; ++q) h[q] = S2[q * PP + at];
    eo_split<A, NQ>(h, he, ho);
    skew_parts<A, NQ, true>(tab.Dtd, he, ho, te, to);
    eo_parts<A, NP, NQ>(tab.Nt, te, to, o);
    eo_join<A, NP>(o);
#pragma unroll
    for (int i = 0; i < NP; ++i) T[i * PP + at] = o[i];
  }
  __syncthreads();
  // ---- 8: y pass of N^T ----
  for (int l = ty; l < NQ * NP; l += nty) {
    V* line = T + (l / NQ) * PP + l % NQ;
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
  // ---- 9: x pass of N^T and assembly ----
  if constexpr (!LOCAL) wait_for_earlier_launch();
  if (have <= 0) return;
  for (int l = ty; l < NP * NP; l += nty) {
    const int i2 = l % NP, i3 = l / NP;
    const NodeLine<A, NP> nodes = node_line<A, NP, 0, false>(m, dx, dy, dz, i2, i3, e, nullptr);
    Pack<D, W> old[NP];
    if constexpr (!LOCAL) read_old<A, NP, SC>(nodes, Y, n_vec, vg, have, vec, sc, old);
    V h[NQ], he[HQ], ho[OQ], o[NP];
    const V* src = T + i3 * PP + i2 * RP;
#pragma unroll
    for (int q = 0; q < NQ; ++q) h[q] = src[q];
    eo_split<A, NQ>(h, he, ho);
    eo_parts<A, NP, NQ>(tab.Nt, he, ho, o);
    eo_join<A, NP>(o);
    if constexpr (LOCAL) {
      D* w = Y + ((size_t)e * NP * NP * NP + (size_t)l * NP) * n_vec + vg;
#pragma unroll
      for (int i = 0; i < NP; ++i) store_pack<D, W>(w + (size_t)i * n_vec, A::to(o[i]), have, vec);
    } else {
      scatter_line<A, NP, SC>(nodes, o, old, X, Y, n_vec, vg, have, vec, sc);
    }
  }
}

template <typename V, int NP, int NQ, bool SC>
__global__ void __launch_bounds__(256) cell_apply_general_kernel(
    const GeneralTables<typename Arith<V>::C, NP, NQ> tab, const MeshDev m, const Geom<typename Arith<V>::G> geo,
    const int* __restrict__ cells, int n_vec, int n_vb, bool vec, const typename Arith<V>::D* __restrict__ X,
    typename Arith<V>::D* __restrict__ Y, const Scale<typename Arith<V>::D> sc) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  let_next_launch_start();
  cell_body_general<V, NP, NQ, SC>(tab, m, geo, cells[blockIdx.x / n_vb], blockIdx.x % n_vb, blockDim.x, threadIdx.x,
                                   threadIdx.y, blockDim.y, n_vec, vec, X, Y, reinterpret_cast<V*>(smem_raw), sc);
}

// Small meshes: every cell in one launch, results to the per-cell scratch.
template <typename V, int NP, int NQ>
__global__ void __launch_bounds__(256) cell_apply_general_local_kernel(
    const GeneralTables<typename Arith<V>::C, NP, NQ> tab, const MeshDev m, const Geom<typename Arith<V>::G> geo,
    int n_vec, int n_vb, bool vec, const typename Arith<V>::D* __restrict__ X, typename Arith<V>::D* __restrict__ Wk) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  let_next_launch_start();
  cell_body_general<V, NP, NQ, false, true>(tab, m, geo, blockIdx.x / n_vb, blockIdx.x % n_vb, blockDim.x, threadIdx.x,
                                            threadIdx.y, blockDim.y, n_vec, vec, X, Wk,
                                            reinterpret_cast<V*>(smem_raw), Scale<typename Arith<V>::D>{});
}

// Host: tables of the skew matrix M (rows o, columns i).  `in` and `out` say
// what a part stands for on that side: 1 = a value's part (v = e +- o), 2 =
// the mirrored sums and differences of the values, twice the part.
template <typename C, int NQ>
void make_skewtab(SkewTab<C, NQ>& t, const double* M, int in, int out) {
  constexpr int H = NQ / 2, HE = (NQ + 1) / 2;
  for (int o = 0; o < HE; ++o)
    for (int i = 0; i < H; ++i) {
      const double f = (in == 1 ? 1.0 : 0.5) * (out == 2 && o < H ? 2.0 : 1.0);
      t.E[o][i] = (C)(f * (M[o * NQ + i] - M[o * NQ + NQ - 1 - i]));
    }
  for (int o = 0; o < H; ++o) {
    const double g = out == 2 ? 2.0 : 1.0;
    for (int i = 0; i < H; ++i) t.O[o][i] = (C)(g * (in == 1 ? 1.0 : 0.5) * (M[o * NQ + i] + M[o * NQ + NQ - 1 - i]));
    if (HE > H) t.O[o][H] = (C)(g * M[o * NQ + H]);
  }
}

template <typename C, int NP, int NQ>
GeneralTables<C, NP, NQ> make_generaltables(const fe_ctx* c) {
  GeneralTables<C, NP, NQ> t;
  double Nt[NP * NQ], Dt[NQ * NQ];
  for (int q = 0; q < NQ; ++q) {
    for (int i = 0; i < NP; ++i) Nt[i * NQ + q] = c->Nf[q * NP + i];
    for (int k = 0; k < NQ; ++k) Dt[k * NQ + q] = c->Df[q * NQ + k];
  }
  make_eotab(t.N, c->Nf.data());
  make_eotab(t.Nt, Nt);
  make_skewtab(t.D, c->Df.data(), 1, 1);
  make_skewtab(t.Dt, Dt, 2, 1);
  make_skewtab(t.Dtd, Dt, 2, 2);
  return t;
}

template <typename V, int NP, int NQ, bool SC = false>
cudaError_t launch_general(const fe_ctx* c, const typename Arith<V>::D* X, typename Arith<V>::D* Y, int n_vec,
                           cudaStream_t s, LineTile want, const Geom<typename Arith<V>::G>& geo,
                           const Scale<typename Arith<V>::D>& sc = Scale<typename Arith<V>::D>{}) {
  using D = typename Arith<V>::D;
  constexpr int W = Arith<V>::W;
  const bool vec = vec_ok<V>(X, Y, n_vec);
  const auto tab = make_generaltables<typename Arith<V>::C, NP, NQ>(c);
  if constexpr (!SC) {   // small meshes, as in launch_box
    const bool fits = (size_t)n_vec * NP * NP * NP * c->n_cells * sizeof(D) <= c->small.bytes();
    if (void* scratch = fits ? c->small.block(s) : nullptr) {
      auto lk = cell_apply_general_local_kernel<V, NP, NQ>;
      int lanes = 1;
      size_t lsm = 0;
      cudaError_t e = small_shape<V, NQ, 3>(c->n_cells, n_vec, &lanes, &lsm);
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
  auto kern = cell_apply_general_kernel<V, NP, NQ, SC>;
  const BoxShape sh = box_shape<V, NQ, 3>(want, Arith<V>::general_tile(NQ), n_vec);
  cudaError_t e = ensure_dyn_smem(reinterpret_cast<const void*>(kern), sh.smem);
  if (e != cudaSuccess) return e;
  const int n_vb = (n_vec + sh.lanes * W - 1) / (sh.lanes * W);
  bool overlap = false;
  for (int k = 0; k < c->colors.n_colors; ++k) {
    const int n = c->colors.offset[k + 1] - c->colors.offset[k];
    if (n == 0) continue;
    e = launch_kernel(kern, (size_t)n * n_vb, dim3(sh.lanes, sh.lines), sh.smem, s, overlap, tab, c->mdev, geo,
                      c->d_cells + c->colors.offset[k], n_vec, n_vb, vec, X, Y, sc);
    if (e != cudaSuccess) return e;
    overlap = true;
  }
  return cudaSuccess;
}

}  // namespace fe
