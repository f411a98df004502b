// What the cell kernels share (box cells: fe_box.cuh, trilinear cells:
// fe_general.cuh): 1D contractions in even-odd form, the shared-memory shape,
// the gather of X and the colour-ordered scatter into Y.
//
// Even-odd decomposition.  The 1D matrices are (skew-)centrosymmetric: GLL
// nodes and the quadrature points are symmetric about 0, so N(n_q-1-q, n_p-1-i)
// = N(q, i) and D~(n_q-1-q, n_q-1-k) = -D~(q, k); folding sqrt(w) keeps both
// symmetries.  A line's values are then split into (even, odd) parts,
//   e_i = in_i + in_{n-1-i},  o_i = in_i - in_{n-1-i},
// which such a matrix does not mix: half the multiply-adds of the plain
// product, plus the sums that split and join (the paper's scheme for its CPU
// kernels, Sec. 3.2.4; it kept the plain form on V100 because of warp stalls --
// on GB300 the FP64 pipe is the bound, so the saved operations are the saved
// time).  Transposed products use the tables of M^T, which has the same symmetry.
#pragma once

#include <algorithm>
#include <type_traits>

#include "fe_arith.cuh"
#include "fe_dispatch.cuh"

namespace fe {

// Tables of out = M in for an NO x NI matrix M with M(NO-1-o, NI-1-i) = S M(o, i).
template <typename T, int NO, int NI>
struct EOTab {
  static constexpr int HO = (NO + 1) / 2;   // outputs computed directly
  static constexpr int HE = (NI + 1) / 2;   // even inputs (with the middle one)
  static constexpr int HOD = NI / 2 > 0 ? NI / 2 : 1;
  T E[HO][HE];
  T O[HO][HOD];
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
// error of a p = 6 product was 1.2e-14 this way, 1.4e-14 the other, with the
// stiffness as one matrix).  FP64
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

template <typename A, int NO, int NI>
__device__ __forceinline__ void eo_parts(const EOTab<typename A::C, NO, NI>& t, const typename A::V* e,
                                         const typename A::V* o, typename A::V* out) {
  constexpr int HI = NI / 2, HE = (NI + 1) / 2, HO = (NO + 1) / 2;
#pragma unroll
  for (int k = 0; k < HO; ++k) eo_row<A, HE, false>(t.E[k], e, out[k]);
#pragma unroll
  for (int k = 0; k < NO / 2; ++k) {
    if constexpr (HI > 0) eo_row<A, HI, false>(t.O[k], o, out[HO + k]);
    else out[HO + k] = A::zero();
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

// Y rows of one line of n_p nodes, or X values of it.
template <typename A, int NP>
struct NodeLine {
  size_t node[NP];
  bool con[NP], first[NP];
};

// Nodes of the x-line (i2, i3) (DIR 0) or the z-line (i1, i2) (DIR 2) of a cell.
template <typename A, int NP, int DIR, bool MAP>
__device__ __forceinline__ NodeLine<A, NP> node_line(const MeshDev& m, const BoxDir& dx, const BoxDir& dy,
                                                     const BoxDir& dz, int a, int b, int e,
                                                     const int* __restrict__ map) {
  constexpr int P = NP - 1;
  NodeLine<A, NP> n;
  if constexpr (MAP) {
#pragma unroll
    for (int i = 0; i < NP; ++i) {
      const int local = DIR == 0 ? (b * NP + a) * NP + i : (i * NP + b) * NP + a;
      const int code = __ldg(map + (size_t)e * NP * NP * NP + local);
      n.node[i] = (size_t)(code & kMapIndex);
      n.con[i] = (code & kMapConstrained) != 0;
      n.first[i] = (code & kMapFirst) != 0;
    }
  } else {
    const BoxDir& d = DIR == 0 ? dx : dz;     // along the line
    const BoxDir& da = DIR == 0 ? dy : dx;    // index a
    const BoxDir& db = DIR == 0 ? dz : dy;    // index b
    const size_t Nx = m.Nx, plane = (size_t)m.Nx * m.Ny, step = DIR == 0 ? 1 : plane;
    const size_t base = DIR == 0 ? Nx * da.at(a, P) + plane * db.at(b, P) : da.at(a, P) + Nx * db.at(b, P);
    const bool con = da.con(a, P) || db.con(b, P), first = da.first(a, P) && db.first(b, P);
#pragma unroll
    for (int i = 0; i < NP; ++i) {
      n.node[i] = base + step * d.at(i, P);
      n.con[i] = con || d.con(i, P);
      n.first[i] = first && d.first(i, P);
    }
  }
  return n;
}

// X on a line (constrained nodes read as 0; SC: times M^-1/2).
template <typename A, int NP, bool SC>
__device__ __forceinline__ void gather_line(const NodeLine<A, NP>& n, const typename A::D* __restrict__ X, int n_vec,
                                            int vg, int have, bool vec, const Scale<typename A::D>& sc,
                                            typename A::V* u) {
  constexpr int W = A::W;
#pragma unroll
  for (int i = 0; i < NP; ++i) {
    if (have > 0 && !n.con[i]) {
      Pack<typename A::D, W> x = load_pack<typename A::D, W>(X + n.node[i] * n_vec + vg, have, vec);
      if constexpr (SC) {
        const typename A::D ms = __ldg(sc.msq + n.node[i]);
#pragma unroll
        for (int k = 0; k < W; ++k) x.a[k] *= ms;
      }
      u[i] = A::from(x);
    } else {
      u[i] = A::zero();
    }
  }
}

// The values of Y that this cell adds to (a later colour than the node's
// first, or the c Y term of the scaled product): read before the line's last
// contraction, and all of them before the first store.
template <typename A, int NP, bool SC>
__device__ __forceinline__ void read_old(const NodeLine<A, NP>& n, const typename A::D* Y, int n_vec, int vg, int have,
                                         bool vec, const Scale<typename A::D>& sc, Pack<typename A::D, A::W>* old) {
  using D = typename A::D;
#pragma unroll
  for (int i = 0; i < NP; ++i)
    if (!n.con[i] && (!n.first[i] || (SC && sc.c != D(0))))
      old[i] = load_pack<D, A::W>(Y + n.node[i] * n_vec + vg, have, vec);
}

// Colour-ordered assembly of a line: the node's first colour stores (0 on
// constrained nodes), later ones add.  SC: the first writer stores
// a M^-1/2 (cell sum) + b X + c Y_old, later ones add their a M^-1/2 (cell sum).
template <typename A, int NP, bool SC>
__device__ __forceinline__ void scatter_line(const NodeLine<A, NP>& n, const typename A::V* o,
                                             const Pack<typename A::D, A::W>* old, const typename A::D* __restrict__ X,
                                             typename A::D* Y, int n_vec, int vg, int have, bool vec,
                                             const Scale<typename A::D>& sc) {
  using D = typename A::D;
  constexpr int W = A::W;
#pragma unroll
  for (int i = 0; i < NP; ++i) {
    Pack<D, W> r = A::to(o[i]);
    if constexpr (SC) {
      const D ams = sc.a * __ldg(sc.msq + n.node[i]);
      const bool own = n.first[i] && !n.con[i];
      Pack<D, W> x;
      if (own && sc.b != D(0)) x = load_pack<D, W>(X + n.node[i] * n_vec + vg, have, vec);
#pragma unroll
      for (int k = 0; k < W; ++k) {
        r.a[k] *= ams;
        if (own && sc.b != D(0)) r.a[k] += sc.b * x.a[k];
        if (own && sc.c != D(0)) r.a[k] += sc.c * old[i].a[k];
      }
    }
    if (n.first[i]) {
      if (n.con[i]) {
#pragma unroll
        for (int k = 0; k < W; ++k) r.a[k] = D(0);
      }
      store_pack<D, W>(Y + n.node[i] * n_vec + vg, r, have, vec);
    } else if (!n.con[i]) {
#pragma unroll
      for (int k = 0; k < W; ++k) r.a[k] = old[i].a[k] + r.a[k];
      store_pack<D, W>(Y + n.node[i] * n_vec + vg, r, have, vec);
    }
  }
}

// Whether a group of W vectors of X and Y can move in one access.
template <typename V>
__host__ __device__ inline bool vec_ok(const void* X, const void* Y, int n_vec) {
  constexpr size_t bytes = sizeof(typename Arith<V>::D) * Arith<V>::W;
  return n_vec % Arith<V>::W == 0 && reinterpret_cast<size_t>(X) % bytes == 0 && reinterpret_cast<size_t>(Y) % bytes == 0;
}

// CTA of a small mesh: every line of a pass has a thread, and B vector groups
// share a CTA, B chosen so that the fullest SM has the fewest warps: with few
// cells a CTA's time is its passes' latency, and partly filled warps cost the
// FP64 pipe as much as full ones (4^3 cells, n_q = 6, 8 vectors: 128 CTAs of 4 x
// 36 threads put 5 warps on an SM, 512 CTAs of one 36-line vector put 8).
template <typename V, int NQ, int TILES>
cudaError_t small_shape(size_t cells, int n_vec, int* lanes, size_t* smem) {
  int dev = 0, sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  const int groups = (n_vec + Arith<V>::W - 1) / Arith<V>::W;
  size_t best = 0;
  *lanes = 1;
  for (int b = 1; b == 1 || (b * NQ * NQ <= 256 && b / 2 < groups); b *= 2) {
    const size_t bytes = (size_t)TILES * b * BoxTile<NQ>::pitch(b, sizeof(V)) * sizeof(V);
    if (bytes > 100 * 1024 && b > 1) break;
    const size_t ctas = cells * ((groups + b - 1) / b);
    const size_t cost = (ctas + sms - 1) / sms * ((b * NQ * NQ + 31) / 32);
    if (best == 0 || cost < best) {
      best = cost;
      *lanes = b;
      *smem = bytes;
    }
  }
  return cudaSuccess;
}

// Lanes (vector groups) x lines of a CTA, and its shared memory: the tile set
// with fe_set_tile, or (want.vb = 0) the default one, whose threads a narrow
// block keeps by taking more lines.
struct BoxShape {
  int lanes, lines;
  size_t smem;
};

template <typename V, int NQ, int TILES>
BoxShape box_shape(LineTile want, LineTile usual, int n_vec) {
  constexpr int W = Arith<V>::W;
  const LineTile t = want.vb > 0 ? want : usual;
  const int groups = (n_vec + W - 1) / W;
  int b = 1;
  while (b * 2 * W <= t.vb) b *= 2;
  const int lanes0 = b;
  auto bytes = [](int k) { return (size_t)TILES * k * BoxTile<NQ>::pitch(k, sizeof(V)) * sizeof(V); };
  while (b > 1 && bytes(b) > 200 * 1024) b /= 2;
  while (b > 1 && b / 2 >= groups) b /= 2;
  int lines = t.lines;
  if (want.vb <= 0 && b < lanes0) lines = std::min(lines * (lanes0 / b), NQ * NQ);
  if (b * lines > 256) lines = 256 / b;
  while ((b * lines) % 32 != 0 && b * lines < 256) ++lines;
  return BoxShape{b, lines, bytes(b)};
}

// The cells sharing a node along one direction (one, or two at a cell
// boundary), as (cell coordinate, local index), ordered by the direction's
// cell colour.
__device__ __forceinline__ int node_cells(int g, int n, int P, int periodic, int last_odd, int* c, int* l) {
  int k;
  if (periodic) {
    c[0] = g / P;
    l[0] = g - c[0] * P;
    k = 1;
    if (l[0] == 0) { c[1] = c[0] > 0 ? c[0] - 1 : n - 1; l[1] = P; k = 2; }
  } else {
    c[0] = g / P < n - 1 ? g / P : n - 1;
    l[0] = g - c[0] * P;
    k = 1;
    if (l[0] == 0 && c[0] > 0) { c[1] = c[0] - 1; l[1] = P; k = 2; }
  }
  if (k == 2 && dir_color(c[1], n, last_odd) < dir_color(c[0], n, last_odd)) {
    int t = c[0]; c[0] = c[1]; c[1] = t;
    t = l[0]; l[0] = l[1]; l[1] = t;
  }
  return k;
}

// Y[dof][v] = sum over the cells sharing dof of W[cell][local][v], added in
// ascending cell colour (z colour slowest, x fastest), which is the order of
// the colour-ordered launches: the result equals theirs bit for bit.
// Dirichlet rows are 0.
template <typename T, int NP>
__global__ void assemble_local_kernel(const MeshDev m, const T* __restrict__ W, T* __restrict__ Y, size_t n_dofs,
                                      int n_vec) {
  constexpr int P = NP - 1, NP3 = NP * NP * NP;
  const size_t total = n_dofs * n_vec;
  wait_for_earlier_launch();
  for (size_t idx = blockIdx.x * (size_t)blockDim.x + threadIdx.x; idx < total;
       idx += (size_t)gridDim.x * blockDim.x) {
    const size_t dof = idx / n_vec;
    const int v = (int)(idx - dof * n_vec);
    const int gx = (int)(dof % m.Nx), gy = (int)((dof / m.Nx) % m.Ny), gz = (int)(dof / ((size_t)m.Nx * m.Ny));
    if (on_boundary(gx, m.Nx, m.periodic) || on_boundary(gy, m.Ny, m.periodic) ||
        on_boundary(gz, m.Nz, m.periodic)) {
      Y[idx] = T(0);
      continue;
    }
    int cx[2], lx[2], cy[2], ly[2], cz[2], lz[2];
    const int kx = node_cells(gx, m.nx, P, m.periodic, m.last_odd_x, cx, lx);
    const int ky = node_cells(gy, m.ny, P, m.periodic, m.last_odd_y, cy, ly);
    const int kz = node_cells(gz, m.nz, P, m.periodic, m.last_odd_z, cz, lz);
    T acc = T(0);
    bool first = true;
    for (int a = 0; a < kz; ++a)
      for (int b = 0; b < ky; ++b)
        for (int d = 0; d < kx; ++d) {
          const size_t e = cx[d] + (size_t)m.nx * (cy[b] + (size_t)m.ny * cz[a]);
          const T val = W[(e * NP3 + (lz[a] * NP + ly[b]) * NP + lx[d]) * n_vec + v];
          acc = first ? val : acc + val;
          first = false;
        }
    Y[idx] = acc;
  }
}

// Host: even-odd tables of an NO x NI row-major matrix M with symmetry S.
template <typename T, int NO, int NI>
void make_eotab(EOTab<T, NO, NI>& t, const double* M) {
  constexpr int HI = NI / 2, HO = (NO + 1) / 2, HE = (NI + 1) / 2;
  for (int o = 0; o < HO; ++o) {
    for (int i = 0; i < HI; ++i) {
      t.E[o][i] = (T)(0.5 * (M[o * NI + i] + M[o * NI + NI - 1 - i]));
      t.O[o][i] = (T)(0.5 * (M[o * NI + i] - M[o * NI + NI - 1 - i]));
    }
    if (HE > HI) t.E[o][HI] = (T)M[o * NI + HI];
  }
}


}  // namespace fe
