// Launch glue for the CUDA-core cell kernels: one instantiation per
// (p, n_q, geometry kind), selected at run time.
#pragma once

#include <cstdio>

#include "fe_cell_kernel.cuh"

namespace fe {

// The colour launches of one product overlap: a launch made with `overlap` may
// start as soon as every CTA of the one before it has started (programmatic
// dependent launch), and its CTAs gather and contract their cells while the
// earlier colour finishes.  They touch Y only after wait_for_earlier_launch(),
// which returns once the earlier launch has completed (and with it, since
// each launch waits in the same way, all before it).  A product's first
// launch is an ordinary one.
__device__ __forceinline__ void let_next_launch_start() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void wait_for_earlier_launch() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

template <typename... P, typename... Args>
cudaError_t launch_kernel_2d(void (*kern)(P...), dim3 grid, dim3 threads, size_t smem, cudaStream_t s, bool overlap,
                             Args... args) {
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid;
  cfg.blockDim = threads;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cfg.attrs = &at;
  cfg.numAttrs = overlap ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kern, static_cast<P>(args)...);
}

template <typename... P, typename... Args>
cudaError_t launch_kernel(void (*kern)(P...), size_t blocks, dim3 threads, size_t smem, cudaStream_t s, bool overlap,
                          Args... args) {
  if (blocks > 0x7fffffffull) return cudaErrorInvalidConfiguration;
  return launch_kernel_2d(kern, dim3((unsigned)blocks), threads, smem, s, overlap, args...);
}

// A cell along one direction: only its first and last nodes can be shared,
// wrapped or constrained.
struct BoxDir {
  int g0, gP;                    // global coordinates of its nodes 0 and P
  bool con0, conP, first0, firstP, shared0, sharedP;
  __device__ __forceinline__ BoxDir(int c, int n, int N, int P, int periodic, int last_odd)
      : g0(c * P), gP(node_coord(c, P, P, N, periodic)), con0(!periodic && c == 0), conP(!periodic && c == n - 1),
        first0(first_along(c, n, 0, P, periodic, last_odd)), firstP(first_along(c, n, P, P, periodic, last_odd)),
        shared0(c > 0 || periodic), sharedP(c < n - 1 || periodic) {}
  __device__ __forceinline__ int at(int i, int P) const { return i == P ? gP : g0 + i; }
  __device__ __forceinline__ bool con(int i, int P) const { return (i == 0 && con0) || (i == P && conP); }
  __device__ __forceinline__ bool first(int i, int P) const { return (i != 0 || first0) && (i != P || firstP); }
  // whether a second cell of the direction holds the node
  __device__ __forceinline__ bool shared(int i, int P) const { return (i == 0 && shared0) || (i == P && sharedP); }
};

template <typename T, int NP, int NQ>
Tables<T, NP, NQ> make_tables(const fe_ctx* c) {
  Tables<T, NP, NQ> t;
  for (int q = 0; q < NQ; ++q) {
    for (int i = 0; i < NP; ++i) t.N[q][i] = (T)c->Nf[q * NP + i];
    for (int k = 0; k < NQ; ++k) t.D[q][k] = (T)c->Df[q * NQ + k];
  }
  return t;
}

template <typename T>
Geom<T> make_geom(const fe_ctx* c);
template <>
inline Geom<double> make_geom<double>(const fe_ctx* c) {
  return Geom<double>{c->d_cellG64, c->d_ptG64, c->d_ptC64};
}
template <>
inline Geom<float> make_geom<float>(const fe_ctx* c) {
  return Geom<float>{c->d_cellG32, c->d_ptG32, c->d_ptC32};
}
template <>
inline Geom<ff> make_geom<ff>(const fe_ctx* c) {
  return Geom<ff>{c->d_cellGff, c->d_ptGff, c->d_ptCff};
}

// Vectors per CTA: the largest power of two not above `want`, the padded
// n_vec, and what three n_q^3 x B tiles allow in 200 KB of shared memory.
template <typename T, int NQ>
inline int pick_vb(int want, int n_vec) {
  int vb = 1;
  while (vb * 2 <= want) vb *= 2;
  while (vb > 1 && (size_t)3 * NQ * NQ * NQ * vb * sizeof(T) > 200 * 1024) vb /= 2;
  while (vb > 1 && vb / 2 >= n_vec) vb /= 2;
  return vb;
}

template <typename T, int NP, int NQ, bool GEN>
cudaError_t launch_apply(const fe_ctx* c, const T* X, T* Y, int n_vec, cudaStream_t s, int want_vb, int want_lines) {
  const auto kern = cell_apply_kernel<T, NP, NQ, GEN>;
  const int vb = pick_vb<T, NQ>(want_vb, n_vec);
  int nty = want_lines;
  if (vb * nty > 256) nty = 256 / vb;
  while ((vb * nty) % 32 != 0 && vb * nty < 256) ++nty;
  const size_t smem = (size_t)3 * NQ * NQ * NQ * vb * sizeof(T);
  {
    cudaError_t e = ensure_dyn_smem(reinterpret_cast<const void*>(kern), smem);
    if (e != cudaSuccess) return e;
  }
  const Tables<T, NP, NQ> tab = make_tables<T, NP, NQ>(c);
  const Geom<T> geo = make_geom<T>(c);
  const int n_vb = (n_vec + vb - 1) / vb;
  for (int k = 0; k < c->colors.n_colors; ++k) {
    const int n = c->colors.offset[k + 1] - c->colors.offset[k];
    if (n == 0) continue;
    const long long blocks = (long long)n * n_vb;
    if (blocks > 0x7fffffffLL) return cudaErrorInvalidConfiguration;
    kern<<<(unsigned)blocks, dim3(vb, nty), smem, s>>>(tab, c->mdev, geo, c->d_cells + c->colors.offset[k], n_vec, n_vb,
                                                       X, Y);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

template <int NP, int NQ, bool GEN>
cudaError_t launch_diag(const fe_ctx* c, double* diag, cudaStream_t s) {
  const Tables<double, NP, NQ> tab = make_tables<double, NP, NQ>(c);
  const Geom<double> geo = make_geom<double>(c);
  constexpr int NP3 = NP * NP * NP;
  for (int k = 0; k < c->colors.n_colors; ++k) {
    const int n = c->colors.offset[k + 1] - c->colors.offset[k];
    if (n == 0) continue;
    const long long threads = (long long)n * NP3;
    cell_diag_kernel<NP, NQ, GEN><<<(unsigned)((threads + 127) / 128), 128, 0, s>>>(
        tab, c->mdev, geo, c->d_cells + c->colors.offset[k], n, diag);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

}  // namespace fe

// Expands F(P, NQ) for every supported degree and quadrature size.
#define FE_FOR_EACH_P_NQ(F) \
  F(1, 2) F(1, 3) F(1, 4)   \
  F(2, 3) F(2, 4) F(2, 5)   \
  F(3, 4) F(3, 5) F(3, 6)   \
  F(4, 5) F(4, 6) F(4, 7)   \
  F(5, 6) F(5, 7) F(5, 8)   \
  F(6, 7) F(6, 8) F(6, 9)   \
  F(7, 8) F(7, 9) F(7, 10)  \
  F(8, 9) F(8, 10) F(8, 11)
