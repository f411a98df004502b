// The product on refined meshes with hanging nodes (Sec. 3.2.2):
//   1. distribute: Xc = X with every slave row replaced by sum_m w_sm X_m
//      (u_S = W u_M; Dirichlet masters are already dropped from W);
//   2. the cell kernels with the explicit cell -> DoF map, colour by colour,
//      on Xc (first writers store, later colours add, Dirichlet rows 0);
//   3. condense: Y_m += sum_s w_sm Y_s for every master m (master rows, no
//      write conflicts);
//   4. slave rows of Y set to 0.
// Together Y = C^T A C X on the free rows, 0 on slave and Dirichlet rows.
#include "fe_dispatch.cuh"
#include "fe_box.cuh"

namespace fe {

namespace {

template <typename T, typename W>
__global__ void distribute_kernel(const T* __restrict__ X, T* __restrict__ Xc, const int* __restrict__ row_slave,
                                  const int* __restrict__ ptr, const int* __restrict__ idx, const W* __restrict__ w,
                                  size_t n, int nv) {
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n * nv; i += (size_t)gridDim.x * blockDim.x) {
    const size_t r = i / nv;
    const int v = (int)(i - r * nv);
    const int s = __ldg(row_slave + r);
    if (s < 0) {
      Xc[i] = X[i];
      continue;
    }
    T acc = T(0);
    for (int k = __ldg(ptr + s); k < __ldg(ptr + s + 1); ++k) acc += (T)__ldg(w + k) * X[(size_t)__ldg(idx + k) * nv + v];
    Xc[i] = acc;
  }
}

template <typename T, typename W>
__global__ void condense_kernel(T* __restrict__ Y, const int* __restrict__ rows, const int* __restrict__ ptr,
                                const int* __restrict__ idx, const W* __restrict__ w, int n_rows, int nv) {
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < (size_t)n_rows * nv;
       i += (size_t)gridDim.x * blockDim.x) {
    const int j = (int)(i / nv), v = (int)(i - (size_t)j * nv);
    T acc = T(0);
    for (int k = __ldg(ptr + j); k < __ldg(ptr + j + 1); ++k) acc += (T)__ldg(w + k) * Y[(size_t)__ldg(idx + k) * nv + v];
    Y[(size_t)__ldg(rows + j) * nv + v] += acc;
  }
}

template <typename T>
__global__ void zero_rows_kernel(T* __restrict__ Y, const int* __restrict__ rows, int n_rows, int nv) {
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < (size_t)n_rows * nv;
       i += (size_t)gridDim.x * blockDim.x) {
    const int j = (int)(i / nv), v = (int)(i - (size_t)j * nv);
    Y[(size_t)__ldg(rows + j) * nv + v] = T(0);
  }
}

cudaError_t cells_refined(const fe_ctx* c, const void* X, void* Y, int n_vec, cudaStream_t s) {
#define FE_CASE(P, NQ)                                                                                       \
  if (c->p == P && c->nq == NQ) {                                                                            \
    if (c->mode == FE_FP32)                                                                                  \
      return launch_box<F2, P + 1, NQ, false, true>(c, static_cast<const float*>(X), static_cast<float*>(Y), \
                                                       n_vec, s, c->tile32(), make_geom<float>(c));            \
    const double* X64 = static_cast<const double*>(X);                                                       \
    double* Y64 = static_cast<double*>(Y);                                                                   \
    return c->mode == FE_FP64                                                                                \
               ? launch_box<double, P + 1, NQ, false, true>(c, X64, Y64, n_vec, s, c->tile64(),               \
                                                            make_geom<double>(c))                            \
               : launch_box<ff, P + 1, NQ, false, true>(c, X64, Y64, n_vec, s, c->tiledf(), make_geom<ff>(c)); \
  }
  FE_FOR_EACH_P_NQ(FE_CASE)
#undef FE_CASE
  return cudaErrorInvalidValue;
}

template <typename T, typename W>
cudaError_t constrained(fe_ctx* c, const void* X, void* Y, int n_vec, cudaStream_t s, const W* sl_w, const W* ma_w,
                        void* xc) {
  const size_t n = c->n_dofs, tot = n * (size_t)n_vec;
  const void* Xin = X;
  if (c->n_slaves > 0) {
    const size_t bytes = tot * sizeof(T);
    if (!xc && c->xc_bytes < bytes) {
      cudaFree(c->d_xc);
      c->d_xc = nullptr;
      c->xc_bytes = 0;
      cudaError_t e = cudaMalloc(&c->d_xc, bytes);
      if (e != cudaSuccess) return e;
      c->xc_bytes = bytes;
    }
    if (!xc) xc = c->d_xc;
    const unsigned grid = (unsigned)std::min<size_t>((tot + 255) / 256, 152 * 16);
    distribute_kernel<T, W><<<grid, 256, 0, s>>>(static_cast<const T*>(X), static_cast<T*>(xc), c->d_row_slave,
                                                 c->d_sl_ptr, c->d_sl_idx, sl_w, n, n_vec);
    Xin = xc;
  }
  cudaError_t e = cells_refined(c, Xin, Y, n_vec, s);
  if (e != cudaSuccess) return e;
  if (c->n_masters > 0) {
    const size_t t = (size_t)c->n_masters * n_vec;
    condense_kernel<T, W><<<(unsigned)std::min<size_t>((t + 255) / 256, 152 * 16), 256, 0, s>>>(
        static_cast<T*>(Y), c->d_ma_rows, c->d_ma_ptr, c->d_ma_idx, ma_w, c->n_masters, n_vec);
  }
  if (c->n_slaves > 0) {
    const size_t t = (size_t)c->n_slaves * n_vec;
    zero_rows_kernel<T><<<(unsigned)std::min<size_t>((t + 255) / 256, 152 * 16), 256, 0, s>>>(
        static_cast<T*>(Y), c->d_slaves, c->n_slaves, n_vec);
  }
  return cudaGetLastError();
}

}  // namespace

cudaError_t apply_refined(fe_ctx* c, const void* X, void* Y, int n_vec, cudaStream_t s, void* xc_scratch) {
  if (c->mode == FE_FP32) return constrained<float, float>(c, X, Y, n_vec, s, c->d_sl_w32, c->d_ma_w32, xc_scratch);
  return constrained<double, double>(c, X, Y, n_vec, s, c->d_sl_w, c->d_ma_w, xc_scratch);
}

}  // namespace fe
