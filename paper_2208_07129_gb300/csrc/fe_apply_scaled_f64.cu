// FP64 instantiations of the scaled product of the Chebyshev filter,
// Y = a M^-1/2 A M^-1/2 X + b X + c Y (box and trilinear kernels).
#include "fe_dispatch.cuh"
#include "fe_box.cuh"
#include "fe_general.cuh"

namespace fe {

cudaError_t apply_scaled_f64(const fe_ctx* c, const double* X, double* Y, int n_vec, const Scale<double>& sc,
                             cudaStream_t s) {
#define FE_CASE(P, NQ)                                                                                        \
  if (c->p == P && c->nq == NQ)                                                                         \
    return c->general ? launch_general<double, P + 1, NQ, true>(c, X, Y, n_vec, s, c->tile64(), make_geom<double>(c), sc) \
                      : launch_box<double, P + 1, NQ, true>(c, X, Y, n_vec, s, c->tile64(), make_geom<double>(c), sc);
  FE_FOR_EACH_P_NQ(FE_CASE)
#undef FE_CASE
  return cudaErrorInvalidValue;
}

}  // namespace fe
