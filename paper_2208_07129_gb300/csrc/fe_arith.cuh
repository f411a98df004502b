// Arithmetic of the box-cell kernel (fe_box.cuh), one struct per value type.
// A thread works on values of type V (W vectors of the block per thread), the
// 1D coefficients are of type C, and D is the element type of X and Y in
// global memory.  Every operation is an explicitly rounded one, so the
// compiler neither contracts nor reassociates and every instantiation of the
// body (launch per colour, small meshes, batch) gives the same bits.
#pragma once

#include <cuda_runtime.h>

#include "fe_ff.cuh"

namespace fe {

template <typename V>
struct Arith;

template <>
struct Arith<double> {
  using V = double;
  using C = double;
  using D = double;
  using Acc = double;
  static constexpr int W = 1;
  static constexpr bool kSumApart = false;   // see eo_row
  static __device__ __forceinline__ V zero() { return 0.0; }
  static __device__ __forceinline__ V add(V a, V b) { return __dadd_rn(a, b); }
  static __device__ __forceinline__ V sub(V a, V b) { return __dsub_rn(a, b); }
  static __device__ __forceinline__ Acc first(C c, V v) { return __dmul_rn(c, v); }
  static __device__ __forceinline__ Acc init(V v) { return v; }
  static __device__ __forceinline__ void fma(Acc& a, C c, V v) { a = __fma_rn(c, v, a); }
  static __device__ __forceinline__ V value(Acc a) { return a; }
  // g s + c v: the middle point of an odd rule
  static __device__ __forceinline__ V point(C c, V v, C g, V s) { return __fma_rn(g, s, __dmul_rn(c, v)); }
  // e = c1 v1 + c2 v2 + g se,  o = c1 v1 - c2 v2 + g so
  static __device__ __forceinline__ void point_pair(C c1, V v1, C c2, V v2, C g, V se, V so, V& e, V& o) {
    const V m = __dmul_rn(c2, v2);
    e = __fma_rn(g, se, __fma_rn(c1, v1, m));
    o = __fma_rn(g, so, __fma_rn(c1, v1, -m));
  }
  static __device__ __forceinline__ C twice(C g) { return 2.0 * g; }
  static __device__ __forceinline__ V load(const D* p, int) { return __ldg(p); }
  static __device__ __forceinline__ V scale(V v, D m) { return __dmul_rn(v, m); }
  static __device__ __forceinline__ D get(V v, int) { return v; }
};

template <>
struct Arith<float> {
  using V = float;
  using C = float;
  using D = float;
  using Acc = float;
  static constexpr int W = 1;
  static constexpr bool kSumApart = true;   // see eo_row
  static __device__ __forceinline__ V zero() { return 0.f; }
  static __device__ __forceinline__ V add(V a, V b) { return __fadd_rn(a, b); }
  static __device__ __forceinline__ V sub(V a, V b) { return __fsub_rn(a, b); }
  static __device__ __forceinline__ Acc first(C c, V v) { return __fmul_rn(c, v); }
  static __device__ __forceinline__ Acc init(V v) { return v; }
  static __device__ __forceinline__ void fma(Acc& a, C c, V v) { a = __fmaf_rn(c, v, a); }
  static __device__ __forceinline__ V value(Acc a) { return a; }
  static __device__ __forceinline__ V point(C c, V v, C g, V s) { return __fmaf_rn(g, s, __fmul_rn(c, v)); }
  static __device__ __forceinline__ void point_pair(C c1, V v1, C c2, V v2, C g, V se, V so, V& e, V& o) {
    const V m = __fmul_rn(c2, v2);
    e = __fmaf_rn(g, se, __fmaf_rn(c1, v1, m));
    o = __fmaf_rn(g, so, __fmaf_rn(c1, v1, -m));
  }
  static __device__ __forceinline__ C twice(C g) { return 2.f * g; }
  static __device__ __forceinline__ V load(const D* p, int) { return __ldg(p); }
  static __device__ __forceinline__ V scale(V v, D m) { return __fmul_rn(v, m); }
  static __device__ __forceinline__ D get(V v, int) { return v; }
};

// FP64 data in double-float arithmetic.
template <>
struct Arith<ff> {
  using V = ff;
  using C = ff;
  using D = double;
  using Acc = ffacc;
  static constexpr int W = 1;
  static constexpr bool kSumApart = true;   // see eo_row
  static __device__ __forceinline__ V zero() { return ff(0.f, 0.f); }
  static __device__ __forceinline__ V add(V a, V b) { return ff_add(a, b); }
  static __device__ __forceinline__ V sub(V a, V b) { return ff_sub(a, b); }
  static __device__ __forceinline__ Acc first(C c, V v) { return acc_first(c, v); }
  static __device__ __forceinline__ Acc init(V v) { return Acc{v.hi, v.lo}; }
  static __device__ __forceinline__ void fma(Acc& a, C c, V v) { acc_fma(a, c, v); }
  static __device__ __forceinline__ V value(const Acc& a) { return acc_value(a); }
  static __device__ __forceinline__ V point(C c, V v, C g, V s) {
    Acc a = acc_first(c, v);
    acc_fma(a, g, s);
    return acc_value(a);
  }
  static __device__ __forceinline__ void point_pair(C c1, V v1, C c2, V v2, C g, V se, V so, V& e, V& o) {
    Acc a = acc_first(c1, v1), b = a;
    acc_fma(a, c2, v2);
    acc_fma(b, ff(-c2.hi, -c2.lo), v2);
    acc_fma(a, g, se);
    acc_fma(b, g, so);
    e = acc_value(a);
    o = acc_value(b);
  }
  static __device__ __forceinline__ C twice(C g) { return ff(2.f * g.hi, 2.f * g.lo); }
  // the M^-1/2 scaling of the filter's product is applied to the FP64 value
  static __device__ __forceinline__ double load(const D* p, int) { return __ldg(p); }
  static __device__ __forceinline__ double scale(double v, D m) { return v * m; }
  static __device__ __forceinline__ D get(V v, int) { return ff_to_double(v); }
};

}  // namespace fe
