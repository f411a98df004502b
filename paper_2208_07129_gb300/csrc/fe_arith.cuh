// Arithmetic of the box-cell kernel (fe_box.cuh), one struct per value type.
// A thread works on values of type V, each W vectors of the block; the 1D
// coefficients are of type C, the geometry of type G, and D is the element
// type of X and Y in global memory.  Every operation is an explicitly rounded
// one, so the compiler neither contracts nor reassociates, and every
// instantiation of the body (launch per colour, small meshes, batch) gives
// the same bits.
#pragma once

#include <cuda_runtime.h>

#include "fe_ff.cuh"

namespace fe {

// W elements moved by one access.
template <typename D, int W>
struct alignas(sizeof(D) * W) Pack {
  D a[W];
};

// The `have` first of W consecutive elements (the others 0); with `vec` the
// address is aligned to W elements and all of them exist.
template <typename D, int W>
__device__ __forceinline__ Pack<D, W> load_pack(const D* p, int have, bool vec) {
  if (W > 1 && !vec) {
    Pack<D, W> r;
#pragma unroll
    for (int k = 0; k < W; ++k) r.a[k] = k < have ? p[k] : D(0);
    return r;
  }
  return *reinterpret_cast<const Pack<D, W>*>(p);
}

template <typename D, int W>
__device__ __forceinline__ void store_pack(D* p, const Pack<D, W>& v, int have, bool vec) {
  if (W > 1 && !vec) {
#pragma unroll
    for (int k = 0; k < W; ++k)
      if (k < have) p[k] = v.a[k];
    return;
  }
  *reinterpret_cast<Pack<D, W>*>(p) = v;
}

template <typename V>
struct Arith;

// Vectors per CTA and 1D lines in flight.
struct LineTile {
  int vb, lines;
};

template <>
struct Arith<double> {
  using V = double;
  using C = double;
  using G = double;
  using D = double;
  using Acc = double;
  static constexpr int W = 1;
  static constexpr bool kSumApart = false;   // see eo_row
  // Default tile of the box kernel, from sweeps of vb x lines at n_q = 4..10 (64
  // vectors).  A pass has n_p^2 to n_q^2 lines: few of them want many vectors per
  // CTA (n_q = 5: 6.18 ms at 32 x 8, 6.68 at 8 x 16), many of them fill the CTA,
  // and the tiles of three CTAs have to fit one SM (n_q = 10: 11.8 ms at 4 x 32,
  // 12.6 at 8 x 32).
  static constexpr LineTile box_tile(int nq) {
    return nq <= 5 ? LineTile{32, 8} : nq <= 7 ? LineTile{16, 8} : nq == 8 ? LineTile{8, 16} : nq == 9 ? LineTile{8, 24} : LineTile{4, 32};
  }
  // Default tile of the trilinear kernel (three tiles of shared memory), swept the same way.
  static constexpr LineTile general_tile(int nq) {
    return nq <= 5 ? LineTile{32, 8} : nq == 6 ? LineTile{16, 16} : nq <= 8 ? LineTile{8, 16} : LineTile{4, 32};
  }
  static __device__ __forceinline__ V zero() { return 0.0; }
  static __device__ __forceinline__ V add(V a, V b) { return __dadd_rn(a, b); }
  static __device__ __forceinline__ V sub(V a, V b) { return __dsub_rn(a, b); }
  static __device__ __forceinline__ Acc first(C c, V v) { return __dmul_rn(c, v); }
  static __device__ __forceinline__ Acc init(V v) { return v; }
  static __device__ __forceinline__ void fma(Acc& a, C c, V v) { a = __fma_rn(c, v, a); }
  static __device__ __forceinline__ V value(Acc a) { return a; }
  static __device__ __forceinline__ V muladd(G c, V v, V a) { return __fma_rn(c, v, a); }
  // c v + g s: the middle point of an odd rule
  static __device__ __forceinline__ V point(G c, V v, G g, V s) { return __fma_rn(g, s, __dmul_rn(c, v)); }
  // e = c1 v1 + c2 v2 + g se,  o = c1 v1 - c2 v2 + g so
  static __device__ __forceinline__ void point_pair(G c1, V v1, G c2, V v2, G g, V se, V so, V& e, V& o) {
    const V m = __dmul_rn(c2, v2);
    e = __fma_rn(g, se, __fma_rn(c1, v1, m));
    o = __fma_rn(g, so, __fma_rn(c1, v1, -m));
  }
  static __device__ __forceinline__ G twice(G g) { return 2.0 * g; }
  static __device__ __forceinline__ V from(const Pack<D, W>& p) { return p.a[0]; }
  static __device__ __forceinline__ Pack<D, W> to(V v) { return Pack<D, W>{{v}}; }
};

// Two FP32 vectors per value, on the packed FP32 instructions of sm_100: one
// issue slot for two operations, and half the shared-memory and global accesses.
// A lane's results are those of the scalar operations (a product that is -0
// comes out as +0).  FP32 was bound by
// issue: 16^3 p = 6, n_q = 8, 64 vectors 0.728 -> 0.464 ms.  Four vectors per
// value take 118 registers and gained only for n_q <= 6 (0.36 -> 0.32 ms at
// 20^3 p = 4, but 0.46 -> 0.49 ms at p = 6).  Double-float stays on one vector:
// packed pairs measured 2.64 against 2.56 ms (16^3 p = 6) and 3.39 against
// 3.19 ms (12^3 p = 8), their registers halving the warps in flight.
using f32x2 = unsigned long long;

__device__ __forceinline__ f32x2 pack2(float a, float b) {
  f32x2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ void unpack2(f32x2 v, float& a, float& b) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
}
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) {
  f32x2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f32x2 sub2(f32x2 a, f32x2 b) {
  f32x2 r;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
  f32x2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
// A product is an FMA with 0: the assembler merges mul.rn.f32x2 with a
// dependent add or sub, and the separately rounded product is then lost.
__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b) { return fma2(a, b, 0ull); }

struct F2 {
  f32x2 v;
};

template <>
struct Arith<F2> {
  using V = F2;
  using C = float;
  using G = float;
  using D = float;
  using Acc = f32x2;
  static constexpr int W = 2;
  static constexpr bool kSumApart = true;   // see eo_row
  static __device__ __forceinline__ f32x2 bc(float c) { return pack2(c, c); }
  // see Arith<double>::box_tile; n_q = 4: 0.33 ms at 32 x 8, 0.74 at 8 x 32; n_q = 8:
  // 0.464 at 16 x 32, 0.483 at 8 x 32; n_q = 10: 0.543 at 8 x 32, 0.55 at 8 x 50
  static constexpr LineTile box_tile(int nq) {
    return nq <= 4 ? LineTile{32, 8} : nq <= 6 ? LineTile{16, 16} : nq <= 8 ? LineTile{16, 32} : LineTile{8, 32};
  }
  static constexpr LineTile general_tile(int nq) {
    return nq <= 4 ? LineTile{32, 8} : nq == 5 ? LineTile{16, 16} : nq <= 8 ? LineTile{8, 32} : LineTile{8, 40};
  }
  static __device__ __forceinline__ V zero() { return V{0ull}; }
  static __device__ __forceinline__ V add(V a, V b) { return V{add2(a.v, b.v)}; }
  static __device__ __forceinline__ V sub(V a, V b) { return V{sub2(a.v, b.v)}; }
  static __device__ __forceinline__ Acc first(C c, V v) { return mul2(bc(c), v.v); }
  static __device__ __forceinline__ Acc init(V v) { return v.v; }
  static __device__ __forceinline__ void fma(Acc& a, C c, V v) { a = fma2(bc(c), v.v, a); }
  static __device__ __forceinline__ V value(Acc a) { return V{a}; }
  static __device__ __forceinline__ V muladd(G c, V v, V a) { return V{fma2(bc(c), v.v, a.v)}; }
  static __device__ __forceinline__ V point(G c, V v, G g, V s) { return V{fma2(bc(g), s.v, mul2(bc(c), v.v))}; }
  static __device__ __forceinline__ void point_pair(G c1, V v1, G c2, V v2, G g, V se, V so, V& e, V& o) {
    const f32x2 gg = bc(g), p = mul2(bc(c1), v1.v);
    e = V{fma2(gg, se.v, fma2(bc(c2), v2.v, p))};
    o = V{fma2(gg, so.v, fma2(bc(-c2), v2.v, p))};
  }
  static __device__ __forceinline__ G twice(G g) { return 2.f * g; }
  static __device__ __forceinline__ V from(const Pack<D, W>& p) { return V{pack2(p.a[0], p.a[1])}; }
  static __device__ __forceinline__ Pack<D, W> to(V v) {
    Pack<D, W> p;
    unpack2(v.v, p.a[0], p.a[1]);
    return p;
  }
};

// FP64 data in double-float arithmetic.
template <>
struct Arith<ff> {
  using V = ff;
  using C = ff;
  using G = ff;
  using D = double;
  using Acc = ffacc;
  static constexpr int W = 1;
  static constexpr bool kSumApart = true;   // see eo_row
  // see Arith<double>::box_tile; n_q = 5: 1.42 ms at 16 x 8, 2.0 at 8 x 32; n_q = 6: 1.73
  // at 16 x 16, 2.2 at 8 x 32; n_q = 9: 2.85 at 8 x 32, 4.0 at 4 x 64
  static constexpr LineTile box_tile(int nq) {
    return nq <= 5 ? LineTile{16, 8} : nq <= 7 ? LineTile{16, 16} : nq <= 9 ? LineTile{8, 32} : LineTile{4, 64};
  }
  static constexpr LineTile general_tile(int nq) {
    return nq <= 4 ? LineTile{16, 8} : nq <= 6 ? LineTile{16, 16} : nq <= 8 ? LineTile{8, 32} : LineTile{4, 32};
  }
  static __device__ __forceinline__ V zero() { return ff(0.f, 0.f); }
  static __device__ __forceinline__ V add(V a, V b) { return ff_add(a, b); }
  static __device__ __forceinline__ V sub(V a, V b) { return ff_sub(a, b); }
  static __device__ __forceinline__ Acc first(C c, V v) { return acc_first(c, v); }
  static __device__ __forceinline__ Acc init(V v) { return Acc{v.hi, v.lo}; }
  static __device__ __forceinline__ void fma(Acc& a, C c, V v) { acc_fma(a, c, v); }
  static __device__ __forceinline__ V value(const Acc& a) { return acc_value(a); }
  static __device__ __forceinline__ V muladd(G c, V v, V a) { return ff_add(acc_value(acc_first(c, v)), a); }
  static __device__ __forceinline__ V point(G c, V v, G g, V s) {
    Acc a = acc_first(c, v);
    acc_fma(a, g, s);
    return acc_value(a);
  }
  static __device__ __forceinline__ void point_pair(G c1, V v1, G c2, V v2, G g, V se, V so, V& e, V& o) {
    Acc a = acc_first(c1, v1), b = a;
    acc_fma(a, c2, v2);
    acc_fma(b, ff(-c2.hi, -c2.lo), v2);
    acc_fma(a, g, se);
    acc_fma(b, g, so);
    e = acc_value(a);
    o = acc_value(b);
  }
  static __device__ __forceinline__ G twice(G g) { return ff(2.f * g.hi, 2.f * g.lo); }
  static __device__ __forceinline__ V from(const Pack<D, W>& p) { return ff(p.a[0]); }
  static __device__ __forceinline__ Pack<D, W> to(V v) { return Pack<D, W>{{ff_to_double(v)}}; }
};

}  // namespace fe
