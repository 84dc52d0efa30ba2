// Derivatives of a KMV triangle's nodal field in symmetry-adapted coordinates.
//
// The element's stiffness action is y = sum_q D_q^T w_q c_q^2 H D_q u with D_q the two
// derivatives at node q (Section 3.2). As dense matrices the two contractions are 4 NN^2
// multiply-adds (3600 at KMV5). The node set is invariant under the triangle's six symmetries,
// so with u written in coordinates that transform by the group's irreducible representations
// and the derivatives taken in each node's own frame (along and across the median of its
// vertex v) they are a few small blocks (Schur's lemma): 26, 80, 180, 500 multiply-adds per
// contraction for k = 2..5 instead of 98, 288, 648, 1800.
//
// Three-vectors x_v (one value per vertex; sym_layout.h) have a sum and a two-component part:
//   even  s = x0 + x1 + x2,  e1 = x0 - (x1 + x2) / 2,   e2 = x1 - x2
//   odd   s = x0 + x1 + x2,  e1 = 3/4 (x2 - x1),        e2 = x0 - (x1 + x2) / 2
// scaled so that both components of every block share their coefficients and every other
// factor is exact in binary. Outputs are put together by the matching inverses:
//   even  x0 = S + E1, x1 = S - E1/2 + 3/4 E2, x2 = S - E1/2 - 3/4 E2
//   odd   x0 = S + E2, x1 = S - E2/2 - E1,     x2 = S - E2/2 + E1
// (the scales are in the coefficient table, kmvtab::sym_tables). The frame of vertex v: radial
// derivative d/db_v - (d/db_v+1 + d/db_v+2) / 2, tangential d/db_v+1 - d/db_v+2.
//
// The coefficients sit at compile-time positions of constant arrays of at most 300 values, once
// plain and once as pairs for the packed multiply-add. Include after declaring, in namespace fwi,
// the unit's __constant__ float c_sym[] and float2 c_sym2[].
#pragma once
#include "sym_layout.h"

namespace fwi {

// A value V is one lane (float) or a pair (float2: two shots of one element), whose multiply-adds
// are packed FP32x2 instructions: half the instructions for the same multiply-adds.
__device__ __forceinline__ float add2(float a, float b) { return a + b; }
__device__ __forceinline__ float sub2(float a, float b) { return a - b; }
__device__ __forceinline__ float mul2(float a, float b) { return a * b; }
__device__ __forceinline__ float fma2(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return __ffma2_rn(b, make_float2(-1.f, -1.f), a); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
template <class V>
__device__ __forceinline__ V dup(float a) {
  if constexpr (sizeof(V) == 8) return make_float2(a, a);
  else return a;
}
template <class V>
__device__ __forceinline__ V coef(int i) {
  if constexpr (sizeof(V) == 8) return c_sym2[i];
  else return c_sym[i];
}

template <class V, int NN>
struct TriCoef {  // a nodal field in the adapted coordinates
  using T = TriSym<NN>;
  V s1[T::NA1], s2[T::NA2 > 0 ? T::NA2 : 1], e1[T::NV], e2[T::NV];
};

template <class V, int NN>
__device__ __forceinline__ void tri_zero(TriCoef<V, NN>& c) {
  using T = TriSym<NN>;
#pragma unroll
  for (int i = 0; i < T::NA1; ++i) c.s1[i] = dup<V>(0.f);
#pragma unroll
  for (int i = 0; i < (T::NA2 > 0 ? T::NA2 : 1); ++i) c.s2[i] = dup<V>(0.f);
#pragma unroll
  for (int i = 0; i < T::NV; ++i) c.e1[i] = c.e2[i] = dup<V>(0.f);
}

// nodal values (load(q) of local node q) to adapted coordinates
template <class V, int NN, int O = 0, class F>
__device__ __forceinline__ void tri_analyse(TriCoef<V, NN>& c, F load) {
  using T = TriSym<NN>;
  if constexpr (O < T::NO) {
    constexpr char K = T::kind(O);
    constexpr int QB = T::base(O), I = T::vec(O), J = T::odd(O);
    if constexpr (K == 'C') {
      c.s1[O] = load(QB + T::place(K, 0, 0));
    } else if constexpr (K == 'X') {
      V p[3], m[3];
#pragma unroll
      for (int v = 0; v < 3; ++v) {
        const V a = load(QB + T::place(K, v, 0)), b = load(QB + T::place(K, v, 1));
        p[v] = add2(a, b);
        m[v] = sub2(a, b);
      }
      const V h = add2(p[1], p[2]), g = add2(m[1], m[2]);
      c.s1[O] = add2(p[0], h);
      c.e1[I] = fma2(dup<V>(-0.5f), h, p[0]);
      c.e2[I] = sub2(p[1], p[2]);
      c.s2[J] = add2(m[0], g);
      c.e1[I + 1] = mul2(dup<V>(0.75f), sub2(m[2], m[1]));
      c.e2[I + 1] = fma2(dup<V>(-0.5f), g, m[0]);
    } else {
      const V x0 = load(QB + T::place(K, 0, 0)), x1 = load(QB + T::place(K, 1, 0)), x2 = load(QB + T::place(K, 2, 0));
      const V h = add2(x1, x2);
      c.s1[O] = add2(x0, h);
      c.e1[I] = fma2(dup<V>(-0.5f), h, x0);
      c.e2[I] = sub2(x1, x2);
    }
    tri_analyse<V, NN, O + 1>(c, load);
  }
}

// the transpose of tri_analyse: store(q, value) for every local node
template <class V, int NN, int O = 0, class F>
__device__ __forceinline__ void tri_gather_back(const TriCoef<V, NN>& c, F store) {
  using T = TriSym<NN>;
  if constexpr (O < T::NO) {
    constexpr char K = T::kind(O);
    constexpr int QB = T::base(O), I = T::vec(O), J = T::odd(O);
    if constexpr (K == 'C') {
      store(QB + T::place(K, 0, 0), c.s1[O]);
    } else {
      const V t = fma2(dup<V>(-0.5f), c.e1[I], c.s1[O]);
      const V p[3] = {add2(c.s1[O], c.e1[I]), add2(t, c.e2[I]), sub2(t, c.e2[I])};
      if constexpr (K == 'X') {
        const V s = c.s2[J];
        const V r = fma2(dup<V>(-0.5f), c.e2[I + 1], s);
        const V m[3] = {add2(s, c.e2[I + 1]), fma2(dup<V>(-0.75f), c.e1[I + 1], r), fma2(dup<V>(0.75f), c.e1[I + 1], r)};
#pragma unroll
        for (int v = 0; v < 3; ++v) {
          store(QB + T::place(K, v, 0), add2(p[v], m[v]));
          store(QB + T::place(K, v, 1), sub2(p[v], m[v]));
        }
      } else {
#pragma unroll
        for (int v = 0; v < 3; ++v) store(QB + T::place(K, v, 0), p[v]);
      }
    }
    tri_gather_back<V, NN, O + 1>(c, store);
  }
}

// The NV coefficients at position `at` of c_sym times the vector coordinates, and the transpose.
template <class V, int NN>
__device__ __forceinline__ void tri_dot(int at, const TriCoef<V, NN>& c, V& E1, V& E2) {
  E1 = E2 = dup<V>(0.f);
#pragma unroll
  for (int i = 0; i < TriSym<NN>::NV; ++i) {
    E1 = fma2(coef<V>(at + i), c.e1[i], E1);
    E2 = fma2(coef<V>(at + i), c.e2[i], E2);
  }
}
template <class V, int NN>
__device__ __forceinline__ void tri_axpy(int at, V E1, V E2, TriCoef<V, NN>& c) {
#pragma unroll
  for (int i = 0; i < TriSym<NN>::NV; ++i) {
    c.e1[i] = fma2(coef<V>(at + i), E1, c.e1[i]);
    c.e2[i] = fma2(coef<V>(at + i), E2, c.e2[i]);
  }
}

// One output three-vector whose coefficients start at position `at`.
template <class V, int NN, bool ODD>
__device__ __forceinline__ void tri_out(int at, const TriCoef<V, NN>& c, V (&x)[3]) {
  using T = TriSym<NN>;
  constexpr int NA = ODD ? T::NA2 : T::NA1;
  V S = dup<V>(0.f), E1, E2;
#pragma unroll
  for (int i = 0; i < NA; ++i) S = fma2(coef<V>(at + i), ODD ? c.s2[i] : c.s1[i], S);
  tri_dot<V, NN>(at + NA, c, E1, E2);
  if constexpr (ODD) {
    const V t = NA > 0 ? fma2(dup<V>(-0.5f), E2, S) : mul2(dup<V>(-0.5f), E2);
    x[0] = NA > 0 ? add2(S, E2) : E2;
    x[1] = sub2(t, E1);
    x[2] = add2(t, E1);
  } else {
    const V t = fma2(dup<V>(-0.5f), E1, S);
    x[0] = add2(S, E1);
    x[1] = fma2(dup<V>(0.75f), E2, t);
    x[2] = fma2(dup<V>(-0.75f), E2, t);
  }
}

// The transpose: adds the three-vector f to the coordinates.
template <class V, int NN, bool ODD>
__device__ __forceinline__ void tri_in(int at, const V (&f)[3], TriCoef<V, NN>& c) {
  using T = TriSym<NN>;
  constexpr int NA = ODD ? T::NA2 : T::NA1;
  const V h = add2(f[1], f[2]), S = add2(f[0], h), t = fma2(dup<V>(-0.5f), h, f[0]);
  const V E1 = ODD ? sub2(f[2], f[1]) : t, E2 = ODD ? t : mul2(dup<V>(0.75f), sub2(f[1], f[2]));
#pragma unroll
  for (int i = 0; i < NA; ++i) {
    if (ODD) c.s2[i] = fma2(coef<V>(at + i), S, c.s2[i]);
    else c.s1[i] = fma2(coef<V>(at + i), S, c.s1[i]);
  }
  tri_axpy<V, NN>(at + NA, E1, E2, c);
}

// Radial and tangential derivatives r[side][v], t[side][v] at the nodes of an orbit of kind K whose
// coefficients start at position `at`.
template <class V, int NN, char K>
__device__ __forceinline__ void tri_grad(int at, const TriCoef<V, NN>& c, V (&r)[2][3], V (&t)[2][3]) {
  using T = TriSym<NN>;
  if constexpr (K == 'C') {
    tri_dot<V, NN>(at, c, r[0][0], t[0][0]);
  } else if constexpr (K == 'X') {
    V p[3], m[3];
    tri_out<V, NN, false>(at, c, p);
    tri_out<V, NN, true>(at + T::EVEN, c, m);
#pragma unroll
    for (int v = 0; v < 3; ++v) {
      r[0][v] = add2(p[v], m[v]);
      r[1][v] = sub2(p[v], m[v]);
    }
    tri_out<V, NN, true>(at + T::EVEN + T::ODD, c, p);
    tri_out<V, NN, false>(at + T::EVEN + 2 * T::ODD, c, m);
#pragma unroll
    for (int v = 0; v < 3; ++v) {
      t[0][v] = add2(p[v], m[v]);
      t[1][v] = sub2(p[v], m[v]);
    }
  } else {
    tri_out<V, NN, false>(at, c, r[0]);
    tri_out<V, NN, true>(at + T::EVEN, c, t[0]);
  }
}

// The transpose of tri_grad: adds the nodes' fluxes to the coordinates of y.
template <class V, int NN, char K>
__device__ __forceinline__ void tri_div(int at, const V (&r)[2][3], const V (&t)[2][3], TriCoef<V, NN>& c) {
  using T = TriSym<NN>;
  if constexpr (K == 'C') {
    tri_axpy<V, NN>(at, r[0][0], t[0][0], c);
  } else if constexpr (K == 'X') {
    V p[3], m[3];
#pragma unroll
    for (int v = 0; v < 3; ++v) {
      p[v] = add2(r[0][v], r[1][v]);
      m[v] = sub2(r[0][v], r[1][v]);
    }
    tri_in<V, NN, false>(at, p, c);
    tri_in<V, NN, true>(at + T::EVEN, m, c);
#pragma unroll
    for (int v = 0; v < 3; ++v) {
      p[v] = add2(t[0][v], t[1][v]);
      m[v] = sub2(t[0][v], t[1][v]);
    }
    tri_in<V, NN, true>(at + T::EVEN + T::ODD, p, c);
    tri_in<V, NN, false>(at + T::EVEN + 2 * T::ODD, m, c);
  } else {
    tri_in<V, NN, false>(at, r[0], c);
    tri_in<V, NN, true>(at + T::EVEN, t[0], c);
  }
}

// B_v^T M of a 2 x m matrix M given on the reference derivatives (d/dx, d/dy): its rows for
// the (radial, tangential) derivatives of frame v, since (d/dx, d/dy) = B_v (radial, tangential)
//   B_0 = [-1 1/2; -1 -1/2], B_1 = [1 1/2; 0 1], B_2 = [0 -1; 1 -1/2].
template <int FR, class V>
__device__ __forceinline__ void tri_frame(V x, V y, V& r, V& t) {
  if (FR == 0) {
    r = mul2(dup<V>(-1.f), add2(x, y));
    t = mul2(dup<V>(0.5f), sub2(x, y));
  } else if (FR == 1) {
    r = x;
    t = fma2(dup<V>(0.5f), x, y);
  } else {
    r = y;
    t = mul2(dup<V>(-1.f), fma2(dup<V>(0.5f), y, x));
  }
}

// H_v = B_v^T Ghat B_v (rr, rt, tt) for the three frames, from Ghat's xx, xy, yy
template <class V>
__device__ __forceinline__ void tri_metric(V xx, V xy, V yy, V (&H)[3][3]) {
  const V h = dup<V>(0.5f), q = dup<V>(0.25f), m = dup<V>(-1.f), s = add2(xx, yy);
  H[0][0] = fma2(dup<V>(2.f), xy, s);
  H[0][1] = mul2(h, sub2(yy, xx));
  H[0][2] = fma2(dup<V>(-0.5f), xy, mul2(q, s));
  H[1][0] = xx;
  H[1][1] = fma2(h, xx, xy);
  H[1][2] = fma2(q, xx, add2(xy, yy));
  H[2][0] = yy;
  H[2][1] = mul2(m, fma2(h, yy, xy));
  H[2][2] = fma2(q, yy, add2(xy, xx));
}

}  // namespace fwi
