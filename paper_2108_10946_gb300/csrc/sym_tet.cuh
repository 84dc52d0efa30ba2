// Derivatives of a KMV tetrahedron's nodal field in symmetry-adapted coordinates (sym_layout.h):
// the counterpart of sym_tri.cuh for the four-group of the tetrahedron, whose characters are all
// one-dimensional. With u in character sums u_x(o) = sum_h x(h) u(node(o, h)) and the derivatives
// along the axes of the cube around the tetrahedron, the derivative along axis d takes character
// x to x ^ d: per contraction 162 (KMV2) and 768 (KMV3) multiply-adds instead of 675 and 3072.
// The sums are butterflies of additions. A third of the coefficients are distinct (54 and 256).
#pragma once
#include "sym_tri.cuh"

namespace fwi {

template <class V, int NN>
struct TetCoef {
  using T = TetSym<NN>;
  V m0[T::M0], m1[3][T::M1];
  __device__ __forceinline__ V& at(int x, int i) { return x == 0 ? m0[i] : m1[x - 1][i]; }
  __device__ __forceinline__ const V& at(int x, int i) const { return x == 0 ? m0[i] : m1[x - 1][i]; }
};
template <class V, int NN>
__device__ __forceinline__ void tet_zero(TetCoef<V, NN>& c) {
  using T = TetSym<NN>;
#pragma unroll
  for (int i = 0; i < T::M0; ++i) c.m0[i] = dup<V>(0.f);
#pragma unroll
  for (int x = 0; x < 3; ++x)
#pragma unroll
    for (int i = 0; i < T::M1; ++i) c.m1[x][i] = dup<V>(0.f);
}

// v[h] to v[x] = sum_h x(h) v[h] (its own transpose)
template <class V>
__device__ __forceinline__ void tet_butterfly(V (&v)[4]) {
  const V p = add2(v[0], v[1]), q = sub2(v[0], v[1]), r = add2(v[2], v[3]), s = sub2(v[2], v[3]);
  v[0] = add2(p, r);
  v[1] = sub2(p, r);
  v[2] = add2(q, s);
  v[3] = sub2(q, s);
}

template <class V, int NN, int O = 0, class F>
__device__ __forceinline__ void tet_analyse(TetCoef<V, NN>& c, F load) {
  using T = TetSym<NN>;
  if constexpr (O < T::NO) {
    if constexpr (T::kind(O) == 'R') {
      V v[4] = {load(T::node(O, 0)), load(T::node(O, 1)), load(T::node(O, 2)), load(T::node(O, 3))};
      tet_butterfly(v);
#pragma unroll
      for (int x = 0; x < 4; ++x) c.at(x, T::mode(O, x)) = v[x];
    } else if constexpr (T::kind(O) == 'P') {
      const V p = load(T::node(O, 0)), m = load(T::node(O, 1));
      c.at(0, T::mode(O, 0)) = add2(p, m);
      c.at(T::axis(O), T::mode(O, T::axis(O))) = sub2(p, m);
    } else {
      c.at(0, T::mode(O, 0)) = load(T::node(O, 0));
    }
    tet_analyse<V, NN, O + 1>(c, load);
  }
}

// the transpose of tet_analyse
template <class V, int NN, int O = 0, class F>
__device__ __forceinline__ void tet_gather_back(const TetCoef<V, NN>& c, F store) {
  using T = TetSym<NN>;
  if constexpr (O < T::NO) {
    if constexpr (T::kind(O) == 'R') {
      V v[4];
#pragma unroll
      for (int x = 0; x < 4; ++x) v[x] = c.at(x, T::mode(O, x));
      tet_butterfly(v);
#pragma unroll
      for (int h = 0; h < 4; ++h) store(T::node(O, h), v[h]);
    } else if constexpr (T::kind(O) == 'P') {
      const V s = c.at(0, T::mode(O, 0)), d = c.at(T::axis(O), T::mode(O, T::axis(O)));
      store(T::node(O, 0), add2(s, d));
      store(T::node(O, 1), sub2(s, d));
    } else {
      store(T::node(O, 0), c.at(0, T::mode(O, 0)));
    }
    tet_gather_back<V, NN, O + 1>(c, store);
  }
}

// Output Z of the derivative along axis D + 1 at orbit O: its input character and its number of modes.
template <int NN, int O, int D, int Z>
struct TetRow {
  using T = TetSym<NN>;
  static constexpr int Y = T::kind(O) == 'P' ? (Z ? (D + 1) ^ T::axis(O) : D + 1) : Z ^ (D + 1);
  static constexpr int N = Y == 0 ? T::M0 : T::M1;
};
template <class V, int NN, int O, int D, int Z>
__device__ __forceinline__ V tet_dot(const TetCoef<V, NN>& c) {
  using R = TetRow<NN, O, D, Z>;
  V s = mul2(coef<V>(tet_at<NN>(O, D, Z, R::Y, 0)), c.at(R::Y, 0));
#pragma unroll
  for (int i = 1; i < R::N; ++i) s = fma2(coef<V>(tet_at<NN>(O, D, Z, R::Y, i)), c.at(R::Y, i), s);
  return s;
}
template <class V, int NN, int O, int D, int Z>
__device__ __forceinline__ void tet_axpy(V f, TetCoef<V, NN>& c) {
  using R = TetRow<NN, O, D, Z>;
#pragma unroll
  for (int i = 0; i < R::N; ++i) c.at(R::Y, i) = fma2(coef<V>(tet_at<NN>(O, D, Z, R::Y, i)), f, c.at(R::Y, i));
}

template <int NN, int O>
struct TetSize {
  static constexpr int N = TetSym<NN>::kind(O) == 'R' ? 4 : TetSym<NN>::kind(O) == 'P' ? 2 : 1;
};

// Derivative along axis D + 1 at the nodes of orbit O.
template <class V, int NN, int O, int D>
__device__ __forceinline__ void tet_grad(const TetCoef<V, NN>& c, V (&g)[4]) {
  using T = TetSym<NN>;
  if constexpr (T::kind(O) == 'R') {
    g[0] = tet_dot<V, NN, O, D, 0>(c);
    g[1] = tet_dot<V, NN, O, D, 1>(c);
    g[2] = tet_dot<V, NN, O, D, 2>(c);
    g[3] = tet_dot<V, NN, O, D, 3>(c);
    tet_butterfly(g);
  } else if constexpr (T::kind(O) == 'P') {
    const V s = tet_dot<V, NN, O, D, 0>(c), d = tet_dot<V, NN, O, D, 1>(c);
    g[0] = add2(s, d);
    g[1] = sub2(s, d);
  } else {
    g[0] = tet_dot<V, NN, O, D, 0>(c);
  }
}

// The transpose: adds the nodes' flux along axis D + 1 to the coordinates.
template <class V, int NN, int O, int D>
__device__ __forceinline__ void tet_div(const V (&f)[4], TetCoef<V, NN>& c) {
  using T = TetSym<NN>;
  if constexpr (T::kind(O) == 'R') {
    V v[4] = {f[0], f[1], f[2], f[3]};
    tet_butterfly(v);
    tet_axpy<V, NN, O, D, 0>(v[0], c);
    tet_axpy<V, NN, O, D, 1>(v[1], c);
    tet_axpy<V, NN, O, D, 2>(v[2], c);
    tet_axpy<V, NN, O, D, 3>(v[3], c);
  } else if constexpr (T::kind(O) == 'P') {
    tet_axpy<V, NN, O, D, 0>(add2(f[0], f[1]), c);
    tet_axpy<V, NN, O, D, 1>(sub2(f[0], f[1]), c);
  } else {
    tet_axpy<V, NN, O, D, 0>(f[0], c);
  }
}

}  // namespace fwi
