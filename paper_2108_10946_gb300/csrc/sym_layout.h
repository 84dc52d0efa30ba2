// Symmetry layout of the KMV elements, shared by the host tabulation (kmv_tab.cpp) and the
// kernels (sym_tri.cuh, sym_tet.cuh).
//
// The node sets of the KMV elements (Section 3.2) do not change under permutations of the
// simplex's vertices, so in coordinates adapted to (a subgroup of) that symmetry group the
// derivative matrices fall apart into small blocks. What a node set needs to say for that is
// its orbits, in the library's local node order.
//
// Triangles: the full group S3. Orbit kinds:
//   'T' (a, a, b): one node on each median, slot base + 2 - v on the median of vertex v (the
//       vertices, first, are numbered the other way round in the local order: sym_slot_node)
//   'X' (g0, g1, g2): two nodes for every vertex v, mirror images in its median
//   'C' the centroid
// Tetrahedra: the four-group of the even pair swaps, h = 0..3 = identity, (01)(23), (02)(13),
// (03)(12). In the cube whose alternate corners are the vertices, (1,1,1), (1,-1,-1), (-1,1,-1),
// (-1,-1,1), its elements are the half turns about the axes, so each derivative along an axis
// takes one of the four characters to another. (The third turn about the diagonal of vertex 0
// permutes the axes cyclically: one axis's coefficients are all.) Orbit kinds:
//   'R' four nodes, one per h; 'P' two nodes on an axis; 'C' the centroid
//
// Every V and T orbit is one "three-vector" x_v, v = 0..2, even under the mirror of each
// median; an X orbit is two, the pair sums (even) and the pair differences (odd).
#pragma once

#ifdef __CUDACC__
#define FWI_HD __host__ __device__
#else
#define FWI_HD
#endif

namespace fwi {

template <int NN>
struct TriOrbits;
template <>
struct TriOrbits<7> {
  static constexpr int NO = 3;
  FWI_HD static constexpr char kind(int o) { return "TTC"[o]; }
};
template <>
struct TriOrbits<12> {
  static constexpr int NO = 3;
  FWI_HD static constexpr char kind(int o) { return "TXT"[o]; }
};
template <>
struct TriOrbits<18> {
  static constexpr int NO = 5;
  FWI_HD static constexpr char kind(int o) { return "TTXTT"[o]; }
};
template <>
struct TriOrbits<30> {
  static constexpr int NO = 7;
  FWI_HD static constexpr char kind(int o) { return "TXXTTTX"[o]; }
};

template <int NN>
struct TriSym : TriOrbits<NN> {
  using B = TriOrbits<NN>;
  static constexpr int NO = B::NO;
  FWI_HD static constexpr int size_of(char k) { return k == 'X' ? 6 : k == 'C' ? 1 : 3; }
  FWI_HD static constexpr int vecs_of(char k) { return k == 'X' ? 2 : k == 'C' ? 0 : 1; }
  // first local node, first three-vector and number of odd three-vectors before orbit o
  // (loops, not recursion: a device function that is not folded must not call itself)
  FWI_HD static constexpr int base(int o) {
    int n = 0;
    for (int i = 0; i < o; ++i) n += size_of(B::kind(i));
    return n;
  }
  FWI_HD static constexpr int vec(int o) {
    int n = 0;
    for (int i = 0; i < o; ++i) n += vecs_of(B::kind(i));
    return n;
  }
  FWI_HD static constexpr int odd(int o) {
    int n = 0;
    for (int i = 0; i < o; ++i) n += B::kind(i) == 'X';
    return n;
  }
  // coordinates: NA1 symmetric sums (one per orbit), NA2 antisymmetric sums (one per odd
  // three-vector) and NV two-component vectors
  static constexpr int NA1 = NO, NA2 = odd(NO), NV = vec(NO);
  static_assert(base(NO) == NN, "orbits cover the node set");
  // slot of orbit o's node at vertex v (side 0 / 1: the two nodes of an X orbit)
  FWI_HD static constexpr int place(char k, int v, int side) {  // in its orbit
    return k == 'T' ? 2 - v
           : k == 'C' ? 0
                      : side == 0 ? (v == 0 ? 4 : v == 1 ? 3 : 0) : (v == 0 ? 5 : v == 1 ? 1 : 2);
  }
  FWI_HD static constexpr int node(int o, int v, int side = 0) { return base(o) + place(B::kind(o), v, side); }
  // Coefficient table, output three-vector by output three-vector. An even output has NA1
  // coefficients for its sum and NV for its vector part, an odd one NA2 and NV; the centroid's
  // gradient is one vector (NV). A T orbit gives the radial (even) and the tangential
  // (odd) derivative; an X orbit radial sums (even) and differences (odd), tangential sums
  // (odd) and differences (even).
  static constexpr int EVEN = NA1 + NV, ODD = NA2 + NV;
  FWI_HD static constexpr int tab(int o) {
    int n = 0;
    for (int i = 0; i < o; ++i) n += B::kind(i) == 'X' ? 2 * (EVEN + ODD) : B::kind(i) == 'C' ? NV : EVEN + ODD;
    return n;
  }
  static constexpr int TAB = tab(NO);
  // Rolled form (KMV5): the table holds the X orbits' coefficients, then the T orbits'; first slots
  // of the k-th X and T orbit.
  static constexpr bool ROLL = NN == 30;
  static constexpr int NX = NA2, NT = NO - NA2, XTAB = 2 * (EVEN + ODD), TTAB = EVEN + ODD;
  FWI_HD static constexpr int roll_x(int k) { return k == 2 ? 24 : 3 + 6 * k; }
  FWI_HD static constexpr int roll_t(int k) { return k == 0 ? 0 : 12 + 3 * k; }
};

// Tetrahedra. Character x: 0 trivial, k = 1..3 (+1 on h = 0 and h = k, -1 on the others); products
// of characters are the XOR of their numbers. u_x(o) = sum_h x(h) u(node(o, h)).
template <int NN>
struct TetSym;
template <>
struct TetSym<15> {  // V, F (faces, by the opposite vertex), the edge midpoints on axes 1..3, centroid
  static constexpr int NO = 6, M0 = 6, M1 = 3, TAB = 54;
  FWI_HD static constexpr char kind(int o) { return "RRPPPC"[o]; }
  FWI_HD static constexpr int axis(int o) { return o >= 2 && o <= 4 ? o - 1 : 0; }
  FWI_HD static constexpr int node(int o, int h) {
    return o == 0 ? h : o == 1 ? 13 - h : o == 5 ? 14 : h == 0 ? 2 + o : 11 - o;
  }
  // mode i of character x is orbit ...; orbit o's mode in character x
  FWI_HD static constexpr int mode(int o, int x) { return x == 0 ? o : o < 2 ? o : 2; }
  FWI_HD static constexpr bool has(int o, int x) { return x == 0 || o < 2 || axis(o) == x; }
  // the orbit and the mode that the cyclic turn takes d steps back
  FWI_HD static constexpr int turn(int o, int d) { return axis(o) ? 2 + (axis(o) - 1 + 3 - d) % 3 : o; }
  FWI_HD static constexpr int turn_mode(int i, int x, int d) { return x == 0 ? turn(i, d) : i; }
  // coefficients of the derivative along axis 1 at orbit o: output character z takes input z ^ 1
  FWI_HD static constexpr int at(int o, int z) {
    return o < 2 ? 15 * o + (z == 0 ? 0 : z == 1 ? 3 : z == 2 ? 9 : 12)
           : o == 2 ? 30 + (z ? 3 : 0)
           : o == 3 ? 39 + (z ? 3 : 0)
           : o == 4 ? 45 + (z ? 3 : 0)
                    : 51;
  }
};
template <>
struct TetSym<32> {  // V; the edge nodes next to vertex 0's edge 01, 02, 03; the face nodes next to
                     // vertex 0 in the faces opposite 1, 2, 3; interior
  static constexpr int NO = 8, M0 = 8, M1 = 8, TAB = 256;
  FWI_HD static constexpr char kind(int) { return 'R'; }
  FWI_HD static constexpr int axis(int) { return 0; }
  FWI_HD static constexpr int node(int o, int h) {
    return o == 0 ? h
           : o == 1 ? (h == 0 ? 4 : h == 1 ? 7 : h == 2 ? 14 : 15)
           : o == 2 ? (h == 0 ? 5 : h == 1 ? 11 : h == 2 ? 8 : 13)
           : o == 3 ? (h == 0 ? 6 : h == 1 ? 10 : h == 2 ? 12 : 9)
           : o == 4 ? (h == 0 ? 24 : h == 1 ? 27 : h == 2 ? 16 : 17)
           : o == 5 ? (h == 0 ? 23 : h == 1 ? 18 : h == 2 ? 26 : 20)
           : o == 6 ? (h == 0 ? 22 : h == 1 ? 19 : h == 2 ? 21 : 25)
                    : 31 - h;
  }
  FWI_HD static constexpr int mode(int o, int) { return o; }
  FWI_HD static constexpr bool has(int, int) { return true; }
  FWI_HD static constexpr int turn(int o, int d) {
    return o >= 1 && o <= 3 ? 1 + (o - 1 + 3 - d) % 3 : o >= 4 && o <= 6 ? 4 + (o - 4 + 3 - d) % 3 : o;
  }
  FWI_HD static constexpr int turn_mode(int i, int, int d) { return turn(i, d); }
  FWI_HD static constexpr int at(int o, int z) { return (o * 4 + z) * 8; }
};
// Character x turned d steps back.
FWI_HD constexpr int tet_turn(int x, int d) { return x == 0 ? 0 : 1 + (x - 1 + 3 - d) % 3; }
// Position of the coefficient of mode i of character y in output z (y = z ^ (d + 1)) of the
// derivative along axis d + 1 at orbit o. At a 'P' orbit outputs are 0 (sum) and 1 (difference).
template <int NN>
FWI_HD constexpr int tet_at(int o, int d, int z, int y, int i) {
  return TetSym<NN>::at(TetSym<NN>::turn(o, d), TetSym<NN>::kind(o) == 'R' ? tet_turn(z, d) : z) +
         TetSym<NN>::turn_mode(i, y, d);
}

// Places between a chunk's owned DoFs and its halo DoFs in every table of the chunk kernels. The owned
// range arrives in whole 16-byte groups, whose last may end up to three floats past it; the halo DoFs
// are copied by other threads meanwhile, in no order to that, so they start where no group ends.
constexpr int SYM_GAP = 3;

// Order of an element's nodes in the chunk tables (local node at slot j): the local order, but a
// triangle's vertices backwards, like its other T orbits; at KMV3 tetrahedra orbit by orbit (slot
// 4 o + h; the interior orbit last). So a loop over like orbits need not be unrolled.
FWI_HD constexpr int sym_slot_node(int dim, int nn, int j) {
  return dim == 3 ? (nn == 32 ? TetSym<32>::node(j / 4, j % 4) : j) : j < 3 ? 2 - j : j;
}

}  // namespace fwi
