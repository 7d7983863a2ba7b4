// Symmetry of the reference tetrahedron used by the CUDA-core stage
// (sym_body.cuh): the node orbits under a subgroup of the vertex permutations
// and the butterflies that take nodal values to symmetry-adapted ones.
//
// V4 = {e, (01)(23), (02)(13), (03)(12)} maps the equispaced nodes, the four
// faces and every fully symmetric volume rule onto themselves.  Its characters
// chi_x(g_y) are the signs of the 4 x 4 Hadamard matrix, and chi_x chi_y =
// chi_{x xor y}.  In the coordinates xi in which the vertices are (1,1,1),
// (1,-1,-1), (-1,1,-1), (-1,-1,1), d/dxi_a transforms with chi_a.  So in values
// adapted to the characters (one sum and three signed sums per orbit) V_q, P_q
// and LIFT fall into four diagonal blocks, and d/dxi_a takes block x to block
// x xor a: a quarter of the dense products' multiplications.
// Z2 = {e, (01)} does the same with two blocks for the conical-product rule,
// which is only symmetric in its innermost collapsed direction.
#pragma once

#ifdef __CUDACC__
#define WADG_HD __host__ __device__
#else
#define WADG_HD
#endif

namespace wadg {

// vertex that g_y of V4 takes vertex v to
WADG_HD constexpr int v4_image(int y, int v) { return v ^ y; }
// sign chi_x(g_y)
WADG_HD constexpr int v4_sign(int x, int y) {
  return (x == 0 || y == 0 || x == y) ? 1 : -1;
}

// Orbits of the order-N equispaced nodes (index order: k outermost, i
// fastest; barycentric numerators (N-i-j-k, i, j, k)).  Adapted values are
// ordered by character: all orbits for chi_0, then those that carry chi_1, ...
//   V4: NFul orbits of four nodes (every character), three of two nodes
//       (stabilised by g_a: chi_0 and chi_a) when N is even, one fixed node
//       (chi_0) when N is a multiple of four
//   Z2: NFul orbits of two nodes (both characters), NFix fixed nodes (chi_0)
template <int N>
struct NodeOrbits {
  static constexpr int Np = (N + 1) * (N + 2) * (N + 3) / 6;
  WADG_HD static constexpr int node(int i, int j, int k) {
    int n = 0;
    for (int kk = 0; kk < k; ++kk) n += (N - kk + 1) * (N - kk + 2) / 2;
    for (int jj = 0; jj < j; ++jj) n += N - k - jj + 1;
    return n + i;
  }
  // V4
  int ful[Np][4] = {};   // nodes of the free orbits, by group element
  int hal[3][2] = {};    // nodes of the orbit stabilised by g_{a+1}
  int sin = -1;          // the node fixed by V4
  int nful = 0;
  // Z2
  int pr[Np][2] = {};
  int fx[Np] = {};
  int npr = 0, nfx = 0;
  WADG_HD constexpr NodeOrbits() {
    for (int k = 0; k <= N; ++k)
      for (int j = 0; j + k <= N; ++j)
        for (int i = 0; i + j + k <= N; ++i) {
          const int b[4] = {N - i - j - k, i, j, k};
          int im[4] = {};
          for (int y = 0; y < 4; ++y)   // the image node's coordinates: b permuted
            im[y] = node(b[v4_image(y, 1)], b[v4_image(y, 2)], b[v4_image(y, 3)]);
          bool first = true;
          for (int y = 1; y < 4; ++y) first = first && im[0] <= im[y];
          if (first) {
            if (im[1] == im[0] && im[2] == im[0]) {
              sin = im[0];
            } else if (im[1] == im[0]) {
              hal[0][0] = im[0]; hal[0][1] = im[2];
            } else if (im[2] == im[0]) {
              hal[1][0] = im[0]; hal[1][1] = im[1];
            } else if (im[3] == im[0]) {
              hal[2][0] = im[0]; hal[2][1] = im[1];
            } else {
              for (int y = 0; y < 4; ++y) ful[nful][y] = im[y];
              ++nful;
            }
          }
          const int sw = node(b[0], b[2], b[3]);   // (01)
          if (sw == im[0]) fx[nfx++] = im[0];
          else if (im[0] < sw) { pr[npr][0] = im[0]; pr[npr][1] = sw; ++npr; }
        }
  }
};

// block sizes: G = 4 (V4), 2 (Z2)
template <int N, int G>
struct Blocks {
  static constexpr NodeOrbits<N> O{};
  static constexpr int NFul = G == 4 ? O.nful : O.npr;
  static constexpr int NH = G == 4 && N % 2 == 0 ? 1 : 0;   // two-node orbits per axis
  static constexpr int NS = G == 4 ? (N % 4 == 0 ? 1 : 0) : O.nfx;
  static constexpr int D0 = NFul + 3 * NH + NS;   // chi_0
  static constexpr int D1 = NFul + NH;            // every other character
  static constexpr int Np = NodeOrbits<N>::Np;
  static_assert(D0 + (G - 1) * D1 == Np, "block sizes");
  WADG_HD static constexpr int dim(int x) { return x == 0 ? D0 : D1; }
  WADG_HD static constexpr int off(int x) { return x == 0 ? 0 : D0 + (x - 1) * D1; }
  // offsets with every block padded to an even size (FP32 multiplies pairs)
  static constexpr int E0 = (D0 + 1) & ~1, E1 = (D1 + 1) & ~1;
  WADG_HD static constexpr int poff(int x) { return x == 0 ? 0 : E0 + (x - 1) * E1; }
  static constexpr int PO = E0 + (G - 1) * E1;
  // coefficients per group of four volume points: of 4 / G point orbits
  static constexpr int CP = (PO * (4 / G) + 3) & ~3;
};

// Layout of the operator table of the symmetric stage (in Reals): the
// derivative blocks by output character x and direction a = 1..3, columns
// (input value j of character x xor a) of RP(x) rows; the LIFT blocks by x,
// columns (face-node orbit m) of RP(x) rows; then per group of four volume
// points (an orbit of V4, or two orbits of Z2) Blocks<N, G>::CP coefficients
// of V_q (value j of character x of orbit o at o PO + poff(x) + j), and the
// same of P_q.
template <int N>
struct SymLayout {
  using B = Blocks<N, 4>;
  static constexpr int Nfp = (N + 1) * (N + 2) / 2;
  static constexpr int RP0 = (B::D0 + 3) & ~3, RP1 = (B::D1 + 3) & ~3;
  WADG_HD static constexpr int RP(int x) { return x == 0 ? RP0 : RP1; }
  static constexpr int DX0 = 3 * B::D1 * RP0;                 // derivative blocks of x = 0
  static constexpr int DX1 = (B::D0 + 2 * B::D1) * RP1;       // ... of one x > 0
  WADG_HD static constexpr int d_off(int x, int a) {
    int o = x == 0 ? 0 : DX0 + (x - 1) * DX1;
    for (int k = 1; k < a; ++k) o += B::dim(x ^ k) * RP(x);
    return o;
  }
  static constexpr int oL = DX0 + 3 * DX1;
  WADG_HD static constexpr int l_off(int x) {
    return oL + (x == 0 ? 0 : Nfp * RP0 + (x - 1) * Nfp * RP1);
  }
  static constexpr int oV = oL + Nfp * (RP0 + 3 * RP1);
};
// Blocks<N, G>::CP
template <int N>
WADG_HD constexpr int sym_cp_n(int G) {
  return G == 4 ? Blocks<N, 4>::CP : Blocks<N, 2>::CP;
}
WADG_HD constexpr int sym_cp(int N, int G) {
  return N == 1 ? sym_cp_n<1>(G) : N == 2 ? sym_cp_n<2>(G) : N == 3 ? sym_cp_n<3>(G)
       : N == 4 ? sym_cp_n<4>(G) : sym_cp_n<5>(G);
}
// largest number of groups of four points that the kernels hold: the compact
// rules have 1, 5, 6, 13 and 24 orbits under V4 (those of fewer than four
// points padded); the conical rule of (N + 1)^3 points has N/2 + 1 (rounded
// down) or (N + 1)/2 pairs per line of N + 1 points
WADG_HD constexpr int sym_groups(int N, int G) {
  if (G == 4) return N == 1 ? 1 : N == 2 ? 5 : N == 3 ? 6 : N == 4 ? 13 : 24;
  return (((N + 2) / 2) * (N + 1) * (N + 1) + 1) / 2;
}

}  // namespace wadg
