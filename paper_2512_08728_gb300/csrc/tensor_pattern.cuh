// Zero pattern of the blocks of a DG operator on a Cartesian grid in a total-degree tensor
// basis (modes ordered by total degree, then by decreasing power of x, then of y).
//
// A face term normal to e_k integrates products of the one-dimensional factors of the other
// directions, which are orthonormal, so it couples two modes only if their degrees agree in
// every direction but k; a volume term couples two modes only if they differ in at most one
// direction.  In three dimensions at degree 2 that leaves 20 of the 100 entries of a coupling
// block and 40 of a diagonal block, at degree 3 50 and 110 of 400.  The pattern is a property
// of the operator that a caller passes, not an assumption: setup checks every block and keeps
// the dense kernels for operators that have entries outside it.
#pragma once

namespace kcmg {

template <int NP, int DIM> struct TensorPattern {
  static constexpr int S = 2 * DIM + 1;
  static constexpr int P = NP == 3 || NP == 4 ? 1 : (NP == 6 || (NP == 10 && DIM == 3)) ? 2 : 3;
  struct Modes { int e[NP][3]; };
  static __host__ __device__ constexpr Modes make_modes() {
    Modes m{};
    int c = 0;
    for (int n = 0; n <= P; ++n)
      for (int x = n; x >= 0; --x)
        for (int y = n - x; y >= 0; --y) {
          const int z = n - x - y;
          if (DIM == 2 && z != 0) continue;
          m.e[c][0] = x;
          m.e[c][1] = y;
          m.e[c][2] = z;
          ++c;
        }
    return m;
  }
  // whether entry (i, j) of the block of slot s can be nonzero
  static __host__ __device__ constexpr bool nz(const Modes& m, int s, int i, int j) {
    int differ = 0;
    for (int k = 0; k < DIM; ++k) {
      if (m.e[i][k] == m.e[j][k]) continue;
      if (s > 0 && (s - 1) / 2 != k) return false;
      ++differ;
    }
    return differ <= 1;
  }

  // The entries that one of PARTS warps applies (rows i = Q mod PARTS), in the order it applies
  // them: slot by slot, column by column, then row by row, so that consecutive multiplications
  // go to different rows.  Every row still sees its entries in the order (slot, column).
  template <int PARTS, int Q> struct Part {
    static constexpr int ROWS = (NP - Q + PARTS - 1) / PARTS;
    struct Tab {
      short n;                  // entries, slot 0 padded to an even number
      short begin[S + 1];       // first entry of each slot
      signed char i[S * NP * NP + 2], j[S * NP * NP + 2];   // row and column (row -1: padding)
    };
    static constexpr Tab make() {
      const Modes m = make_modes();
      Tab t{};
      int c = 0;
      for (int s = 0; s < S; ++s) {
        t.begin[s] = (short)c;
        for (int j = 0; j < NP; ++j)
          for (int i = Q; i < NP; i += PARTS)
            if (nz(m, s, i, j)) {
              t.i[c] = (signed char)i;
              t.j[c] = (signed char)j;
              ++c;
            }
        if (s == 0 && (c & 1)) {
          t.i[c] = -1;
          ++c;
        }
      }
      t.begin[S] = (short)c;
      t.n = (short)c;
      return t;
    }
    static constexpr Tab tab = make();
    static constexpr int PAIRS = (tab.n + 1) / 2;
  };
  // pairs of stored values per 32 cells and lane: the largest part's, for every part
  template <int PARTS> static constexpr int max_pairs() {
    int m = Part<PARTS, 0>::PAIRS;
    if constexpr (PARTS > 1) m = m > Part<PARTS, 1>::PAIRS ? m : Part<PARTS, 1>::PAIRS;
    if constexpr (PARTS > 2) {
      m = m > Part<PARTS, 2>::PAIRS ? m : Part<PARTS, 2>::PAIRS;
      m = m > Part<PARTS, 3>::PAIRS ? m : Part<PARTS, 3>::PAIRS;
    }
    return m;
  }
  // columns of row i outside the pattern of slot s, one bit each
  struct Zeros { unsigned m[S][NP]; };
  static constexpr Zeros make_zeros() {
    const Modes m = make_modes();
    Zeros z{};
    for (int s = 0; s < S; ++s)
      for (int i = 0; i < NP; ++i)
        for (int j = 0; j < NP; ++j)
          if (!nz(m, s, i, j)) z.m[s][i] |= 1u << j;
    return z;
  }

  // warps that share a group of 32 cells, each with every PARTS-th row
  static constexpr int PARTS = NP == 20 ? 4 : (NP == 10 || NP == 6) ? 2 : 1;
  static constexpr int PAIRS = max_pairs<PARTS>();
  // pairs of inverse entries of the largest part
  static constexpr int INV_PAIRS = (((NP + PARTS - 1) / PARTS) * NP + 1) / 2;
};

}  // namespace kcmg
