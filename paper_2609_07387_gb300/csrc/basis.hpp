// Monomial basis of the reconstruction polynomial (Eq. 3): psi_k = xi^e_k,
// xi = (x - x_i)/h_i, h_i = |V_i|^(1/3), k = 0 .. K(r) - 1 with
// K(r) = (r+1)(r+2)(r+3)/6 - 1 non-constant modes (3, 9, 19, 34 for r = 1..4).
// Shared by the host precompute and the kernels.
#pragma once

#ifdef __CUDACC__
#define UCNS_HD __host__ __device__
#else
#define UCNS_HD
#endif

namespace ucns {

constexpr int kMaxOrder = 4;

UCNS_HD constexpr int basis_count(int r) { return (r + 1) * (r + 2) * (r + 3) / 6 - 1; }

// exponent of coordinate d in basis monomial k: the nine of P2 in the order
// x y z xx yy zz xy xz yz, then the cubics and the quartics, each by
// descending power of x, then of y
UCNS_HD constexpr int basis_exp(int k, int d) {
  constexpr signed char t[34][3] = {
      {1, 0, 0}, {0, 1, 0}, {0, 0, 1}, {2, 0, 0}, {0, 2, 0}, {0, 0, 2}, {1, 1, 0}, {1, 0, 1}, {0, 1, 1},
      {3, 0, 0}, {2, 1, 0}, {2, 0, 1}, {1, 2, 0}, {1, 1, 1}, {1, 0, 2}, {0, 3, 0}, {0, 2, 1}, {0, 1, 2}, {0, 0, 3},
      {4, 0, 0}, {3, 1, 0}, {3, 0, 1}, {2, 2, 0}, {2, 1, 1}, {2, 0, 2}, {1, 3, 0}, {1, 2, 1}, {1, 1, 2}, {1, 0, 3},
      {0, 4, 0}, {0, 3, 1}, {0, 2, 2}, {0, 1, 3}, {0, 0, 4}};
  return t[k][d];
}

UCNS_HD constexpr int basis_degree(int k) { return basis_exp(k, 0) + basis_exp(k, 1) + basis_exp(k, 2); }

// the mode with exponents (a, b, c), of degree 1 or more
UCNS_HD constexpr int basis_index(int a, int b, int c) {
  const int deg = a + b + c, i = b + c;
  if (deg == 2) return a == 2 ? 3 : (b == 2 ? 4 : (c == 2 ? 5 : (c == 0 ? 6 : (b == 0 ? 7 : 8))));
  return basis_count(deg - 1) + i * (i + 1) / 2 + (i - b);
}

// the mode of basis monomial k divided by coordinate d (k of degree 2 or more, with exponent of d at least 1)
UCNS_HD constexpr int basis_lower(int k, int d) {
  return basis_index(basis_exp(k, 0) - (d == 0), basis_exp(k, 1) - (d == 1), basis_exp(k, 2) - (d == 2));
}

// Place of a monomial (k = -1: the constant) in the order in which a nested Horner
// evaluation of degree r reads the coefficients: by descending power of z, then of
// y, then of x, the constant last
UCNS_HD constexpr int horner_place(int k, int r) {
  const int e[3] = {k < 0 ? 0 : basis_exp(k, 0), k < 0 ? 0 : basis_exp(k, 1), k < 0 ? 0 : basis_exp(k, 2)};
  const int D = r - e[2], E = D - e[1];  // degrees left in (x, y) and in x
  // levels above in z: sum of (d+1)(d+2)/2 for d < D; in y: sum of (d+1) for d < E
  return D * (D + 1) * (D + 2) / 6 + E * (E + 1) / 2 + E - e[0];
}

}  // namespace ucns
