"""The fixed-point sums of csrc/fixed.cuh on the host, against exact rational
arithmetic: differences, contractions, polynomial coefficients and conversions
of FP64 values of one magnitude, spread over many binades, at and beside powers
of two, subnormal and near the largest, and non-finite ones.
The bounds are those of the header: a sum is off by at most (2^-57 + M 2^-56.5)
sum|P| max|u_m - u_0| and the final rounding."""
import os
import shutil
import subprocess
from fractions import Fraction

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2609_07387_gb300", "csrc")

PROGRAM = r"""
#include "basis.hpp"
#include "fixed.cuh"
#include <cstdio>
#include <random>
using namespace ucns;
std::mt19937_64 g(5);
double u() { return 2.0 * (double)(g() >> 11) / 9007199254740992.0 - 1.0; }
template <int M> void sums(double scale, double spread) {
  for (int t = 0; t < 40; t++) {
    double P[M], U[M], l1 = 0.0, u0 = scale * (1.0 + spread * u());
    for (int m = 0; m < M; m++) {
      P[m] = u() * std::exp(2.0 * u());
      U[m] = scale * (1.0 + spread * u());
      l1 += std::fabs(P[m]);
    }
    printf("sum %d %a", M, u0);
    for (int m = 0; m < M; m++) printf(" %a %a", P[m], U[m]);
    const int E = fx_row_exponent(l1);
    int2 q[M];
    int e;
    fx_differences<M>(U, u0, q, e);
    FxAcc acc;
    for (int m = 0; m < M; m++) fx_mac(acc, fx_limbs(fx_round(std::ldexp(P[m], 60 - E))), q[m]);
    printf(" %a\n", fx_double(fx_sum(acc), E + e - 2 - fx_bits_of(M)));
  }
}
// one sum of edge values: members that are signed powers of two, their neighbours in
// FP64, or of many decades, against centres far below (dir 0), or the reverse (dir 1)
template <int M> void edge(int k, int j, int kind, int dir, double sign) {
  double P[M], U[M], l1 = 0.0;
  const double big = sign * std::ldexp(1.0, k), small = (j % 2 ? -1.0 : 1.0) * std::ldexp(1.0 + 0.7 * (j % 3), k - j);
  double u0 = dir ? big : small;
  if (kind == 1 && dir) u0 = std::nextafter(big, 0.0);
  for (int m = 0; m < M; m++) {
    double x = dir ? small : big;
    if (m % 3 == 1) x = dir ? -small : small;
    if (kind == 1 && !dir) x = m % 2 ? std::nextafter(x, 0.0) : std::nextafter(x, 2.0 * x);
    if (kind == 2 && m % 3) x = u() * std::ldexp(1.0, k - (int)(g() % 120));
    U[m] = x;
    P[m] = u();
    l1 += std::fabs(P[m]);
  }
  printf("edge %d %a", M, u0);
  for (int m = 0; m < M; m++) printf(" %a %a", P[m], U[m]);
  const int E = fx_row_exponent(l1);
  int2 q[M];
  int e;
  fx_differences<M>(U, u0, q, e);
  FxAcc acc;
  for (int m = 0; m < M; m++) fx_mac(acc, fx_limbs(fx_round(std::ldexp(P[m], 60 - E))), q[m]);
  printf(" %a\n", fx_double(fx_sum(acc), E + e - 2 - fx_bits_of(M)));
}
template <int M> void edges() {
  for (int k : {0, 8, -3})
    for (int j = 50; j <= 66; j++)
      for (int kind = 0; kind < 3; kind++)
        for (int dir = 0; dir < 2; dir++)
          for (double sign : {1.0, -1.0}) edge<M>(k, j, kind, dir, sign);
}
// the coefficients of a polynomial on a cell of axis scale 2^h: about 2^u each in scaled
// coordinates, so of 2^(u - deg h), some zero
template <int ORDER> void coefficients(int h, int u2, bool zeros) {
  constexpr int K = basis_count(ORDER), B = ORDER == 4 ? 57 : 58;
  double c[K];
  int off[K], e;
  for (int k = 0; k < K; k++) {
    off[k] = basis_degree(k) * h;
    c[k] = std::ldexp(u(), u2 - off[k] - (int)(g() % 12));
    if (zeros && (k >= 3 || g() % 2)) c[k] = 0.0;
    if (!std::isfinite(c[k])) return;
  }
  double in[K];
  for (int k = 0; k < K; k++) in[k] = c[k];
  const int eb = fx_align_scaled<K>(c, off, e);
  printf("poly %d %d", B, e);
  for (int k = 0; k < K; k++) printf(" %a %d %lld", in[k], off[k], fx_value(fx_operand<B>(c[k], eb - off[k])));
  printf("\n");
}
int main() {
  for (int h : {-180, -20, 0, 12, 40, 90, 170})
    for (int u2 : {0, 300, -330, -700, -860, -960, -1030})
      for (int t = 0; t < 8; t++) {
        coefficients<2>(h, u2, t % 2);
        coefficients<3>(h, u2, t % 2);
        coefficients<4>(h, u2, t % 2);
      }
  edges<6>();
  edges<18>();
  edges<38>();
  edges<68>();
  for (double spread : {1e-9, 0.1, 10.0})
    for (double scale : {1.0, 1e-200, 1e200, 0x1p-1000}) { sums<6>(scale, spread); sums<18>(scale, spread); sums<68>(scale, spread); }
  for (int t = 0; t < 4000; t++) {
    const long long s = (long long)g() >> (g() % 63);
    const int e = (int)(g() % 2100) - 1080;
    printf("double %lld %d %a\n", s, e, fx_double(s, e));
    const double a = u() * std::ldexp(1.0, (int)(g() % 200) - 100), b = u() * std::ldexp(1.0, (int)(g() % 200) - 100);
    printf("add %a %a %a\n", a, b, fx_double(fx_add(fx_of(a), fx_of(b))));
  }
  double w[6] = {1.0, NAN, 1.0, 1.0, 1.0, 1.0}, z[6] = {3.0, 3.0, 3.0, 3.0, 3.0, 3.0};
  int2 q[6];
  int e;
  fx_differences<6>(w, 1.0, q, e);
  printf("nan %a %a %a\n", fx_double(fx_value(q[0]), e - 58), fx_double(fx_add(fx_of(INFINITY), fx_of(1.0))), fx_double(fx_add(fx_of(1.0), fx_of(NAN))));
  fx_differences<6>(z, 3.0, q, e);
  printf("zero %a\n", fx_double(fx_value(q[2]), e - 58));
}
"""


@pytest.fixture(scope="module")
def lines(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not found")
    d = tmp_path_factory.mktemp("fixed")
    (d / "t.cu").write_text(PROGRAM)
    subprocess.run([nvcc, "-O2", "-std=c++17", "-gencode", "arch=compute_103a,code=sm_103a", "-I", CSRC, "-o", str(d / "t"),
                    str(d / "t.cu")], check=True, capture_output=True)
    return [x.split() for x in subprocess.run([str(d / "t")], check=True, capture_output=True, text=True).stdout.splitlines()]


def _exact(x):
    return Fraction(float.fromhex(x))


def test_contractions(lines):
    n = 0
    for w in (w for w in lines if w[0] == "sum"):
        M, u0 = int(w[1]), _exact(w[2])
        P, U = [_exact(x) for x in w[3:-1:2]], [_exact(x) for x in w[4:-1:2]]
        exact = sum(p * (x - u0) for p, x in zip(P, U))
        scale = sum(abs(p) for p in P) * max(abs(x - u0) for x in U)
        bound = scale * (Fraction(1, 1 << 57) + M * Fraction(3, 1 << 58)) + abs(exact) / (1 << 53) + Fraction(1, 1 << 1074)
        assert abs(_exact(w[-1]) - exact) <= bound, (M, float(abs(_exact(w[-1]) - exact) / scale))
        n += 1
    assert n == 40 * 3 * 4 * 3


def _check(w):
    M, u0 = int(w[1]), _exact(w[2])
    P, U = [_exact(x) for x in w[3:-1:2]], [_exact(x) for x in w[4:-1:2]]
    exact = sum(p * (x - u0) for p, x in zip(P, U))
    scale = sum(abs(p) for p in P) * max(abs(x - u0) for x in U)
    bound = scale * (Fraction(1, 1 << 57) + M * Fraction(3, 1 << 58)) + abs(exact) / (1 << 53)
    return M, w[2], float(abs(_exact(w[-1]) - exact) / scale) if abs(_exact(w[-1]) - exact) > bound else 0.0


def test_contractions_at_powers_of_two(lines):
    """Differences within a few units of a power of two: members that are signed powers
    of two (or next to one, or spread over 120 binades) and centres 2^-50 to 2^-66 of
    them, either way round, in the header's bound (test_contractions states it)."""
    off = [_check(w) for w in lines if w[0] == "edge"]
    assert len(off) == 4 * 3 * 17 * 3 * 2 * 2
    assert [x for x in off if x[2]] == []


def test_coefficients(lines):
    """Polynomial coefficients c_k scaled by 2^off_k and aligned to the largest of them
    (csrc/kernels.cuh, store_fixed): half a unit 2^(e - B) of error each, the unit not more
    than that of the largest; cells of any size, states that make some coefficients
    subnormal or zero."""
    n = 0
    for w in (w for w in lines if w[0] == "poly"):
        B, e = int(w[1]), int(w[2])
        exact = [_exact(c) * Fraction(2) ** int(off) for c, off in zip(w[3::3], w[4::3])]
        q = [int(x) for x in w[5::3]]
        big = max(abs(x) for x in exact)
        if big == 0:
            assert q == [0] * len(q)
            continue
        unit = Fraction(2) ** (e - B)
        assert unit <= 2 * big / (1 << B), (e, float(big))
        assert all(abs(x - y * unit) <= unit / 2 and abs(y) <= 1 << B for x, y in zip(exact, q)), (w[:3], float(big))
        n += 1
    assert n > 800


def test_conversions(lines):
    for w in (w for w in lines if w[0] == "double"):
        exact = int(w[1]) * Fraction(2) ** int(w[2])
        if abs(exact) < Fraction(2) ** 1024:  # one rounding to nearest, or a subnormal result
            assert abs(_exact(w[3]) - exact) <= abs(exact) / (1 << 53) + Fraction(1, 1 << 1074)
        else:
            assert float.fromhex(w[3]) in (float("inf"), float("-inf"))
    for w in (w for w in lines if w[0] == "add"):
        a, b = _exact(w[1]), _exact(w[2])
        assert abs(_exact(w[3]) - (a + b)) <= abs(a + b) / (1 << 53) + max(abs(a), abs(b)) / (1 << 59)


def test_special_values(lines):
    nan = next(w for w in lines if w[0] == "nan")
    assert all(x.strip("-") == "nan" for x in nan[1:])
    assert float.fromhex(next(w for w in lines if w[0] == "zero")[1]) == 0.0
