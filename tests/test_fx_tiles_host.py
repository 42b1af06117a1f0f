"""The host conversion of the precompute's rows into the FP64 form's tiles
(csrc/fx_tiles.hpp): no allocation inside the OpenMP region that calls it (an
exception there would end the process instead of becoming an error code), and
entries, stencils and row exponents at their places, on a ragged last tile."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2609_07387_gb300", "csrc")

PROGRAM = r"""
#include <atomic>
#include <cstdio>
#include <cstdlib>
#include <new>
#include <random>
#include "fx_tiles.hpp"
using namespace ucns;
std::atomic<int> armed{0}, allocations{0};
void* operator new(size_t n) {
#ifndef __CUDA_ARCH__
  if (armed) allocations++;
#endif
  return malloc(n);
}
void operator delete(void* p) noexcept { free(p); }
void operator delete(void* p, size_t) noexcept { free(p); }

std::mt19937_64 rng(3);
const int64_t N = 24 + 7;
void fill(std::vector<double>& v, size_t n) {
  v.resize(n);
  for (double& x : v) x = (2.0 * (double)(rng() >> 11) / 9007199254740992.0 - 1.0) * std::ldexp(1.0, (int)(rng() % 30));
}
void fill(std::vector<int32_t>& v, size_t n) {
  v.resize(n);
  for (int32_t& x : v) x = (int32_t)(rng() % N);
}
double back(int2 q, int E) { return std::ldexp((double)fx_value(q), E - 60); }
// entry (q, E) of a row whose largest sum is below 2^E against the value x
int off(int2 q, int E, double x) { return !(std::fabs(back(q, E) - x) <= std::ldexp(1.0, E - 60)); }

int p2(int nd) {
  using T = FxTile;
  HostArrays h;
  fill(h.Pc, (size_t)T::K * T::MC * N);
  fill(h.sc, (size_t)T::MC * N);
  fill(h.Pd, (size_t)nd * 3 * T::MD * N);
  fill(h.sd, (size_t)nd * T::MD * N);
  std::vector<unsigned char> r(T::record(nd), 0);
  armed = 1;
  fx_tile(h, nd, N, 0, r.data());
  armed = 0;
  int bad = 0;
  const int2* P = reinterpret_cast<const int2*>(r.data());
  const int16_t* E = reinterpret_cast<const int16_t*>(r.data() + T::C_EXP);
  const unsigned char* dr = r.data() + T::CENTRAL;
  for (int c = 0; c < T::TC; c++) {
    for (int k = 0; k < T::K; k++)
      for (int m = 0; m < T::MC; m++)
        bad += off(P[(k * T::MC + m) * T::TC + c], E[k * T::TC + c], c < N ? h.Pc[((size_t)k * T::MC + m) * N + c] : 0.0);
    for (int k = 0; k < nd * 3; k++)
      for (int m = 0; m < T::MD; m++)
        bad += off(reinterpret_cast<const int2*>(dr)[(k * T::MD + m) * T::TC + c],
                   reinterpret_cast<const int16_t*>(dr + T::d_exp(nd))[k * T::TC + c],
                   c < N ? h.Pd[((size_t)k * T::MD + m) * N + c] : 0.0);
    for (int m = 0; m < nd * T::MD; m++)
      bad += reinterpret_cast<const int32_t*>(dr + T::d_id(nd))[m * T::TC + c] != (c < N ? h.sd[(size_t)m * N + c] : 0);
  }
  return bad;
}

template <int ORDER> int ho() {
  using T = HOFxTile<ORDER>;
  HostArrays h;
  fill(h.Pc, (size_t)T::K * T::MC * N);
  fill(h.sc, (size_t)T::MC * N);
  fill(h.Pd, (size_t)6 * T::KD * T::MD * N);
  fill(h.sd, (size_t)6 * T::MD * N);
  fill(h.Msi, (size_t)T::K * (T::K + 1) / 2 * N);
  int bad = 0;
  for (int t = 0; t < 2; t++) {
    std::vector<unsigned char> r(T::record(true), 0);
    std::vector<int32_t> id(T::IDS * T::TC, 0);
    std::vector<int16_t> ex(T::EXPS * T::TC, 0);
    armed = 1;
    ho_fx_tile<ORDER>(h, true, N, t, r.data(), id.data(), ex.data());
    armed = 0;
    const int2* q = reinterpret_cast<const int2*>(r.data());
    const int2* si = q + T::CENTRAL / 8;
    for (int g = 0; g < T::NG; g++) {
      for (int p = 0; p < T::NP; p++)
        for (int rr = 0; rr < 4; rr++)
          for (int mm = 0; mm < T::MCH; mm++, q += T::TC)
            for (int c = 0; c < T::TC; c++) {
              const int k = 4 * g + rr, m = p * T::MCH + mm;
              const bool in = k < T::K && t * T::TC + c < N;
              bad += off(q[c], in ? ex[k * T::TC + c] : 0, in ? h.Pc[((size_t)k * T::MC + m) * N + t * T::TC + c] : 0.0);
            }
      for (int p = 0; p < T::si_pieces(g); p++)
        for (int rr = 0; rr < 4; rr++)
          for (int mm = 0; mm < T::si_columns(g, p); mm++, si += T::TC)
            for (int c = 0; c < T::TC; c++) {
              const int k = 4 * g + rr, l = 4 * g + p * T::MCH + mm;
              const bool in = k < T::K && l >= k && t * T::TC + c < N;
              const double x = in ? h.Msi[(size_t)(k * T::K - k * (k - 1) / 2 + l - k) * N + t * T::TC + c] : 0.0;
              bad += off(si[c], in ? ex[(T::K + k) * T::TC + c] : 0, l == k ? x : 2.0 * x);
            }
    }
    for (int k = 0; k < 6 * T::KD; k++)
      for (int m = 0; m < T::MD; m++, si += T::TC)
        for (int c = 0; c < T::TC; c++) {
          const bool in = t * T::TC + c < N;
          bad += off(si[c], in ? ex[(2 * T::K + k) * T::TC + c] : 0, in ? h.Pd[((size_t)k * T::MD + m) * N + t * T::TC + c] : 0.0);
        }
    for (int c = 0; c < T::TC; c++)
      for (int m = 0; m < T::IDS; m++) {
        const std::vector<int32_t>& s = m < T::MC ? h.sc : h.sd;
        bad += id[m * T::TC + c] != (t * T::TC + c < N ? s[(size_t)(m < T::MC ? m : m - T::MC) * N + t * T::TC + c] : 0);
      }
  }
  return bad;
}

// a sum over a row of two cells, the second's with one entry bad, times members 1, ..., 6
void non_finite(double bad) {
  double x[6][2], U[6];
  int2 P[6][2], q[6];
  int16_t E[2];
  int e;
  for (int m = 0; m < 6; m++) {
    x[m][0] = x[m][1] = 0.25 * m;
    U[m] = 1.0 + m;
  }
  x[4][1] = bad;
  fixed_row([&](int m) { return x[m]; }, 6, 2, [&](int m) { return P[m]; }, E);
  fx_differences<6>(U, 0.0, q, e);
  for (int c = 0; c < 2; c++) {
    FxAcc acc;
    for (int m = 0; m < 6; m++) fx_mac(acc, P[m][c], q[m]);
    printf(" %g", fx_double(fx_sum(acc), E[c] + e - 2 - fx_bits_of(6)));
  }
}

int main() {
  const int a = p2(0) + p2(6), b = ho<3>(), c = ho<4>();
  printf("%d %d %d %d", a, b, c, (int)allocations);
  non_finite(NAN);
  non_finite(INFINITY);
  non_finite(-INFINITY);
  printf("\n");
}
"""


@pytest.fixture(scope="module")
def out(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not found")
    d = tmp_path_factory.mktemp("tiles")
    (d / "t.cu").write_text(PROGRAM)
    subprocess.run([nvcc, "-O1", "-std=c++17", "-gencode", "arch=compute_103a,code=sm_103a", "-I", CSRC, "-o", str(d / "t"),
                    str(d / "t.cu")], check=True, capture_output=True)
    return subprocess.run([str(d / "t")], check=True, capture_output=True, text=True).stdout.split()


def test_tiles(out):
    assert out[:3] == ["0", "0", "0"]  # misplaced entries at P2, P3, P4
    assert out[3] == "0"  # allocations while a tile is converted


def test_non_finite_rows_give_nan(out):
    """As FP64 sums do: 17.5 over the sound row, NaN over one with a NaN or an infinity."""
    assert [x.strip("-") for x in out[4:]] == ["17.5", "nan"] * 3
