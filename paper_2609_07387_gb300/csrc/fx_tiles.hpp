// The FP64 form's reconstruction tiles from P2 on, built on the host from the
// precompute's rows: limb pairs and row exponents (fixed.cuh) in the order in
// which the kernels stream them (FxTile, HOFxTile).  The functions run inside
// OpenMP regions, which an exception must not leave: they allocate nothing.
#pragma once

#include <algorithm>
#include <cmath>
#include <cstdint>

#include "host_arrays.hpp"
#include "kernels.cuh"
#include "kernels_ho.cuh"

namespace ucns {

// One matrix row of nc <= 32 consecutive cells, entry m of cell c at row(m)[c], as
// limb pairs at(m)[c] and exponents E[c] (fixed.cuh); a row with a NaN or an infinity
// (a smoothness matrix whose moments left FP64's range) has zeros and the NaN exponent
template <class Row, class At>
void fixed_row(const Row& row, int M, int nc, const At& at, int16_t* E) {
  double l1[32] = {0.0}, up[32], more[32];
  for (int m = 0; m < M; m++) {
    const double* x = row(m);
    for (int c = 0; c < nc; c++) l1[c] += std::fabs(x[c]);
  }
  for (int c = 0; c < nc; c++) {
    const int e = fx_row_exponent(l1[c]);
    E[c] = (int16_t)e;
    up[c] = std::ldexp(1.0, std::min(60 - e, 1000));
    more[c] = std::ldexp(1.0, std::max(60 - e - 1000, 0));
  }
  for (int m = 0; m < M; m++) {
    const double* x = row(m);
    int2* q = at(m);
    for (int c = 0; c < nc; c++) q[c] = E[c] == kFxNan - 1 ? make_int2(0, 0) : fx_limbs(fx_round(x[c] * up[c] * more[c]));
  }
}

// record r of tile t of the P2 reconstruction (zero on entry)
inline void fx_tile(const HostArrays& h, int nd, int64_t N, int64_t t, unsigned char* r) {
  using T = FxTile;
  const int64_t i0 = t * T::TC;
  const int nc = (int)std::min<int64_t>(T::TC, N - i0);
  auto rows = [&](const std::vector<double>& src, int K, int M, int2* P, int16_t* E) {
    for (int k = 0; k < K; k++)
      fixed_row([&](int mm) { return src.data() + ((size_t)k * M + mm) * N + i0; }, M, nc,
                [&](int mm) { return P + (k * M + mm) * T::TC; }, E + k * T::TC);
  };
  auto stencils = [&](const std::vector<int32_t>& src, int M, int32_t* id) {
    for (int mm = 0; mm < M; mm++) std::copy_n(src.data() + (size_t)mm * N + i0, nc, id + mm * T::TC);
  };
  rows(h.Pc, T::K, T::MC, reinterpret_cast<int2*>(r), reinterpret_cast<int16_t*>(r + T::C_EXP));
  stencils(h.sc, T::MC, reinterpret_cast<int32_t*>(r + T::C_ID));
  if (nd == 0) return;
  unsigned char* dr = r + T::CENTRAL;
  rows(h.Pd, nd * 3, T::MD, reinterpret_cast<int2*>(dr), reinterpret_cast<int16_t*>(dr + T::d_exp(nd)));
  stencils(h.sd, nd * T::MD, reinterpret_cast<int32_t*>(dr + T::d_id(nd)));
}

// record rec of tile t of the P3/P4 reconstruction, its stencils id and row exponents ex (zero on entry)
template <int ORDER>
void ho_fx_tile(const HostArrays& h, bool weno, int64_t N, int64_t t, unsigned char* rec, int32_t* id, int16_t* ex) {
  using T = HOFxTile<ORDER>;
  constexpr int K = T::K, MC = T::MC, KD = T::KD, MD = T::MD, TC = T::TC;
  int2* r = reinterpret_cast<int2*>(rec);
  const int64_t i0 = t * TC;
  const int nc = (int)std::min<int64_t>(TC, N - i0);
  for (int mm = 0; mm < MC; mm++) std::copy_n(h.sc.data() + (size_t)mm * N + i0, nc, id + mm * TC);
  for (int k = 0; k < K; k++)
    fixed_row([&](int mm) { return h.Pc.data() + ((size_t)k * MC + mm) * N + i0; }, MC, nc,
              [&](int mm) {
                return r + (((k / 4) * T::NP + mm / T::MCH) * 4 * T::MCH + (k % 4) * T::MCH + mm % T::MCH) * TC;
              },
              ex + k * TC);
  if (!weno) return;
  int2* at = r + T::CENTRAL / 8;
  for (int g = 0; g < T::NG; g++) {
    const int cols = K - 4 * g;  // columns from the group's first row on, in pieces of MCH
    for (int rr = 0; rr < 4 && 4 * g + rr < K; rr++) {
      const int k = 4 * g + rr;  // row k: zero below the diagonal, off-diagonal entries doubled
      double x[(size_t)K * TC] = {0.0};
      for (int l = k; l < K; l++)
        for (int c = 0; c < nc; c++)
          x[(size_t)(l - 4 * g) * TC + c] =
              (l == k ? 1.0 : 2.0) * h.Msi[(size_t)(k * K - k * (k - 1) / 2 + l - k) * N + i0 + c];
      fixed_row([&](int l) { return x + (size_t)l * TC; }, cols, nc,
                [&](int l) {
                  const int p = l / T::MCH;
                  return at + (4 * p * T::MCH + rr * T::si_columns(g, p) + l % T::MCH) * TC;
                },
                ex + (K + k) * TC);
    }
    at += 4 * cols * TC;
  }
  for (int mm = 0; mm < 6 * MD; mm++) std::copy_n(h.sd.data() + (size_t)mm * N + i0, nc, id + (MC + mm) * TC);
  for (int k = 0; k < 6 * KD; k++)  // row k % KD of stencil k / KD
    fixed_row([&](int mm) { return h.Pd.data() + ((size_t)k * MD + mm) * N + i0; }, MD, nc,
              [&](int mm) { return at + ((k / 3) * 3 * MD + (k % 3) * MD + mm) * TC; }, ex + (2 * K + k) * TC);
}

}  // namespace ucns
