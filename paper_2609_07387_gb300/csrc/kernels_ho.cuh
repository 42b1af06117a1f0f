// P3 and P4 reconstruction and face kernels (FP64), hexahedra.
//
//   k_recon_ho  tile by tile, thread = (cell, variable): central least-squares
//               contraction (K = 19 or 34 modes over 2K members, Eq. 4) in
//               fixed point; with CWENOZ the six directional candidates
//               (linear at P3, quadratic over 18 members at P4, Sec. 2.2), the
//               smoothness indicators as the quadratic forms a^T M a of each
//               cell's precomputed matrix M (Eq. 6 reading), the nonlinear
//               weights and the combination.
//   k_face_ho   ORDER^2 Gauss points per face on ORDER^2 lanes (9 at P3, 16
//               at P4; 32 / ORDER^2 faces per warp); values and gradients of
//               the monomial-form polynomials, HLLC, penalised viscous flux
//               (Eq. 7), and each (face, variable) total summed by a lane of
//               its own in point order (deterministic).
//   k_recon_ho_mx the same in the mixed form, tile by tile (32 cells): the
//               stencil ids and FP32 pseudo-inverses stream through shared
//               memory in bulk-copied chunks, thread = (cell, variable).
//   (the mixed face kernel of every order is k_face_mx, kernels_mixed.cuh)
#pragma once

#include "basis.hpp"
#include "kernels.cuh"
#include "kernels_mixed.cuh"

namespace ucns {

template <int ORDER>
struct HO {
  static constexpr int K = basis_count(ORDER);
  static constexpr int MC = 2 * K;
  static constexpr int KD = ORDER == 4 ? 9 : 3;  // modes of a directional candidate
  static constexpr int MD = 2 * KD;
  static constexpr int NQ = ORDER * ORDER;
};

// The FP64 form's reconstruction data, tile by tile (24 cells: four warps of (cell,
// variable) threads, one on each scheduler), in fixed point (fixed.cuh).  Streamed
// chunks: the central rows in groups of four, each in pieces of MCH members, [4][MCH][24]
// limb pairs; with CWENOZ the smoothness matrix's rows in groups of four, upper
// triangle (off-diagonal entries doubled), columns from the group's first row on in
// pieces of MCH, [4][columns][24]; then per directional stencil its rows in groups of
// three, [3][MD][24].  Rows past K and cells past N are zero.
template <int ORDER>
struct HOFxTile {
  using H = HO<ORDER>;
  static constexpr int K = H::K, MC = H::MC, KD = H::KD, MD = H::MD, TC = 24;
  static constexpr int LANES = 128, THREADS = LANES + 32;  // 120 (cell, variable) threads and 8 spare ones, a copying warp
  static constexpr int MCH = ORDER == 4 ? 17 : 19, NP = MC / MCH, NG = (K + 3) / 4, NGD = KD / 3;
  static constexpr int CHUNK = 4 * MCH * TC * 8;  // bytes of a stage
  static constexpr int DCHUNK = 3 * MD * TC * 8;
  static constexpr int S = 3;
  static constexpr int QB = MC * LANES * 8;  // operands of the sum at hand, one column per thread
  // per tile: stencil ids [MC + 6 MD][24], row exponents [2 K + 6 KD][24] (central, matrix, directional)
  static constexpr int IDS = MC + 6 * MD, EXPS = 2 * K + 6 * KD, EB = EXPS * TC * 2;
  static constexpr int SMEM = QB + S * CHUNK + EB + 2 * S * 8 + 8;
  UCNS_HD static constexpr int si_pieces(int g) { return (K - 4 * g + MCH - 1) / MCH; }
  UCNS_HD static constexpr int si_columns(int g, int p) { return K - 4 * g - p * MCH < MCH ? K - 4 * g - p * MCH : MCH; }
  // bytes of the smoothness matrix, and of a tile's record
  UCNS_HD static constexpr int si_bytes() {
    int n = 0;
    for (int g = 0; g < NG; g++) n += 4 * (K - 4 * g) * TC * 8;
    return n;
  }
  static constexpr int CENTRAL = NG * NP * CHUNK;
  UCNS_HD static constexpr int record(bool weno) { return CENTRAL + (weno ? si_bytes() + 6 * NGD * DCHUNK : 0); }
  static_assert(MC % MCH == 0 && EB % 16 == 0 && 6 * KD <= MC && DCHUNK <= CHUNK && CHUNK % 16 == 0 && DCHUNK % 16 == 0 && QB % 16 == 0, "whole chunks");
};

struct ReconArgsHO {
  const double* __restrict__ U;     // [5][N]
  const unsigned char* __restrict__ tiles;  // records (HOFxTile)
  const int32_t* __restrict__ ids;          // [tiles][IDS][24]
  const int16_t* __restrict__ exps;         // [tiles][EXPS][24]
  const double* __restrict__ Msi;   // [KD(KD+1)/2][N]: the smoothness-indicator matrix's leading block, upper triangle by rows
  const double* __restrict__ psib;  // [K-3][N]: cell means of the basis monomials of degree >= 2
  const double* __restrict__ inv_h; // [N]
  const short4* __restrict__ hexp;  // [N] exponents of the cell's axis scales
  double* __restrict__ coef;        // [K+1][N][5] physical-unit monomial coefficients, the non-constant ones in fixed point
  int32_t* __restrict__ cexp;       // [N][5] their exponents
  int* err;                         // bit 1: a copy wait gave up
  int N;
  double lam0, lams, eps;
};

// a^T M a (M: K x K symmetric, upper triangle stored by rows: entry (k, l >= k) at
// q = k K - k (k - 1) / 2 + l - k)
template <int K>
__device__ __forceinline__ double si_form(const double* __restrict__ M, size_t N, int i, const double (&a)[K]) {
  double s = 0.0;
#pragma unroll
  for (int k = 0; k < K; k++) {
    double t = 0.0;
#pragma unroll
    for (int l = k + 1; l < K; l++) t = fma(__ldg(&M[(size_t)(k * K - k * (k - 1) / 2 + l - k) * N + i]), a[l], t);
    const double mkk = __ldg(&M[(size_t)(k * K - k * (k - 1) / 2) * N + i]);
    s = fma(a[k], fma(2.0, t, mkk * a[k]), s);
  }
  return s;
}

// One block per 24-cell tile: thread (cell c, variable v) = 5 c + v, plus a copying
// warp that streams the tile's chunks through a ring of S shared-memory stages, every
// wait bounded.  The differences of a stencil wait in shared memory as operands while
// its rows pass; the central coefficients (xi units) wait in the output array.
// Bound by latency at two warps per scheduler (P4: issue 28 %, FP64 pipe 42 %): 11
// thousand integer multiply-adds a thread at P4.  P4 CWENOZ at 24^3, us: FP64
// contractions from global memory 852, this 329 (418 with the directional
// contractions run twice and the row exponents read from global memory).
template <int ORDER, bool WENO>
__global__ void __launch_bounds__(HOFxTile<ORDER>::THREADS, 2) k_recon_ho(ReconArgsHO a) {
  using T = HOFxTile<ORDER>;
  constexpr int K = T::K, MC = T::MC, KD = T::KD, MD = T::MD, ND = 6, TC = T::TC, S = T::S, L = T::LANES;
  extern __shared__ __align__(128) unsigned char smem[];
  long long* sQ = reinterpret_cast<long long*>(smem);
  unsigned char* ring = smem + T::QB;
  unsigned char* sE = ring + S * T::CHUNK;  // the row exponents
  uint64_t* full = reinterpret_cast<uint64_t*>(sE + T::EB);
  uint64_t* empty = full + S;
  uint64_t* ebar = empty + S;
  const int t = threadIdx.x, lane = t & 31, tile = blockIdx.x;
  if (t < S) {
    bar_init(&full[t]);
    bar_init(&empty[t], L / 32);
  }
  if (t == S) bar_init(ebar);
  __syncthreads();
  if (t >= L) {  // the copying warp
    if (lane != 0) return;
    bar_expect(ebar, T::EB);
    bulk_load(sE, a.exps + (size_t)tile * T::EXPS * TC, T::EB, ebar);
    const unsigned char* rec = a.tiles + (size_t)tile * T::record(WENO);
    int q = 0;
    bool ok = true;
    auto put = [&](const unsigned char* src, int bytes) {
      ok = ok && (q < S || bar_wait(&empty[q % S], (uint32_t)(q / S + 1) & 1u));
      if (!ok) return;
      bar_expect(&full[q % S], (uint32_t)bytes);
      bulk_load(ring + (q % S) * T::CHUNK, src, (uint32_t)bytes, &full[q % S]);
      q++;
    };
    for (int n = 0; n < T::NG * T::NP && ok; n++) put(rec + (size_t)n * T::CHUNK, T::CHUNK);
    if constexpr (WENO) {
      const unsigned char* src = rec + T::CENTRAL;
      for (int g = 0; g < T::NG; g++)
        for (int p = 0; p < T::si_pieces(g) && ok; p++) {
          const int bytes = 4 * T::si_columns(g, p) * TC * 8;
          put(src, bytes);
          src += bytes;
        }
      for (int n = 0; n < ND * T::NGD && ok; n++) put(src + (size_t)n * T::DCHUNK, T::DCHUNK);
    }
    if (!ok) atomicOr(a.err, 2);
    bar_wait(ebar, 0);
    // the last copies into each stage land before the block's shared memory is released
    for (int n = q - 1; n >= 0 && n >= q - S; n--) bar_wait(&full[n % S], (uint32_t)(n / S) & 1u);
    return;
  }
  const int c = t < 5 * TC ? t / 5 : 0, v = t < 5 * TC ? t - 5 * c : 0;
  const bool live = t < 5 * TC && tile * TC + c < a.N;
  const int i = min(tile * TC + c, a.N - 1);
  const size_t N = a.N;
  const double* __restrict__ Uv = a.U + (size_t)v * N;
  const double ui = Uv[i];
  const int32_t* __restrict__ ids = a.ids + (size_t)tile * T::IDS * TC + c;
  const int16_t* exps = reinterpret_cast<const int16_t*>(sE) + c;
  double* out = a.coef + (size_t)i * 5 + v;
  const size_t st = N * 5;
  int q = 0;
  bool ok = __all_sync(0xffffffffu, bar_wait(ebar, 0));
  auto take = [&]() {  // wait for chunk q
    ok = ok && __all_sync(0xffffffffu, bar_wait(&full[q % S], (uint32_t)(q / S) & 1u));
    return reinterpret_cast<const int2*>(ring + (q % S) * T::CHUNK) + c;
  };
  auto give = [&]() {  // this warp is done with chunk q
    __syncwarp();
    if (lane == 0) bar_arrive(&empty[q % S]);
    q++;
  };
  // the differences of the central stencil as operands (fx_differences, by way of shared memory)
  constexpr int B = fx_bits_of(MC);
  int ec;
  {
    long long* col = sQ + t;
    int eb = fx_exponent(ui);
#pragma unroll 17
    for (int m = 0; m < MC; m++) {
      const double u = Uv[ids[m * TC]];
      col[m * L] = __double_as_longlong(u);
      eb = max(eb, fx_exponent(u));
    }
    const bool low = eb < 64;
    const double up = low ? 0x1p512 : 1.0;
    if (low) {
      eb = fx_exponent(ui * up);
      for (int m = 0; m < MC; m++) {
        const double u = __longlong_as_double(col[m * L]) * up;
        col[m * L] = __double_as_longlong(u);
        eb = max(eb, fx_exponent(u));
      }
    }
    const long long f0 = fx_integer(low ? ui * up : ui, eb);
    unsigned long long any = 1;
#pragma unroll 4
    for (int m = 0; m < MC; m++) {
      const long long d = fx_integer(__longlong_as_double(col[m * L]), eb) - f0;
      col[m * L] = d;
      any |= (unsigned long long)(d ^ (d >> 63));
    }
    const int lz = fx_clz(any);
#pragma unroll 4
    for (int m = 0; m < MC; m++) *reinterpret_cast<int2*>(&col[m * L]) = fx_normalised<B>(col[m * L], lz);
    ec = eb == 2047 ? kFxNan : eb - 1020 - lz - (low ? 512 : 0);
  }
  const int2* op = reinterpret_cast<const int2*>(sQ) + t;
  int ea = 0;  // largest biased exponent of the central coefficients
#pragma unroll 1
  for (int g = 0; g < T::NG; g++) {
    FxAcc acc[4];
#pragma unroll 1
    for (int p = 0; p < T::NP; p++) {
      const int2* ch = take();
      if (!ok) break;
#pragma unroll
      for (int m = 0; m < T::MCH; m++) {
        const int2 w = op[(p * T::MCH + m) * L];
#pragma unroll
        for (int r = 0; r < 4; r++) fx_mac(acc[r], ch[(r * T::MCH + m) * TC], w);
      }
      give();
    }
    if (!ok) break;
#pragma unroll
    for (int r = 0; r < 4; r++)
      if (4 * g + r < K) {
        const double x = fx_double(fx_sum(acc[r]), (int)exps[(4 * g + r) * TC] + ec - 2 - B);
        ea = max(ea, fx_exponent(x));
        if (live) out[(4 * g + r + 1) * st] = x;
      }
  }
  double r0 = 1.0;
  double cd[KD];  // the leading modes' part of the directional candidates
#pragma unroll
  for (int k = 0; k < KD; k++) cd[k] = 0.0;
  if constexpr (WENO) {
    // a^T M a of the central coefficients, rows t_k = sum_{l >= k} M_kl a_l in integers
    // (coefficients below 2^-959 have no square in FP64: the sum is zero)
    constexpr int BA = fx_bits_of(K);
#pragma unroll
    for (int k = 0; k < K; k++)
      *reinterpret_cast<int2*>(&sQ[k * L + t]) = fx_operand<BA>(live ? out[(k + 1) * st] : 0.0, ea);
    const int es = ea == 2047 ? kFxNan : ea - 1022;
    double SI0 = 0.0;
#pragma unroll 1
    for (int g = 0; g < T::NG && ok; g++) {
      FxAcc acc[4];
      double ak[4];
#pragma unroll
      for (int r = 0; r < 4; r++) ak[r] = 4 * g + r < K && live ? out[(4 * g + r + 1) * st] : 0.0;
#pragma unroll 1
      for (int p = 0; p < T::si_pieces(g); p++) {
        const int2* ch = take();
        if (!ok) break;
        const int nc = T::si_columns(g, p);
#pragma unroll 4
        for (int m = 0; m < nc; m++) {
          const int2 w = op[(4 * g + p * T::MCH + m) * L];
#pragma unroll
          for (int r = 0; r < 4; r++) fx_mac(acc[r], ch[(r * nc + m) * TC], w);
        }
        give();
      }
#pragma unroll
      for (int r = 0; r < 4; r++)
        if (4 * g + r < K && ea >= 64)
          SI0 = fma(ak[r], fx_double(fx_sum(acc[r]), (int)exps[(K + 4 * g + r) * TC] + es - 2 - BA), SI0);
    }
    // directional candidate s: b = P_s (U_m - U_i) over its members
    constexpr int BD = fx_bits_of(MD);
    auto candidate = [&](int s, double (&b)[KD]) {
      double u[MD];
#pragma unroll
      for (int m = 0; m < MD; m++) u[m] = Uv[ids[(MC + s * MD + m) * TC]];
      int2 w[MD];
      int e;
      fx_differences<MD>(u, ui, w, e);
#pragma unroll
      for (int g = 0; g < T::NGD; g++) {
        const int2* ch = take();
        if (!ok) return;
#pragma unroll
        for (int r = 0; r < 3; r++) {
          FxAcc acc;
#pragma unroll
          for (int m = 0; m < MD; m++) fx_mac(acc, ch[(r * MD + m) * TC], w[m]);
          b[3 * g + r] = fx_double(fx_sum(acc), (int)exps[(2 * K + s * KD + 3 * g + r) * TC] + e - 2 - BD);
        }
        give();
      }
    };
    double SI[ND];
    double tau = 0.0;
    double* sB = reinterpret_cast<double*>(sQ) + t;  // the candidates wait where the operands were
#pragma unroll 1
    for (int s = 0; s < ND && ok; s++) {
      double b[KD];
      candidate(s, b);
      if (!ok) break;
#pragma unroll
      for (int k = 0; k < KD; k++) sB[(s * KD + k) * L] = b[k];
      SI[s] = si_form<KD>(a.Msi, N, i, b);
      tau += fabs(SI0 - SI[s]);
    }
    tau *= (1.0 / ND);
    // omega~_s = lambda_s (1 + tau / (eps + SI_s)), normalised
    const double w0 = a.lam0 * (1.0 + tau / (a.eps + SI0));
    double ws[ND];
    double wsum = w0;
#pragma unroll
    for (int s = 0; s < ND; s++) {
      ws[s] = a.lams * (1.0 + tau / (a.eps + SI[s]));
      wsum += ws[s];
    }
    const double iws = 1.0 / wsum;
    // p = omega_0 p_1 + sum_s omega_s p_s with p_1 = (p_opt - sum lambda_s p_s)/lambda_0
    r0 = (w0 * iws) / a.lam0;
#pragma unroll
    for (int s = 0; s < ND; s++) {
      const double e = ws[s] * iws - r0 * a.lams;
#pragma unroll
      for (int k = 0; k < KD; k++) cd[k] = fma(e, sB[(s * KD + k) * L], cd[k]);
    }
  }
  if (!ok) {
    if (lane == 0) atomicOr(a.err, 2);
    return;
  }
  if (!live) return;
  double cf[K];
#pragma unroll
  for (int k = 0; k < K; k++) {
    const double ao = out[(k + 1) * st];
    cf[k] = WENO ? fma(r0, ao, k < KD ? cd[k < KD ? k : 0] : 0.0) : ao;
  }
  // monomial form in physical units: p = c0 + sum_k (c_k / h^deg_k) (x - x_i)^e_k,
  // c0 = U_i - sum_{deg >= 2} c_k mean(psi_k)
  double c0 = ui;
#pragma unroll
  for (int k = 3; k < K; k++) c0 = fma(-cf[k], __ldg(&a.psib[(size_t)(k - 3) * N + i]), c0);
  const double ih = __ldg(&a.inv_h[i]);
  double ihp[ORDER + 1];
  ihp[0] = 1.0;
#pragma unroll
  for (int e = 1; e <= ORDER; e++) ihp[e] = ihp[e - 1] * ih;
  out[0] = c0;
#pragma unroll
  for (int k = 0; k < K; k++) cf[k] *= ihp[basis_degree(k)];
  store_fixed<ORDER>(cf, a.hexp[i], out, st, a.cexp + (size_t)i * 5 + v);
}

// The point values and gradients are computed variable by variable in a loop that
// stays rolled (its body is 1500 instructions at P4; unrolled over sides and
// variables the kernel ran out of the instruction cache and of registers) and wait
// in shared memory, one column per thread, for the flux.  Bound by the FP64 pipe and
// its latency.  P4 at 24^3, us: evaluation in FP64 1635, in integers unrolled 969
// (8 warps per SM), in this loop 548 (6, 8, 10 blocks per SM: 637, 548, 595), the
// constant term added as an integer 534, with the face sums shared out 453.
constexpr int kFaceHoThreads = 64;
template <int ORDER, bool VISC>
__global__ void __launch_bounds__(kFaceHoThreads, 8) k_face_ho(FaceArgs a) {
  constexpr int NQ = ORDER * ORDER, FPW = 32 / NQ;  // faces per warp
  const int gw = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
  const int grp = lane / NQ, q = lane - NQ * (lane / NQ);
  const bool in_group = grp < FPW;
  const int f = gw * FPW + (in_group ? grp : 0);
  const bool live = in_group && f < a.F;
  const int fc = live ? f : a.F - 1, qc = in_group ? q : 0;
  const size_t F = a.F;
  const double* __restrict__ fq = a.fq + (size_t)qc * 10 * F + fc;
  const int2* __restrict__ fx = reinterpret_cast<const int2*>(fq);
  const double n[3] = {fq[6 * F], fq[7 * F], fq[8 * F]};
  const double area = fq[9 * F];
  const int o = a.fo[fc], nb = a.fn[fc];
  __shared__ double sv[25][kFaceHoThreads];  // U_L, U_R, then grad U_L + grad U_R of each variable
  const int t = threadIdx.x;
  const size_t st = (size_t)a.N * 5;
#pragma unroll 1
  for (int side = 0; side < 2; side++) {
    const int cell = side ? nb : o;
    const int2* w = fx + (size_t)side * 3 * F;
    const FxPoint<ORDER> pt(w[0], w[F], w[2 * F]);
    const short4 h = __ldg(&a.hexp[cell]);
    const double* p = a.coef + (size_t)cell * 5;
#pragma unroll 1
    for (int v = 0; v < 5; v++) {
      double u;
      FxSum g[3];
      pt.eval(p + v, st, a.cexp[(size_t)cell * 5 + v], h, u, g);
      sv[side * 5 + v][t] = u;
#pragma unroll
      for (int d = 0; d < 3; d++) {
        const double x = fx_double(g[d]);
        sv[10 + 3 * v + d][t] = side ? sv[10 + 3 * v + d][t] + x : x;
      }
    }
  }
  double UL[5], UR[5], gs[5][3];
#pragma unroll
  for (int v = 0; v < 5; v++) {
    UL[v] = sv[v][t];
    UR[v] = sv[5 + v][t];
#pragma unroll
    for (int d = 0; d < 3; d++) gs[v][d] = sv[10 + 3 * v + d][t];
  }
  double flux[5];
  point_flux<VISC>(UL, UR, gs, n, VISC ? 2.0 * a.fpen[fc] : 0.0, a.c, flux);
#pragma unroll
  for (int v = 0; v < 5; v++) flux[v] *= area;
  // each (face, variable) of the warp on a lane of its own, summed in point order
#pragma unroll
  for (int v = 0; v < 5; v++) sv[v][t] = flux[v];
  __syncwarp();
  const int g = lane / 5, v = lane - 5 * (lane / 5), fs = gw * FPW + g;
  if (g < FPW && fs < a.F) {
    const double* x = &sv[v][(t & ~31) + g * NQ];
    double tot = x[0];
#pragma unroll
    for (int k = 1; k < NQ; k++) tot += x[k];
    a.G[(size_t)v * F + fs] = tot;
  }
}

// ------------------------------------------------------- mixed P3 / P4
// The mixed form at P3 / P4 (the arithmetic split of the mixed form at P2):
// stencil differences from the float pairs of the FP64 state, FP32
// pseudo-inverses, contractions, smoothness forms and weights; the constant
// term written relative to the reference state U_ref; coefficients FP32
// rows [N][cs]; FP32 HLLC and viscous flux on reference-relative states, FP32
// face totals (k_rk<s, nfc, float> sums them as float pairs into FP64).
struct ReconArgsHOMx {
  const float* __restrict__ Uhl;    // [N][5][2] float pairs (hi, lo) of the state
  const float* __restrict__ tiles;  // per 32-cell tile its stencil chunks (HOTile)
  const float* __restrict__ Msi;    // [K(K+1)/2][N]
  const float* __restrict__ psib;   // [K-3][N]
  const float* __restrict__ inv_h;  // [N]
  float* __restrict__ coef;         // [N][cs] rows, entries cidx(v, horner_place(k), K + 1): the constant relative
                                    // to U_ref, the others in physical units
  int* err;                         // bit 1: a copy wait gave up
  int N, cs;
  float lam0, lams, eps;
  float eref_hi, eref_lo;  // E_ref = p_ref/(gamma-1) as a float pair
};

// The P3/P4 mixed reconstruction's data, tile by tile (32 cells): the central
// stencil in NCC chunks of MCH members, then each of the six directional
// stencils in NDC chunks of MDH members.  A chunk is [members][32] stencil ids
// (int32) followed by its pseudo-inverse entries as pairs of consecutive
// members, [modes][members / 2][32][2]; every chunk is one bulk copy.  Cells
// past N in the last tile have ids 0 and zero entries.
template <int ORDER>
struct HOTile {
  using H = HO<ORDER>;
  static constexpr int K = H::K, MC = H::MC, KD = H::KD, MD = H::MD;
  static constexpr int TC = 32;
  static constexpr int MCH = ORDER == 4 ? 4 : 2, MDH = 6;
  static constexpr int NCC = MC / MCH, NDC = MD / MDH;
  static constexpr int CCS = MCH * TC + K * MCH * TC;  // floats per central chunk
  static constexpr int DCS = MDH * TC + KD * MDH * TC;  // floats per directional chunk
  static constexpr int CENTRAL = NCC * CCS;
  static constexpr int STAGE = CCS > DCS ? CCS : DCS;
  // with CWENOZ the smoothness matrices follow the central chunks: [K(K+1)/2][32]
  // entries in chunks of MSR rows, then the directional chunks
  static constexpr int NQS = K * (K + 1) / 2, MSR = STAGE / TC, NMC = (NQS + MSR - 1) / MSR;
  static constexpr int SMAT = NQS * TC;
  UCNS_HD static constexpr int tile_floats(bool weno) { return CENTRAL + (weno ? SMAT + 6 * NDC * DCS : 0); }
  static constexpr int S = ORDER == 4 ? 3 : 4;  // stages of the copy ring (6 at P4 measured slower)
  static constexpr int THREADS = 5 * TC + 32;   // (cell, variable) threads and one copying warp
  // the ring, its barriers, then (CWENOZ) the directional candidates, one column per thread
  static constexpr size_t smem(bool weno) {
    return (size_t)S * STAGE * 4 + (size_t)2 * S * 8 + (weno ? (size_t)6 * KD * 5 * TC * 4 : 0);
  }
  static constexpr int blocks(bool weno) { return ORDER == 4 ? (weno ? 2 : 4) : 4; }
  static_assert(MC % MCH == 0 && MD % MDH == 0 && MCH % 2 == 0 && MDH % 2 == 0, "whole member pairs");
  static_assert(CCS % 4 == 0 && DCS % 4 == 0, "16-byte chunks");
};

// a^T M a over the first KK modes of one variable (M: K x K, stored as in si_form), FP32
template <int K, int KK>
__device__ __forceinline__ float si_form_f(const float* __restrict__ M, size_t N, int i, const float (&a)[KK]) {
  float s = 0.f;
#pragma unroll
  for (int k = 0; k < KK; k++) {
    float t = 0.f;
#pragma unroll
    for (int l = k + 1; l < KK; l++) t = fmaf(__ldg(&M[(size_t)(k * K - k * (k - 1) / 2 + l - k) * N + i]), a[l], t);
    const float mkk = __ldg(&M[(size_t)(k * K - k * (k - 1) / 2) * N + i]);
    s = fmaf(a[k], fmaf(2.f, t, mkk * a[k]), s);
  }
  return s;
}

// U_j - U_i of variable v from the float pairs (the leading parts subtract exactly)
__device__ __forceinline__ float pair_diff_ho(const float* __restrict__ hl, int j, int v, float hi_i, float lo_i) {
  const float2 p = __ldg(reinterpret_cast<const float2*>(hl + (size_t)j * 10 + 2 * v));
  return (p.x - hi_i) + (p.y - lo_i);
}

// one chunk's contraction into acc[0 .. KK): members in pairs, in order
template <int KK, int MM>
__device__ __forceinline__ void chunk_contract(const float* chunk, int c, const float* __restrict__ hl, int v,
                                               float hi_i, float lo_i, float (&acc)[KK]) {
  constexpr int TC = 32;
  const float2* P = reinterpret_cast<const float2*>(chunk + MM * TC);
#pragma unroll
  for (int mp = 0; mp < MM / 2; mp++) {
    const int j0 = reinterpret_cast<const int*>(chunk)[(2 * mp) * TC + c];
    const int j1 = reinterpret_cast<const int*>(chunk)[(2 * mp + 1) * TC + c];
    const float d0 = pair_diff_ho(hl, j0, v, hi_i, lo_i), d1 = pair_diff_ho(hl, j1, v, hi_i, lo_i);
#pragma unroll
    for (int k = 0; k < KK; k++) {
      const float2 p = P[(k * (MM / 2) + mp) * TC + c];
      acc[k] = fmaf(p.y, d1, fmaf(p.x, d0, acc[k]));
    }
  }
}

// One block per 32-cell tile: thread (cell c, variable v) = 5 c + v, plus a
// copying warp that streams the tile's chunks (central; with CWENOZ the
// smoothness matrices, then the directional chunks) through a ring of S
// shared-memory stages, every wait bounded; the directional candidates wait in
// shared memory for the weights.  Per variable the arithmetic is that of the
// FP64 form in FP32, members and modes in the same order.  Bound by the latency of
// the state gathers.  CWENOZ at P3 40^3 / P4 32^3, us: 64-cell tiles, the directional
// chunks streamed and contracted twice 89 / 182, 32-cell tiles 88 / 166, the candidates
// kept 79 / 158 (P3 at 4, 5, 6 blocks per SM 79, 82, 87; P4 at 1 and 2 173, 158).
template <int ORDER, bool WENO>
__global__ void __launch_bounds__(HOTile<ORDER>::THREADS, HOTile<ORDER>::blocks(WENO)) k_recon_ho_mx(ReconArgsHOMx a) {
  using T = HOTile<ORDER>;
  constexpr int K = T::K, KD = T::KD, ND = 6, TC = T::TC, S = T::S;
  constexpr int NQ = T::NCC + (WENO ? T::NMC + ND * T::NDC : 0);  // chunks streamed per tile
  extern __shared__ __align__(128) unsigned char smem[];
  float* st = reinterpret_cast<float*>(smem);
  uint64_t* full = reinterpret_cast<uint64_t*>(st + S * T::STAGE);
  uint64_t* empty = full + S;
  float* sB = reinterpret_cast<float*>(empty + S) + threadIdx.x;  // this thread's column of candidates
  const int t = threadIdx.x, lane = t & 31, tile = blockIdx.x;
  if (t < S) {
    bar_init(&full[t]);
    bar_init(&empty[t], 5 * TC / 32);
  }
  __syncthreads();
  if (t >= 5 * TC) {  // the copying warp
    if (lane != 0) return;
    const float* base = a.tiles + (size_t)tile * T::tile_floats(WENO);
    int q = 0;
    bool ok = true;
    for (; q < NQ; q++) {
      if (q >= S && !bar_wait(&empty[q % S], (uint32_t)(q / S + 1) & 1u)) {
        ok = false;
        break;
      }
      // chunk q: central chunks first, then the smoothness matrices, then the directional ones
      const float* src;
      uint32_t bytes;
      if (q < T::NCC) {
        src = base + (size_t)q * T::CCS;
        bytes = T::CCS * 4u;
      } else if (q < T::NCC + T::NMC) {
        const int r0 = (q - T::NCC) * T::MSR;
        src = base + T::CENTRAL + (size_t)r0 * TC;
        bytes = (uint32_t)(min(T::MSR, T::NQS - r0) * TC) * 4u;
      } else {
        const int qd = q - T::NCC - T::NMC;
        src = base + T::CENTRAL + T::SMAT + (size_t)qd * T::DCS;
        bytes = T::DCS * 4u;
      }
      bar_expect(&full[q % S], bytes);
      bulk_load(st + (q % S) * T::STAGE, src, bytes, &full[q % S]);
    }
    if (!ok) atomicOr(a.err, 2);
    // the last copies into each stage land before the block's shared memory is released
    for (int qq = q - 1; qq >= 0 && qq >= q - S; qq--) bar_wait(&full[qq % S], (uint32_t)(qq / S) & 1u);
    return;
  }
  const int c = t / 5, v = t - 5 * (t / 5);
  const int i0 = tile * TC + c;
  const bool live = i0 < a.N;
  const int i = live ? i0 : a.N - 1;
  const size_t N = a.N;
  const float* __restrict__ hl = a.Uhl;
  const float2 pi = __ldg(reinterpret_cast<const float2*>(hl + (size_t)i * 10 + 2 * v));
  const float hi_i = pi.x, lo_i = pi.y;
  int q = 0;
  bool ok = true;
  auto take = [&]() -> const float* {  // wait for chunk q
    ok = ok && __all_sync(0xffffffffu, bar_wait(&full[q % S], (uint32_t)(q / S) & 1u));
    return st + (q % S) * T::STAGE;
  };
  auto give = [&]() {  // this warp is done with chunk q
    __syncwarp();
    if (lane == 0) bar_arrive(&empty[q % S]);
    q++;
  };
  float ao[K];
#pragma unroll
  for (int k = 0; k < K; k++) ao[k] = 0.f;
#pragma unroll 1
  for (int ch = 0; ch < T::NCC; ch++) {
    const float* chunk = take();
    if (!ok) break;
    chunk_contract<K, T::MCH>(chunk, c, hl, v, hi_i, lo_i, ao);
    give();
  }
  float cf[K];
  if constexpr (!WENO) {
#pragma unroll
    for (int k = 0; k < K; k++) cf[k] = ao[k];
  } else {
    // a^T M a of the central coefficients, M's entries from the streamed
    // chunks in row order (each row's diagonal entry read first; the
    // arithmetic as in si_form)
    float SI0 = 0.f;
    {
      const float* mc = take();
#pragma unroll
      for (int k = 0; k < K; k++) {
        const int q0 = k * K - k * (k - 1) / 2;
        auto M = [&](int qq) -> float {
          if (qq % T::MSR == 0 && qq != 0) {
            give();
            mc = take();
          }
          return mc[(qq % T::MSR) * TC + c];
        };
        const float mkk = M(q0);
        float tk = 0.f;
#pragma unroll
        for (int l = k + 1; l < K; l++) tk = fmaf(M(q0 + l - k), ao[l], tk);
        SI0 = fmaf(ao[k], fmaf(2.f, tk, mkk * ao[k]), SI0);
      }
      give();
    }
    float SI[ND];
    float tau = 0.f;
#pragma unroll 1
    for (int s = 0; s < ND && ok; s++) {
      float b[KD];
#pragma unroll
      for (int k = 0; k < KD; k++) b[k] = 0.f;
#pragma unroll 1
      for (int h = 0; h < T::NDC; h++) {
        const float* chunk = take();
        if (!ok) break;
        chunk_contract<KD, T::MDH>(chunk, c, hl, v, hi_i, lo_i, b);
        give();
      }
#pragma unroll
      for (int k = 0; k < KD; k++) sB[(s * KD + k) * 5 * TC] = b[k];
      SI[s] = si_form_f<K, KD>(a.Msi, N, i, b);
      tau += fabsf(SI0 - SI[s]);
    }
    tau *= (1.f / ND);
    const float w0 = a.lam0 * (1.f + fdiv(tau, a.eps + SI0));
    float ws[ND];
    float wsum = w0;
#pragma unroll
    for (int s = 0; s < ND; s++) {
      ws[s] = a.lams * (1.f + fdiv(tau, a.eps + SI[s]));
      wsum += ws[s];
    }
    const float iws = fdiv(1.f, wsum);
    const float r0 = fdiv(w0 * iws, a.lam0);
#pragma unroll
    for (int k = 0; k < K; k++) cf[k] = r0 * ao[k];
#pragma unroll
    for (int s = 0; s < ND; s++) {
      const float e = ws[s] * iws - r0 * a.lams;
#pragma unroll
      for (int k = 0; k < KD; k++) cf[k] = fmaf(e, sB[(s * KD + k) * 5 * TC], cf[k]);
    }
  }
  if (!ok) {
    if (lane == 0) atomicOr(a.err, 2);
    return;
  }
  if (!live) return;
  // the constant term relative to U_ref = (1, 0, 0, 0, E_ref), less the means of
  // the non-linear monomials; coefficients in physical units
  float c0 = v == 0 ? (hi_i - 1.f) + lo_i : (v == 4 ? (hi_i - a.eref_hi) + (lo_i - a.eref_lo) : hi_i + lo_i);
#pragma unroll
  for (int k = 3; k < K; k++) c0 = fmaf(-cf[k], __ldg(&a.psib[(size_t)(k - 3) * N + i]), c0);
  const float ih = __ldg(&a.inv_h[i]);
  float ihp[ORDER + 1];
  ihp[0] = 1.f;
#pragma unroll
  for (int e = 1; e <= ORDER; e++) ihp[e] = ihp[e - 1] * ih;
  float* out = a.coef + (size_t)i * a.cs;
  out[cidx(v, horner_place(-1, ORDER), K + 1)] = c0;
#pragma unroll
  for (int k = 0; k < K; k++) out[cidx(v, horner_place(k, ORDER), K + 1)] = cf[k] * ihp[basis_degree(k)];
}

}  // namespace ucns
