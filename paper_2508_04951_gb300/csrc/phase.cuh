// Ionospheric phase phi_k = 4 pi K2 / (c f_k) of the FFT correction
// (Eqs. 15-16) in cycles, phi / 2 pi = C / f_k, evaluated and reduced in
// double-float arithmetic before the FP32 sincos.  phi reaches thousands of
// radians at TEC ~ 1e2 TECU and f ~ 1 GHz, where one float ulp is ~2.4e-4 rad;
// the double-float path keeps ~48 bits, so the reduced angle is good to float
// rounding.  Working in cycles makes the reduction two exact subtractions of
// an integer; a bin costs 24 to 30 instructions with its sincos and product, so
// the transform kernels evaluate every bin where it lies in registers (bins
// 256 rows apart) instead of regrouping runs of neighbours to step the phase
// from one to the next.
#pragma once

#include "common.cuh"

namespace dc {

// Per-pulse constants, split on the host from FP64 into hi + lo floats.
struct PhaseParams {
  float c_hi, c_lo;     // C = 2 kappa E / c         [cycles Hz]
  float fc_hi, fc_lo;   // carrier fc                [Hz]; 0 = RF sampling
  float d_hi, d_lo;     // bin spacing fs / L        [Hz]
  int log2L;            // transform length L = 2^log2L
  // 0 when E == 0 (identity).  kPhasePlain where every f_k > 0, fc and fs / L are
  // floats exactly (baseband at round frequencies) and |C / f| max(1, fs / 2f) <
  // kPlainCycles at the lowest f: the evaluation leaves out the terms that are zero then
  // and the second reduction.
  int enabled;
};
constexpr int kPhasePlain = 2;
// q2 below is at most 2.75 ulps of C / f (2^-23 each: the reciprocal one, its product 1/2, f's
// low part 1/2 and as much times fs / 2f, C's low part 1/4): 0.086 cycles here, so that the
// phase stays within 0.59 cycles, where the approximate sine is specified (to 2^-20.5
// within a cycle).  1e4 TECU at a carrier of 300 MHz are 9e4 cycles.
constexpr double kPlainCycles = 1 << 18;

// kt of bin k of an L-point DFT (fftfreq order): k below L/2, else k - L.
DC_DEV float bin_kt(const PhaseParams& P, int k) {
  const int L = 1 << P.log2L;
  return (float)(k < (L >> 1) ? k : k - L);
}

// Reduced phase in cycles, about [-1/2, 1/2], at f = fc + (fs/L) kt.  A bin at
// f == 0 (DC under RF sampling) gets 0.
template <bool PLAIN> DC_DEV float iono_cycles(const PhaseParams& P, float kt) {
  // f = fh + fl: fc is 0 or above fs / 2 >= |d kt|, so the sum's rounding
  // error is exact by one subtraction each way
  const df p = two_prod(P.d_hi, kt);
  const float fh = __fadd_rn(P.fc_hi, p.hi);
  const float fe = __fsub_rn(p.hi, __fsub_rn(fh, P.fc_hi));
  const float fl = PLAIN ? __fadd_rn(p.lo, fe)
                         : __fadd_rn(fmaf(P.d_lo, kt, p.lo), __fadd_rn(fe, P.fc_lo));
  // C / f = q1 + q2: q1 to a couple of ulps, the remainder C - q1 f formed
  // exactly, its quotient q2 to float accuracy relative to itself
  const float rb = fast_rcp(fh);
  const float q1 = __fmul_rn(P.c_hi, rb);
  float r = fmaf(-q1, fh, P.c_hi);
  r = fmaf(-q1, fl, __fadd_rn(r, P.c_lo));
  const float q2 = __fmul_rn(r, rb);
  float x = __fadd_rn(__fsub_rn(q1, rintf(q1)), q2);   // q1 - rint(q1) is exact
  if constexpr (PLAIN) return x;                       // within [-0.59, 0.59]: kPlainCycles
  x = __fsub_rn(x, rintf(x));                          // |q2| passes 1/2 for |C / f| > 2^22
  return fh == 0.f ? 0.f : x;
}

// Correction factor exp(-i phi) (Eq. 16) at kt, and at bin k.
template <bool PLAIN = false> DC_DEV float2 iono_factor_kt(const PhaseParams& P, float kt) {
  float s, c;
  __sincosf(iono_cycles<PLAIN>(P, kt) * 6.28318530717958648f, &s, &c);
  return make_float2(c, -s);
}
// The same by sincospif, for transforms below 4096 points and for factor tables: the
// angle is not rounded again by 2 pi, and __sincosf's 2^-21 is more than half of a short
// transform's distance from 64 bits (2048 points: 2.59e-7, now 1.81e-7; a 10001-sample
// bank 2.79e-7, now 2.00e-7).  It costs plans of thousands of short pulses 4 to 9 %
// (10000 x 300 samples 41.4 us, now 45.3) and nothing elsewhere.  The transforms from 4096
// points on, bound by issue, keep the form above.
DC_DEV float2 iono_factor_full(const PhaseParams& P, float kt) {
  float s, c;
  sincospif(2.f * iono_cycles<false>(P, kt), &s, &c);
  return make_float2(c, -s);
}
DC_DEV float2 iono_factor(const PhaseParams& P, int k) { return iono_factor_full(P, bin_kt(P, k)); }

}  // namespace dc
