// Doppler resampling y[n] = x(alpha n Ts) (Eq. 2) by windowed and exact
// Whittaker-Shannon interpolation (Eq. 17; Sec. III-B; Table I).
#pragma once

#include "common.cuh"

namespace dc {

constexpr int kMaxHalf = 32;      // taps <= 64
constexpr int kWCoef = 8;         // window polynomial coefficients per tap (degree 7)

// One pulse of a windowed-resample launch.
struct RsItem {
  const float2* x;     // input samples [n_in]
  float2* y;           // output samples [n_out]
  int n_in, n_out;
  float dl_hi, dl_lo;  // delta = alpha - 1 as a double-float
  int tile_begin;      // first kRsTile-output tile of this item in the launch
  // Output n is multiplied by exp(2 pi i g n), g = rot_hi + rot_lo cycles per
  // sample (0: no rotation): the carrier term fc (alpha - 1) / fs of a
  // passband dilation, or the tone of frequency conversion.
  float rot_hi, rot_lo;
};

struct RsArgs {
  const RsItem* items;
  int n_items;
  int n_tiles;         // total tiles of the launch
  int half;            // R = taps / 2
  // Kaiser window of tap k at fractional delay e in [0, 1]:
  //   w(e - k) = sum_d wpoly[t * kWCoef + d] e^d,  t = k + R - 1
  // (fitted per tap in FP64 on the host; |error| <= 6e-8 for beta <= 20).
  const float* wpoly;
  int* err;            // device error flag (bounded waits)
  RsItem one;          // with items null: the single pulse (no upload, no search)
};
DC_DEV RsItem rs_item(const RsArgs& a, int i) { return a.items ? a.items[i] : a.one; }

// One alpha of an exact-sinc launch (config: n_pulses pulses share alpha).
struct ExItem {
  const float2* x;     // [n_pulses][n_in]
  float2* y;           // [n_pulses][n_out]
  float dl_hi, dl_lo;
  float rot_hi, rot_lo;  // carrier term, as in RsItem (0: none)
};
struct ExArgs {
  const ExItem* items; // one per alpha (grid.z)
  int n_in, n_out, n_pulses;
  // Scratch of the near and far form (null: every sample term by term):
  // block moments [groups][n_pulses][16 blocks(n_in)] and node values
  // [groups][n_pulses][16 blocks(n_out)], groups = 1 when every alpha has
  // the same pulses (`shared`), else one per alpha.
  float2 *mom, *loc;
  int shared;
  ExItem one;          // with items null: the single alpha
};
DC_DEV ExItem ex_item(const ExArgs& a, int i) { return a.items ? a.items[i] : a.one; }
// Float2 elements of that scratch for n samples a pulse, and whether a call
// takes the form at all (delta_max: the largest |alpha - 1|).
size_t exact_fp32_far_elems(long long pulses, int n);
bool exact_fp32_far(int n_in, int n_out, int n_pulses, int n_alpha, double delta_max);

// v exp(2 pi i g n) (the item's carrier rotation), or v when g = 0.
DC_DEV float2 rotate(float2 v, float g_hi, float g_lo, int n) {
  if (g_hi == 0.f && g_lo == 0.f) return v;
  return cmul(v, cycles_rot(g_hi, g_lo, n));
}

// One launch of the tensor-core bank resampler (rs_tc.cu): one pulse x[n_in]
// for n_slots range rates, slot s holding delta = dl[2s] + dl[2s+1] and
// writing y + vidx[s] * n_out (vidx < 0: an empty slot).  Slots are grouped
// 32 per CTA; within a group the range rates' integer offsets
// floor(delta n) over any 128-output tile must span at most
// rs_tc_max_span() samples (the host orders the slots by delta and checks).
struct RsTcArgs {
  const float2* x;
  int n_in, n_out;
  float2* y;
  const float* dl;
  const int* vidx;
  int n_slots;
  const float* wpoly;  // 32-tap window polynomials and their first two
                       // derivatives: [tap][3][kWCoef] (w, w', w'' in e)
  int* err;
  // launched with programmatic serialization behind a kernel whose results it
  // does not read; it waits for that kernel before it ends, so that work behind
  // it in the stream finds both done
  int pdl;
};
int rs_tc_max_span();
cudaError_t launch_resample_tc(const RsTcArgs& a, cudaStream_t s);

constexpr int kRsTile = 1024;     // outputs per CTA of the resampling kernels
constexpr float kRsTiledMaxDelta = 0.01f;
// The tiled kernel's warp tile is 32 q outputs (q = 8 or 4 per lane); its
// per-tap quadratic weights need e to move at most kRsQuadSpan across it,
// else the tile falls back to exact weights: q = 8 while
// |delta| (256 - 1) <= kRsQuadSpan, q = 4 above.
constexpr float kRsQuadSpan = 0.015f;
inline int resample_q(double delta_abs) { return delta_abs * 255.0 <= 0.98 * kRsQuadSpan ? 8 : 4; }

cudaError_t launch_resample_tiled32(const RsArgs& a, int q, cudaStream_t s);
// Frequency conversion (Sec. I, Table I): y[n] = x[n] exp(2 pi i g n) for
// n < n_out, x = 0 beyond n_in; g from the items' rotation fields.
cudaError_t launch_freqconv(const RsArgs& a, cudaStream_t s);
cudaError_t launch_resample_direct(const RsArgs& a, cudaStream_t s);
cudaError_t launch_exact_fp32(const ExArgs& a, int n_alpha, cudaStream_t s);
inline int exact_fp32_kernels(const ExArgs& a) { return a.mom ? 3 : 1; }   // launched by it

}  // namespace dc
