// Windowed Whittaker-Shannon resampling kernels (Eq. 17, Sec. III-B).
//
// Windowed: y[n] = sum_i x[i] h(alpha n - i), h(u) = sinc(u) w(u), w a Kaiser
// window of half width R, support |u| < R, x zero outside [0, N).  With
// alpha n = n + delta n = m + e (e in [0,1)) the sum runs over i = m + k,
// k = -R+1..R, and sinc(e - k) = (-1)^k sin(pi e) / (pi (e - k)).
//
// Two kernels:
//  * direct (any alpha): one output per thread, every weight evaluated.  This
//    is the paper's Algorithm 1 shape and the library's general path.
//  * tiled (|alpha - 1| <= 0.01, 32 taps): a CTA owns 1024 consecutive outputs;
//    each warp loads its own slice of the input into shared memory; each
//    lane owns Q = 8 consecutive outputs (a warp 256) while e moves by at most
//    0.015 of a sample across a warp tile (|alpha - 1| <= 5.8e-5, |v_r| <=
//    8.7 km/s), else Q = 4 (|alpha - 1| <= 1.1e-4, |v_r| <= 17 km/s); each tap
//    weight is then the quadratic through its exact values at the warp tile's
//    first, middle and last output (error <= 2e-7), with one more tap where
//    floor(delta n) steps inside the tile.  Other warp tiles use exact
//    per-output weights read against the same slice (taken at every step
//    they cost a short pulse 18.4 instead of 6.2 us).
#include "resample.cuh"

namespace dc {

constexpr float kInvPi = 0.318309886183790672f;
constexpr int kRsThreads = 256;

// w(e - k) from the per-tap polynomial, t = k + R - 1.
DC_DEV float window_at(const float* __restrict__ wp, int t, float e) {
  const float4 lo = __ldg(reinterpret_cast<const float4*>(wp + t * kWCoef));
  const float4 hi = __ldg(reinterpret_cast<const float4*>(wp + t * kWCoef + 4));
  float w = fmaf(hi.w, e, hi.z);
  w = fmaf(w, e, hi.y);
  w = fmaf(w, e, hi.x);
  w = fmaf(w, e, lo.w);
  w = fmaf(w, e, lo.z);
  w = fmaf(w, e, lo.y);
  return fmaf(w, e, lo.x);
}

// h(e - k) for tap k; s_e = sin(pi e)/pi.
DC_DEV float tap_weight(const RsArgs& a, float e, float s_e, int k) {
  const float u = e - (float)k;
  if (u == 0.f) return 1.f;
  const float sc = fast_div((k & 1) ? -s_e : s_e, u);
  return sc * window_at(a.wpoly, k + a.half - 1, e);
}

// The item owning a tile: the last item with tile_begin <= tile (tile_begin
// strictly increases).  One warp probes 32 evenly spaced items per round, so
// the search takes ceil(log32 n_items) dependent loads instead of log2.
// Every lane of the warp calls it and gets the answer.
DC_DEV int find_item(const RsArgs& a, int tile) {
  const int lane = threadIdx.x & 31;
  if (!a.items) return 0;
  int lo = 0, hi = a.n_items;                  // items[lo].tile_begin <= tile < items[hi]
  while (hi - lo > 1) {
    const int step = (hi - lo + 31) >> 5;
    const int idx = lo + lane * step;
    const bool ok = idx < hi && a.items[idx].tile_begin <= tile;
    const unsigned m = __ballot_sync(0xffffffffu, ok);   // lane 0 always set
    lo += (31 - __clz((int)m)) * step;
    hi = min(hi, lo + step);
  }
  return lo;
}

// ------------------------------------------------------------- direct
__global__ void __launch_bounds__(kRsThreads) resample_direct_kernel(RsArgs a) {
  pdl_release();                        // the transform that follows may start its set-up
  __shared__ int s_item;
  const int tile = blockIdx.x;
  if (threadIdx.x < 32) {
    const int it = find_item(a, tile);
    if (threadIdx.x == 0) s_item = it;
  }
  __syncthreads();
  const RsItem I = rs_item(a, s_item);
  const int o0 = (tile - I.tile_begin) * kRsTile;
  for (int q = 0; q < kRsTile / kRsThreads; ++q) {
    const int i = o0 + q * kRsThreads + threadIdx.x;
    if (i >= I.n_out) break;
    int fl;
    float e;
    rs_delay(I.dl_hi, I.dl_lo, (float)i, fl, e);
    const int m = i + fl;
    float2 acc = make_float2(0.f, 0.f);
    if (e == 0.f) {
      if (m >= 0 && m < I.n_in) acc = __ldg(I.x + m);
    } else {
      const float s_e = sinpif(e) * kInvPi;
      for (int k = -a.half + 1; k <= a.half; ++k) {
        const int idx = m + k;
        if ((unsigned)idx >= (unsigned)I.n_in) continue;
        const float h = tap_weight(a, e, s_e, k);
        const float2 v = __ldg(I.x + idx);
        acc.x = fmaf(v.x, h, acc.x);
        acc.y = fmaf(v.y, h, acc.y);
      }
    }
    I.y[i] = rotate(acc, I.rot_hi, I.rot_lo, i);
  }
}

// ---------------------------------------------------- frequency conversion
__global__ void __launch_bounds__(kRsThreads) freqconv_kernel(RsArgs a) {
  pdl_release();                        // the transform that follows may start its set-up
  __shared__ int s_item;
  const int tile = blockIdx.x;
  if (threadIdx.x < 32) {
    const int it = find_item(a, tile);
    if (threadIdx.x == 0) s_item = it;
  }
  __syncthreads();
  const RsItem I = rs_item(a, s_item);
  const int o0 = (tile - I.tile_begin) * kRsTile;
#pragma unroll
  for (int q = 0; q < kRsTile / kRsThreads; ++q) {
    const int i = o0 + q * kRsThreads + threadIdx.x;
    if (i >= I.n_out) break;
    const float2 v = i < I.n_in ? __ldg(I.x + i) : make_float2(0.f, 0.f);
    __stcs(I.y + i, rotate(v, I.rot_hi, I.rot_lo, i));
  }
}

// ------------------------------------------------------------- tiled
// Q consecutive outputs per lane (4 or 8): a warp tile is 32 Q outputs and
// kRsTile / Q threads cover the 1024-output CTA tile.
// Largest move of e across a warp tile for the quadratic weights: the
// interpolation error is about 0.064 |h'''| (span/2)^3 <= 2e-7 per weight.
constexpr float kQuadSpan = kRsQuadSpan;

// Bank-spread window layout: element i at i + i / Q, so that lane l's
// first tap input (Q l + const) lands on bank pair (Q + 1) l + const.
template <int LQ> DC_DEV int wpad(int i) { return i + (i >> LQ); }

// Inner product loop of one lane over all taps: outputs ow + Q lane + q,
// inputs at padded slice positions m + (m >> log2 Q) from the lane's base
// (the slice starts at the warp tile's first input, so every offset is a
// compile-time constant).  The Q inputs of a tap slide by one per tap, so
// each tap loads one new input and one weight quadruple.  The tile's
// quadratic weight h(s) = w.x + w.y s + w.z s^2 (w.w = 2 w.z) is evaluated
// once per lane at its centre sl, value and slope, and the Q outputs
// sl + u, |u| <= (Q - 1) / 2, take the tangent: the term w.z u^2 left out
// is about |h''| / 2 (u de/ds)^2 <= 7.1e-8 per weight (|h''| <= 3.32 for
// the 32-tap Kaiser(8) sinc; |de/ds| <= kRsQuadSpan / (32 Q - 1), so
// |u de/ds| <= 2.06e-4 at Q = 8 and 1.77e-4 at Q = 4).
template <int TAPS, int LQ>
DC_DEV void tap_loop(const float2* __restrict__ w0, const float4* __restrict__ wts,
                     float sl, bool step, unsigned lower, float2 (&acc)[1 << LQ]) {
  constexpr int Q = 1 << LQ;
  float2 xw[Q];
#pragma unroll
  for (int q = 0; q < Q; ++q) xw[q] = w0[q + (q >> LQ)];
#pragma unroll
  for (int t = 0; t < TAPS; ++t) {
    const float4 w = wts[t];
    const float hl = fmaf(fmaf(w.z, sl, w.y), sl, w.x);
    const float dl = fmaf(w.w, sl, w.y);
    // packed two-lane FMAs, each lane rounding as fmaf does: the weight h
    // in both lanes, then both parts of the output at once
    const float2 hl2 = make_float2(hl, hl), dl2 = make_float2(dl, dl);
#pragma unroll
    for (int q = 0; q < Q; ++q) {
      const float u = (float)q - 0.5f * (float)(Q - 1);
      const float2 h2 = __ffma2_rn(dl2, make_float2(u, u), hl2);
      acc[q] = __ffma2_rn(xw[q], h2, acc[q]);
    }
#pragma unroll
    for (int q = 0; q + 1 < Q; ++q) xw[q] = xw[q + 1];
    if (t == 0 && step) {
      // the lowest tap has left the support of the upper cell's outputs
#pragma unroll
      for (int q = 0; q < Q; ++q)
        if (!(lower >> q & 1)) acc[q] = make_float2(0.f, 0.f);
    }
    if (t + 1 < TAPS) {
      const int m = Q + t;
      xw[Q - 1] = w0[m + (m >> LQ)];
    }
  }
}

// h(e - k) for a tap of a warp tile whose nodes may lie in two unit cells: k is
// relative to the node's own cell, and the taps just outside its support (k =
// -R and R + 1) continue the neighbouring tap's window polynomial, so that a
// tap's quadratic in the position is smooth across the step.
DC_DEV float tap_weight_ext(const RsArgs& a, float e, float s_e, int k) {
  const float u = e - (float)k;
  if (u == 0.f) return 1.f;
  const float sc = fast_div((k & 1) ? -s_e : s_e, u);
  const int t = k + a.half - 1;
  if (t < 0) return sc * window_at(a.wpoly, 0, e + 1.f);
  if (t >= 2 * a.half) return sc * window_at(a.wpoly, 2 * a.half - 1, e - 1.f);
  return sc * window_at(a.wpoly, t, e);
}

template <int HALF, int LQ>
__global__ void __launch_bounds__(kRsTile >> LQ, LQ == 3 ? 8 : 3) resample_tiled_kernel(RsArgs a) {
  pdl_release();                        // the transform that follows may start its set-up
  constexpr int Q = 1 << LQ;
  constexpr int NT = kRsTile / Q;          // threads
  constexpr int W = 32 * Q;                // outputs per warp tile
  constexpr int TAPS = 2 * HALF;
  constexpr int NW = NT / 32;
  constexpr int WWIN = W + TAPS + 3;                   // a warp's slice (|f2 - f0| <= 4)
  constexpr int WSTRIDE = ((WWIN + (WWIN >> LQ) + 1) | 1) + 1;   // even: 16-byte aligned slices
  constexpr int NLD = (WWIN + 31) / 32;
  static_assert(WSTRIDE >= W, "a slice stages the warp's outputs");
  __shared__ __align__(16) float2 win[NW * WSTRIDE];
  __shared__ float4 wts[NW][TAPS + 1];
  __shared__ int s_item;

  const int tile = blockIdx.x;
  if (a.items) {
    if (threadIdx.x < 32) {
      const int it = find_item(a, tile);
      if (threadIdx.x == 0) s_item = it;
    }
    __syncthreads();                           // the only one: the warps go their own ways
  }
  const RsItem I = rs_item(a, s_item);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int ow = (tile - I.tile_begin) * kRsTile + warp * W;
  if (ow >= I.n_out) return;                   // warp-uniform: nothing to write
  constexpr float H = 0.5f * (W - 1);
  // the warp tile's first, centre and last positions: one per lane 0..2
  int fl_l;
  float e_l;
  rs_delay(I.dl_hi, I.dl_lo, lane == 0 ? (float)ow : lane == 1 ? (float)ow + H : (float)(ow + W - 1),
           fl_l, e_l);
  const float s_l = sinpif(e_l) * kInvPi;
  const int f0 = __shfl_sync(0xffffffffu, fl_l, 0), f1 = __shfl_sync(0xffffffffu, fl_l, 1),
            f2 = __shfl_sync(0xffffffffu, fl_l, 2);
  const float e0 = __shfl_sync(0xffffffffu, e_l, 0), e1 = __shfl_sync(0xffffffffu, e_l, 1),
              e2 = __shfl_sync(0xffffffffu, e_l, 2);
  if (abs(f2 - f0) > 4) {                      // |delta| too large for the slice
    if (lane == 0) atomicMax(a.err, 2);
    return;
  }
  // The warp's slice of the input -- positions G .. G + WWIN - 1, zero outside
  // the pulse -- goes from global memory into a private, bank-spread region of
  // shared memory (compile-time tap offsets, no CTA barrier; the region then
  // stages the warp's outputs).  Its loads are in flight while the weights are
  // formed.  (Staged for the whole CTA by one bulk copy first, the slice waits for
  // the copy, a barrier and a second pass through shared memory.)
  const int fmin = min(f0, f2);
  const int G = ow + fmin - HALF + 1;
  float2* ww = win + warp * WSTRIDE;
  float2 ld[NLD];
  if (G >= 0 && G + 32 * NLD <= I.n_in) {      // all inside the pulse
#pragma unroll
    for (int i = 0; i < NLD; ++i) ld[i] = __ldg(I.x + G + lane + 32 * i);
  } else {
#pragma unroll
    for (int i = 0; i < NLD; ++i) {
      const int gi = G + lane + 32 * i;
      ld[i] = gi >= 0 && gi < I.n_in ? __ldg(I.x + gi) : make_float2(0.f, 0.f);
    }
  }
  // Quadratic weights per tap through the three nodes s = -H, 0, +H, taps
  // counted from the lower of the tile's (at most two) unit cells; a tile across
  // a step of floor(delta n) has one more tap.
  const bool step = f0 != f2;
  const bool quad = abs(f2 - f0) <= 1 && fabsf((e2 - e0) + (float)(f2 - f0)) <= kQuadSpan;
  if (quad) {
    const float s0 = __shfl_sync(0xffffffffu, s_l, 0), s1 = __shfl_sync(0xffffffffu, s_l, 1),
                s2 = __shfl_sync(0xffffffffu, s_l, 2);
    for (int t = lane; t < TAPS + (step ? 1 : 0); t += 32) {
      const int k = t - HALF + 1;
      const float hA = tap_weight_ext(a, e0, s0, k - (f0 - fmin));
      const float hB = tap_weight_ext(a, e1, s1, k - (f1 - fmin));
      const float hC = tap_weight_ext(a, e2, s2, k - (f2 - fmin));
      const float q1 = (hC - hA) * (0.5f / H);
      const float q2 = (hC - 2.f * hB + hA) * (0.5f / (H * H));
      wts[warp][t] = make_float4(hB, q1, q2, 2.f * q2);
    }
  }
#pragma unroll
  for (int i = 0; i < NLD; ++i) {
    const int p = lane + 32 * i;
    if (p < WWIN && DC_IN_BOUNDS(wpad<LQ>(p) < WSTRIDE, a.err)) ww[wpad<LQ>(p)] = ld[i];
  }
  __syncwarp();

  float2 acc[Q];
#pragma unroll
  for (int q = 0; q < Q; ++q) acc[q] = make_float2(0.f, 0.f);
  if (quad) {
    // Output ow + Q lane + q at tap t reads slice position Q lane + q + t,
    // padded (Q + 1) lane + m + (m >> log2 Q) with m = q + t.
    const float sl = (float)(lane * Q) + 0.5f * (float)(Q - 1) - H;   // the lane's centre
    unsigned lower = (1u << Q) - 1;              // outputs in the tile's lower cell
    if (step) {
#pragma unroll
      for (int q = 0; q < Q; ++q) {
        int fl;
        float e;
        rs_delay(I.dl_hi, I.dl_lo, (float)(ow + lane * Q + q), fl, e);
        if (fl != fmin) lower &= ~(1u << q);
      }
    }
    tap_loop<TAPS, LQ>(ww + (Q + 1) * lane, wts[warp], sl, step, lower, acc);
    if (step) {
      // ... and one more tap has entered it
      const float4 w1 = wts[warp][TAPS];
#pragma unroll
      for (int q = 0; q < Q; ++q) {
        if (lower >> q & 1) continue;
        const float s = (float)(lane * Q + q) - H;
        const float h1 = fmaf(fmaf(w1.z, s, w1.y), s, w1.x);
        const float2 x1 = ww[wpad<LQ>(lane * Q + q + TAPS)];
        acc[q].x = fmaf(x1.x, h1, acc[q].x);
        acc[q].y = fmaf(x1.y, h1, acc[q].y);
      }
    }
  } else {
    // floor(delta n) steps more than once inside this warp tile, or e moves
    // too far: exact weights per output.
#pragma unroll
    for (int q = 0; q < Q; ++q) {
      const int i = ow + lane * Q + q;
      int fl;
      float e;
      rs_delay(I.dl_hi, I.dl_lo, (float)i, fl, e);
      const int base = (i - ow) + (fl - fmin) + HALF - 1;   // slice position of tap k = 0
      if (e == 0.f) {
        acc[q] = ww[wpad<LQ>(base)];
      } else {
        const float s_e = sinpif(e) * kInvPi;
        for (int k = -HALF + 1; k <= HALF; ++k) {
          const float h = tap_weight(a, e, s_e, k);
          const float2 v = ww[wpad<LQ>(base + k)];
          acc[q].x = fmaf(v.x, h, acc[q].x);
          acc[q].y = fmaf(v.y, h, acc[q].y);
        }
      }
    }
  }
  // Stage the warp's W outputs in its slice (16-byte slots, XOR-swizzled so
  // lanes 4 slots apart use distinct banks), then store them coalesced.
  __syncwarp();
  float4* s4 = reinterpret_cast<float4*>(ww);
#pragma unroll
  for (int q = 0; q < Q / 2; ++q) {
    const int f = lane * (Q / 2) + q;
    s4[f ^ ((f >> 3) & 7)] = make_float4(acc[2 * q].x, acc[2 * q].y, acc[2 * q + 1].x, acc[2 * q + 1].y);
  }
  __syncwarp();
  const int n_here = min(W, I.n_out - ow);
  float2* y = I.y + ow;
  const bool rot = I.rot_hi != 0.f || I.rot_lo != 0.f;    // carrier term
  if ((reinterpret_cast<uintptr_t>(y) & 15) == 0) {
    for (int p = lane; 2 * p + 1 < n_here; p += 32) {
      float4 t = s4[p ^ ((p >> 3) & 7)];
      if (rot) {
        const float2 u = rotate(make_float2(t.x, t.y), I.rot_hi, I.rot_lo, ow + 2 * p);
        const float2 w = rotate(make_float2(t.z, t.w), I.rot_hi, I.rot_lo, ow + 2 * p + 1);
        t = make_float4(u.x, u.y, w.x, w.y);
      }
      __stcs(reinterpret_cast<float4*>(y) + p, t);
    }
    if ((n_here & 1) && lane == 0) {
      const int p = (n_here - 1) >> 1;
      const float4 t = s4[p ^ ((p >> 3) & 7)];
      y[n_here - 1] = rotate(make_float2(t.x, t.y), I.rot_hi, I.rot_lo, ow + n_here - 1);
    }
  } else {
    for (int p = lane; p < n_here; p += 32) {
      const int f = p >> 1;
      const float4 t = s4[f ^ ((f >> 3) & 7)];
      y[p] = rotate((p & 1) ? make_float2(t.z, t.w) : make_float2(t.x, t.y), I.rot_hi, I.rot_lo,
                    ow + p);
    }
  }
}

cudaError_t launch_resample_tiled32(const RsArgs& a, int q, cudaStream_t s) {
  if (a.n_tiles <= 0) return cudaSuccess;
  if (q == 8) resample_tiled_kernel<16, 3><<<a.n_tiles, kRsTile / 8, 0, s>>>(a);
  else if (q == 4) resample_tiled_kernel<16, 2><<<a.n_tiles, kRsTile / 4, 0, s>>>(a);
  else return cudaErrorInvalidValue;
  return cudaGetLastError();
}

cudaError_t launch_freqconv(const RsArgs& a, cudaStream_t s) {
  if (a.n_tiles <= 0) return cudaSuccess;
  freqconv_kernel<<<a.n_tiles, kRsThreads, 0, s>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_resample_direct(const RsArgs& a, cudaStream_t s) {
  if (a.n_tiles <= 0) return cudaSuccess;
  resample_direct_kernel<<<a.n_tiles, kRsThreads, 0, s>>>(a);
  return cudaGetLastError();
}

}  // namespace dc
