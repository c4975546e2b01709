// 4096-point rows in registers: 256 threads, 16 points each, one padded
// shared-memory buffer and one CTA barrier per direction.
#pragma once

#include "fft.cuh"

namespace dc {

constexpr int kRowN = 4096;             // row length
constexpr int kRowThreads = 256;        // threads per row (one radix-16 butterfly each)
constexpr int kRowPitch = kRowN + kRowN / 16;

DC_DEV int pad16(int p) { return p + (p >> 4); }

// Twiddles of a 4096-point row: W256^(r k), k = 0..15 (s2) and W4096^(r j), j =
// 0..255 (s3), forward values.  Only the table rows r = 1, 2, 4, 8 are read;
// the other powers are their products (apply_powers).
struct GlobalTw {                 // the context's table (coalesced across the warp)
  static constexpr int kBases = 4;
  const float2* __restrict__ tw;
  DC_DEV void s2(float2 (&b)[4], int k) const {
    const float2* t = tw + kTwS2 + k;             // row r at (r - 1) * 16
    b[0] = __ldg(t), b[1] = __ldg(t + 16), b[2] = __ldg(t + 48), b[3] = __ldg(t + 112);
  }
  DC_DEV void s3(float2 (&b)[4], int j) const {
    const float2* t = tw + kTwS3 + j;             // row r at (r - 1) * 256
    b[0] = __ldg(t), b[1] = __ldg(t + 256), b[2] = __ldg(t + 768), b[3] = __ldg(t + 1792);
  }
};
struct SharedTw {                 // a persistent CTA's copies of those rows, [4][16] and [4][256]
  static constexpr int kBases = 4;
  const float2 *t2, *t3;
  DC_DEV void s2(float2 (&b)[4], int k) const {
#pragma unroll
    for (int q = 0; q < 4; ++q) b[q] = t2[q * 16 + k];
  }
  DC_DEV void s3(float2 (&b)[4], int j) const {
#pragma unroll
    for (int q = 0; q < 4; ++q) b[q] = t3[q * 256 + j];
  }
};
struct HeldTw {                   // loaded ahead by the caller, for this thread
  static constexpr int kBases = 4;
  const float2 (&f2)[4], (&f3)[4];
  DC_DEV void s2(float2 (&b)[4], int) const {
#pragma unroll
    for (int q = 0; q < 4; ++q) b[q] = f2[q];
  }
  DC_DEV void s3(float2 (&b)[4], int) const {
#pragma unroll
    for (int q = 0; q < 4; ++q) b[q] = f3[q];
  }
};
// The rows r = 1, 2, 3, 4, 8, 12, for the middle rows of long transforms: a power is one
// product at most, of two table values, and fewer are live at a time (16 bytes spilled
// instead of 40).  RF pulse of 2^19 samples 3.65e-7 from 64 bits, now 3.52e-7; batch of
// 4096 uneven pulses 3435 us, now 3417.  All 15 rows of both tables: 3.42e-7, but the batch takes
// 3481 us; the cluster kernels, whose error is no larger with four rows, lose 1 to 3 %.
struct FineTw {
  static constexpr int kBases = 6;
  const float2* __restrict__ tw;
  static __host__ __device__ constexpr int row(int q) { return q < 3 ? q + 1 : 4 * (q - 2); }
  DC_DEV void s2(float2 (&b)[6], int k) const {
#pragma unroll
    for (int q = 0; q < 6; ++q) b[q] = __ldg(tw + kTwS2 + (row(q) - 1) * 16 + k);
  }
  DC_DEV void s3(float2 (&b)[6], int j) const {
#pragma unroll
    for (int q = 0; q < 6; ++q) b[q] = __ldg(tw + kTwS3 + (row(q) - 1) * 256 + j);
  }
};
template <int DIR, int N> DC_DEV void orient(float2 (&b)[N]) {
#pragma unroll
  for (int q = 0; q < N; ++q) b[q] = conj_if<DIR>(b[q]);
}

// 4096-point rows, thread j = 16 s + t of 256, with one CTA barrier each.  The
// split 4096 = 16 x 16 x 16: n = 256 p + 16 u + w, k = s + 16 a + 256 r.
//
// Forward: v[p] = x[256 p + j] in, v[r] = X[s + 16 t + 256 r] out.
//   length-16 DFT over p (thread q = 16 u + w), W4096^(q s); a CTA-wide exchange
//   gives half-warp s the 256 values of its sub-problem; DFT over u in thread w =
//   t, W256^(w a); a 16 x 16 transpose inside the half-warp; DFT over w in thread
//   a = t.
// Inverse: the mirror image, v[r] = Y[s + 16 t + 256 r] in, v[p] = y[256 p + j]
// out: DFT over r, W256^(-w a), half-warp transpose, DFT over a, CTA-wide
// exchange, W4096^(-q s), DFT over s.
//
// So a forward row, factors on the bins and an inverse row need two CTA barriers
// between them, and the bins meet their factors in registers.  b is one padded
// buffer (element n at n + n / 16): half-warp s keeps to its own 272 elements
// except in the CTA-wide exchange, where the forward row writes element 256 p +
// j (thread j of every p: what that thread may itself have read there before)
// and the inverse row reads it.  Callers: before the forward row nobody else may
// still read elements 256 p + j, before the inverse row nobody may still read
// b; on return from the inverse row other threads may still read b.
template <class TW>
DC_DEV void row_forward(float2 (&v)[16], float2* b, int j, const TW& tw) {
  const int s = j >> 4, t = j & 15;
  float2 w[TW::kBases];
  tw.s3(w, j);                                             // issued ahead of the DFT
  dft16<-1>(v);                                            // over p
  apply_powers(v, w);                                       // W4096^(q s), q = j
#pragma unroll
  for (int r = 0; r < 16; ++r) b[pad16(256 * r + j)] = v[r];
  tw.s2(w, t);
  __syncthreads();
  float2* reg = b + 272 * s;                               // = pad16(256 s)
#pragma unroll
  for (int u = 0; u < 16; ++u) v[u] = reg[17 * u + t];     // q = 16 u + t
  dft16<-1>(v);                                            // over u
  apply_powers(v, w);                                       // W256^(w a)
  __syncwarp();                                            // its reads of the region are done
#pragma unroll
  for (int a = 0; a < 16; ++a) reg[17 * a + t] = v[a];     // V[w = t][a]
  __syncwarp();
#pragma unroll
  for (int q = 0; q < 16; ++q) v[q] = reg[17 * t + q];     // thread a = t: V[w = q][a]
  dft16<-1>(v);                                            // over w
}

// ARRIVE: arrive at the cluster barrier (release) once this thread's last read
// of b is done: peers may overwrite the buffer after their wait.
// FROM: the outputs of thread j also take the factor from (a thread's own
// constant, folded into the last twiddle).
template <bool ARRIVE, bool FROM = false, class TW>
DC_DEV void row_inverse(float2 (&v)[16], float2* b, int j, const TW& tw, float2 from = float2{1.f, 0.f}) {
  const int s = j >> 4, t = j & 15;
  float2 w[TW::kBases];
  tw.s2(w, t);
  dft16<+1>(v);                                            // over r
  orient<+1>(w);
  apply_powers(v, w);                                       // W256^(-w a), a = t
  float2* reg = b + 272 * s;
  __syncwarp();                                            // a forward row's reads of the region
#pragma unroll
  for (int q = 0; q < 16; ++q) reg[17 * q + t] = v[q];     // V[a = t][w]
  __syncwarp();
#pragma unroll
  for (int a = 0; a < 16; ++a) v[a] = reg[17 * t + a];     // thread w = t: V[a][w]
  dft16<+1>(v);                                            // over a
  __syncwarp();
#pragma unroll
  for (int u = 0; u < 16; ++u) reg[17 * u + t] = v[u];     // q = 16 u + t of sub-problem s
  tw.s3(w, j);
  __syncthreads();
#pragma unroll
  for (int q = 0; q < 16; ++q) v[q] = b[pad16(256 * q + j)];
  if constexpr (ARRIVE) asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  orient<+1>(w);
  if constexpr (FROM) apply_powers_from(v, from, w);       // W4096^(-q s), q = j
  else apply_powers(v, w);
  dft16<+1>(v);                                            // over s
}

// A stored row (16-byte aligned; plain loads: it may have been written by the kernel
// a pdl_wait waited for) as 16-byte pairs: thread j's bins 2 i, 2 i + 1 are
// pair spec_pair(j) + 16 i (spec_index).
DC_DEV int spec_pair(int j) { return ((j >> 4) << 7) + (j & 15); }
DC_DEV void load_bins(const float2* row, int j, float2 (&v)[16]) {
  const float4* t = reinterpret_cast<const float4*>(row) + spec_pair(j);
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const float4 q = t[16 * i];
    v[2 * i] = make_float2(q.x, q.y);
    v[2 * i + 1] = make_float2(q.z, q.w);
  }
}
DC_DEV void mul_bins(const float2* row, int j, float2 (&v)[16]) {
  const float4* t = reinterpret_cast<const float4*>(row) + spec_pair(j);
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const float4 q = t[16 * i];
    v[2 * i] = cmul(v[2 * i], make_float2(q.x, q.y));
    v[2 * i + 1] = cmul(v[2 * i + 1], make_float2(q.z, q.w));
  }
}
DC_DEV void store_bins(float2* row, int j, const float2 (&v)[16]) {
  float4* t = reinterpret_cast<float4*>(row) + spec_pair(j);
#pragma unroll
  for (int i = 0; i < 8; ++i) t[16 * i] = make_float4(v[2 * i].x, v[2 * i].y, v[2 * i + 1].x, v[2 * i + 1].y);
}

// v[r] *= the factor of bin k1 + L1 (s + 16 t + 256 r), r = 0..15 (L1 =
// 2^log2L1): the item's table (exp(-i phi_k) times anything else the call
// bundles into the frequency domain, e.g. a matched filter's conjugate
// replica spectrum) when there is one, else exp(-i phi_k) of Eq. 16.
DC_DEV void bin_factors(const FftItem& I, int k1, int log2L1, int j, float2 (&v)[16]) {
  if (I.ptab) {
    mul_bins(I.ptab + (size_t)k1 * kRowN, j, v);
  } else if (I.ph.enabled) {
    // bins r >= 8 are the upper half of the transform: kt = k - L
    const PhaseParams& P = I.ph;
    const float kt0 = (float)(k1 + (((j >> 4) + ((j & 15) << 4)) << log2L1));
    const float step = (float)(256 << log2L1);
    if (P.enabled == kPhasePlain) {
#pragma unroll
      for (int r = 0; r < 16; ++r)
        v[r] = cmul(v[r], iono_factor_kt<true>(P, fmaf((float)(r < 8 ? r : r - 16), step, kt0)));
    } else {
#pragma unroll
      for (int r = 0; r < 16; ++r)
        v[r] = cmul(v[r], iono_factor_kt(P, fmaf((float)(r < 8 ? r : r - 16), step, kt0)));
    }
  }
}

// The whole correction of one L = 4096 transform: zero-padded input, forward row,
// factors, inverse row, 1 / L, truncation.  Every stage base of both rows is loaded up
// front, beside the input: one CTA per transform leaves nothing to hide a load issued
// per stage.  The input is read after pdl_wait, by plain loads (a non-coherent load may
// be scheduled ahead of the wait).
DC_DEV void full_4096(const FftItem& I, float2* b, int j, const float2* tw) {
  float2 f2[4], f3[4];
  GlobalTw{tw}.s2(f2, j & 15);
  GlobalTw{tw}.s3(f3, j);
  pdl_wait();                                   // the input's producer has finished
  float2 v[16];
#pragma unroll
  for (int r = 0; r < 16; ++r) {
    const int n = j + 256 * r;
    v[r] = n < I.n_valid ? I.src[n] : make_float2(0.f, 0.f);
  }
  row_forward(v, b, j, HeldTw{f2, f3});
  bin_factors(I, 0, 0, j, v);
  const float invL = 1.0f / (float)kRowN;
#pragma unroll
  for (int r = 0; r < 16; ++r) v[r] = cscale(v[r], invL);
  row_inverse<false>(v, b, j, HeldTw{f2, f3});
#pragma unroll
  for (int r = 0; r < 16; ++r) {
    const int n = j + 256 * r;
    if (n < I.n_out) __stcs(I.dst + n, v[r]);
  }
}

}  // namespace dc
