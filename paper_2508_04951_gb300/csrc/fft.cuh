// FFT passes and the ionospheric correction built on them
// (Sec. II-B, Eqs. 15-16: forward DFT, multiply by exp(-i phi_k), inverse DFT).
//
// Transform lengths L = 2^m up to 2^20.  L <= 4096 runs as one "row" pass in
// registers.  Larger L uses the four-step split L = L1 x L2 with
// L2 = 4096, n = n2 + L2 n1, k = k1 + L1 k2:
//   F1  (column pass): DFT over n1 of x[n2 + L2 n1], times W_L^(n2 k1),
//                      stored at T[n2 + L2 k1]
//   F2  (row pass)   : DFT over n2 of row k1 of T  -> bins k1 + L1 k2 of row k1
//                      (transposed spectrum, never reordered; stored spectra and
//                      factor tables keep bin k2 of a row at spec_index(k2))
//   phase multiply on that layout, then the inverse in mirror order:
//   A   (row pass)   : inverse DFT over k2, times W_L^(-n2 k1), back to T
//   B   (column pass): inverse DFT over k1, times 1/L, out[n2 + L2 n1]
// F2, the phase multiply and A run in one row kernel, so a corrected pulse
// costs three passes over the data.
#pragma once

#include "common.cuh"
#include "phase.cuh"

namespace dc {

// Order of the bins of a 4096-point row in stored spectra and factor tables: bin
// k2 = s + 16 a + 256 r (nibbles r, a, s) at index 256 s + 32 (r / 2) + 2 a + r % 2.
// Thread (s, a) of a row transform holds exactly those 16 bins (r = 0..15) after
// the forward row and before the inverse one, so both read and write them
// straight from registers, two bins per 16-byte access.  Rows below 4096 points
// keep natural order.
__host__ __device__ constexpr int spec_index(int k2) {
  return ((k2 & 15) << 8) | ((k2 >> 9) << 5) | (((k2 >> 4) & 15) << 1) | ((k2 >> 8) & 1);
}
__host__ __device__ constexpr int spec_bin(int idx) {
  return (idx >> 8) | (((idx >> 1) & 15) << 4) | ((idx & 1) << 8) | (((idx >> 5) & 7) << 9);
}

// One transform of a launch.  64 bytes: read whole by four 16-byte loads (ldg_item).
struct alignas(16) FftItem {
  PhaseParams ph;
  const float2* src;     // input of this pass
  float2* dst;           // output of this pass
  const float2* ptab;    // per-bin factors (length L): exp(-i phi_k), times a
                         // matched filter's conjugate replica spectrum when
                         // compressing, in the spectrum's layout (bin
                         // k1 + L1 k2 at k1*4096 + spec_index(k2) for L >=
                         // 4096, natural order below); null -> exp(-i phi_k)
                         // computed from `ph`
  int n_valid;           // samples of src that are data (zero beyond), first pass
  int n_out;             // samples stored by the last pass (truncation)
};
static_assert(sizeof(FftItem) == 64, "four 16-byte loads");

// An item by non-coherent loads, which the compiler may move over stores to
// shared memory (it cannot prove those apart from a generic pointer's target).
DC_DEV FftItem ldg_item(const FftItem* p) {
  union {
    uint4 q[4];
    FftItem it;
  } u = {};
#pragma unroll
  for (int i = 0; i < 4; ++i) u.q[i] = __ldg(reinterpret_cast<const uint4*>(p) + i);
  return u.it;
}

enum RowOp : int {
  ROW_FULL = 0,   // L <= 4096: load (zero-pad), fwd, phase, inv, 1/L, store n < n_out
  ROW_MID = 1,    // four-step middle: fwd, phase, inv, W_L^(-n2 k1); in place on T
  ROW_SPEC = 2,   // forward only: L <= 4096 from y (zero-pad), else row of T (F2)
  ROW_APPLY = 3,  // phase + inverse: L <= 4096 -> 1/L, store n < n_out; else twiddle, store T
};
enum ColOp : int {
  COL_F1 = 0,     // forward first pass, from y (zero-pad) to T
  COL_B = 1,      // inverse last pass, from T to out (1/L, n < n_out)
};

// Items of a launch: an array on the device or, null, the one item in the
// arguments themselves (a single transform: no upload, no load).
struct RowArgs {
  const FftItem* items;
  int n_items;
  int log2L;       // transform length
  int log2L1;      // rows per transform (0 for L <= 4096)
  const float2* tw;
  FftItem one;
  int pdl;         // Pdl, ROW_MID: launched programmatically behind the pass before it
};
// The full correction (ROW_FULL) of several length classes L = 2^m, m <= 12, in
// one launch: class m's transforms are items [first[m], first[m + 1]), its CTAs
// blocks [block[m], block[m + 1]).
struct RowClasses {
  const FftItem* items;
  int first[14], block[14];
  const float2* tw;
  FftItem one;
};
struct ColArgs {
  const FftItem* items;
  int n_items;
  int log2L;
  int log2L1;      // column length M = L1
  const float2* tw;
  FftItem one;
  int pdl;         // Pdl: launched programmatically behind the pass before it
};
// Programmatic launches of the three-pass path's second and third pass and of the
// short transforms (`pdl` below): a pass's launch and set-up then run under the one
// before.  With at most one CTA per SM the passes of a single pulse are latency.
// A pass that starts so is placed where there is room, which piles its CTAs on the
// few SMs the first has left; above 64 CTAs (PDL_SPREAD) each therefore asks for so
// much shared memory that two row CTAs never share an SM's 227 KiB, a row and a
// column CTA do.  iono_correct, us, without / with / with spread: n = 2^17: 16.7 /
// 12.3 / 12.3; 2^18: 18.2 / 12.9 / 14.3; 2^19: 18.4 / 22.5 / 14.4.  From two full
// waves on (1216 CTAs) the next pass's CTAs only take slots that the last wave
// leaves empty: 24 x 4 bank of 200000 samples, three chunks: 232 -> 214.
enum Pdl : int { PDL_NONE = 0, PDL_ON = 1, PDL_SPREAD = 2 };
constexpr int kPdlColSmem = 100 << 10, kPdlRowSmem = 120 << 10;
inline int pdl_for(long long ctas) {
  return ctas <= 64 || ctas >= 1216 ? PDL_ON : ctas <= 152 ? PDL_SPREAD : PDL_NONE;
}

template <class A> DC_DEV FftItem item_of(const A& a, int i) { return a.items ? a.items[i] : a.one; }

// Launchers (fft.cu).  Return cudaSuccess or the launch error.
cudaError_t launch_row(int op, const RowArgs& a, cudaStream_t s);
cudaError_t launch_row_classes(RowClasses a, cudaStream_t s);   // block[] filled here
cudaError_t launch_col(int op, const ColArgs& a, cudaStream_t s);

}  // namespace dc
