// Exact-sinc resampling on tcgen05 tensor cores with hi/lo split operands
// (see exact_tc.cu).
#pragma once

#include "common.cuh"

namespace dc {

struct ExTcArgs {
  int n_in, n_out, n_pulses;
  int rows_per_alpha;      // rows of the split planes between alpha groups (0: shared pulses)
  float2* y;               // [n_alpha][n_pulses][n_out]
  const float* dl;         // per alpha: (alpha - 1) as hi, lo floats
  int* err;                // device error flag (bounded waits)
  // far-field pass only: its output planes [rows of the pulses][n_out]
  uint16_t *loc_hi, *loc_lo;
  // near and far field: blocks either side taken term by term; whether the
  // output's own block is summed first
  int near, own_first;
  // fp16x3 with far field: largest |component| of each two blocks, [pulses][n_peaks],
  // and the inverse of the node values' scale, one per alpha group and column tile
  const float* peak;
  int n_peaks;
  float* loc_inv;
};

// Device scratch of one call: the split planes (exact_tc_plane_bytes each)
// and, with `far`, the planes of block moments (exact_tc_far_plane_bytes of
// n), of node values (exact_tc_far_plane_bytes of n_out) and the pulses' peaks with
// the scales from them (exact_tc_peak_bytes; `groups` of n_pulses).
struct ExTcPlanes {
  void *hi, *lo;
  bool far;
  void *mom_hi, *mom_lo, *loc_hi, *loc_lo, *peak;
};

// Bytes of one 16-bit split plane for `rows` real rows of n samples.
size_t exact_tc_plane_bytes(long long rows, int n);

// Whether blocks away from an output are summed through their moments:
// n_in long enough, and every output within 63 samples of its own index
// (delta_max: the largest |alpha - 1|).
bool exact_tc_far(bool fp16, int n_in, int n_out, double delta_max);
size_t exact_tc_far_plane_bytes(long long rows, int n);
size_t exact_tc_peak_bytes(bool fp16, long long groups, int n_pulses, int n);

// Split x (x_rows_c complex pulses of n samples) into the planes, then run the
// contraction.
cudaError_t launch_exact_tc(bool fp16, const float2* x, long long x_rows_c, int n, const ExTcPlanes& planes,
                            const ExTcArgs& args, int n_alpha, cudaStream_t s);
inline int exact_tc_kernels(const ExTcPlanes& p) { return p.far ? 3 : 2; }   // launched by it

}  // namespace dc
