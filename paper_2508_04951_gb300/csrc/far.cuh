// Far field of the exact sinc sum (Eq. 17): geometry and Chebyshev bases of
// the block moments and node values, shared by the tensor-core and the FP32
// kernels (the method is described at the head of exact_tc.cu).
#pragma once

#include "common.cuh"

namespace dc {

constexpr int kFarBlock = 256;                       // samples per block, both sides
constexpr int kFarP = 16;                            // nodes per block, both sides
constexpr int kFarMargin = 64;                       // widening of the target interval
inline int far_blocks(int n) { return (n + kFarBlock - 1) / kFarBlock; }
constexpr float kSrcHalf = 127.5f;                   // source interval [0, 255] about 127.5
constexpr float kTgtHalf = 128.f + kFarMargin;       // target interval about 127.5
// Chebyshev node i of kFarP on [-1, 1], and T_k there.
DC_DEV float far_node(int i) { return cospif((2 * i + 1) / (2.f * kFarP)); }
DC_DEV float far_cheb(int i, int k) {
  return cospif((float)((2 * i + 1) * k % (4 * kFarP)) / (2.f * kFarP));
}
// Lagrange basis of the nodes at z from the Chebyshev polynomials T_k(z):
// l_i(z) = (1/p) sum_k d_k T_k(z_i) T_k(z), d_0 = 1, d_k = 2; D[i][k] holds
// d_k T_k(z_i) / p.
DC_DEV void far_fill_table(float* D, int tid, int threads) {
  for (int q = tid; q < kFarP * kFarP; q += threads) {
    const int i = q / kFarP, k = q % kFarP;
    D[q] = far_cheb(i, k) * ((k ? 2.f : 1.f) / kFarP);
  }
}
DC_DEV void far_polys(float z, float (&T)[kFarP]) {
  T[0] = 1.f;
  T[1] = z;
#pragma unroll
  for (int k = 2; k < kFarP; ++k) T[k] = fmaf(2.f * z, T[k - 1], -T[k - 2]);
}
DC_DEV float far_basis(const float* D, int i, const float (&T)[kFarP]) {
  float v = 0.f;
#pragma unroll
  for (int k = 0; k < kFarP; ++k) v = fmaf(D[i * kFarP + k], T[k], v);
  return v;
}

// Shared table of the moment weights l_j(m) (-1)^m scale at [j][m], one thread
// per sample m of a block (256 threads); D from far_fill_table.
DC_DEV void far_fill_weights(float* w, const float* D, int m, float scale) {
  float T[kFarP];
  far_polys(((float)m - 127.5f) * (1.f / kSrcHalf), T);
#pragma unroll 1
  for (int j = 0; j < kFarP; ++j)
    w[j * kFarBlock + m] = far_basis(D, j, T) * ((m & 1) ? -scale : scale);
}

// Moments of two consecutive blocks by one warp: lane l holds samples
// 64 q + 2 l, + 1 of block b in v[b][q]; it forms its share of the 2 x 16
// complex moments (packed FMAs, the weights from shared memory), and a halving
// exchange over the lanes leaves moment l % 16 of block l / 16 in lane l.
DC_DEV void far_moments(const float* w, int lane, const float2 (&v)[2][4][2], float2& out) {
  float acc[64];                                       // [block][node][re, im]
#pragma unroll
  for (int j = 0; j < kFarP; ++j) {
    float2 s[2] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const float2 u = *reinterpret_cast<const float2*>(w + j * kFarBlock + 64 * q + 2 * lane);
      const float2 u0 = make_float2(u.x, u.x), u1 = make_float2(u.y, u.y);
#pragma unroll
      for (int b = 0; b < 2; ++b) {
        s[b] = __ffma2_rn(v[b][q][0], u0, s[b]);
        s[b] = __ffma2_rn(v[b][q][1], u1, s[b]);
      }
    }
#pragma unroll
    for (int b = 0; b < 2; ++b) {
      acc[b * 32 + 2 * j] = s[b].x;
      acc[b * 32 + 2 * j + 1] = s[b].y;
    }
  }
  // after the step over lane bit o, a lane keeps the half of its values that
  // its bit selects, summed with its partner's
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const bool up = lane & o;
#pragma unroll
    for (int i = 0; i < 2 * o; ++i) {
      const float keep = up ? acc[i + 2 * o] : acc[i];
      const float send = up ? acc[i] : acc[i + 2 * o];
      acc[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
    }
  }
  out = make_float2(acc[0], acc[1]);
}

}  // namespace dc
