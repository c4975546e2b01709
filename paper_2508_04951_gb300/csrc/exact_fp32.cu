// Exact-sinc resampling on the FP32 cores (Eq. 17):
//
//   Y[p][n] = sum_m X[p][m] S[n][m],  S[n][m] = sinc(alpha n - m)
//           = (-1)^(m + m_n) sin(pi e_n) / (pi ((m_n - m) + e_n)),  alpha n = m_n + e_n.
//
// Two kernels form that Cauchy sum: ex_tile_kernel for many pulses (S in shared
// memory, reused by up to 64 pulses) and ex_gemv_kernel for at most 8 (one warp per
// output).  Each runs in three roles (ExJob): the whole sum term by term; the
// three 256-sample blocks about an output term by term and the others through
// their moments (the near and far form described at the head of exact_tc.cu,
// here with moments and node values in FP32); and the moments-to-nodes product of
// that form, which is a Cauchy sum as well.
#include "far.cuh"
#include "resample.cuh"

namespace dc {

namespace {

constexpr float kInvPi = 0.318309886183790672f;

enum ExJob : int {
  EX_DENSE = 0,   // every input sample
  EX_NEAR = 1,    // blocks b - 1 .. b + 1 and the node values of block b
  EX_NODES = 2,   // block moments -> node values (outputs (b, i), inputs (B, j))
};

// One output of the sum: its position (or target node) and the weights.
struct ExRow {
  int mn;         // alpha n = mn + e, or the row's block
  float e;        // or the target node, relative to the block's centre
  float sg;       // (-1)^mn sin(pi e) / pi
};
template <int JOB> DC_DEV ExRow ex_row(const ExItem& I, int n) {
  ExRow r;
  if constexpr (JOB == EX_NODES) {
    r.mn = n / kFarP;
    r.e = kTgtHalf * far_node(n % kFarP);
    r.sg = 1.f;
  } else {
    rs_delay(I.dl_hi, I.dl_lo, (float)n, r.mn, r.e);
    r.mn += n;
    const float s = sinpif(r.e) * kInvPi;
    r.sg = (r.mn & 1) ? -s : s;
  }
  return r;
}
// 1 / (tau - s_j) of blocks b and B, s = the source node, zero for near blocks.
DC_DEV float node_weight(const ExRow& r, int B, float s) {
  const int db = r.mn - B;
  return db < -1 || db > 1 ? fast_div(1.f, (float)(db * kFarBlock) + r.e - s) : 0.f;
}

// ------------------------------------------------------------- moments
// M_B[j] = sum_m l_j(m) (-1)^m x[m], one warp per two consecutive blocks.
__global__ void __launch_bounds__(kFarBlock, 2) ex_moments_kernel(ExArgs a, int groups) {
  pdl_release();
  __shared__ float s_w[kFarP * kFarBlock];
  __shared__ float s_D[kFarP * kFarP];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  far_fill_table(s_D, threadIdx.x, blockDim.x);
  __syncthreads();
  far_fill_weights(s_w, s_D, threadIdx.x, 1.f);
  __syncthreads();
  const int nb = (a.n_in + kFarBlock - 1) / kFarBlock;
  const int n_pair = (nb + 1) / 2;
  const long long total = (long long)groups * a.n_pulses * n_pair;
  for (long long g = blockIdx.x * 8LL + warp; g < total; g += gridDim.x * 8LL) {
    const long long pr = g / n_pair;
    const int grp = (int)(pr / a.n_pulses);
    const float2* x = ex_item(a, grp).x + (pr - (long long)grp * a.n_pulses) * a.n_in;
    const int m0 = (int)(g - pr * n_pair) * 2 * kFarBlock + 2 * lane;
    float2 v[2][4][2];
#pragma unroll
    for (int b = 0; b < 2; ++b)
#pragma unroll
      for (int q = 0; q < 4; ++q)
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          const int m = m0 + b * kFarBlock + 64 * q + i;
          v[b][q][i] = m < a.n_in ? __ldg(x + m) : make_float2(0.f, 0.f);
        }
    float2 mom;
    far_moments(s_w, lane, v, mom);
    const int e = (m0 - 2 * lane) / kFarBlock * kFarP + lane;
    if (e < nb * kFarP) a.mom[pr * nb * kFarP + e] = mom;
  }
}

// --------------------------------------------------------------- tiles
// CTA tile: TN (64 or 32) outputs x PT pulses, 4 x 4 per thread, K in chunks of 16.  Input
// chunks arrive by cp.async two chunks ahead (three buffers), the next chunk's
// weights are formed after the current one's products (two buffers): one barrier
// per chunk.  A complex multiply-add is one packed FMA with the weight in both
// lanes.  What bounds the products is shared memory's return path, four cycles of the
// SM per wide load of a warp against eight for the packed FMAs of one input and
// four weights; so four weights travel in one load and a move doubles each (stored
// twice side by side they took two: 48 pulses x 8 rates x 4096 samples 175 us, now
// 153).  8 x 4 per thread (4 loads for 32 FMAs, half the warps): 165.  The 16 node
// values of the far field are one more chunk, taken first (its basis evaluation
// then holds no accumulators).
constexpr int kTK = 16, kXS = 3;
static_assert(kTK == kFarP, "the node values are one chunk");

// 8-byte copy from global to shared memory, zero where !valid.
DC_DEV void cp_async8(float2* dst, const float2* src, bool valid) {
  const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(d), "l"(src), "r"(valid ? 8 : 0) : "memory");
}
DC_DEV void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N> DC_DEV void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

template <int PT, int TN, int JOB>
__global__ void __launch_bounds__(TN * PT / 16, (PT <= 32 ? 9216 : 12288) / (TN * PT)) ex_tile_kernel(ExArgs a) {
  constexpr int NT = TN * PT / 16;
  constexpr int XR = kTK * PT / NT;                    // inputs per thread and chunk
  constexpr int SR = (kTK * TN + NT - 1) / NT;        // weights per thread and chunk
  __shared__ __align__(16) float Ss[2][kTK][TN];
  __shared__ __align__(16) float2 Xs[kXS][kTK][PT + 2];
  __shared__ float s_D[JOB == EX_NEAR ? kFarP * kFarP : 1];
  const int al = blockIdx.z, n0 = blockIdx.x * TN, p0 = blockIdx.y * PT;
  const ExItem I = ex_item(a, al);
  const int tid = threadIdx.x;
  const int blk = n0 / kFarBlock;
  const int kb = (a.n_in + kFarBlock - 1) / kFarBlock * kFarP;
  const int ob = (a.n_out + kFarBlock - 1) / kFarBlock * kFarP;
  const long long grp = a.shared ? 0 : al;
  const float2* X = JOB == EX_NODES ? a.mom + grp * a.n_pulses * kb : I.x;
  const float2* L = JOB == EX_NEAR ? a.loc + grp * a.n_pulses * ob : nullptr;
  float2* Y = JOB == EX_NODES ? a.loc + grp * a.n_pulses * ob : I.y;
  const int n_in = JOB == EX_NODES ? kb : a.n_in;
  const int n_out = JOB == EX_NODES ? ob : a.n_out;

  const int on = tid % TN, ok = tid / TN;            // the weights this thread forms
  const ExRow row = ex_row<JOB>(I, n0 + on);
  const int xk = tid % kTK, xp = tid / kTK;            // the input it copies: 4 pulses, 16 samples a half-warp
  int lo = 0, hi = n_in, far = 0;
  if constexpr (JOB == EX_NEAR) {
    // chunk 0: node values and bases.  A pulse with a sample that is not
    // finite (or near overflow) far away has node values that are not finite:
    // its tile then takes every term.
    bool bad = false;
#pragma unroll
    for (int r = 0; r < XR; ++r) {
      const int p = p0 + xp + NT / kTK * r;
      float2 v = make_float2(0.f, 0.f);
      if (p < a.n_pulses) v = __ldcg(L + (size_t)p * ob + blk * kFarP + xk);
      bad = bad || !(isfinite(v.x) && isfinite(v.y));
      Xs[0][xk][xp + NT / kTK * r] = v;
    }
    far_fill_table(s_D, tid, NT);
    far = !__syncthreads_or(bad);
    if (far) {
      lo = max(0, (blk - 1) * kFarBlock);
      hi = max(lo, min(n_in, (blk + 2) * kFarBlock));
      float T[kFarP];
      far_polys(((float)(row.mn - blk * kFarBlock) - 127.5f + row.e) * (1.f / kTgtHalf), T);
#pragma unroll 1
      for (int k = ok; k < kTK; k += NT / TN) Ss[0][k][on] = row.sg * far_basis(s_D, k, T);
    }
  }
  const int n_chunk = (hi - lo + kTK - 1) / kTK + far;

  // chunk c's weights into buffer c % 2, its input into buffer c % 3
  const float sgk = (ok & 1) ? -row.sg : row.sg;       // (-1)^k of this thread's first k
  auto weights = [&](int c) {
    const int m0 = lo + (c - far) * kTK;
    const float d0 = (float)(row.mn - m0 - ok);
#pragma unroll
    for (int r = 0; r < SR; ++r) {
      constexpr int KS = NT / TN;
      const int k = ok + KS * r;
      if (SR * KS == kTK || k < kTK) {
        float w;
        if constexpr (JOB == EX_NODES) {
          w = m0 + k < n_in ? node_weight(row, (m0 + k) / kFarP, kSrcHalf * far_node(k)) : 0.f;
        } else {
          // (m_n - m) exactly, then + e; samples past n_in are zero, their
          // weights finite; e = 0 (sigma = 0) leaves weight 1 at m = m_n alone
          const float den = (d0 - (float)(KS * r)) + row.e;
          w = fast_div((KS * r) & 1 ? -sgk : sgk, den);
          if (den == 0.f) w = 1.f;
        }
        Ss[c & 1][k][on] = w;
      }
    }
  };
  auto fetch = [&](int c) {
    if (c < n_chunk) {
      const int m = lo + (c - far) * kTK + xk;
#pragma unroll
      for (int r = 0; r < XR; ++r) {
        const int p = p0 + xp + NT / kTK * r;
        const bool in = p < a.n_pulses && m < n_in;
        cp_async8(&Xs[c % kXS][xk][xp + NT / kTK * r], in ? X + (size_t)p * n_in + m : X, in);
      }
    }
    cp_async_commit();
  };

  // a warp covers 32 outputs x 16 pulses: its three wide loads per k read 128
  // distinct bytes at most; four consecutive outputs, pulses 2 tp, + 1 and 8 more
  const int warp = tid >> 5, lane = tid & 31;
  const int wn = (TN == 64 ? (warp & 1) * 32 : 0) + 4 * (lane & 7);
  const int wp = (TN == 64 ? warp >> 1 : warp) * 16 + 2 * (lane >> 3);
  float2 acc[4][4];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = make_float2(0.f, 0.f);
  if (!far) {
    __syncthreads();                                   // chunk 0's buffers may hold node values
    fetch(0);
    if (n_chunk > 0) weights(0);
  } else {
    cp_async_commit();
  }
  fetch(1);
  for (int c = 0; c < n_chunk; ++c) {
    cp_async_wait<1>();                                // this thread's copies of chunk c
    __syncthreads();                                   // everyone's, and everyone is done with chunk c - 1
    fetch(c + 2);
    const int b = c & 1, x3 = c % kXS;
    // few warps (PT <= 32): the next k's operands are loaded ahead of this
    // k's products; more warps hide the loads (48 pulses x 8 rates x 4096: 153
    // against 165 us)
    constexpr bool AHEAD = PT <= 32;
    float4 f[AHEAD ? 2 : 1][3];
    auto load = [&](int k) {
      float4 (&q)[3] = f[AHEAD ? k & 1 : 0];
      q[0] = *reinterpret_cast<const float4*>(&Ss[b][k][wn]);
      q[1] = *reinterpret_cast<const float4*>(&Xs[x3][k][wp]);
      q[2] = *reinterpret_cast<const float4*>(&Xs[x3][k][wp + 8]);
    };
    if constexpr (AHEAD) load(0);
#pragma unroll
    for (int k = 0; k < kTK; ++k) {
      if (AHEAD ? k + 1 < kTK : true) load(AHEAD ? k + 1 : k);
      const float4 (&q)[3] = f[AHEAD ? k & 1 : 0];
      const float2 s[4] = {{q[0].x, q[0].x}, {q[0].y, q[0].y}, {q[0].z, q[0].z}, {q[0].w, q[0].w}};
      const float2 x[4] = {{q[1].x, q[1].y}, {q[1].z, q[1].w}, {q[2].x, q[2].y}, {q[2].z, q[2].w}};
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = __ffma2_rn(x[j], s[i], acc[i][j]);
    }
    if (c + 1 < n_chunk) weights(c + 1);
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int n = n0 + wn + i;
    if (n >= n_out) continue;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int p = p0 + wp + (j >> 1) * 8 + (j & 1);
      if (p < a.n_pulses)
        Y[(size_t)p * n_out + n] = JOB == EX_NODES ? acc[i][j] : rotate(acc[i][j], I.rot_hi, I.rot_lo, n);
    }
  }
}

// ------------------------------------------------------------ few pulses
// A matrix-vector product (one pulse per call of the single-pulse entry
// points): one warp per output sample, lanes striding the input, the weight
// computed once per (n, m) and applied to every pulse, lanes combined by a fixed
// shuffle tree (deterministic).
// One lane's share of the sum: terms m = lo + lane, + 32, ... (FAST: m_n - m
// converted by exact_i2f, valid for |m_n - m| < 2^22).  A round's loads are
// issued together, ahead of its weights (the kernel is bound by their latency);
// the terms are still added in the order m = lo + lane, + 32, ...
template <bool FAST> DC_DEV float gemv_weight(int mn, int m, float e, float sgl) {
  const float den = (FAST ? exact_i2f(mn - m) : (float)(mn - m)) + e;
  return fast_div(sgl, den);
}
template <int P, class W>
DC_DEV void gemv_terms(const float2* __restrict__ x, int n_in, int np, int m, int hi, W&& weight,
                       float2 (&acc)[P]) {
  constexpr int U = P <= 2 ? 8 : 4;                    // loads of a pulse in flight
  for (; m + 32 * (U - 1) < hi; m += 32 * U) {
    float2 xv[P][U];
#pragma unroll
    for (int p = 0; p < P; ++p)
#pragma unroll
      for (int u = 0; u < U; ++u) xv[p][u] = __ldg(x + (size_t)min(p, np - 1) * n_in + m + 32 * u);
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const float w = weight(m + 32 * u);
#pragma unroll
      for (int p = 0; p < P; ++p) {
        acc[p].x = fmaf(xv[p][u].x, w, acc[p].x);
        acc[p].y = fmaf(xv[p][u].y, w, acc[p].y);
      }
    }
  }
  for (; m < hi; m += 32) {
    const float w = weight(m);
#pragma unroll
    for (int p = 0; p < P; ++p) {
      if (p < np) {
        const float2 xv = __ldg(x + (size_t)p * n_in + m);
        acc[p].x = fmaf(xv.x, w, acc[p].x);
        acc[p].y = fmaf(xv.y, w, acc[p].y);
      }
    }
  }
}

template <int P, int JOB>
__global__ void __launch_bounds__(256) ex_gemv_kernel(ExArgs a) {
  pdl_release();                        // the kernel that follows may start its set-up
  const ExItem I = ex_item(a, blockIdx.y);
  const int n = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  const int kb = (a.n_in + kFarBlock - 1) / kFarBlock * kFarP;
  const int ob = (a.n_out + kFarBlock - 1) / kFarBlock * kFarP;
  if (n >= (JOB == EX_NODES ? ob : a.n_out)) return;
  const int p0 = blockIdx.z * P, np = min(P, a.n_pulses - p0);   // z > 0: node values only
  const long long row0 = (a.shared ? 0 : (long long)blockIdx.y * a.n_pulses) + p0;
  const ExRow row = ex_row<JOB>(I, n);
  float2 acc[P];
#pragma unroll
  for (int p = 0; p < P; ++p) acc[p] = make_float2(0.f, 0.f);
  auto reduce = [&] {
#pragma unroll
    for (int p = 0; p < P; ++p) {
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        acc[p].x += __shfl_xor_sync(0xffffffffu, acc[p].x, o);
        acc[p].y += __shfl_xor_sync(0xffffffffu, acc[p].y, o);
      }
    }
  };
  if constexpr (JOB == EX_NODES) {
    const float s = kSrcHalf * far_node(lane % kFarP);   // j = m % 16 of every term of this lane
    pdl_wait();
    const float2* M = a.mom + row0 * kb;
#pragma unroll 2
    for (int m = lane; m < kb; m += 32) {
      const float w = node_weight(row, m / kFarP, s);
      float2 xv[P];                     // all loads of a round in flight together
#pragma unroll
      for (int p = 0; p < P; ++p) xv[p] = M[(size_t)min(p, np - 1) * kb + m];
#pragma unroll
      for (int p = 0; p < P; ++p) {
        acc[p].x = fmaf(xv[p].x, w, acc[p].x);
        acc[p].y = fmaf(xv[p].y, w, acc[p].y);
      }
    }
    reduce();
    if (lane == 0) {
#pragma unroll
      for (int p = 0; p < P; ++p)
        if (p < np) a.loc[(row0 + p) * ob + n] = acc[p];
    }
    return;
  } else {
    const int mn = row.mn;
    const float e = row.e;
    int lo = 0, hi = a.n_in;
    float2 far[P];
    if constexpr (JOB == EX_NEAR) {
      // lane i < 16: u_i(t_n) L_b[i]; l_i(z) = (1/p) sum_k d_k T_k(z_i) T_k(z)
      const int blk = n / kFarBlock;
      const float z = ((float)(mn - blk * kFarBlock) - 127.5f + e) * (1.f / kTgtHalf);
      const float zi = far_node(lane % kFarP);
      float t0 = 1.f, t1 = z, c0 = 1.f, c1 = zi, u = fmaf(z + z, zi, 1.f);
#pragma unroll
      for (int k = 2; k < kFarP; ++k) {
        const float t = fmaf(2.f * z, t1, -t0), c = fmaf(2.f * zi, c1, -c0);
        u = fmaf(t + t, c, u);
        t0 = t1, t1 = t, c0 = c1, c1 = c;
      }
      u *= lane < kFarP ? row.sg / kFarP : 0.f;
      pdl_wait();
      bool ok = true;
#pragma unroll
      for (int p = 0; p < P; ++p) {
        far[p] = make_float2(0.f, 0.f);
        if (p < np) {
          const float2 v = __ldcg(a.loc + (row0 + p) * ob + blk * kFarP + lane % kFarP);
          ok = ok && isfinite(v.x) && isfinite(v.y);
          far[p] = make_float2(u * v.x, u * v.y);
        }
      }
      // a pulse with a sample that is not finite (or near overflow) far away has
      // node values that are not finite: its outputs then take every term
      if (__all_sync(0xffffffffu, ok)) {
        lo = max(0, (blk - 1) * kFarBlock);
        hi = min(a.n_in, (blk + 2) * kFarBlock);
#pragma unroll
        for (int p = 0; p < P; ++p) acc[p] = far[p];
      }
    }
    if (e == 0.f) {                                // alpha n on a sample: copy it
      if (lane < np) {
        const bool in = mn >= 0 && mn < a.n_in;
        const float2 v = in ? __ldg(I.x + (size_t)lane * a.n_in + mn) : make_float2(0.f, 0.f);
        I.y[(size_t)lane * a.n_out + n] = rotate(v, I.rot_hi, I.rot_lo, n);
      }
      return;
    }
    const float sgl = (lane & 1) ? -row.sg : row.sg;   // (-1)^m: m steps by 32 from lo + lane, lo even
    // m_n - m lies in (m_n - n_in, m_n]; below 2^22 in size (any Doppler
    // range rate) it converts exactly without the quarter-rate instruction
    if (mn < (1 << 22))
      gemv_terms<P>(I.x, a.n_in, np, lo + lane, hi, [&](int m) { return gemv_weight<true>(mn, m, e, sgl); }, acc);
    else
      gemv_terms<P>(I.x, a.n_in, np, lo + lane, hi, [&](int m) { return gemv_weight<false>(mn, m, e, sgl); }, acc);
    reduce();
    if (lane == 0) {
#pragma unroll
      for (int p = 0; p < P; ++p)
        if (p < np) I.y[(size_t)p * a.n_out + n] = rotate(acc[p], I.rot_hi, I.rot_lo, n);
    }
  }
}

// -------------------------------------------------------------- launches
constexpr int kMaxGrid = 65535;                        // CTAs of a grid in y and z

template <class K>
cudaError_t launch(K k, dim3 grid, int threads, bool pdl, const ExArgs& a, cudaStream_t s) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(threads);
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = pdl ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, k, a);
}

template <int JOB>
cudaError_t launch_gemv(const ExArgs& a, int rows, int n_alpha, cudaStream_t s) {
  const dim3 grid((rows + 7) / 8, n_alpha, (a.n_pulses + 7) / 8);
  const bool pdl = JOB != EX_DENSE;
  if (a.n_pulses == 1) return launch(ex_gemv_kernel<1, JOB>, grid, 256, pdl, a, s);
  if (a.n_pulses <= 2) return launch(ex_gemv_kernel<2, JOB>, grid, 256, pdl, a, s);
  if (a.n_pulses <= 4) return launch(ex_gemv_kernel<4, JOB>, grid, 256, pdl, a, s);
  return launch(ex_gemv_kernel<8, JOB>, grid, 256, pdl, a, s);
}

template <int TN, int JOB>
cudaError_t launch_tile_n(const ExArgs& a, int pt, dim3 grid, cudaStream_t s) {
  // no programmatic launch: tiles placed while the kernel before still holds
  // most SMs pile up on the free ones (48 pulses x 3072 samples: 138 against 76 us)
  const bool pdl = false;
  if (pt == 64) return launch(ex_tile_kernel<64, TN, JOB>, grid, TN * 4, pdl, a, s);
  if (pt == 48) return launch(ex_tile_kernel<48, TN, JOB>, grid, TN * 3, pdl, a, s);
  if (pt == 32) return launch(ex_tile_kernel<32, TN, JOB>, grid, TN * 2, pdl, a, s);
  return launch(ex_tile_kernel<16, TN, JOB>, grid, TN, pdl, a, s);
}

// 32 instead of 64 outputs per tile while those then fill at most one CTA per SM:
// 64 against 32, us, pulses x rates x samples: 48 x 1 x 4096: 61 / 49, 64 x 4 x 1024:
// 62 / 43, 48 x 8 x 512: 33 / 25, 12 x 1 x 4096: 41 / 43; beyond, the inputs are
// fetched twice as often for nothing (64 x 4 x 2048: 62 / 64, 48 x 8 x 4096: 154 / 160).
template <int JOB>
cudaError_t launch_tile(const ExArgs& a, int rows, int n_alpha, cudaStream_t s) {
  // the pulse tile that pads the pulses least, the widest among equals, of those
  // whose tiles a grid takes
  int pt = 64, least = (a.n_pulses + 63) / 64 * 64;
  for (int t : {48, 32, 16}) {
    const int tiles = (a.n_pulses + t - 1) / t;
    if (tiles <= kMaxGrid && tiles * t < least) pt = t, least = tiles * t;
  }
  const dim3 wide((rows + 63) / 64, (a.n_pulses + pt - 1) / pt, n_alpha);
  if (pt <= 16 || 2LL * wide.x * wide.y * wide.z > 152) return launch_tile_n<64, JOB>(a, pt, wide, s);
  return launch_tile_n<32, JOB>(a, pt, dim3((rows + 31) / 32, wide.y, wide.z), s);
}

// The node values of many pulses take the warp-per-output form while the
// product is small: a tile's chain of blocks(n_in) chunks is latency.
constexpr int kNodesGemvMax = 1024;                    // moments per pulse
template <int JOB>
cudaError_t launch_sum(const ExArgs& a, int rows, int n_alpha, cudaStream_t s) {
  const bool gemv = a.n_pulses <= 8 || (JOB == EX_NODES && kFarP * far_blocks(a.n_in) <= kNodesGemvMax &&
                                        (a.n_pulses + 7) / 8 <= kMaxGrid);
  return gemv ? launch_gemv<JOB>(a, rows, n_alpha, s) : launch_tile<JOB>(a, rows, n_alpha, s);
}

}  // namespace

size_t exact_fp32_far_elems(long long pulses, int n) { return (size_t)pulses * kFarP * far_blocks(n); }

// The near and far form adds two launches and replaces n_in terms by at most 768
// and 16.  Measured, far against dense, in us:
//   tiles (more than 8 pulses), pulses x rates: 12 x 1: n = 1024: 39 / 35, 1536: 39 /
//   51, 4096: 41 / 129; 48 x 8: 1024: 64 / 59, 1536: 83 / 139, 4096: 154 /
//   670; so from 1536 on.
//   one warp per output: 1 x 1: 4096: 12.3 / 10.3, 6000: 12.4 / 16.4, 16384: 19 / 81;
//   2 x 4: 1536: 16.4 / 12.8, 2048: 18.0 / 18.2; 8 x 1: 2048: 22.6 / 24.9; 8 x 8:
//   1024: 36 / 31, 1536: 46 / 58, 4096: 97 / 312; so from 2^25 terms on.
bool exact_fp32_far(int n_in, int n_out, int n_pulses, int n_alpha, double delta_max) {
  const double terms = (double)n_in * n_out * n_pulses * n_alpha;
  return n_in >= 1536 && (n_pulses > 8 || terms >= (double)(1 << 25)) &&
         delta_max * (double)n_out <= (double)(kFarMargin - 1);
}

cudaError_t launch_exact_fp32(const ExArgs& a, int n_alpha, cudaStream_t s) {
  if (n_alpha <= 0 || a.n_out <= 0 || a.n_pulses <= 0) return cudaSuccess;
  if (a.n_pulses > 64 * kMaxGrid) return cudaErrorInvalidConfiguration;   // before the first launch
  if (!a.mom) return launch_sum<EX_DENSE>(a, a.n_out, n_alpha, s);
  const int groups = a.shared ? 1 : n_alpha;
  const long long pairs = (long long)groups * a.n_pulses * ((far_blocks(a.n_in) + 1) / 2);
  const int grid = (int)((pairs + 7) / 8 < 152 * 2 ? (pairs + 7) / 8 : 152 * 2);
  ex_moments_kernel<<<grid, kFarBlock, 0, s>>>(a, groups);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  if ((e = launch_sum<EX_NODES>(a, kFarP * far_blocks(a.n_out), groups, s)) != cudaSuccess) return e;
  return launch_sum<EX_NEAR>(a, a.n_out, n_alpha, s);
}

}  // namespace dc
