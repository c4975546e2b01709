// Exact-sinc resampling as a tensor-core contraction (Eq. 17, Table I row 1):
//
//   Y_a[p][n] = sum_m X[p][m] S_a[n][m],   S_a[n][m] = sinc(a n - m),
//
// for many pulses p sharing one range rate a.  Treating the re/im parts of the
// pulses as 2P real columns this is the GEMM  C[n][c] = sum_m S[n][m] X^T[m][c].
// It runs on the 5th-generation tensor cores (tcgen05.mma, kind::f16) with
// split operands: every FP32 value v is written as hi + lo with hi = rn(v) in
// bf16 (or fp16) and lo = rn(v - hi); the product keeps the three significant
// terms  S_hi X_hi + S_hi X_lo + S_lo X_hi  (dropping S_lo X_lo, ~2^-16 of the
// result for bf16) with FP32 accumulation in tensor memory.  For fp16 the lo
// parts are scaled by 2^11 (they would underflow fp16's range) and summed in a
// second accumulator, C = acc1 + 2^-11 acc2.
//
// One CTA computes a 256 x 256 tile of C for bf16 (two 128-row MMA halves
// sharing each X tile, halving the X traffic per flop) or 128 x 256 for fp16:
//   warp 0     TMA: X_hi / X_lo tiles (256 columns x 32 samples, 64B swizzle)
//   warp 1     TMEM allocation (512 columns); one thread issues the MMAs
//   warps 2-17 generate the S tile (rows x 32) in the same swizzled K-major
//              layout, hi and lo, from the Cauchy form
//              S[n][m] = (-1)^(m + m_n) sin(pi e_n) / (pi ((m_n - m) + e_n)),
//              a n = m_n + e_n -- one division per element, no table
//   epilogue   TMEM -> registers (tcgen05.ld) -> complex64 outputs
// Three (bf16) or four (fp16) pipeline stages of 64 / 48 KiB, mbarriers
// between the producers and the MMA thread, every wait bounded.
//
// Near and far field.  S is a Cauchy matrix, sigma_n (-1)^m / (t_n - m), so a
// block of sources seen from a distance has low rank: the sum over it needs 16
// numbers per pulse instead of its samples (Chebyshev interpolation of 1/(t - m)
// in both arguments; Fong & Darve, "The black-box fast multipole method", J.
// Comput. Phys. 228, 2009).  Inputs and outputs are cut into blocks of
// kFarBlock = 256 samples, and output block b sums
//   near   blocks b-1, b, b+1 (or b-3 .. b+3, below) term by term, as the dense
//          contraction does;
//   far    every other block B through its moments
//            M_B[j] = sum_m l_j(m) (-1)^m x[m]           (16 source nodes s_j)
//          turned into 16 values at the target nodes tau_i of block b,
//            L_b[i] = sum_{B far} sum_j M_B[j] / (tau_i - s_j),
//          and read at every output as sigma_n sum_i u_i(t_n) L_b[i].
// The nodes are fixed in each block (the target interval is 64 samples wider
// on both sides, so that t_n of any output stays inside while |delta| n_out <=
// 63), so both interpolation errors are below 2e-9 of the far sum (Chebyshev
// ratio rho >= 3.7 at 16 nodes), itself 3 % of a typical output.  Three
// launches: far_split_kernel writes the 16-bit planes and, in FP32 from the
// values the planes hold, the moments; the tile kernel runs the moments-to-nodes
// product (JOB_FAR: the same Cauchy form, K = 16 per block); the tile kernel
// runs the near chunks and one more K = 16 step for the far field (JOB_NEAR).
//
// The accumulators round toward zero at every MMA, so a long sum loses a little of
// each output (about 3e-8 per K = 16 step after its largest terms): the dense
// contraction of 8192 samples is 2.3e-5 off in bf16x3 and 9e-6 in fp16x3, the
// near and far form 4e-6 and 9e-7.  bf16x3 above 4096 samples takes the blocks
// within three of its own, its own first (1.0e-5 off): with one block either
// side the results would be more than 2e-5 from the dense contraction's.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cudaTypedefs.h>

#include <algorithm>

#include "exact_tc.cuh"
#include "far.cuh"
#include "tc.cuh"

namespace dc {

namespace {

constexpr int BN = 256, BK = 32;                     // N columns, K per stage
constexpr int kHalfRows = 128;                       // rows per MMA (M = 128)
constexpr int kAPlane = kHalfRows * BK * 2;          // 8 KiB: one 128-row A plane
constexpr int kBPlane = BN * BK * 2;                 // 16 KiB: one B plane
constexpr int kProducerWarps = 16;                   // S-tile producers (4 per scheduler)
constexpr int kThreads = 64 + 32 * kProducerWarps;

// bf16x3: two 128-row halves share every X tile (one accumulator each);
// fp16x3: one half with two accumulators (hi*hi and the 2^11-scaled cross
// terms).  Either way the 512 TMEM columns hold exactly the accumulators.
template <bool FP16> struct Cfg {
  static constexpr int MH = FP16 ? 1 : 2;            // 128-row halves per CTA
  static constexpr int BM = MH * kHalfRows;
  static constexpr int STAGES = FP16 ? 4 : 3;
  static constexpr int A_BYTES = 2 * MH * kAPlane;   // hi + lo planes of all halves
  static constexpr int STAGE = A_BYTES + 2 * kBPlane;
  static constexpr int SMEM = STAGES * STAGE + 1024; // + alignment slack
};
constexpr float kInvPi = 0.318309886183790672f;

// Instruction descriptor of this kernel's MMAs: N = 256, M = 128.
template <bool FP16> __host__ __device__ constexpr uint32_t instr_desc() {
  return f16_instr_desc(!FP16, kHalfRows, BN);
}

// Split 8 floats into 8 hi and 8 lo 16-bit values (one 16-byte chunk each).
template <bool FP16> DC_DEV void split8(const float (&v)[8], uint4& hi, uint4& lo) {
  uint32_t h[4], l[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    if constexpr (FP16) {
      const __half2 a = __floats2half2_rn(v[2 * i], v[2 * i + 1]);
      const __half2 b = __floats2half2_rn((v[2 * i] - __low2float(a)) * 2048.f,
                                          (v[2 * i + 1] - __high2float(a)) * 2048.f);
      h[i] = *reinterpret_cast<const uint32_t*>(&a);
      l[i] = *reinterpret_cast<const uint32_t*>(&b);
    } else {
      const __nv_bfloat162 a = __floats2bfloat162_rn(v[2 * i], v[2 * i + 1]);
      const __nv_bfloat162 b = __floats2bfloat162_rn(v[2 * i] - __low2float(a),
                                                     v[2 * i + 1] - __high2float(a));
      h[i] = *reinterpret_cast<const uint32_t*>(&a);
      l[i] = *reinterpret_cast<const uint32_t*>(&b);
    }
  }
  hi = make_uint4(h[0], h[1], h[2], h[3]);
  lo = make_uint4(l[0], l[1], l[2], l[3]);
}

// One value into its hi and lo halves (lo times 2^11 for fp16).
template <bool FP16> DC_DEV void split1(float v, uint16_t& hi, uint16_t& lo) {
  if constexpr (FP16) {
    const __half a = __float2half_rn(v);
    hi = __half_as_ushort(a);
    lo = __half_as_ushort(__float2half_rn((v - __half2float(a)) * 2048.f));
  } else {
    const __nv_bfloat16 a = __float2bfloat16_rn(v);
    hi = __bfloat16_as_ushort(a);
    lo = __bfloat16_as_ushort(__float2bfloat16_rn(v - __bfloat162float(a)));
  }
}
template <bool FP16> DC_DEV float join1(uint16_t hi, uint16_t lo) {
  if constexpr (FP16)
    return fmaf(__half2float(__ushort_as_half(lo)), 1.f / 2048, __half2float(__ushort_as_half(hi)));
  else
    return __bfloat162float(__ushort_as_bfloat16(hi)) + __bfloat162float(__ushort_as_bfloat16(lo));
}

// a n = m_n + e_n with a - 1 a double-float (same arithmetic as the FP32 path).
DC_DEV void position(float dl_hi, float dl_lo, int n, int& m, float& e) {
  rs_delay(dl_hi, dl_lo, (float)n, m, e);
  m += n;
}

// Powers of two that keep the 16-bit moments and node values inside fp16's
// range for any pulse inside it (|M| <= 32 max|x|, |L| <= 17 max|x|):
// planes hold M / 32 and L times loc_scale, the Cauchy elements are taken times 256.
constexpr float kMomScale = 1.f / 32, kCauchyScale = 256.f;
// 2^-e, e the exponent of the largest component of the tile's pulses, in [1/32, 1]: 1/32
// throughout left node values of pulses below 1e-4 32 times coarser than their
// samples, as fp16's spacing ends at 2^-24 (pulses of 1e-6 x 2000 samples: up to 3.0 times
// the dense sum's distance from 64 bits, now below it; 512 pulses x 16 rates x 8192:
// 542 us, now 546).  bf16, with FP32's range, keeps 1/32.
constexpr float kLocScale = 1.f / 32;
DC_DEV float loc_scale(uint32_t peak_bits) {
  const int e = (int)(peak_bits >> 23) - 127;                   // 128 for inf and NaN
  return __uint_as_float((uint32_t)(127 - min(max(e, 0), 5)) << 23);
}

constexpr int kFarMinIn = 1536, kFarMinInFp16 = 1792;   // see exact_tc_far
constexpr int kFarWideIn = 4096;                     // bf16x3 above: near = 3 blocks either side

// What one launch of the tile kernel contracts.
enum Job : int {
  JOB_DENSE = 0,   // every input sample
  JOB_NEAR = 1,    // the blocks around the output's own, and the far field from the node values
  JOB_FAR = 2,     // block moments -> node values (rows (b, i), columns of K (B, j))
};

template <bool FP16, int JOB>
__global__ void __launch_bounds__(kThreads, 1)
    exact_tc_kernel(const __grid_constant__ CUtensorMap map_hi,
                    const __grid_constant__ CUtensorMap map_lo,
                    const __grid_constant__ CUtensorMap map_far_hi,
                    const __grid_constant__ CUtensorMap map_far_lo, ExTcArgs a) {
  using C = Cfg<FP16>;
  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(8) unsigned long long full_bar[C::STAGES], empty_bar[C::STAGES], acc_bar;
  __shared__ uint32_t tmem_base;
  __shared__ float s_sig[C::BM], s_e[C::BM];
  __shared__ int s_m[C::BM];
  __shared__ float s_far[JOB == JOB_DENSE ? 1 : kFarP * kFarP];   // basis table, or source nodes
  constexpr bool PEAK = FP16 && JOB == JOB_FAR;
  __shared__ uint32_t s_peak[PEAK ? kThreads / 32 : 1];   // the warps' shares of the pulses' peak

  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                             ~(uintptr_t)1023);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int n0 = blockIdx.x * C::BM;
  const int c0 = blockIdx.y * BN;
  const int alpha = blockIdx.z;
  // the K chunks of this tile: all of the planes' chunks, or (JOB_NEAR) those
  // of the blocks around the tile's own and then one chunk of node values
  const int blk = n0 / kFarBlock;              // output block of the tile
  int k0 = 0, nk = (a.n_in + BK - 1) / BK, own = 0;
  if constexpr (JOB == JOB_NEAR) {
    constexpr int kPer = kFarBlock / BK;
    k0 = max(0, (blk - a.near) * kPer);
    const int planes = max(0, min(nk, (blk + a.near + 1) * kPer) - k0);
    if (a.own_first) own = min(blk * kPer - k0, planes);
    nk = planes + 1;
  }
  // plane chunk of step kc (own_first: the output's own block first, then
  // those above it, then those below)
  auto chunk_of = [&](int kc) {
    if constexpr (JOB != JOB_NEAR) return kc;
    const int c = kc + own;
    return k0 + (c < nk - 1 ? c : c - (nk - 1));
  };
  constexpr uint32_t kCols = 512;

  if (threadIdx.x == 0) {
    for (int s = 0; s < C::STAGES; ++s) {
      mbar_init(&full_bar[s], 1 + kProducerWarps);   // TMA arrival + one per producer warp
      mbar_init(&empty_bar[s], 1);
    }
    mbar_init(&acc_bar, 1);
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_addr(&tmem_base)),
                 "r"(kCols));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  if (warp >= 2 && threadIdx.x - 64 < C::BM) {
    const int nl = threadIdx.x - 64;
    if constexpr (JOB == JOB_FAR) {
      // row (b, i): target node i of block b, relative to the block's centre
      s_m[nl] = (n0 + nl) / kFarP;
      s_e[nl] = kTgtHalf * far_node((n0 + nl) % kFarP);
    } else {
      int m;
      float e;
      position(a.dl[2 * alpha], a.dl[2 * alpha + 1], n0 + nl, m, e);
      const float s = sinpif(e) * kInvPi;
      s_m[nl] = m;
      s_e[nl] = e;
      s_sig[nl] = (m & 1) ? -s : s;
    }
  }
  if constexpr (JOB == JOB_NEAR) far_fill_table(s_far, threadIdx.x, kThreads);
  if constexpr (JOB == JOB_FAR) {
    if (threadIdx.x < kFarP) s_far[threadIdx.x] = kSrcHalf * far_node(threadIdx.x);
  }
  if constexpr (PEAK) {
    // non-negative floats (inf and NaN above all) in the order of their bits
    const long long first = (long long)alpha * (a.rows_per_alpha / 2) + c0 / 2;
    const int count = min(BN / 2, a.n_pulses - c0 / 2) * a.n_peaks;
    uint32_t m = 0;
    for (int i = threadIdx.x; i < count; i += kThreads)
      m = max(m, __float_as_uint(__ldg(a.peak + first * a.n_peaks + i)));
    m = __reduce_max_sync(0xffffffffu, m);
    if (lane == 0) s_peak[warp] = m;
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  // node values' scale: formed where they are, read where they are used
  float* const tile_inv = a.loc_inv + (a.rows_per_alpha ? alpha : 0) * gridDim.y + blockIdx.y;
  float loc = kLocScale;
  if constexpr (PEAK) {
    uint32_t m = 0;
    for (int i = 0; i < kThreads / 32; ++i) m = max(m, s_peak[i]);
    loc = loc_scale(m);
    if (blockIdx.x == 0 && threadIdx.x == 0) *tile_inv = 1.f / loc;
  }
  const uint32_t tmem = tmem_base;
  bool ok = true;

  if (warp == 0) {
    // ---------------------------------------------------------------- TMA
    if (lane == 0) {
      const int row0 = alpha * a.rows_per_alpha + c0;
      for (int kc = 0; kc < nk && ok; ++kc) {
        const int s = kc % C::STAGES;
        const uint32_t ph = (kc / C::STAGES) & 1;
        if (!mbar_wait_bounded(&empty_bar[s], ph ^ 1, a.err)) { ok = false; break; }
        uint8_t* st = smem + s * C::STAGE;
        mbar_expect_tx(&full_bar[s], 2 * kBPlane);
        if (JOB == JOB_NEAR && kc == nk - 1) {       // the block's 16 node values (the first half)
          tma_load_2d(st + C::A_BYTES, &map_far_hi, blk * kFarP, row0, &full_bar[s]);
          tma_load_2d(st + C::A_BYTES + kBPlane, &map_far_lo, blk * kFarP, row0, &full_bar[s]);
        } else {
          tma_load_2d(st + C::A_BYTES, &map_hi, chunk_of(kc) * BK, row0, &full_bar[s]);
          tma_load_2d(st + C::A_BYTES + kBPlane, &map_lo, chunk_of(kc) * BK, row0, &full_bar[s]);
        }
      }
    }
  } else if (warp == 1) {
    // ---------------------------------------------------------------- MMA
    if (lane == 0) {
      constexpr uint32_t idesc = instr_desc<FP16>();
      for (int kc = 0; kc < nk && ok; ++kc) {
        const int s = kc % C::STAGES;
        const uint32_t ph = (kc / C::STAGES) & 1;
        if (!mbar_wait_bounded(&full_bar[s], ph, a.err)) { ok = false; break; }
        tc_fence_after();
        const uint32_t st = smem_addr(smem + s * C::STAGE);
        const uint32_t b_hi = st + C::A_BYTES, b_lo = b_hi + kBPlane;
#pragma unroll
        for (int kk = 0; kk < BK / 16; ++kk) {
          if (JOB == JOB_NEAR && kk > 0 && kc == nk - 1) break;   // 16 node values only
          const uint32_t off = kk * 32;     // 16 elements of K = 32 bytes inside the swizzle atom
          const uint32_t acc = (kc > 0 || kk > 0) ? 1u : 0u;
#pragma unroll
          for (int h = 0; h < C::MH; ++h) {
            const uint32_t a_hi = st + h * kAPlane, a_lo = st + (C::MH + h) * kAPlane;
            const uint32_t d = tmem + h * 256;
            if constexpr (FP16) {
              mma_f16(d, sw64_desc(a_hi + off), sw64_desc(b_hi + off), idesc, acc);
              mma_f16(d + 256, sw64_desc(a_hi + off), sw64_desc(b_lo + off), idesc, acc);
              mma_f16(d + 256, sw64_desc(a_lo + off), sw64_desc(b_hi + off), idesc, 1u);
            } else {
              mma_f16(d, sw64_desc(a_hi + off), sw64_desc(b_hi + off), idesc, acc);
              mma_f16(d, sw64_desc(a_hi + off), sw64_desc(b_lo + off), idesc, 1u);
              mma_f16(d, sw64_desc(a_lo + off), sw64_desc(b_hi + off), idesc, 1u);
            }
          }
        }
        mma_commit(&empty_bar[s]);
      }
      mma_commit(&acc_bar);
    }
  } else {
    // ------------------------------------------------- S tile producers
    // thread -> one of the BM rows and CHUNKS of its 4 chunks of 8 (bf16:
    // 256 rows, 2 chunks; fp16: 128 rows, 1 chunk)
    constexpr int NP = 32 * kProducerWarps;
    constexpr int CHUNKS = 4 * C::BM / NP;
    static_assert(CHUNKS >= 1 && 4 * C::BM == CHUNKS * NP, "producers cover the tile");
    const int p = threadIdx.x - 64;            // 0..NP-1
    const int nl = p % C::BM;
    const int cbase = (p / C::BM) * CHUNKS;
    const int h = nl >> 7, r = nl & 127;       // half and row inside it
    const int mn = s_m[nl];
    const float en = s_e[nl], sg = s_sig[nl];
    const float loc_inv = FP16 && JOB == JOB_NEAR ? __ldg(tile_inv) : 1.f / kLocScale;
    for (int kc = 0; kc < nk && ok; ++kc) {
      const int s = kc % C::STAGES;
      const uint32_t ph = (kc / C::STAGES) & 1;
      if (!mbar_wait_bounded(&empty_bar[s], ph ^ 1, a.err)) { ok = false; break; }
      uint8_t* st = smem + s * C::STAGE;
      const bool far = JOB == JOB_NEAR && kc == nk - 1;
#pragma unroll
      for (int q = 0; q < CHUNKS; ++q) {
        const int k8 = cbase + q;              // 16-byte chunk of the 64-byte row
        float v[8];
        const int m0 = chunk_of(kc) * BK + k8 * 8;
        if (far) {
          // sigma_n u_i(t_n), i = 8 k8 .. + 7, at t_n relative to the block's centre
          if (k8 >= kFarP / 8) continue;       // the MMA reads 16 columns of this chunk
          float T[kFarP];
          far_polys(((float)(mn - blk * kFarBlock) - 127.5f + en) * (1.f / kTgtHalf), T);
          const float sc = sg * loc_inv;
#pragma unroll
          for (int i = 0; i < 8; ++i) v[i] = sc * far_basis(s_far, k8 * 8 + i, T);
        } else if (JOB == JOB_FAR) {
          // 1 / (tau_i - s_j) of blocks b (the row's) and B = m0 / 16, times 2^8
          const int db = mn - m0 / kFarP;
          const float c = exact_i2f(db * kFarBlock) + en;
          const bool live = db < -a.near || db > a.near;
#pragma unroll
          for (int i = 0; i < 8; ++i)
            v[i] = live ? fast_div(kCauchyScale, c - s_far[(m0 + i) % kFarP]) : 0.f;
        } else {
        // (m_n - m) + e_n with the integer part formed exactly first
        // ((m_n - m0) - i, integers below 2^22) and e_n added last, so the
        // denominator near m = m_n is e_n itself even when e_n is far below
        // the rounding unit of m_n - m0
        // (samples past n_in are zero in X: their weights only need to be finite)
        const float di0 = exact_i2f(mn - m0);
        if (en != 0.f) {
#pragma unroll
          for (int i = 0; i < 8; ++i) v[i] = fast_div((i & 1) ? -sg : sg, (di0 - (float)i) + en);
        } else {
#pragma unroll
          for (int i = 0; i < 8; ++i) v[i] = m0 + i == mn ? 1.f : 0.f;
        }
        }
        // (-1)^m: m = kc*32 + k8*8 + i has the parity of i
        uint4 hi, lo;
        split8<FP16>(v, hi, lo);
        const int off = r * 64 + ((k8 ^ ((r >> 1) & 3)) << 4);
        if (DC_IN_BOUNDS((C::MH + h) * kAPlane + off + 16 <= C::A_BYTES && off + 16 <= kAPlane, a.err)) {
          *reinterpret_cast<uint4*>(st + h * kAPlane + off) = hi;
          *reinterpret_cast<uint4*>(st + (C::MH + h) * kAPlane + off) = lo;
        }
      }
      async_proxy_fence();                     // our generic-proxy writes -> async proxy
      __syncwarp();
      if (lane == 0) bar_arrive(&full_bar[s]);
    }
    // ----------------------------------------------------------- epilogue
    if (warp < 2 + 4 * C::MH) {
      const int q = warp & 3;                   // TMEM lanes 32q .. 32q+31
      const int hh = (warp - 2) >> 2;           // accumulator half
      const bool ready = mbar_wait_bounded(&acc_bar, 0, a.err);
      tc_fence_after();
      const int n = n0 + hh * kHalfRows + 32 * q + lane;
      if (ready) {
        for (int cc = 0; cc < BN / 16; ++cc) {
          float f[16];
          const uint32_t taddr = tmem + hh * 256 + ((uint32_t)(32 * q) << 16) + cc * 16;
          tmem_ld16(taddr, f);
          if constexpr (FP16) {
            float g[16];
            tmem_ld16(taddr + 256, g);
#pragma unroll
            for (int i = 0; i < 16; ++i) f[i] = fmaf(g[i], 1.0f / 2048.f, f[i]);
          }
          if (JOB == JOB_FAR) {
            if (n < a.n_out) {
#pragma unroll
              for (int i = 0; i < 16; ++i) {
                const int col = c0 + cc * 16 + i;
                if (col >= 2 * a.n_pulses) break;
                uint16_t hi, lo;
                split1<FP16>(f[i] * (loc / (kMomScale * kCauchyScale)), hi, lo);
                const size_t o = ((size_t)alpha * 2 * a.n_pulses + col) * a.n_out + n;
                a.loc_hi[o] = hi;
                a.loc_lo[o] = lo;
              }
            }
          } else if (n < a.n_out) {
#pragma unroll
            for (int i = 0; i < 8; ++i) {
              const int pulse = (c0 + cc * 16) / 2 + i;
              if (pulse < a.n_pulses)
                a.y[((size_t)alpha * a.n_pulses + pulse) * a.n_out + n] = make_float2(f[2 * i], f[2 * i + 1]);
            }
          }
        }
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kCols));
  }
}

// X (complex64, pulses of n samples) -> hi / lo 16-bit planes, row 2p = re,
// row 2p + 1 = im, samples contiguous with row stride `ld` (lo scaled by 2^11
// for fp16).
template <bool FP16>
__global__ void split_planes_kernel(const float2* __restrict__ x, int n, long long rows_c, int ld,
                                    uint16_t* hi, uint16_t* lo) {
  const long long total = rows_c * n;
  for (long long g = blockIdx.x * (long long)blockDim.x + threadIdx.x; g < total;
       g += (long long)gridDim.x * blockDim.x) {
    const long long pr = g / n;
    const int m = (int)(g - pr * n);
    const float2 v = x[g];
    const float vv[2] = {v.x, v.y};
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      uint16_t h, l;
      split1<FP16>(vv[c], h, l);
      const long long o = (2 * pr + c) * (long long)ld + m;
      hi[o] = h;
      lo[o] = l;
    }
  }
}

// The planes as split_planes_kernel writes them, and the block moments
// M_B[j] = sum_m l_j(m) (-1)^m x[m] of the values the planes hold, in FP32,
// written as planes too (row 2p / 2p + 1, element 16 B + j, times kMomScale).
// One warp per two consecutive blocks of a pulse (far_moments).
constexpr int kFsWarps = 8;
template <bool FP16>
__global__ void __launch_bounds__(32 * kFsWarps, 2)
    far_split_kernel(const float2* __restrict__ x, int n, long long rows_c, int ld, uint16_t* hi,
                     uint16_t* lo, int ld_mom, uint16_t* mom_hi, uint16_t* mom_lo, float* peak) {
  __shared__ float s_w[kFarP * kFarBlock];             // l_j(m) (-1)^m kMomScale at [j][m]
  __shared__ float s_D[kFarP * kFarP];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  far_fill_table(s_D, threadIdx.x, blockDim.x);
  __syncthreads();
  static_assert(32 * kFsWarps == kFarBlock, "one thread per sample of a block");
  far_fill_weights(s_w, s_D, threadIdx.x, kMomScale);
  __syncthreads();
  const int nb = (n + kFarBlock - 1) / kFarBlock;
  const int n_pair = (nb + 1) / 2;                     // block pairs of a pulse
  const long long total = rows_c * n_pair;
  for (long long g = blockIdx.x * (long long)kFsWarps + warp; g < total;
       g += (long long)gridDim.x * kFsWarps) {
    const long long pr = g / n_pair;
    const int m0 = (int)(g - pr * n_pair) * 2 * kFarBlock + 2 * lane;
    const float2* xp = x + pr * n;
    float2 v[2][4][2];
    const bool al = (reinterpret_cast<uintptr_t>(xp) & 15) == 0;   // m0 is even
#pragma unroll
    for (int b = 0; b < 2; ++b)
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int m = m0 + b * kFarBlock + 64 * q;
        v[b][q][0] = v[b][q][1] = make_float2(0.f, 0.f);
        if (al && m + 1 < n) {
          const float4 t = __ldcs(reinterpret_cast<const float4*>(xp + m));
          v[b][q][0] = make_float2(t.x, t.y);
          v[b][q][1] = make_float2(t.z, t.w);
        } else {
          if (m < n) v[b][q][0] = __ldcs(xp + m);
          if (m + 1 < n) v[b][q][1] = __ldcs(xp + m + 1);
        }
      }
    if constexpr (FP16) {                              // g = pr * n_pair + pair
      uint32_t top = 0;
#pragma unroll
      for (int b = 0; b < 2; ++b)
#pragma unroll
        for (int q = 0; q < 4; ++q)
#pragma unroll
          for (int i = 0; i < 2; ++i)
            top = max(top, max(__float_as_uint(v[b][q][i].x) & 0x7fffffffu, __float_as_uint(v[b][q][i].y) & 0x7fffffffu));
      top = __reduce_max_sync(0xffffffffu, top);
      if (lane == 0) peak[g] = __uint_as_float(top);
    }
#pragma unroll
    for (int b = 0; b < 2; ++b)
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int m = m0 + b * kFarBlock + 64 * q;
        uint16_t h[2][2], l[2][2];                     // [re, im][sample]
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          split1<FP16>(v[b][q][i].x, h[0][i], l[0][i]);
          split1<FP16>(v[b][q][i].y, h[1][i], l[1][i]);
          v[b][q][i] = make_float2(join1<FP16>(h[0][i], l[0][i]), join1<FP16>(h[1][i], l[1][i]));
        }
        if (m < n) {                                   // m + 1 < ld: the row pitch is even
#pragma unroll
          for (int c = 0; c < 2; ++c) {
            const long long o = (2 * pr + c) * (long long)ld + m;
            *reinterpret_cast<uint32_t*>(hi + o) = h[c][0] | ((uint32_t)h[c][1] << 16);
            *reinterpret_cast<uint32_t*>(lo + o) = l[c][0] | ((uint32_t)l[c][1] << 16);
          }
        }
      }
    float2 mom;
    far_moments(s_w, lane, v, mom);
    const float acc[2] = {mom.x, mom.y};
    const int e = (m0 - 2 * lane) / kFarBlock * kFarP + lane;   // node lane % 16 of block lane / 16
    if (e < nb * kFarP) {
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        uint16_t h, l;
        split1<FP16>(acc[c], h, l);
        const long long o = (2 * pr + c) * (long long)ld_mom + e;
        mom_hi[o] = h;
        mom_lo[o] = l;
      }
    }
  }
}

PFN_cuTensorMapEncodeTiled_v12000 encode_fn() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  if (!fn) {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
            cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
  }
  return fn;
}

bool make_map(CUtensorMap* m, void* base, bool fp16, long long rows, int n, int ld) {
  auto fn = encode_fn();
  if (!fn) return false;
  cuuint64_t dims[2] = {(cuuint64_t)n, (cuuint64_t)rows};
  cuuint64_t strides[1] = {(cuuint64_t)ld * 2};
  cuuint32_t box[2] = {BK, BN};      // 32 x 16-bit = 64 bytes inner: 64-byte swizzle
  cuuint32_t estr[2] = {1, 1};
  CUresult r = fn(m, fp16 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT16 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, base,
                  dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_64B,
                  CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS;
}

}  // namespace

namespace {

template <bool FP16, int JOB>
cudaError_t launch_tiles(const CUtensorMap& mh, const CUtensorMap& ml, const CUtensorMap& fh,
                         const CUtensorMap& fl, const ExTcArgs& args, int n_alpha, cudaStream_t s) {
  using C = Cfg<FP16>;
  dim3 grid((args.n_out + C::BM - 1) / C::BM, (2 * args.n_pulses + BN - 1) / BN, n_alpha);
  auto k = exact_tc_kernel<FP16, JOB>;
  cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, C::SMEM);
  if (e != cudaSuccess) return e;
  k<<<grid, kThreads, C::SMEM, s>>>(mh, ml, fh, fl, args);
  return cudaGetLastError();
}

template <bool FP16>
cudaError_t run_exact_tc(const float2* x, long long x_rows_c, int n, const ExTcPlanes& pl,
                         const ExTcArgs& args, int n_alpha, cudaStream_t s) {
  const int ld = (n + 7) / 8 * 8;
  CUtensorMap mh, ml;
  if (!make_map(&mh, pl.hi, FP16, 2 * x_rows_c, n, ld) || !make_map(&ml, pl.lo, FP16, 2 * x_rows_c, n, ld))
    return cudaErrorInvalidValue;
  if (!pl.far) {
    const long long total = x_rows_c * n;
    const int grid_c = (int)std::min<long long>((total + 255) / 256, 152LL * 32);
    split_planes_kernel<FP16><<<grid_c, 256, 0, s>>>(x, n, x_rows_c, ld, (uint16_t*)pl.hi, (uint16_t*)pl.lo);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    return launch_tiles<FP16, JOB_DENSE>(mh, ml, mh, ml, args, n_alpha, s);
  }
  // moments of the pulses' blocks, node values of the outputs' blocks
  const int kb = kFarP * far_blocks(n), ob = kFarP * far_blocks(args.n_out);
  CUtensorMap qh, ql, fh, fl;
  if (!make_map(&qh, pl.mom_hi, FP16, 2 * x_rows_c, kb, kb) || !make_map(&ql, pl.mom_lo, FP16, 2 * x_rows_c, kb, kb) ||
      !make_map(&fh, pl.loc_hi, FP16, 2 * x_rows_c, ob, ob) || !make_map(&fl, pl.loc_lo, FP16, 2 * x_rows_c, ob, ob))
    return cudaErrorInvalidValue;
  const long long pairs = x_rows_c * ((far_blocks(n) + 1) / 2);
  const int grid_c = (int)std::min<long long>((pairs + kFsWarps - 1) / kFsWarps, 152LL * 2);
  far_split_kernel<FP16><<<grid_c, 32 * kFsWarps, 0, s>>>(x, n, x_rows_c, ld, (uint16_t*)pl.hi, (uint16_t*)pl.lo, kb,
                                                          (uint16_t*)pl.mom_hi, (uint16_t*)pl.mom_lo, (float*)pl.peak);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  ExTcArgs g = args;
  g.near = !FP16 && n > kFarWideIn ? 3 : 1;
  g.own_first = g.near > 1;
  g.peak = (const float*)pl.peak;
  g.n_peaks = (far_blocks(n) + 1) / 2;
  g.loc_inv = (float*)pl.peak + x_rows_c * g.n_peaks;
  ExTcArgs f = g;
  f.n_in = kb;
  f.n_out = ob;
  f.loc_hi = (uint16_t*)pl.loc_hi;
  f.loc_lo = (uint16_t*)pl.loc_lo;
  // the node values depend on the pulses only: one set per group of pulses
  if ((e = launch_tiles<FP16, JOB_FAR>(qh, ql, qh, ql, f, args.rows_per_alpha ? n_alpha : 1, s))) return e;
  return launch_tiles<FP16, JOB_NEAR>(mh, ml, fh, fl, g, n_alpha, s);
}

}  // namespace

size_t exact_tc_plane_bytes(long long rows, int n) {
  const long long ld = (n + 7) / 8 * 8;
  return (size_t)rows * ld * 2;
}

// The near and far form replaces n_in / 32 chunks by at most 25 (bf16x3 above
// 4096: 57) and adds two launches.  Measured, far against dense, in us (8 pulses x 1
// rate, 64 x 4, 512 x 1): bf16x3: n = 1025: 43 / 39, 50 / 41, 56 / 43; 1536: 43 / 51,
// 49 / 54, 55 / 57; 2048: 45 / 63, 49 / 68, 57 / 70; 4097: 75 / 114, 83 / 121, 91 /
// 126; 8192 at 512 x 16: 1023 / 3383.  fp16x3: 1536: 35 / 34, 38 /
// 37, 44 / 42; 2048: 35 / 43, 40 / 47, 46 / 49; 8192: 41 / 133, 69 / 275, 85 / 285.
bool exact_tc_far(bool fp16, int n_in, int n_out, double delta_max) {
  return n_in >= (fp16 ? kFarMinInFp16 : kFarMinIn) && delta_max * (double)n_out <= (double)(kFarMargin - 1);
}
size_t exact_tc_far_plane_bytes(long long rows, int n) {
  return (size_t)rows * kFarP * far_blocks(n) * 2;
}

size_t exact_tc_peak_bytes(bool fp16, long long groups, int n_pulses, int n) {
  const size_t tiles = (2 * (size_t)n_pulses + BN - 1) / BN;
  return fp16 ? (size_t)groups * (n_pulses * (size_t)((far_blocks(n) + 1) / 2) + tiles) * sizeof(float) : 0;
}

cudaError_t launch_exact_tc(bool fp16, const float2* x, long long x_rows_c, int n, const ExTcPlanes& pl,
                            const ExTcArgs& args, int n_alpha, cudaStream_t s) {
  return fp16 ? run_exact_tc<true>(x, x_rows_c, n, pl, args, n_alpha, s)
              : run_exact_tc<false>(x, x_rows_c, n, pl, args, n_alpha, s);
}

}  // namespace dc
