// FFT passes with the fused ionospheric phase multiply.
// Index conventions and the four-step split are described in fft.cuh.
#include <algorithm>

#include "fft.cuh"
#include "fused.cuh"
#include "rows.cuh"

namespace dc {

constexpr int kThreads = 256;

// Twiddles w^1 .. w^15 of a thread from table rows of PITCH entries, and v[q] *= w^q (its
// conjugate for DIR > 0): table values, each rounded once, in rows that a warp reads
// consecutively.  Products of four powers of two instead, gathered from the 4096-point
// table, round up to three times more (2048 points: 2.93e-7 from 64 bits, now 2.60e-7) and
// gained nothing: plans of 10000 pulses of 300 samples 43.5 us, now 41.4, 4000 of 2000:
// 82.6, 79.9, a lone pulse 8 us either way.
template <int PITCH> DC_DEV void load_powers(float2 (&w)[16], const float2* __restrict__ row) {
#pragma unroll
  for (int q = 1; q < 16; ++q) w[q] = __ldg(row + (q - 1) * PITCH);
}
template <int DIR> DC_DEV void mul_powers(float2 (&v)[16], const float2 (&w)[16]) {
#pragma unroll
  for (int q = 1; q < 16; ++q) v[q] = cmul(v[q], conj_if<DIR>(w[q]));
}

// Transforms of M = 16 R points, R = 2, 4 or 8, in registers: R threads of 16
// points per transform, which exchange once in each direction behind a warp
// barrier.  The split n = R p + t, k = s + 16 a (p, s < 16; t, a < R): DFT over p in
// thread t, W_M^(t s); exchange; DFT over t (16 / R of them, s = t + R i, in each
// thread); the inverse mirrored.  Point t of sub-problem s of transform q lies at
// (t * 16 + s) * pitch + q.  With M <= 16 (R = 1) a thread holds a transform whole.
// Latency bounds a few transforms, the accesses of 64 (R = 8) to 8 bytes many.  Radix-16
// stages through shared memory, with two CTA barriers and table loads per element
// each, took 8.2 us for a pulse of 128 (now 4.5), 6.2 for one of 16 (2.3), 52 for
// 20000 transforms of 128 (22).
template <int M, int OP>
DC_DEV void tiny_pass(float2* sm, const FftItem* items, const FftItem& one, int n_items, int block,
                      const float2* __restrict__ tw) {
  constexpr int R = M > 16 ? M / 16 : 1, N = M > 16 ? 16 : M;      // threads, points of each
  constexpr int NT = kThreads / R, PITCH = NT + 16 / R, NI = 16 / R;
  const int q = threadIdx.x / R, t = threadIdx.x % R;
  const int g = block * NT + q;
  const bool live = g < n_items;
  const FftItem I = items ? ldg_item(items + (live ? g : 0)) : one;
  float2 wt[16];                                // W_M^(t s)
  if constexpr (R > 1) load_powers<R>(wt, tw + kTwSub(R) + t);
  pdl_wait();                                   // the input's producer has finished
  float2 v[N];
  // v[i R + a] = bin t + R i + 16 a once the forward transform is done
  auto bin = [&](int x) { return R > 1 ? t + R * (x / R) + 16 * (x % R) : x; };
  if constexpr (OP == ROW_APPLY) {
#pragma unroll
    for (int x = 0; x < N; ++x) v[x] = live ? I.src[bin(x)] : make_float2(0.f, 0.f);
  } else {
#pragma unroll
    for (int p = 0; p < N; ++p) v[p] = live && R * p + t < I.n_valid ? I.src[R * p + t] : make_float2(0.f, 0.f);
    dft<N, -1>(v);                              // over p
    if constexpr (R > 1) {
      mul_powers<-1>(v, wt);
#pragma unroll
      for (int s = 0; s < 16; ++s) sm[(t * 16 + s) * PITCH + q] = v[s];
      __syncwarp();
#pragma unroll
      for (int i = 0; i < NI; ++i) {
        float2 u[R];
#pragma unroll
        for (int k = 0; k < R; ++k) u[k] = sm[(k * 16 + t + R * i) * PITCH + q];
        dft<R, -1>(u);                          // over t
#pragma unroll
        for (int k = 0; k < R; ++k) v[i * R + k] = u[k];
      }
    }
  }
  if constexpr (OP == ROW_SPEC) {
    if (live) {
#pragma unroll
      for (int x = 0; x < N; ++x) I.dst[bin(x)] = v[x];
    }
    return;
  }
  if (OP == ROW_APPLY || I.ptab) {
#pragma unroll
    for (int x = 0; x < N; ++x) v[x] = cmul(v[x], I.ptab[bin(x)]);
  } else if (I.ph.enabled) {
#pragma unroll
    for (int x = 0; x < N; ++x) v[x] = cmul(v[x], iono_factor(I.ph, bin(x)));
  }
  if constexpr (R > 1) {
    __syncwarp();                               // the forward transform's reads
#pragma unroll
    for (int i = 0; i < NI; ++i) {
      float2 u[R];
#pragma unroll
      for (int k = 0; k < R; ++k) u[k] = v[i * R + k];
      dft<R, +1>(u);                            // over a
#pragma unroll
      for (int k = 0; k < R; ++k) sm[(k * 16 + t + R * i) * PITCH + q] = u[k];
    }
    __syncwarp();
#pragma unroll
    for (int s = 0; s < 16; ++s) v[s] = sm[(t * 16 + s) * PITCH + q];
    mul_powers<+1>(v, wt);
  }
  dft<N, +1>(v);                                // over s
  if (live) {
#pragma unroll
    for (int p = 0; p < N; ++p)
      if (R * p + t < I.n_out) __stcs(I.dst + R * p + t, cscale(v[p], 1.0f / (float)M));
  }
}

// Transforms of M = 256 A points, A = 1 .. 8, in registers: 16 A threads of 16 points
// per transform, 16 / A transforms per CTA, one barrier in each direction (the
// 4096-point rows of rows.cuh are A = 16).  The split n = 16 A p + 16 u + w, k =
// s + 16 a + 16 A r (u, a < A; p, w, s, r < 16), thread (s, t) of 16 x A:
//   forward  DFT over p in thread q = 16 u + w, W_M^(q s); exchange; DFT over u (16 / A
//            of them, w = t + A i); transpose among the A threads of sub-problem s;
//            W_16A^(w a) in thread a = t; DFT over w
//   inverse  the mirror image
// Sub-problem s keeps to its own 17 A elements except in the exchange, whose pitch
// 17 A puts a half-warp's accesses on 16 different bank pairs throughout.  Against
// radix-16 stages through shared memory with two barriers each and table loads per
// element a lone pulse of 2048 takes 6.2 instead of 12.3 us.
template <int A, int OP>
DC_DEV void line_pass(float2* sm, const FftItem* items, const FftItem& one, int n_items, int block,
                      const float2* __restrict__ tw) {
  constexpr int M = 256 * A, T = 16 * A, P = 17 * A, NI = 16 / A;
  const int tl = threadIdx.x % T, s = tl / A, t = tl % A;
  const int g = block * NI + threadIdx.x / T;
  const bool live = g < n_items;
  const FftItem I = items ? ldg_item(items + (live ? g : 0)) : one;
  float2* b = sm + (threadIdx.x / T) * 16 * P;
  float2* reg = b + s * P;
  float2 wq[16], wt[16];                        // W_M^(q r), q = tl, and W_16A^(t w)
  load_powers<T>(wq, tw + kTwLine(A) + tl);
  if constexpr (A > 1) load_powers<A>(wt, tw + kTwSub(A) + t);
  pdl_wait();                                   // the input's producer has finished
  float2 v[16];
  if constexpr (OP == ROW_APPLY) {
#pragma unroll
    for (int r = 0; r < 16; ++r) v[r] = live ? I.src[s + 16 * t + T * r] : make_float2(0.f, 0.f);
  } else {
#pragma unroll
    for (int p = 0; p < 16; ++p) {
      const int n = T * p + tl;
      v[p] = live && n < I.n_valid ? I.src[n] : make_float2(0.f, 0.f);
    }
    dft16<-1>(v);                               // over p
    mul_powers<-1>(v, wq);
#pragma unroll
    for (int r = 0; r < 16; ++r) b[r * P + tl] = v[r];
    __syncthreads();
#pragma unroll
    for (int i = 0; i < NI; ++i) {
      float2 u[A];
#pragma unroll
      for (int k = 0; k < A; ++k) u[k] = reg[16 * k + t + A * i];
      dft<A, -1>(u);                            // over u
#pragma unroll
      for (int k = 0; k < A; ++k) v[i * A + k] = u[k];
    }
    __syncwarp();
#pragma unroll
    for (int i = 0; i < NI; ++i)
#pragma unroll
      for (int k = 0; k < A; ++k) reg[17 * k + t + A * i] = v[i * A + k];
    __syncwarp();
#pragma unroll
    for (int w = 0; w < 16; ++w) v[w] = reg[17 * t + w];
    if constexpr (A > 1) mul_powers<-1>(v, wt);
    dft16<-1>(v);                               // over w: v[r] = X[s + 16 t + T r]
  }
  if constexpr (OP == ROW_SPEC) {
    if (live) {
#pragma unroll
      for (int r = 0; r < 16; ++r) I.dst[s + 16 * t + T * r] = v[r];
    }
    return;
  }
  if (OP == ROW_APPLY || I.ptab) {
#pragma unroll
    for (int r = 0; r < 16; ++r) v[r] = cmul(v[r], I.ptab[s + 16 * t + T * r]);
  } else if (I.ph.enabled) {
#pragma unroll
    for (int r = 0; r < 16; ++r)
      v[r] = cmul(v[r], iono_factor_full(I.ph, (float)(s + 16 * t + T * (r < 8 ? r : r - 16))));
  }
  dft16<+1>(v);                                 // over r
  if constexpr (A > 1) mul_powers<+1>(v, wt);
  __syncwarp();
#pragma unroll
  for (int w = 0; w < 16; ++w) reg[17 * t + w] = v[w];
  __syncwarp();
#pragma unroll
  for (int i = 0; i < NI; ++i) {
    float2 u[A];
#pragma unroll
    for (int k = 0; k < A; ++k) u[k] = reg[17 * k + t + A * i];
    dft<A, +1>(u);                              // over a
#pragma unroll
    for (int k = 0; k < A; ++k) v[i * A + k] = u[k];
  }
  __syncwarp();
#pragma unroll
  for (int i = 0; i < NI; ++i)
#pragma unroll
    for (int k = 0; k < A; ++k) reg[16 * k + t + A * i] = v[i * A + k];
  __syncthreads();
#pragma unroll
  for (int r = 0; r < 16; ++r) v[r] = b[r * P + tl];
  mul_powers<+1>(v, wq);
  dft16<+1>(v);                                 // over s
  if (live) {
#pragma unroll
    for (int p = 0; p < 16; ++p)
      if (T * p + tl < I.n_out) __stcs(I.dst + T * p + tl, cscale(v[p], 1.0f / (float)M));
  }
}

// The pass of CTA `block` for transforms of M points, its transforms per CTA and shared memory.
template <int M, int OP>
DC_DEV void short_pass(float2* sm, const FftItem* items, const FftItem& one, int n_items, int block, const float2* tw) {
  if constexpr (M == 4096) full_4096(items ? ldg_item(items + block) : one, sm, threadIdx.x, tw);
  else if constexpr (M >= 256) line_pass<M / 256, OP>(sm, items, one, n_items, block, tw);
  else tiny_pass<M, OP>(sm, items, one, n_items, block, tw);
}
constexpr int short_lines(int M) { return M <= 16 ? kThreads : 4096 / M; }
constexpr size_t short_smem(int M) { return M <= 16 ? 0 : sizeof(float2) * kRowPitch; }

template <int M, int OP>
__global__ void __launch_bounds__(kThreads) row_kernel(RowArgs a) {
  extern __shared__ float2 sm[];
  short_pass<M, OP>(sm, a.items, a.one, a.n_items, blockIdx.x, a.tw);
}

// Short transforms of several length classes in one launch: run one after the
// other, the classes of a small batch leave the chip idle (each is one latency
// chain on a few CTAs).  Launched programmatically: successive calls, and the
// resampling before it, overlap its set-up (iono_correct of 256 to 2048 samples,
// calls back to back: 6.2 -> 4.5 us).
template <int M>
DC_DEV void class_pass(float2* sm, const RowClasses& a, int m) {
  short_pass<M, ROW_FULL>(sm, a.items ? a.items + a.first[m] : nullptr, a.one, a.first[m + 1] - a.first[m],
                        blockIdx.x - a.block[m], a.tw);
}
__global__ void __launch_bounds__(kThreads, 2) row_classes_kernel(const __grid_constant__ RowClasses a) {
  extern __shared__ float2 sm[];
  int m = 0;
  while (m < 12 && (int)blockIdx.x >= a.block[m + 1]) ++m;
  switch (m) {
    case 0: class_pass<1>(sm, a, m); break;
    case 1: class_pass<2>(sm, a, m); break;
    case 2: class_pass<4>(sm, a, m); break;
    case 3: class_pass<8>(sm, a, m); break;
    case 4: class_pass<16>(sm, a, m); break;
    case 5: class_pass<32>(sm, a, m); break;
    case 6: class_pass<64>(sm, a, m); break;
    case 7: class_pass<128>(sm, a, m); break;
    case 8: class_pass<256>(sm, a, m); break;
    case 9: class_pass<512>(sm, a, m); break;
    case 10: class_pass<1024>(sm, a, m); break;
    case 11: class_pass<2048>(sm, a, m); break;
    default: class_pass<4096>(sm, a, m);
  }
}

// ------------------------------------------------------------ column pass
// Column pass for M = L1 in [32, 256]: M = 16 x R, R = M / 16.  A CTA takes C =
// 4096 / M columns (32 KiB of shared memory for every M); consecutive threads take
// consecutive columns, so global rows of C complex are read and written whole.
// Thread (column c, p0 < R) loads rows p0 + R q straight into the radix-16
// butterfly they form, exchanges once through shared memory (element p of column
// c at sm[p*C + c]) and runs 16 / R butterflies of radix R, whose outputs again
// are rows p0 + R i: four trips through the load/store path per element, which
// bounds this pass (with both stages and the transfers through shared memory it
// took eight, at 85 % of that path: 128 pulses of 2^18, forward 106 us, inverse 79).
// Four CTAs per SM: the forward pass at its own 74 registers, three, waited for its
// loads (a batch's forward passes 538 us, now 519).
template <int M, int OP>
__global__ void __launch_bounds__(kThreads, 4) col_kernel_smem(ColArgs a) {
  constexpr int C = 4096 / M, R = M / 16, NB = 16 / R;
  __shared__ float2 sm[4096];
  const int L2 = 1 << (a.log2L - a.log2L1);
  const int cta_per_item = L2 / C;
  const int it = blockIdx.x / cta_per_item;
  const int col0 = (blockIdx.x % cta_per_item) * C;
  const FftItem I = item_of(a, it);
  constexpr int DIR = OP == COL_F1 ? -1 : +1;
  const int c = threadIdx.x % C, p0 = threadIdx.x / C;
  const int n2 = col0 + c;
  pdl_release();
  pdl_wait();                                  // plain loads below: they stay behind it
  float2 v[16];
#pragma unroll
  for (int q = 0; q < 16; ++q) {
    const int p = p0 + R * q;
    if (OP == COL_F1) {
      const int n = n2 + L2 * p;
      v[q] = n < I.n_valid ? I.src[n] : make_float2(0.f, 0.f);
    } else {
      v[q] = I.src[(size_t)p * L2 + n2];
    }
  }
  dft16<DIR>(v);
#pragma unroll
  for (int r = 0; r < 16; ++r) sm[(16 * p0 + r) * C + c] = v[r];
  __syncthreads();
#pragma unroll
  for (int q = 0; q < NB; ++q) {
    const int k = p0 + R * q;                  // butterfly k: rows k + 16 r
    float2 u[R];
#pragma unroll
    for (int r = 0; r < R; ++r) u[r] = sm[(k + 16 * r) * C + c];
#pragma unroll
    for (int r = 1; r < R; ++r) u[r] = cmul(u[r], tw_m<DIR>(a.tw, r * k * (4096 / M)));
    dft<R, DIR>(u);
#pragma unroll
    for (int r = 0; r < R; ++r) v[q + NB * r] = u[r];   // row k + 16 r = p0 + R (q + NB r)
  }
  if (OP == COL_F1) {
    // twiddle W_L^(n2 k1), k1 = p0 + R i: W_L^(n2 p0) times the i-th power of
    // W_L^(n2 R) (powers from the table values for 1, 2, 4, 8)
    const uint32_t mask = (1u << a.log2L) - 1;
    float2 b[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) b[i] = tw_big<-1>(a.tw, (uint32_t)(n2 * (R << i)) & mask, a.log2L);
    apply_powers_from(v, tw_big<-1>(a.tw, (uint32_t)(n2 * p0) & mask, a.log2L), b);
#pragma unroll
    for (int i = 0; i < 16; ++i) I.dst[(size_t)(p0 + R * i) * L2 + n2] = v[i];
  } else {
    const float invL = 1.0f / (float)(1 << a.log2L);
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      const int n = n2 + L2 * (p0 + R * i);
      if (n < I.n_out) __stcs(I.dst + n, cscale(v[i], invL));
    }
  }
}

// Column pass for M = L1 in [2, 16]: one column per thread, all in registers.
template <int M, int OP>
__global__ void __launch_bounds__(kThreads) col_kernel_reg(ColArgs a) {
  const int L2 = 1 << (a.log2L - a.log2L1);
  const int cta_per_item = L2 / kThreads;
  const int it = blockIdx.x / cta_per_item;
  const int n2 = (blockIdx.x % cta_per_item) * kThreads + threadIdx.x;
  const FftItem I = item_of(a, it);
  float2 v[M];
#pragma unroll
  for (int p = 0; p < M; ++p) {
    if (OP == COL_F1) {
      const int n = n2 + L2 * p;
      v[p] = n < I.n_valid ? I.src[n] : make_float2(0.f, 0.f);
    } else {
      v[p] = I.src[(size_t)p * L2 + n2];
    }
  }
  dft<M, OP == COL_F1 ? -1 : +1>(v);
  if (OP == COL_F1) {
#pragma unroll
    for (int p = 0; p < M; ++p)
      I.dst[(size_t)p * L2 + n2] =
          cmul(v[p], tw_big<-1>(a.tw, (uint32_t)(n2 * p) & ((1u << a.log2L) - 1), a.log2L));
  } else {
    const float invL = 1.0f / (float)(1 << a.log2L);
#pragma unroll
    for (int p = 0; p < M; ++p) {
      const int n = n2 + L2 * p;
      if (n < I.n_out) __stcs(I.dst + n, cscale(v[p], invL));
    }
  }
}

// ---------------------------------------------------------------- launchers
template <int M, int OP>
static cudaError_t launch_row_m(const RowArgs& a, cudaStream_t s) {
  const long long grid = ((long long)a.n_items + short_lines(M) - 1) / short_lines(M);
  if (grid <= 0) return cudaSuccess;
  row_kernel<M, OP><<<(unsigned)grid, kThreads, short_smem(M), s>>>(a);
  return cudaGetLastError();
}

template <int OP>
static cudaError_t launch_row_op(const RowArgs& a, cudaStream_t s) {
  const int m = a.log2L - a.log2L1;   // row length log2
  switch (m) {
    case 0: return launch_row_m<1, OP>(a, s);
    case 1: return launch_row_m<2, OP>(a, s);
    case 2: return launch_row_m<4, OP>(a, s);
    case 3: return launch_row_m<8, OP>(a, s);
    case 4: return launch_row_m<16, OP>(a, s);
    case 5: return launch_row_m<32, OP>(a, s);
    case 6: return launch_row_m<64, OP>(a, s);
    case 7: return launch_row_m<128, OP>(a, s);
    case 8: return launch_row_m<256, OP>(a, s);
    case 9: return launch_row_m<512, OP>(a, s);
    case 10: return launch_row_m<1024, OP>(a, s);
    case 11: return launch_row_m<2048, OP>(a, s);
    case 12:
      // one-pass rows of L = 4096 here, the four-step rows in fused.cu
      if constexpr (OP == ROW_FULL) return launch_row_m<4096, OP>(a, s);
      else return launch_row_4096(OP, a, s);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t launch_row_classes(RowClasses a, cudaStream_t s) {
  size_t smem = 0;
  a.block[0] = 0;
  for (int m = 0; m <= 12; ++m) {
    const int n = a.first[m + 1] - a.first[m], lines = short_lines(1 << m);
    a.block[m + 1] = a.block[m] + (n + lines - 1) / lines;
    if (n > 0) smem = std::max(smem, short_smem(1 << m));
  }
  if (a.block[13] == 0) return cudaSuccess;
  // launched programmatically behind the resampling (three-pass rules)
  const int pdl = pdl_for(a.block[13]);
  if (pdl == PDL_SPREAD) {
    smem = kPdlRowSmem;
    cudaError_t e = cudaFuncSetAttribute(row_classes_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)a.block[13]);
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = pdl ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, row_classes_kernel, a);
}

cudaError_t launch_row(int op, const RowArgs& a, cudaStream_t s) {
  switch (op) {
    case ROW_FULL: return launch_row_op<ROW_FULL>(a, s);
    case ROW_MID: return launch_row_4096(op, a, s);
    case ROW_SPEC: return launch_row_op<ROW_SPEC>(a, s);
    case ROW_APPLY: return launch_row_op<ROW_APPLY>(a, s);
    default: return cudaErrorInvalidValue;
  }
}

template <int M, int OP>
static cudaError_t launch_col_m(const ColArgs& a, cudaStream_t s) {
  const int L2 = 1 << (a.log2L - a.log2L1);
  if (a.n_items <= 0) return cudaSuccess;
  if constexpr (M <= 16) {
    const long long grid = (long long)a.n_items * (L2 / kThreads);
    col_kernel_reg<M, OP><<<(unsigned)grid, kThreads, 0, s>>>(a);
  } else {
    const long long grid = (long long)a.n_items * (L2 / (4096 / M));
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3(kThreads);
    cfg.stream = s;
    if (a.pdl == PDL_SPREAD) {
      cfg.dynamicSmemBytes = kPdlColSmem - 4096 * sizeof(float2);
      cudaError_t e = cudaFuncSetAttribute(col_kernel_smem<M, OP>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                           (int)cfg.dynamicSmemBytes);
      if (e != cudaSuccess) return e;
    }
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = a.pdl ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, col_kernel_smem<M, OP>, a);
  }
  return cudaGetLastError();
}

template <int OP>
static cudaError_t launch_col_op(const ColArgs& a, cudaStream_t s) {
  switch (a.log2L1) {
    case 1: return launch_col_m<2, OP>(a, s);
    case 2: return launch_col_m<4, OP>(a, s);
    case 3: return launch_col_m<8, OP>(a, s);
    case 4: return launch_col_m<16, OP>(a, s);
    case 5: return launch_col_m<32, OP>(a, s);
    case 6: return launch_col_m<64, OP>(a, s);
    case 7: return launch_col_m<128, OP>(a, s);
    case 8: return launch_col_m<256, OP>(a, s);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t launch_col(int op, const ColArgs& a, cudaStream_t s) {
  return op == COL_F1 ? launch_col_op<COL_F1>(a, s) : launch_col_op<COL_B>(a, s);
}

}  // namespace dc
