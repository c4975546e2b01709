// Cluster-fused FFT correction kernels; see fused.cuh for the data flow.
#include <algorithm>
#include <cooperative_groups.h>
#include <type_traits>

#include "fused.cuh"
#include "rows.cuh"
#include "tma.cuh"

namespace cg = cooperative_groups;

namespace dc {

namespace {

// Wait half of a split cluster barrier (acquire), after an arrive.release.
template <int CL> DC_DEV void cluster_wait() {
  if constexpr (CL > 1) asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// Transform p of a FUSED_APPLY launch, formed from the grid description.
DC_DEV FftItem apply_item(const FusedArgs& a, int p) {
  FftItem I = {};
  const int i = p / a.grid_n_tec, t = p - i * a.grid_n_tec;
  const size_t L = (size_t)1 << a.log2L;
  I.src = a.grid_src + (size_t)i * L;
  I.ptab = a.grid_ptab + (size_t)t * L;
  I.dst = a.grid_dst + (size_t)p * a.grid_n_out;
  I.n_valid = a.grid_n_out;
  I.n_out = a.grid_n_out;
  return I;
}

// Spectra (FUSED_SPEC): one row k1 of the four-step spectrum per CTA, one
// cluster of L1 CTAs per transform.  Each CTA runs the length-L1 forward
// DFTs of its 4096 / L1 columns straight from global memory, applies
// W_L^(n2 k1) and writes element k1 of column n2 into the shared memory of
// the CTA owning row k1 (plain remote stores between two cluster barriers:
// every peer running before, every column delivered after); the received
// row is transformed in the same buffer.
template <int LOG2L1>
__global__ void __launch_bounds__(kRowThreads, 4) spec_kernel(FusedArgs a) {
  constexpr int L1 = 1 << LOG2L1;
  constexpr int COLS = kRowN / L1;              // columns per CTA
  constexpr int PER = COLS / kRowThreads;       // columns per thread
  extern __shared__ __align__(128) float2 sm[];
  float2* A = sm;                               // [kRowPitch] received row, row FFT buffer
  const int k1 = L1 > 1 ? (int)cg::this_cluster().block_rank() : 0;
  const FftItem I = item_of(a, blockIdx.x >> LOG2L1);
  const int j = threadIdx.x;
  float2 v[16];
  pdl_release();                                // the next pass may start its set-up
  if constexpr (L1 == 1) {
    pdl_wait();                                 // the pulses' producer has finished
#pragma unroll
    for (int r = 0; r < 16; ++r) {
      const int n = j + 256 * r;
      v[r] = n < I.n_valid ? I.src[n] : make_float2(0.f, 0.f);
    }
  } else {
    asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");   // this CTA runs
    const float2* T = a.t4 + kT4Offset(L1);
    pdl_wait();                                 // the pulses' producer has finished
#pragma unroll
    for (int p = 0; p < PER; ++p) {
      const int n2 = k1 * COLS + j + 256 * p;
      float2 col[L1];
#pragma unroll
      for (int n1 = 0; n1 < L1; ++n1) {
        const int n = n2 + kRowN * n1;
        col[n1] = n < I.n_valid ? I.src[n] : make_float2(0.f, 0.f);   // plain: after pdl_wait
      }
      dft<L1, -1>(col);
      float2 w[4];                              // W_L^(2^b n2), conjugates of the table rows
#pragma unroll
      for (int b = 0; b < LOG2L1; ++b) w[b] = conj_if<+1>(__ldg(T + b * kRowN + n2));
      apply_powers<L1>(col, w);
      if (p == 0) cluster_wait<L1>();           // every peer runs: its shared memory exists
      const uint32_t dst = smem_addr(A + pad16(n2));
#pragma unroll
      for (int q = 0; q < L1; ++q) st_cluster_c64(dsmem_map(dst, q), col[q]);
    }
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");   // columns delivered
    cluster_wait<L1>();
#pragma unroll
    for (int r = 0; r < 16; ++r) v[r] = A[pad16(j + 256 * r)];
  }
  row_forward(v, A, j, GlobalTw{a.tw});
  store_bins(I.dst + (size_t)k1 * kRowN, j, v);
}

template <int LOG2L1>
cudaError_t launch_spec(const FusedArgs& a, cudaStream_t s) {
  constexpr int L1 = 1 << LOG2L1;
  if (L1 > 1 && !a.t4) return cudaErrorInvalidValue;
  const size_t smem = sizeof(float2) * kRowPitch;
  auto k = spec_kernel<LOG2L1>;
  cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  if (L1 > 8) {
    e = cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return e;
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(a.n_items * L1));
  cfg.blockDim = dim3(kRowThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = L1;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = a.pdl ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, k, a);
}

// Spectrum apply (FUSED_APPLY): G = 2^LOG2G rows of the transform per CTA
// (256 threads per row), one cluster of CL = L1 / G CTAs per transform.
// Spectrum and factor rows come straight into registers (both stored in the
// inverse row's order); after the inverse row FFTs each thread writes its 16
// outputs X[n2] straight into the shared memory of the CTA that owns column n2
// (plain remote stores, a warp's 32 into one 256-byte block), so no CTA reads
// another's shared memory.  The rows are received into the buffers the row FFTs
// used (one 34 KiB buffer per row, 64 registers: 4 / G CTAs per SM): a first
// cluster barrier after the row FFTs frees every buffer, a second one after the
// stores delivers them.  The owner then applies W_L^(-n2 q) from the table and
// runs its columns.  Two rows per CTA halve the cluster (8 CTAs at L = 65536):
// fewer peers per barrier and exchange, which moves the same bytes faster.
template <int LOG2L1, int LOG2G>
__global__ void __launch_bounds__(kRowThreads << LOG2G, 4 >> LOG2G) apply_kernel(FusedArgs a) {
  constexpr int L1 = 1 << LOG2L1;
  constexpr int G = 1 << LOG2G;                 // rows per CTA
  constexpr int CL = L1 / G;                    // CTAs per transform
  constexpr int NT = kRowThreads * G;
  constexpr int COLS = kRowN / CL;              // columns owned by a CTA
  constexpr int PER = COLS / kRowThreads;       // a row thread's output r goes to CTA r / PER
  constexpr int PERC = COLS / NT;               // columns per thread
  static_assert(G == 1 || CL > 1, "two rows per CTA need a cluster");
  static_assert(G == 1 || L1 * COLS <= G * kRowPitch, "received rows fit the row buffers");
  extern __shared__ __align__(128) float2 sm[];
  float2* R = sm;                               // [L1][COLS] received rows (CL > 1)

  const int rank = CL > 1 ? (int)cg::this_cluster().block_rank() : 0;
  const FftItem I = apply_item(a, blockIdx.x >> (LOG2L1 - LOG2G));
  const int j = threadIdx.x;
  const int h = j / kRowThreads, jj = j % kRowThreads;   // row of the CTA, thread in the row
  const int k1 = rank * G + h;
  float2* A = sm + h * kRowPitch;               // this row's buffer
  float2 v[16];
  pdl_wait();                                   // spectra and factors are written
  load_bins(I.src + (size_t)k1 * kRowN, jj, v);
  mul_bins(I.ptab + (size_t)k1 * kRowN, jj, v);
  row_inverse<(L1 > 1)>(v, A, jj, GlobalTw{a.tw});   // arrives at the cluster barrier

  if constexpr (L1 == 1) {
#pragma unroll
    for (int r = 0; r < 16; ++r) {
      const int n = j + 256 * r;
      if (n < I.n_out) __stcs(I.dst + n, v[r]);
    }
  } else {
    // every peer's row FFTs are done with their buffers (the release arrive
    // is inside the row FFT)
    cluster_wait<L1>();
    const uint32_t r_loc = smem_addr(R + k1 * COLS + jj);
    // the farthest element this thread writes in its owners' buffers
    if (DC_IN_BOUNDS(k1 * COLS + jj + 256 * (PER - 1) < L1 * COLS && 16 / PER <= CL, a.err)) {
#pragma unroll
      for (int r = 0; r < 16; ++r) {
        const int owner = r / PER;              // n2 = jj + 256 r -> owner n2 / COLS
        const uint32_t off = (uint32_t)(256 * (r % PER) * sizeof(float2));
        st_cluster_c64(dsmem_map(r_loc + off, owner), v[r]);
      }
    }
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");   // rows delivered
    const float2* T = a.t4 + kT4Offset(L1);
#pragma unroll
    for (int p = 0; p < PERC; ++p) {
      const int c = j + NT * p;
      const int n2 = rank * COLS + c;
      float2 w[4];
#pragma unroll
      for (int b = 0; b < LOG2L1; ++b) w[b] = __ldg(T + b * kRowN + n2);   // W_L^(-2^b n2)
      if (p == 0) cluster_wait<L1>();           // every peer's stores into R are visible
      float2 col[L1];
#pragma unroll
      for (int q = 0; q < L1; ++q) col[q] = R[q * COLS + c];
      apply_powers<L1>(col, w);
      dft<L1, +1>(col);
#pragma unroll
      for (int n1 = 0; n1 < L1; ++n1) {
        const int n = n2 + kRowN * n1;
        if (n < I.n_out) __stcs(I.dst + n, col[n1]);
      }
    }
  }
}

template <int LOG2L1, int LOG2G>
cudaError_t launch_apply(const FusedArgs& a, cudaStream_t s) {
  constexpr int L1 = 1 << LOG2L1;
  constexpr int G = 1 << LOG2G;
  constexpr int CL = L1 / G;
  if (L1 > 1 && !a.t4) return cudaErrorInvalidValue;
  const size_t smem = sizeof(float2) * kRowPitch * G;
  auto k = apply_kernel<LOG2L1, LOG2G>;
  cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  if (CL > 8) {
    e = cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return e;
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(a.n_items * CL));
  cfg.blockDim = dim3(kRowThreads * G);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = CL;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = a.pdl ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, k, a);
}

// Spectrum apply in two passes through L2 (FUSED_APPLY with a.scratch set):
// no cluster.  A persistent grid takes tasks from one global queue in a
// fixed order.  A row task transforms one 4096-point row of one transform
// (spectrum row times factor row, inverse row) into a scratch slot; a column
// task reads 4096 / L1 columns of one transform back from its slot, applies
// W_L^(-n2 q) and runs the length-L1 inverse columns into the output.  The
// transforms go in chunks of P = a.chunk: the queue alternates the rows of
// chunk i and the columns of chunk i - kApplyLag, and the scratch holds
// (kApplyLag + 2) P transforms (slot = transform mod that), small enough to
// stay in L2 between the passes, so DRAM sees the output once, as with the
// cluster kernel, but no cluster barrier or distributed-shared-memory
// exchange is needed.  A task is counted done by one release reduction
// after a CTA barrier; a column task waits until the L1 rows of its
// transform are counted, a row task until the columns of the slot's
// previous transform are (one thread polls with acquire loads, the others
// wait at a CTA barrier).  The lag keeps both waits on
// tasks queued several blocks earlier (a grid holds about 2.4 blocks of
// tasks at once), so they rarely wait at all.  Every wait is on tasks taken
// from the queue earlier, by CTAs already running, so the order cannot
// deadlock; each wait is bounded (error flag 1 when it runs out, and the
// task goes on).  Counters (a.ctr: queue head, then rows done and columns
// done per transform) start at zero.
constexpr int kApplyLag = kApplyL2Slots - 2;

DC_DEV int ld_acquire_gpu(const int* p) {
  int v;
  asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

// Release add: the writes this thread has made or observed (a CTA barrier
// before it covers the whole CTA's) become visible before the count.
DC_DEV void red_release_gpu(int* p, int v) {
  asm volatile("red.release.gpu.global.add.s32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

// Thread 0: poll *p until it reaches `want`, for about a second at most.
DC_DEV void wait_count(const int* p, int want, int* err) {
  for (int i = 0; i < (1 << 24); ++i) {
    if (ld_acquire_gpu(p) >= want) return;
    __nanosleep(64);
  }
  atomicMax(err, 1);
}

// One task of the two-pass apply as thread 0 decodes it for the CTA.
struct ApplyTask {
  const float2* src;    // the transform's spectrum (row tasks)
  const float2* ptab;   // its factor table (row tasks)
  float2* dst;          // its output (column tasks)
  float2* slot;         // its scratch slot
  int n_out;
  int p;                // transform
  int rq;               // row k1 (row task) or column block q (column task)
  int prev;             // the slot's previous transform, or -1
  int kind;             // 1 row, 2 column, 0 nothing (past the last chunk), -1 queue done
};

template <int LOG2L1>
__global__ void __launch_bounds__(kRowThreads, 4) apply_l2_kernel(FusedArgs a) {
  constexpr int L1 = 1 << LOG2L1;
  constexpr int COLS = kRowN / L1;              // columns of a column task
  constexpr int PER = COLS / kRowThreads;       // columns per thread
  extern __shared__ __align__(128) float2 sm[]; // [kRowPitch] the row buffer
  __shared__ ApplyTask s_ti[2];                 // the task in hand and the next one
  __shared__ float2 s_tw2[64], s_tw3[1024];     // the row's stage-base table rows r = 1, 2, 4, 8
  const int j = threadIdx.x;
  if (j < 64) s_tw2[j] = __ldg(a.tw + kTwS2 + ((1 << (j >> 4)) - 1) * 16 + (j & 15));
#pragma unroll
  for (int q = 0; q < 4; ++q) s_tw3[q * 256 + j] = __ldg(a.tw + kTwS3 + ((1 << q) - 1) * 256 + j);
  const int P = a.chunk;
  const int n_chunks = (a.n_items + P - 1) / P;
  const int per_block = P * L1;                 // the rows (or columns) of one chunk
  // block 2i: rows of chunk i; block 2i + 1: columns of chunk i - kApplyLag
  const int n_tasks = 2 * (n_chunks + kApplyLag) * per_block;
  const int n_slots = (kApplyLag + 2) * P;
  int* head = a.ctr;
  int* row_done = a.ctr + 1;
  int* col_done = a.ctr + 1 + a.n_items;
  const size_t slot_elems = (size_t)L1 * kRowN;
  // each task is decoded once (the divisions stay off the other threads)
  auto decode = [&](int t) {
    ApplyTask d = {};
    if (t >= n_tasks) {
      d.kind = -1;
      return d;
    }
    const int b = t / per_block, w = t % per_block;
    const bool is_col = b & 1;
    const int chunk = is_col ? (b >> 1) - kApplyLag : b >> 1;
    d.p = chunk * P + w / L1;
    d.rq = w % L1;                              // row k1, or column block q
    if (chunk < 0 || chunk >= n_chunks || d.p >= a.n_items) return d;   // kind 0: nothing
    d.kind = is_col ? 2 : 1;
    const FftItem I = apply_item(a, d.p);
    d.src = I.src;
    d.ptab = I.ptab;
    d.dst = I.dst;
    d.n_out = I.n_out;
    d.slot = a.scratch + (size_t)(d.p % n_slots) * slot_elems;
    d.prev = d.p >= n_slots ? d.p - n_slots : -1;
    return d;
  };
  // one thread of the last warp takes tasks from the queue, one ahead, and
  // decodes them while thread 0 counts the finished one: both chains are latency
  // that the CTA waits for between tasks
  const bool taker = j == kRowThreads - 32;
  int t_next = 0;                               // the task taken ahead
  if (taker) s_ti[0] = decode(atomicAdd(head, 1));
  for (int it = 0;; ++it) {
    __syncthreads();                            // s_ti; the last task's reads of sm are done
    const ApplyTask T = s_ti[it & 1];
    if (T.kind < 0) break;
    if (taker) t_next = atomicAdd(head, 1);     // decoded at the end of this task
    const int p = T.p, rq = T.rq;
    if (T.kind > 0 && DC_IN_BOUNDS(rq >= 0 && rq < L1 && p >= 0 && p < a.n_items, a.err)) {
      const bool is_col = T.kind == 2;
      float2* slot = T.slot;
      FftItem I = {};
      I.src = T.src;
      I.ptab = T.ptab;
      I.dst = T.dst;
      I.n_out = T.n_out;
      if (!is_col) {
        float2 v[16];
        load_bins(I.src + (size_t)rq * kRowN, j, v);
        mul_bins(I.ptab + (size_t)rq * kRowN, j, v);
        // the slot is free: the row's CTA barrier orders thread 0's wait
        // before every thread's stores (the others poll nothing)
        if (j == 0 && T.prev >= 0) wait_count(col_done + T.prev, L1, a.err);
        row_inverse<false>(v, sm, j, SharedTw{s_tw2, s_tw3});   // v[r] = Y[j + 256 r]
        float2* yrow = slot + (size_t)rq * kRowN;
#pragma unroll
        for (int r = 0; r < 16; ++r) __stcg(yrow + j + 256 * r, v[r]);
        __syncthreads();
        if (j == 0) red_release_gpu(row_done + p, 1);   // every thread's row stores first
      } else {
        const float2* tw4 = a.t4 + kT4Offset(L1);
        float2 w4[PER][4];                      // W_L^(-2^b n2), loaded ahead of the wait
#pragma unroll
        for (int pp = 0; pp < PER; ++pp)
#pragma unroll
          for (int bb = 0; bb < LOG2L1; ++bb) w4[pp][bb] = __ldg(tw4 + bb * kRowN + rq * COLS + j + 256 * pp);
        if (j == 0) wait_count(row_done + p, L1, a.err);
        __syncthreads();
#pragma unroll
        for (int pp = 0; pp < PER; ++pp) {
          const int n2 = rq * COLS + j + 256 * pp;
          float2 col[L1];
#pragma unroll
          for (int q = 0; q < L1; ++q) col[q] = __ldcg(slot + (size_t)q * kRowN + n2);
          apply_powers<L1>(col, w4[pp]);
          dft<L1, +1>(col);
          if (pp == PER - 1) {
            // every thread's slot reads are done; counted ahead of the output's last
            // stores, which the release would otherwise wait for
            __syncthreads();
            if (j == 0) red_release_gpu(col_done + p, 1);
          }
#pragma unroll
          for (int n1 = 0; n1 < L1; ++n1) {
            const int n = n2 + kRowN * n1;
            if (n < I.n_out) __stcs(I.dst + n, col[n1]);
          }
        }
      }
    }
    if (taker) s_ti[(it + 1) & 1] = decode(t_next);
  }
}

template <int LOG2L1>
cudaError_t launch_apply_l2(const FusedArgs& a, cudaStream_t s) {
  if (!a.t4 || !a.scratch || !a.ctr || a.chunk < 1) return cudaErrorInvalidValue;
  const size_t smem = sizeof(float2) * kRowPitch;
  auto k = apply_l2_kernel<LOG2L1>;
  cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  int dev = 0, sms = 0, per_sm = 0;
  if ((e = cudaGetDevice(&dev)) != cudaSuccess ||
      (e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess ||
      (e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k, kRowThreads, smem)) != cudaSuccess)
    return e;
  const long long tasks = 2LL * (a.n_items + (long long)kApplyLag * a.chunk) * (1 << LOG2L1);
  const int grid = (int)std::max(1LL, std::min<long long>((long long)sms * std::max(per_sm, 1), tasks));
  k<<<grid, kRowThreads, smem, s>>>(a);
  return cudaGetLastError();
}

// Full correction (FUSED_FULL): one row k1 of the transform per CTA, one
// cluster of L1 CTAs per transform, one padded buffer per CTA.  The forward
// columns run straight from global memory (zero past n_valid), take
// W_L^(n2 k1) and go to the row owners by plain remote stores; the forward
// row, exp(-i phi_k) / L on the bins in registers and the inverse row (two CTA
// barriers in all) follow in the same buffer; the
// inverse row's outputs go to the column owners the same way, which apply
// W_L^(-n2 q) and run the inverse columns (out truncated to n_out).  Cluster
// barriers order it all: every CTA running before the first remote store,
// each exchange delivered before it is read, every buffer free before the
// second exchange overwrites it.  At L = 4096 one CTA holds the whole
// transform.
template <int LOG2L1>
__global__ void __launch_bounds__(kRowThreads, LOG2L1 == 0 ? 2 : 4) full_kernel(FusedArgs a) {
  constexpr int L1 = 1 << LOG2L1;
  constexpr int COLS = kRowN / L1;              // columns owned by a CTA
  constexpr int PER = COLS / kRowThreads;       // columns per thread
  constexpr int LOG2L = 12 + LOG2L1;
  extern __shared__ __align__(128) float2 sm[];
  float2* A = sm;                               // [kRowPitch] received row, row FFTs,
  float2* R = sm;                               // then [L1][COLS] received inverse rows
  const int k1 = L1 > 1 ? (int)cg::this_cluster().block_rank() : 0;
  const FftItem I = item_of(a, blockIdx.x >> LOG2L1);
  const int j = threadIdx.x;
  if constexpr (L1 == 1) {
    full_4096(I, A, j, a.tw);
  } else {
    asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");   // this CTA runs
    float2 v[16];
    const float2* T = a.t4 + kT4Offset(L1);
    pdl_wait();                                 // the input's producer has finished
#pragma unroll
    for (int p = 0; p < PER; ++p) {
      const int n2 = k1 * COLS + j + 256 * p;
      float2 col[L1];
#pragma unroll
      for (int n1 = 0; n1 < L1; ++n1) {
        const int n = n2 + kRowN * n1;
        col[n1] = n < I.n_valid ? I.src[n] : make_float2(0.f, 0.f);   // plain: after pdl_wait
      }
      dft<L1, -1>(col);
      float2 w[4];                              // W_L^(2^b n2), conjugates of the table rows
#pragma unroll
      for (int b = 0; b < LOG2L1; ++b) w[b] = conj_if<+1>(__ldg(T + b * kRowN + n2));
      apply_powers<L1>(col, w);
      if (p == 0) cluster_wait<L1>();           // every peer runs: its shared memory exists
      const uint32_t dst = smem_addr(A + pad16(n2));
#pragma unroll
      for (int q = 0; q < L1; ++q) st_cluster_c64(dsmem_map(dst, q), col[q]);
    }
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");   // columns delivered
    cluster_wait<L1>();
#pragma unroll
    for (int r = 0; r < 16; ++r) v[r] = A[pad16(j + 256 * r)];
    row_forward(v, A, j, GlobalTw{a.tw});
    bin_factors(I, k1, LOG2L1, j, v);
    const float invL = 1.0f / (float)(1 << LOG2L);
#pragma unroll
    for (int r = 0; r < 16; ++r) v[r] = cscale(v[r], invL);
    row_inverse<true>(v, A, j, GlobalTw{a.tw});   // arrives at the cluster barrier
    cluster_wait<L1>();                         // every peer's buffer is free
    const uint32_t r_loc = smem_addr(R + k1 * COLS + j);
#pragma unroll
    for (int r = 0; r < 16; ++r) {
      const int owner = r / PER;                // n2 = j + 256 r -> owner n2 / COLS
      const uint32_t off = (uint32_t)(256 * (r % PER) * sizeof(float2));
      st_cluster_c64(dsmem_map(r_loc + off, owner), v[r]);
    }
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");   // rows delivered
#pragma unroll
    for (int p = 0; p < PER; ++p) {
      const int c = j + 256 * p;
      const int n2 = k1 * COLS + c;
      float2 w[4];
#pragma unroll
      for (int b = 0; b < LOG2L1; ++b) w[b] = __ldg(T + b * kRowN + n2);   // W_L^(-2^b n2)
      if (p == 0) cluster_wait<L1>();           // every peer's stores into R are visible
      float2 col[L1];
#pragma unroll
      for (int q = 0; q < L1; ++q) col[q] = R[q * COLS + c];
      apply_powers<L1>(col, w);
      dft<L1, +1>(col);
#pragma unroll
      for (int n1 = 0; n1 < L1; ++n1) {
        const int n = n2 + kRowN * n1;
        if (n < I.n_out) __stcs(I.dst + n, col[n1]);
      }
    }
  }
}

template <int LOG2L1>
cudaError_t launch_full(const FusedArgs& a, cudaStream_t s) {
  constexpr int L1 = 1 << LOG2L1;
  if (L1 > 1 && !a.t4) return cudaErrorInvalidValue;
  const size_t smem = sizeof(float2) * kRowPitch;
  auto k = full_kernel<LOG2L1>;
  cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  if (L1 > 8) {
    e = cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return e;
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(a.n_items * L1));
  cfg.blockDim = dim3(kRowThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  // with a.pdl, programmatic serialization: the launch may begin (items,
  // twiddles) while the kernel before it finishes; the kernel waits for it
  // (pdl_wait) before its first read of the input and its first store
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = L1;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  // L = 4096 (one CTA per transform) is no cluster launch
  cfg.attrs = L1 > 1 ? attr : attr + 1;
  cfg.numAttrs = (L1 > 1 ? 1 : 0) + (a.pdl ? 1 : 0);
  return cudaLaunchKernelEx(&cfg, k, a);
}


// Row passes on 4096-point rows, one per CTA (launch_row_4096): the row comes
// in and goes out coalesced (natural order on the four-step scratch, spec_index
// order on stored spectra), everything between stays in registers and the one
// padded buffer.  34 KiB and 64 registers: 4 CTAs per SM.
template <int OP>
__global__ void __launch_bounds__(kRowThreads, 4) row_4096_kernel(RowArgs a) {
  extern __shared__ __align__(128) float2 sm[];
  const int L1 = 1 << a.log2L1;
  const int g = blockIdx.x;
  const FftItem I = item_of(a, g >> a.log2L1);
  const int k1 = g & (L1 - 1);
  const int j = threadIdx.x;
  const std::conditional_t<OP == ROW_MID, FineTw, GlobalTw> tw{a.tw};
  const float2* src = I.src + (size_t)k1 * kRowN;
  float2* dst = I.dst + (size_t)k1 * kRowN;
  float2 v[16];
  pdl_release();
  pdl_wait();
  if constexpr (OP == ROW_APPLY) {
    load_bins(src, j, v);
  } else {
    // the zero-padded input itself when a row is the whole transform (L = 4096)
    const int valid = OP == ROW_SPEC && L1 == 1 ? I.n_valid : kRowN;
#pragma unroll
    for (int r = 0; r < 16; ++r) v[r] = j + 256 * r < valid ? src[j + 256 * r] : make_float2(0.f, 0.f);
    row_forward(v, sm, j, tw);
  }
  if constexpr (OP == ROW_SPEC) {
    store_bins(dst, j, v);
    return;
  }
  if constexpr (OP == ROW_APPLY) mul_bins(I.ptab + (size_t)k1 * kRowN, j, v);
  else bin_factors(I, k1, a.log2L1, j, v);
  if (OP == ROW_APPLY && L1 == 1) {
    row_inverse<false>(v, sm, j, tw);
    const float invL = 1.0f / (float)kRowN;
#pragma unroll
    for (int r = 0; r < 16; ++r)
      if (j + 256 * r < I.n_out) __stcs(dst + j + 256 * r, cscale(v[r], invL));
    return;
  }
  // four-step twiddle W_L^(-k1 (j + 256 r)): the thread's own W_L^(-k1 j) inside
  // the row, the CTA's W_(16 L1)^(-k1 r) after it
  row_inverse<false, true>(v, sm, j, tw, tw_big<+1>(a.tw, (uint32_t)(j * k1), a.log2L));
  const int m16 = 16 * L1 - 1, step = 256 >> a.log2L1;
#pragma unroll
  for (int r = 1; r < 16; ++r) v[r] = cmul(v[r], tw_m<+1>(a.tw, ((r * k1) & m16) * step));
#pragma unroll
  for (int r = 0; r < 16; ++r) dst[j + 256 * r] = v[r];
}

template <int OP> cudaError_t launch_row_4096_op(const RowArgs& a, cudaStream_t s) {
  const size_t smem = a.pdl == PDL_SPREAD ? kPdlRowSmem : sizeof(float2) * kRowPitch;
  auto k = row_4096_kernel<OP>;
  cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kPdlRowSmem);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(a.n_items << a.log2L1));
  cfg.blockDim = dim3(kRowThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = a.pdl ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, k, a);
}

}  // namespace

cudaError_t launch_row_4096(int op, const RowArgs& a, cudaStream_t s) {
  if (a.n_items <= 0) return cudaSuccess;
  if (a.log2L - a.log2L1 != 12 || a.log2L1 < 0 || a.log2L1 > 8) return cudaErrorInvalidValue;
  switch (op) {
    case ROW_MID: return launch_row_4096_op<ROW_MID>(a, s);
    case ROW_SPEC: return launch_row_4096_op<ROW_SPEC>(a, s);
    case ROW_APPLY: return launch_row_4096_op<ROW_APPLY>(a, s);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t launch_fused(int op, const FusedArgs& a, cudaStream_t s) {
  if (a.n_items <= 0) return cudaSuccess;
  switch (op) {
    case FUSED_APPLY:
      switch (a.log2L) {
        case 12: return launch_apply<0, 0>(a, s);
        case 13: return a.scratch ? launch_apply_l2<1>(a, s) : launch_apply<1, 0>(a, s);
        case 14: return a.scratch ? launch_apply_l2<2>(a, s) : launch_apply<2, 0>(a, s);
        case 15: return a.scratch ? launch_apply_l2<3>(a, s)
                       : a.apply_rows2 ? launch_apply<3, 1>(a, s) : launch_apply<3, 0>(a, s);
        case 16: return a.scratch ? launch_apply_l2<4>(a, s)
                       : a.apply_rows2 ? launch_apply<4, 1>(a, s) : launch_apply<4, 0>(a, s);
        default: return cudaErrorInvalidValue;
      }
    case FUSED_FULL:
      switch (a.log2L) {
        case 12: return launch_full<0>(a, s);
        case 13: return launch_full<1>(a, s);
        case 14: return launch_full<2>(a, s);
        case 15: return launch_full<3>(a, s);
        case 16: return launch_full<4>(a, s);
        default: return cudaErrorInvalidValue;
      }
    case FUSED_SPEC:
      switch (a.log2L) {
        case 12: return launch_spec<0>(a, s);
        case 13: return launch_spec<1>(a, s);
        case 14: return launch_spec<2>(a, s);
        case 15: return launch_spec<3>(a, s);
        case 16: return launch_spec<4>(a, s);
        default: return cudaErrorInvalidValue;
      }
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace dc
