// Dynamic activation quantization (Step 3, Eq. "daq"; b = 8, zero-point 0, clip threshold = the
// token's absolute maximum): bf16 [M][K] -> int8 codes + one fp32 scale per token.
//
// One warp owns one token, or two or four where a row is long (launch_daq_t). The row is read once with 16-byte loads and kept in registers; the
// absolute maximum is taken on the bf16 magnitude bits (monotone for finite values, so integer
// max is exact); the quantizer is one fused multiply-add per element: x * fl(127/a) + 1.5*2^23
// rounds the exact product once, half to even, and leaves the integer in the low mantissa bits.
// HBM-bound: 2 bytes read + 1 byte written per element.
#include <limits.h>

#include "daq_device.cuh"

namespace dp {

constexpr int kDaqWarps = 8;
constexpr int kDaqThreads = 128;  // CTA of the register-resident kernel

// The first launch of a call lets its dependents start only once everything before the call has
// finished (they may read the layers' constants ahead of their own wait, and those may have been written by
// the kernel before the call); later ones let them start at once.
__device__ __forceinline__ void daq_begin(const UnpackJob& job) {
  if (!job.early) pdl_wait();
  pdl_launch_dependents();
}
// The end of a launch's first CTA.
__device__ __forceinline__ void daq_end(const UnpackJob& job) {
  if (job.ahead && blockIdx.x == 0) pdl_wait();
}

// RW warps share a row: MAXV = 16-byte vectors held per lane (a row of up to 256 * RW * MAXV elements in
// registers). SUM: also the row's code sum.
template <int RW, int MAXV, bool EO, bool SUM>
__global__ void __launch_bounds__(kDaqThreads)
daq_rows_kernel(const uint16_t* __restrict__ x, int64_t M, int K, int64_t ldx,
                int8_t* __restrict__ q, int64_t ldq, float* __restrict__ s_a,
                int32_t* __restrict__ rowsum, int tiled_kb, const UnpackJob job) {
  constexpr int kRows = kDaqThreads / 32 / RW;  // rows of a CTA
  constexpr int TPR = 32 * RW;
  __shared__ uint32_t part[kDaqThreads / 32];
  daq_begin(job);
  if (static_cast<int>(blockIdx.x) >= job.first_block) {  // the launch's weight-expansion CTAs
    unpack_units(job, blockIdx.x - job.first_block);
    return;
  }
  if (!job.ahead) pdl_wait();
  const int rw = threadIdx.x / TPR, lane = threadIdx.x % TPR;  // row of the CTA, position in the row
  const int64_t row = static_cast<int64_t>(blockIdx.x) * kRows + rw;
  const bool live = row < M;
  const int nvec = live ? K >> 3 : 0;
  const uint4* xr = reinterpret_cast<const uint4*>(x + row * ldx);
  uint4 v[MAXV];
#pragma unroll
  for (int i = 0; i < MAXV; ++i) {
    const int idx = lane + TPR * i;
    if (idx < nvec) ld_stream_u32x4(xr + idx, v[i]);
    else v[i] = make_uint4(0, 0, 0, 0);
  }
  uint32_t m = 0;
#pragma unroll
  for (int i = 0; i < MAXV; ++i) {
    m = absmax_bits2(m, v[i].x);
    m = absmax_bits2(m, v[i].y);
    m = absmax_bits2(m, v[i].z);
    m = absmax_bits2(m, v[i].w);
  }
  m = warp_max_u32(max(m & 0xFFFFu, m >> 16));
  if constexpr (RW > 1) {
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = m;
    __syncthreads();
#pragma unroll
    for (int w = 0; w < RW; ++w) m = max(m, part[rw * RW + w]);
  }
  if (RW == 1 && !live) return;
  float sc, inv;
  token_scale(m, sc, inv);
  const QRow qr(q, row, ldq, tiled_kb);
  int sum = 0;
#pragma unroll
  for (int i = 0; i < MAXV; ++i) {
    const int idx = lane + TPR * i;
    if (idx < nvec) {
      uint2 o = quant_vec<EO>(v[i], inv);
      qr.store(idx, o);
      if constexpr (SUM) {
        sum = __dp4a(static_cast<int>(o.x), 0x01010101, sum);
        sum = __dp4a(static_cast<int>(o.y), 0x01010101, sum);
      }
    }
  }
  if (lane == 0 && live) s_a[row] = sc;
  if constexpr (SUM) {
    sum = warp_sum_i32(sum);
    if constexpr (RW > 1) {
      __syncthreads();
      if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = static_cast<uint32_t>(sum);
      __syncthreads();
      sum = 0;
#pragma unroll
      for (int w = 0; w < RW; ++w) sum += static_cast<int>(part[rw * RW + w]);
    }
    if (lane == 0 && live) rowsum[row] = sum;
  }
  daq_end(job);
}

// Any K (multiple of 8): two passes over the row, the second served by L1/L2.
template <bool EO>
__global__ void __launch_bounds__(kDaqWarps * 32)
daq_rows_2pass_kernel(const uint16_t* __restrict__ x, int64_t M, int K, int64_t ldx,
                      int8_t* __restrict__ q, int64_t ldq, float* __restrict__ s_a,
                      int32_t* __restrict__ rowsum, int tiled_kb, const UnpackJob job) {
  daq_begin(job);
  const int64_t row = static_cast<int64_t>(blockIdx.x) * kDaqWarps + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (static_cast<int>(blockIdx.x) >= job.first_block) {  // the launch's weight-expansion CTAs
    unpack_units(job, blockIdx.x - job.first_block);
    return;
  }
  if (!job.ahead) pdl_wait();
  if (row >= M) return;
  const int nvec = K >> 3;
  const uint4* xr = reinterpret_cast<const uint4*>(x + row * ldx);
  uint32_t m = 0;
  for (int idx = lane; idx < nvec; idx += 32) {
    const uint4 v = ld_global_v4(xr + idx);
    m = absmax_bits2(absmax_bits2(absmax_bits2(absmax_bits2(m, v.x), v.y), v.z), v.w);
  }
  m = warp_max_u32(max(m & 0xFFFFu, m >> 16));
  float sc, inv;
  token_scale(m, sc, inv);
  const QRow qr(q, row, ldq, tiled_kb);
  int sum = 0;
  for (int idx = lane; idx < nvec; idx += 32) {
    uint2 o = quant_vec<EO>(ld_global_v4(xr + idx), inv);
    qr.store(idx, o);
    sum = __dp4a(static_cast<int>(o.x), 0x01010101, sum);
    sum = __dp4a(static_cast<int>(o.y), 0x01010101, sum);
  }
  if (lane == 0) s_a[row] = sc;
  if (rowsum != nullptr) {
    sum = warp_sum_i32(sum);
    if (lane == 0) rowsum[row] = sum;
  }
  daq_end(job);
}

// ---- DAQ with a percentile clip and a-bit codes: robust_row in daq_device.cuh ------------------------
// RW warps to a token, MAXV vectors a lane, registers for CTAS resident CTAs (see launch_daq_robust).
constexpr int kRobustWarpK = 256 * 6;  // rows that one warp takes in a plan's preparation
template <int RW, int MAXV, int CTAS>
__global__ void __launch_bounds__(kDaqThreads, CTAS)
daq_rows_robust_kernel(const uint16_t* __restrict__ x, int64_t M, int K, int64_t ldx, int8_t* __restrict__ q,
                       int64_t ldq, float* __restrict__ s_a, int32_t* __restrict__ rowsum, int clip_rank,
                       float qmax, int tiled_kb, const UnpackJob job) {
  __shared__ uint2 meet[2 * RW];
  daq_begin(job);
  if (static_cast<int>(blockIdx.x) >= job.first_block) {  // the launch's weight-expansion CTAs
    unpack_units(job, blockIdx.x - job.first_block);
    return;
  }
  if (!job.ahead) pdl_wait();
  const int64_t row = static_cast<int64_t>(blockIdx.x) * (kDaqThreads / 32 / RW) + threadIdx.x / (32 * RW);
  const int lane = threadIdx.x % (32 * RW);
  if (row >= M) return;
  const QRow qr(q, row, ldq, tiled_kb);
  float sc;
  int sum;
  robust_row<RW, MAXV>(x + row * ldx, K, lane, clip_rank, qmax, qr, sc, sum, meet);
  if (lane == 0) s_a[row] = sc;
  if (rowsum != nullptr) {
    sum = warp_sum_i32(sum);
    if constexpr (RW > 1) {
      __syncthreads();  // all have read the last maxima
      if ((lane & 31) == 0) meet[lane >> 5].x = static_cast<uint32_t>(sum);
      __syncthreads();
      sum = 0;
#pragma unroll
      for (int w = 0; w < RW; ++w) sum += static_cast<int>(meet[w].x);
    }
    if (lane == 0) rowsum[row] = sum;
  }
  daq_end(job);
}

__global__ void __launch_bounds__(kDaqWarps * 32)
unpack_kernel(const UnpackJob job) {
  daq_begin(job);
  unpack_units(job, blockIdx.x);
}

// ---- the preparation of a plan's unit of layers (gemm_plan.cu), in one launch -------------------------
// A CTA works on one segment: rows of a layer to quantize, codes to expand, weights to send into L2. It runs beside the
// GEMM kernel of the unit before, which leaves room for a few small CTAs on an SM. So a CTA has 128 threads, holds rows as five
// vectors a lane (longer rows by two or four warps), and keeps four units of 32 codes a thread in flight. With the
// percentile rule a thread takes 48 registers, five CTAs beside a GEMM CTA; with one warp to every row, 18 vectors a lane and 128
// registers there was room for one, and a step of 28 blocks, 1024 tokens, 16-bit layers took 769 us instead of 745.
constexpr int kExpandUnits = 4, kFetchBytes = 32768, kFetchThreads = 4;

template <int BITS>
__device__ __forceinline__ void prep_expand(const PlanPrepSeg& s, int block, bool wait) {
  const int64_t u0 = static_cast<int64_t>(block) * (kDaqThreads * kExpandUnits) + threadIdx.x;
  uint32_t pk[kExpandUnits][BITS];
#pragma unroll
  for (int i = 0; i < kExpandUnits; ++i) {
    const int64_t u = u0 + i * kDaqThreads;
    if (u >= s.count) continue;
    if constexpr (BITS == 4) {
      uint4 v;
      ld_stream_u32x4(static_cast<const uint4*>(s.src) + u, v);
      pk[i][0] = v.x, pk[i][1] = v.y, pk[i][2] = v.z, pk[i][3] = v.w;
    } else {
      const uint32_t* w = static_cast<const uint32_t*>(s.src) + u * 3;
#pragma unroll
      for (int j = 0; j < 3; ++j) pk[i][j] = __ldg(w + j);
    }
  }
  if (wait) pdl_wait();
#pragma unroll
  for (int i = 0; i < kExpandUnits; ++i) {
    const int64_t u = u0 + i * kDaqThreads;
    if (u >= s.count) continue;
    uint32_t w[8];
    expand_unit<BITS>(pk[i], w, 1u << (BITS - 1));
    st_global_v8(reinterpret_cast<uint4*>(s.dst) + u * 2, w);
  }
}

// CTA `block` over the rows of a segment, RW warps to a row, `part` a word per warp: daq_rows_kernel without its options. (One
// function for both costs that kernel registers, 40 -> 42 with four warps to a row, and with them two CTAs of an SM:
// K = 3072, M = 2048 / 8192 4.6 / 13.2 -> 5.0 / 14.1 us. Where ten CTAs an SM hold all rows and twelve leave SMs with fewer, that was
// the better: K = 3072 / 4608, M = 1285 3.5 / 4.5 -> 3.4 / 4.35, but M = 1600 3.6 / 4.8 -> 4.1 / 4.75.)
template <int RW>
__device__ __forceinline__ void prep_rows(const PlanPrepSeg& s, int block, uint32_t* part) {
  constexpr int TPR = 32 * RW, MAXV = 5;
  const int K = s.arg * 8;
  const int rw = threadIdx.x / TPR, lane = threadIdx.x % TPR;
  const int64_t row = static_cast<int64_t>(block) * (kDaqThreads / TPR) + rw;
  const int nvec = row < s.count ? K >> 3 : 0;
  const uint4* xr = reinterpret_cast<const uint4*>(static_cast<const uint16_t*>(s.src) + row * K);
  uint4 v[MAXV];
#pragma unroll
  for (int i = 0; i < MAXV; ++i) {
    const int idx = lane + TPR * i;
    if (idx < nvec) ld_stream_u32x4(xr + idx, v[i]);
    else v[i] = make_uint4(0, 0, 0, 0);
  }
  uint32_t m = 0;
#pragma unroll
  for (int i = 0; i < MAXV; ++i) m = absmax_bits2(absmax_bits2(absmax_bits2(absmax_bits2(m, v[i].x), v[i].y), v[i].z), v[i].w);
  m = warp_max_u32(max(m & 0xFFFFu, m >> 16));
  if constexpr (RW > 1) {
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = m;
    __syncthreads();
#pragma unroll
    for (int w = 0; w < RW; ++w) m = max(m, part[rw * RW + w]);
  }
  if (nvec == 0) return;
  float sc, inv;
  token_scale(m, sc, inv);
  const QRow qr(s.dst, row, K, K >> 7);
#pragma unroll
  for (int i = 0; i < MAXV; ++i) {
    const int idx = lane + TPR * i;
    if (idx < nvec) qr.store(idx, quant_vec<false>(v[i], inv));
  }
  if (lane == 0) s.s_a[row] = sc;
}

template <bool ROBUST>
__global__ void __launch_bounds__(kDaqThreads, ROBUST ? 10 : 12)
plan_prep_kernel(const __grid_constant__ PlanPrepParams p) {
  __shared__ uint32_t part[kDaqThreads / 32];
  __shared__ uint2 meet[2 * kDaqThreads / 32];
  if (!p.early) pdl_wait();
  pdl_launch_dependents();
  // (a search over the segments one by one was a chain of constant-cache misses: 3 us of a CTA's 5)
  int i = 0;
#pragma unroll
  for (int step = kPlanPrepSegs / 2; step > 0; step >>= 1)
    if (static_cast<int>(blockIdx.x) >= p.first_block[i + step]) i += step;
  const PlanPrepSeg& s = p.seg[i];
  const int block = blockIdx.x - p.first_block[i];
  if (s.kind == PlanPrepSeg::EXPAND) {
    if (s.arg == 4) prep_expand<4>(s, block, !p.ahead);
    else prep_expand<3>(s, block, !p.ahead);
  } else if (s.kind == PlanPrepSeg::FETCH) {
    const int64_t at = (static_cast<int64_t>(block) * kFetchThreads + threadIdx.x) * kFetchBytes;
    if (threadIdx.x < kFetchThreads && at < s.count)
      bulk_prefetch_l2(static_cast<const uint8_t*>(s.src) + at,
                       static_cast<uint32_t>(s.count - at < kFetchBytes ? s.count - at : kFetchBytes));
  } else {
    if (!p.ahead) pdl_wait();
    const int K = s.arg * 8;
    if constexpr (ROBUST) {
      const bool one = K <= kRobustWarpK;  // one warp to a row
      const int64_t row = one ? static_cast<int64_t>(block) * (kDaqThreads / 32) + (threadIdx.x >> 5) : block;
      if (row < s.count) {
        const uint16_t* x = static_cast<const uint16_t*>(s.src) + row * K;
        const int lane = one ? threadIdx.x & 31 : threadIdx.x;
        const QRow qr(s.dst, row, K, K >> 7);
        float sc;
        int sum;
        if (one) robust_row<1, 6>(x, K, lane, s.rank, p.qmax, qr, sc, sum);
        else robust_row<kDaqThreads / 32, 5>(x, K, lane, s.rank, p.qmax, qr, sc, sum, meet);
        if (lane == 0) s.s_a[row] = sc;
      }
    } else {
      if (K <= 256 * 5) prep_rows<1>(s, block, part);
      else if (K <= 512 * 5) prep_rows<2>(s, block, part);
      else prep_rows<4>(s, block, part);
    }
  }
  // One CTA of every launch stays until everything before it has finished. Rows and expansion wait by themselves unless `ahead`,
  // but a unit of 16-bit layers has neither, and the GEMM kernel behind this one waits for this one only.
  if (p.early && blockIdx.x == 0) pdl_wait();
}

static unsigned unpack_blocks(const UnpackJob& job, int threads) {
  return static_cast<unsigned>((job.units + threads - 1) / threads);
}

template <int RW, int MAXV, bool EO, bool SUM, typename... A>
static cudaError_t launch_rows(int64_t M, UnpackJob job, cudaStream_t stream, bool pdl, A... a) {
  constexpr int kRows = kDaqThreads / 32 / RW;
  const unsigned daq_blocks = static_cast<unsigned>((M + kRows - 1) / kRows);
  job.first_block = static_cast<int32_t>(daq_blocks);
  const dim3 grid(daq_blocks + unpack_blocks(job, kDaqThreads));
  return launch(daq_rows_kernel<RW, MAXV, EO, SUM>, grid, dim3(kDaqThreads), 0, stream, pdl, a..., job);
}

template <bool EO, bool SUM>
static cudaError_t launch_daq_t(const uint16_t* xp, int64_t M, int k, int64_t ldx, int8_t* q, int64_t ldq,
                                float* s_a, int32_t* rowsum, int tiled_kb, cudaStream_t stream, bool pdl,
                                UnpackJob job) {
#define DP_ROWS(RW, MAXV) launch_rows<RW, MAXV, EO, SUM>(M, job, stream, pdl, xp, M, k, ldx, q, ldq, s_a, rowsum, tiled_kb)
  // As many warps to a row as leave a lane at most five vectors: a row of 4608 held by one warp (18 vectors,
  // ~90 registers) left one CTA beside a running GEMM and a long serial chain per warp. Whole 8-bit layer,
  // K = 4608, N = 1152, M = 256 / 2048 / 32768: one warp 12.1 / 18.8 / 182.5 us, two 12.3 / 17.6 / 182.5,
  // four 12.1 / 17.4 / 181.7. Shorter rows want one: K = 1152 whole layer (N = 1152), M = 2048 / 32768: one
  // 8.8 / 56.8 us, two 9.2 / 58.1, four 8.8 / 70.3 (their warps spend longer starting than working). So do rows of up to
  // 2048 where there are many: DAQ alone, K = 1536, M = 333 / 2048 / 9000: one warp 1.72 / 3.18 / 7.9 us, two 1.66 / 3.58 /
  // 8.7; K = 2048: one 1.88 / 3.66 / 9.98, two 1.72 / 4.10 / 10.1.
  if (k <= 256 * 5) return DP_ROWS(1, 5);
  if (k <= 256 * 6 && M > 512) return DP_ROWS(1, 6);
  if (k <= 256 * 8 && M > 512) return DP_ROWS(1, 8);
  if (k <= 512 * 5) return DP_ROWS(2, 5);
  if (k <= 1024 * 5) return DP_ROWS(4, 5);
#undef DP_ROWS
  const unsigned daq_blocks = static_cast<unsigned>((M + kDaqWarps - 1) / kDaqWarps);
  job.first_block = static_cast<int32_t>(daq_blocks);
  return launch(daq_rows_2pass_kernel<EO>, dim3(daq_blocks + unpack_blocks(job, kDaqWarps * 32)), dim3(kDaqWarps * 32), 0,
                stream, pdl, xp, M, k, ldx, q, ldq, s_a, rowsum, tiled_kb, job);
}

int launch_daq(const void* x, int64_t M, int64_t K, int64_t ldx, int8_t* q, int64_t ldq,
               float* s_a, int32_t* rowsum, int korder, bool tiled, cudaStream_t stream, bool pdl,
               const UnpackJob* unpack) {
  if (M == 0) return DP_OK;
  const uint16_t* xp = static_cast<const uint16_t*>(x);
  const int k = static_cast<int>(K);
  const int tiled_kb = tiled ? k / 128 : 0;
  UnpackJob job;
  if (unpack != nullptr) job = *unpack;
  const cudaError_t e = korder == KORDER_EVEN_ODD
                            ? launch_daq_t<true, false>(xp, M, k, ldx, q, ldq, s_a, nullptr, tiled_kb, stream, pdl, job)
                        : rowsum != nullptr
                            ? launch_daq_t<false, true>(xp, M, k, ldx, q, ldq, s_a, rowsum, tiled_kb, stream, pdl, job)
                            : launch_daq_t<false, false>(xp, M, k, ldx, q, ldq, s_a, rowsum, tiled_kb, stream, pdl, job);
  if (e != cudaSuccess) return fail(DP_ERR_CUDA, "DAQ launch failed: %s", cudaGetErrorString(e));
  return DP_OK;
}

template <int RW, int MAXV, int CTAS, typename... A>
static cudaError_t launch_robust_rows(int64_t M, UnpackJob job, cudaStream_t stream, bool pdl, A... a) {
  constexpr int kRows = kDaqThreads / 32 / RW;
  const unsigned daq_blocks = static_cast<unsigned>((M + kRows - 1) / kRows);
  job.first_block = static_cast<int32_t>(daq_blocks);
  const dim3 grid(daq_blocks + unpack_blocks(job, kDaqThreads));
  return launch(daq_rows_robust_kernel<RW, MAXV, CTAS>, grid, dim3(kDaqThreads), 0, stream, pdl, a..., job);
}

int launch_daq_robust(const void* x, int64_t M, int64_t K, int64_t ldx, int8_t* q, int64_t ldq, float* s_a,
                      int32_t* rowsum, int clip_rank, int act_bits, bool tiled, cudaStream_t stream, bool pdl,
                      const UnpackJob* unpack) {
  if (M == 0) return DP_OK;
  const uint16_t* xp = static_cast<const uint16_t*>(x);
  const int k = static_cast<int>(K);
  const int tiled_kb = tiled ? k / 128 : 0;
  const float qmax = static_cast<float>((1 << (act_bits - 1)) - 1);
  UnpackJob job;
  if (unpack != nullptr) job = *unpack;
#define DP_ROWS(RW, MAXV, CTAS) \
  launch_robust_rows<RW, MAXV, CTAS>(M, job, stream, pdl, xp, M, k, ldx, q, ldq, s_a, rowsum, clip_rank, qmax, tiled_kb)
  // Four warps to a row of more than 2304 elements, and to one of more than 1280 where there are few. One warp, 18 vectors a lane
  // (five peeling rounds, two CTAs of 256 threads on an SM) -> this: K = 4608, p = 99.9, M = 100 / 1024 / 8192 / 32768 6.4 / 7.8 /
  // 32.0 / 108 us -> 2.8 / 7.3 / 28.0 / 100 (threshold of rank 47, p = 99: 23.8 / 25.9 / 101 / 359 -> 9.6 / 22.3 / 98 / 369);
  // K = 3072 5.4 / 5.8 / 25.9 / 89 -> 2.4 / 5.2 / 22.7 / 81. Shorter rows, many of them, spend longer on the exchanges than on
  // the row: K = 2304, one warp and nine vectors in CTAs of 256 / four warps / one warp and nine vectors in CTAs of 128:
  // M = 100 3.3 / 2.2 / -, 1024 3.5 / 4.4 / 3.2, 32768 54 / 68 / 39; K = 1536 (nine, -, six) 2.4 / 1.9 / -, 2.5 / 3.5 / 2.4, 38 / 56 / 26.
  // Few registers, many CTAs to an SM, only from 4096 rows on. Up to there all rows are resident either way and more CTAs of
  // them beside the GEMM before make the GEMM behind wait. Quantization and the GEMM of an 8-bit layer of 1152 channels on its codes,
  // p = 99.9, CTAs of 256 threads and two or three to an SM / ten small ones (K = 2304: six) / this: K = 1152, M = 900 7.27 / 7.95 / 7.33 us,
  // 2048 8.53 / 9.57 / 8.62, 3001 10.05 / 11.08 / 9.94; K = 1536, M = 2048 9.50 / 10.69 / 8.96; K = 2304, M = 2048 11.15 / 12.59 / 11.09.
  // Beyond it the rate of the quantization itself counts: K = 1152, six / eight to an SM, M = 9000 8.61 / 8.06, layer 19.4 / 19.4.
  const bool few = M < 4096;
  const cudaError_t e = k <= 256 * 5               ? few ? DP_ROWS(1, 5, 6) : DP_ROWS(1, 5, 8)
                        : k > 256 * 9 || M <= 512 ? DP_ROWS(kDaqThreads / 32, 5, 10)
                        : k <= 256 * 6            ? few ? DP_ROWS(1, 6, 4) : DP_ROWS(1, 6, 8)
                                                  : few ? DP_ROWS(1, 9, 4) : DP_ROWS(1, 9, 6);
#undef DP_ROWS
  if (e != cudaSuccess) return fail(DP_ERR_CUDA, "robust DAQ launch failed: %s", cudaGetErrorString(e));
  return DP_OK;
}

int launch_plan_prep(PlanPrepParams& p, bool robust, cudaStream_t stream, bool pdl) {
  int64_t at = 0;
  for (int i = 0; i < p.n_seg; ++i) {
    PlanPrepSeg& s = p.seg[i];
    p.first_block[i] = static_cast<int32_t>(at);
    int64_t per = kDaqThreads * kExpandUnits;
    if (s.kind == PlanPrepSeg::FETCH) {
      per = static_cast<int64_t>(kFetchBytes) * kFetchThreads;
    } else if (s.kind == PlanPrepSeg::ROWS) {
      const int K = s.arg * 8;
      per = kDaqThreads / 32 / (robust ? (K <= kRobustWarpK ? 1 : kDaqThreads / 32) : K <= 256 * 5 ? 1 : K <= 512 * 5 ? 2 : 4);
    }
    at += (s.count + per - 1) / per;
  }
  for (int i = p.n_seg; i < kPlanPrepSegs; ++i) p.first_block[i] = INT_MAX;
  const dim3 grid(static_cast<unsigned>(at)), block(kDaqThreads);
  const cudaError_t e = robust ? launch(plan_prep_kernel<true>, grid, block, 0, stream, pdl, p)
                               : launch(plan_prep_kernel<false>, grid, block, 0, stream, pdl, p);
  if (e != cudaSuccess) return fail(DP_ERR_CUDA, "plan preparation launch failed: %s", cudaGetErrorString(e));
  return DP_OK;
}

int launch_unpack(const UnpackJob& job, cudaStream_t stream, bool pdl) {
  if (job.units == 0) return DP_OK;
  const dim3 grid(unpack_blocks(job, kDaqWarps * 32));
  const cudaError_t e = launch(unpack_kernel, grid, dim3(kDaqWarps * 32), 0, stream, pdl, job);
  if (e != cudaSuccess) return fail(DP_ERR_CUDA, "weight expansion launch failed: %s", cudaGetErrorString(e));
  return DP_OK;
}

}  // namespace dp

extern "C" int dp_daq_quantize(const void* x_bf16, int64_t M, int64_t K, int64_t ldx, int8_t* q,
                               int64_t ldq, float* s_a, int32_t* rowsum, dp_stream stream) {
  using namespace dp;
  if (M < 0 || K < 8 || K > 65536) return fail(DP_ERR_SHAPE, "dp_daq_quantize: bad M=%lld K=%lld",
                                                (long long)M, (long long)K);
  if (K % 8) return fail(DP_ERR_SHAPE, "dp_daq_quantize: K=%lld not a multiple of 8", (long long)K);
  if (M == 0) return DP_OK;
  if (!x_bf16 || !q || !s_a) return fail(DP_ERR_INVALID_ARG, "dp_daq_quantize: NULL pointer");
  if (ldx < K || ldq < K) return fail(DP_ERR_SHAPE, "dp_daq_quantize: leading dimension < K");
  if (!aligned16(x_bf16) || !aligned16(q) || (ldx % 8) || (ldq % 16) ||
      (reinterpret_cast<uintptr_t>(s_a) & 3u))
    return fail(DP_ERR_ALIGN, "dp_daq_quantize: pointers/pitches must be 16-byte aligned");
  int st = check_device();
  if (st != DP_OK) return st;
  return launch_daq(x_bf16, M, K, ldx, q, ldq, s_a, rowsum, KORDER_NATURAL, false,
                    static_cast<cudaStream_t>(stream), true);
}

extern "C" int dp_daq_quantize_robust(const void* x_bf16, int64_t M, int64_t K, int64_t ldx, int8_t* q,
                                      int64_t ldq, float* s_a, int32_t* rowsum, int32_t clip_rank,
                                      int32_t act_bits, dp_stream stream) {
  using namespace dp;
  if (M < 0 || K < 8 || K > 4608 || (K % 8))
    return fail(DP_ERR_SHAPE, "dp_daq_quantize_robust: need M >= 0 and K a multiple of 8 in [8, 4608] (M=%lld K=%lld)",
                (long long)M, (long long)K);
  if (clip_rank < 1 || clip_rank > 64 || clip_rank > K)
    return fail(DP_ERR_INVALID_ARG, "dp_daq_quantize_robust: clip_rank=%d not in [1, min(K, 64)]", clip_rank);
  if (act_bits < 2 || act_bits > 8)
    return fail(DP_ERR_BITS, "dp_daq_quantize_robust: act_bits=%d not in [2, 8]", act_bits);
  if (M == 0) return DP_OK;
  if (!x_bf16 || !q || !s_a) return fail(DP_ERR_INVALID_ARG, "dp_daq_quantize_robust: NULL pointer");
  if (ldx < K || ldq < K) return fail(DP_ERR_SHAPE, "dp_daq_quantize_robust: leading dimension < K");
  if (!aligned16(x_bf16) || !aligned16(q) || (ldx % 8) || (ldq % 16) || (reinterpret_cast<uintptr_t>(s_a) & 3u))
    return fail(DP_ERR_ALIGN, "dp_daq_quantize_robust: pointers/pitches must be 16-byte aligned");
  int st = check_device();
  if (st != DP_OK) return st;
  return launch_daq_robust(x_bf16, M, K, ldx, q, ldq, s_a, rowsum, clip_rank, act_bits, false,
                           static_cast<cudaStream_t>(stream), true, nullptr);
}
