// LayerNorm + adaLN modulation taken into dynamic activation quantization.
//
//   Step 3 of the paper keeps LayerNorms in higher precision and quantizes the activations of the
//   wrapped linears on the fly (Eq. "daq"). In a DiT block the qkv and fc1 linears are fed
//   LayerNorm(x) * (1 + scale) + shift with a per-sample adaLN scale and shift; run as separate
//   operators that is a normalization kernel writing bf16, and a quantization kernel reading it
//   back. Here one kernel reads the block's bf16 stream once and writes int8 codes and token scales:
//   the normalized, modulated values exist only in fp32 registers and are never rounded to bf16.
//
// Arithmetic (the oracle's, bit for bit): sums of x and x^2 of a token in double (the terms are bf16
// values and their squares; for activations whose magnitudes span less than ~2^13 every partial sum is
// exact, so the order of summation cannot matter; beyond that the sums differ from a sequential sum
// by double-precision roundings only), mean = S1 / K, var = S2 / K - mean^2, rstd = 1 / sqrt(var +
// eps), all in double with IEEE operations, then rounded to fp32; n = (x - mean) * rstd and
// h = fma(n, 1 + scale, shift) in fp32; DAQ of h as for bf16 inputs (absmax / 127, one rounding of
// the exact product with fl(127 / absmax), half to even).
//
// One to four warps own a token; the row stays in registers as bf16 (16-byte loads), then as fp32 h. Moves
// DAQ's bytes (2 read + 1 written per element) but is bound by the double precision of the statistics: the
// conversions (16 per clock and SM; building the doubles with integer operations was slower), two additions
// per element, a division and a root per token. M = 2048, K = 1152 / 2304 / 4608: 4.6 / 9.0 / 15.1 us with one
// warp, a single chain of additions and the modulation read after the statistics, 4.4 / 7.0 / 11.5 this way;
// M = 32768, K = 1152: 33 us against 18 for DAQ alone (the modulation read at its use there, see the launch).
#include "daq_device.cuh"

namespace dp {

constexpr int kLnThreads = 128;

struct LnArgs {
  const uint16_t* x;
  int64_t M, ldx;
  int K;
  const uint16_t* shift;  // [ceil(M / rows_per_sample)][K] or nullptr (then scale is nullptr too)
  const uint16_t* scale;
  int64_t rows_per_sample;
  float eps;
  int8_t* q;
  int64_t ldq;
  float* s_a;
};

__device__ __forceinline__ float bf16_lo(uint32_t w) { return __uint_as_float(w << 16); }
__device__ __forceinline__ float bf16_hi(uint32_t w) { return __uint_as_float(w & 0xFFFF0000u); }

// two bf16 packed in a word -> two fp32 packed in 64 bits
__device__ __forceinline__ uint64_t bf16x2_to_f32x2(uint32_t w) {
  return (static_cast<uint64_t>(w & 0xFFFF0000u) << 32) | static_cast<uint64_t>(w << 16);
}

// h of the two elements packed in w (modulation words sw, hw when MOD), as packed fp32 operations
// (each half rounded like the scalar instruction); nmean2 = (-mean, -mean), rstd2, one2 likewise.
template <bool MOD>
__device__ __forceinline__ uint64_t ln_pair(uint32_t w, uint32_t sw, uint32_t hw, uint64_t nmean2, uint64_t rstd2,
                                            uint64_t one2) {
  uint64_t h = f32x2_mul(f32x2_add(bf16x2_to_f32x2(w), nmean2), rstd2);  // x - mean is x + (-mean) exactly
  if constexpr (MOD) h = f32x2_fma(h, f32x2_add(one2, bf16x2_to_f32x2(sw)), bf16x2_to_f32x2(hw));
  return h;
}

// RW warps share a row, MAXV = 16-byte vectors held per lane. LATE: the modulation is read where it is used.
template <int RW, int MAXV, bool MOD, bool LATE>
__global__ void __launch_bounds__(kLnThreads) ln_modulate_daq_kernel(const LnArgs a) {
  constexpr int kRows = kLnThreads / 32 / RW, TPR = 32 * RW;
  __shared__ double part1[kLnThreads / 32], part2[kLnThreads / 32];
  __shared__ uint32_t part3[kLnThreads / 32];
  pdl_launch_dependents();
  const int warp = threadIdx.x >> 5;
  const int rw = threadIdx.x / TPR, lane = threadIdx.x % TPR;  // row of the CTA, position in the row
  const int64_t row = static_cast<int64_t>(blockIdx.x) * kRows + rw;
  const bool live = row < a.M;
  const int nvec = live ? a.K >> 3 : 0;
  pdl_wait();
  const uint4* xr = reinterpret_cast<const uint4*>(a.x + row * a.ldx);
  const uint4* shr = nullptr;
  const uint4* scr = nullptr;
  if constexpr (MOD) {
    const int64_t sample = live ? row / a.rows_per_sample : 0;
    shr = reinterpret_cast<const uint4*>(a.shift + sample * a.K);
    scr = reinterpret_cast<const uint4*>(a.scale + sample * a.K);
  }
  uint4 v[MAXV], sh[MAXV], sc[MAXV];  // (unless LATE the modulation's vectors fly beside the row's)
#pragma unroll
  for (int i = 0; i < MAXV; ++i) {
    const int idx = lane + TPR * i;
    v[i] = sh[i] = sc[i] = make_uint4(0, 0, 0, 0);
    if (idx < nvec) {
      ld_stream_u32x4(xr + idx, v[i]);
      if constexpr (MOD && !LATE) {
        sh[i] = ld_global_v4(shr + idx);
        sc[i] = ld_global_v4(scr + idx);
      }
    }
  }
  // ---- token statistics in double, even and odd elements apart (two chains of additions each) ----
  double s1 = 0.0, s2 = 0.0, s1b = 0.0, s2b = 0.0;
#pragma unroll
  for (int i = 0; i < MAXV; ++i) {
    if (lane + TPR * i >= nvec) continue;  // (padding vectors are zero: nothing to add)
    const uint32_t w[4] = {v[i].x, v[i].y, v[i].z, v[i].w};
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const double lo = static_cast<double>(bf16_lo(w[j])), hi = static_cast<double>(bf16_hi(w[j]));
      s1 = __dadd_rn(s1, lo);
      s1b = __dadd_rn(s1b, hi);
      s2 = __fma_rn(lo, lo, s2);
      s2b = __fma_rn(hi, hi, s2b);
    }
  }
  s1 = __dadd_rn(s1, s1b);
  s2 = __dadd_rn(s2, s2b);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    s1 = __dadd_rn(s1, __shfl_xor_sync(0xFFFFFFFFu, s1, o));
    s2 = __dadd_rn(s2, __shfl_xor_sync(0xFFFFFFFFu, s2, o));
  }
  if constexpr (RW > 1) {
    if ((threadIdx.x & 31) == 0) {
      part1[warp] = s1;
      part2[warp] = s2;
    }
    __syncthreads();
    s1 = part1[rw * RW];
    s2 = part2[rw * RW];
#pragma unroll
    for (int w = 1; w < RW; ++w) {
      s1 = __dadd_rn(s1, part1[rw * RW + w]);
      s2 = __dadd_rn(s2, part2[rw * RW + w]);
    }
  }
  const double kd = static_cast<double>(a.K);
  const double mean_d = __ddiv_rn(s1, kd);
  double var_d = __dsub_rn(__ddiv_rn(s2, kd), __dmul_rn(mean_d, mean_d));
  if (var_d < 0.0) var_d = 0.0;
  const float mean = __double2float_rn(mean_d);
  const float rstd = __double2float_rn(__ddiv_rn(1.0, __dsqrt_rn(__dadd_rn(var_d, static_cast<double>(a.eps)))));
  // ---- h and its absmax ----
  const uint64_t nmean2 = f32x2_pack(-mean, -mean), rstd2 = f32x2_pack(rstd, rstd), one2 = f32x2_pack(1.0f, 1.0f);
  uint64_t h[MAXV][4];
  uint32_t amax_bits = 0;  // |h| as an integer: ordered like the value for finite h
#pragma unroll
  for (int i = 0; i < MAXV; ++i) {
    if (lane + TPR * i >= nvec) continue;
    if constexpr (MOD && LATE) {
      sh[i] = ld_global_v4(shr + lane + TPR * i);
      sc[i] = ld_global_v4(scr + lane + TPR * i);
    }
    h[i][0] = ln_pair<MOD>(v[i].x, sc[i].x, sh[i].x, nmean2, rstd2, one2);
    h[i][1] = ln_pair<MOD>(v[i].y, sc[i].y, sh[i].y, nmean2, rstd2, one2);
    h[i][2] = ln_pair<MOD>(v[i].z, sc[i].z, sh[i].z, nmean2, rstd2, one2);
    h[i][3] = ln_pair<MOD>(v[i].w, sc[i].w, sh[i].w, nmean2, rstd2, one2);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      amax_bits = max(amax_bits, static_cast<uint32_t>(h[i][j]) & 0x7FFFFFFFu);
      amax_bits = max(amax_bits, static_cast<uint32_t>(h[i][j] >> 32) & 0x7FFFFFFFu);
    }
  }
  amax_bits = __reduce_max_sync(0xFFFFFFFFu, amax_bits);
  if constexpr (RW > 1) {
    if ((threadIdx.x & 31) == 0) part3[warp] = amax_bits;
    __syncthreads();
#pragma unroll
    for (int w = 0; w < RW; ++w) amax_bits = max(amax_bits, part3[rw * RW + w]);
  }
  if (!live) return;
  const float amax = __uint_as_float(amax_bits);
  float sa = 0.0f, inv = 0.0f;
  if (!(amax < 7.888609052210118e-31f)) {  // 2^-100: below it the token is all-zero, as in the bf16 form
    sa = __fdiv_rn(amax, 127.0f);
    inv = __fdiv_rn(127.0f, amax);
  }
  // ---- quantize: fma(h, inv, 1.5 * 2^23) rounds the exact product once, half to even ----
  const uint64_t inv2 = f32x2_pack(inv, inv), magic2 = f32x2_pack(12582912.0f, 12582912.0f);
  uint2* qrow = reinterpret_cast<uint2*>(a.q + row * a.ldq);
#pragma unroll
  for (int i = 0; i < MAXV; ++i) {
    const int idx = lane + TPR * i;
    if (idx < nvec) {
      uint32_t p[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const uint64_t r = f32x2_fma(h[i][j], inv2, magic2);
        p[j] = __byte_perm(static_cast<uint32_t>(r), static_cast<uint32_t>(r >> 32), 0x0040);  // two codes in the low bytes
      }
      qrow[idx] = make_uint2(__byte_perm(p[0], p[1], 0x5410), __byte_perm(p[2], p[3], 0x5410));
    }
  }
  if (lane == 0) a.s_a[row] = sa;
}

template <int RW, int MAXV, bool LATE = false>
static cudaError_t launch_ln_v(const LnArgs& a, cudaStream_t stream, bool pdl) {
  constexpr int kRows = kLnThreads / 32 / RW;
  const dim3 grid(static_cast<unsigned>((a.M + kRows - 1) / kRows));
  if (a.shift != nullptr) return launch(ln_modulate_daq_kernel<RW, MAXV, true, LATE>, grid, dim3(kLnThreads), 0, stream, pdl, a);
  return launch(ln_modulate_daq_kernel<RW, MAXV, false, LATE>, grid, dim3(kLnThreads), 0, stream, pdl, a);
}

int launch_ln_modulate_daq(const void* x, int64_t M, int64_t K, int64_t ldx, const void* shift, const void* scale,
                           int64_t rows_per_sample, float eps, int8_t* q, int64_t ldq, float* s_a,
                           cudaStream_t stream, bool pdl) {
  if (M == 0) return DP_OK;
  LnArgs a{static_cast<const uint16_t*>(x), M, ldx, static_cast<int>(K), static_cast<const uint16_t*>(shift),
           static_cast<const uint16_t*>(scale), rows_per_sample, eps, q, ldq, s_a};
  // The fewest warps to a row that leave a lane at most five vectors (three for rows that two or four can hold that
  // way), because every warp of a row repeats the statistics' division and root in double. K = 1152, M = 64 / 2056 /
  // 32768: one warp 2.4 / 4.5 / 38 us, two 2.3 / 4.4 / 46, four 2.0 / 5.4 / 62. Up to 512 rows leave SMs idle: four.
  // From 4096 rows on there are warps enough to cover the modulation's way through L2, and what counts is how many fit an
  // SM: it is read where it is used (94 registers otherwise), into as many vectors as the row has. M = 32768, K = 384 /
  // 768 / 1152: read ahead into five vectors 27 / 31 / 37.9 us, this way 18.6 / 23.6 / 33.3 (M = 2048: 2.9 / 3.4 / 4.4 read ahead).
  const cudaError_t e = M <= 512 && K <= 2048 ? launch_ln_v<4, 2>(a, stream, pdl)
                        : M >= 4096 && K <= 256 * 2 ? launch_ln_v<1, 2, true>(a, stream, pdl)
                        : M >= 4096 && K <= 256 * 3 ? launch_ln_v<1, 3, true>(a, stream, pdl)
                        : M >= 4096 && K <= 256 * 4 ? launch_ln_v<1, 4, true>(a, stream, pdl)
                        : M >= 4096 && K <= 256 * 5 ? launch_ln_v<1, 5, true>(a, stream, pdl)
                        : K <= 256 * 5        ? launch_ln_v<1, 5>(a, stream, pdl)
                        : K <= 512 * 3        ? launch_ln_v<2, 3>(a, stream, pdl)
                        : K <= 1024 * 3       ? launch_ln_v<4, 3>(a, stream, pdl)
                                              : launch_ln_v<4, 5>(a, stream, pdl);
  if (e != cudaSuccess) return fail(DP_ERR_CUDA, "LayerNorm + DAQ launch failed: %s", cudaGetErrorString(e));
  return DP_OK;
}

}  // namespace dp
