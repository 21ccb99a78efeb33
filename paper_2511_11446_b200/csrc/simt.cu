// Weight-streaming path of the quantized linear for small row counts (adaLN modulation: M = batch).
//
// The whole layer in one launch, bound by the weight bytes (M <= 32: 2..144 int8 ops per weight
// byte). Form for K > 1152: a CTA owns 32 output channels and up to 8 tokens. Eight lanes share one channel: each
// lane fetches its 32-code units of the packed weight row straight into registers, all loads of a
// pass issued back to back and BEFORE the CTA quantizes its tokens (DAQ, Step 3 Eq. "daq", one
// warp per token, codes to shared memory), so the HBM latency of the weights overlaps the
// prologue. The units are then expanded to int8 in registers, contracted against the shared int8
// tokens with dp4a, reduced over the eight lanes by a transpose-reduction (7 shuffles leave lane j
// with token j's sum) and sent through the dequant epilogue.
//
// For K <= 1152 (every adaLN layer) the contraction instead runs on warp-level int8 matrix
// instructions (m16n8k32 with the tokens as the 16 rows and 8 output channels as the columns), and
// the weights reach the SM as bulk asynchronous copies: eight consecutive weight rows are one
// contiguous run of the packed matrix, which each warp streams through a private ring of
// shared-memory stages, one copy to a stage (completion counted in bytes on its mbarrier), so
// HBM sees a few thousand long sequential streams and the bytes in flight do not depend on
// registers. Lane (g, t) = (lane / 4, lane % 4) reads the units 4j + t of row g from the stage and
// feeds them as B fragments: 8-bit codes as they are; packed 3- and 4-bit codes as UNSIGNED bytes
// that one mask (and at most a short shift) isolates where the field already sits, the power of two
// such a byte carries being common to an accumulator set and shifted out exactly at the end, the
// offset 2^(b-1) leaving as 2^(b-1) times the sum of the token's codes. Because a dot product may
// visit k in any order as long as both operands agree, the A fragments are the same units of tokens
// g and g + 8 from shared memory, staged in the k order the masks produce (row pitch K + 16 keeps
// those 128-bit reads conflict-free).
//
// A single layer of few tokens is a chain of latencies (launch, token, DAQ, contraction, store), not a stream: a
// launch in a chain takes 2.3 us for K = 128, N = 64. K = 1152, N = 6912, one token: 4.7 -> 2.75 us at 4 bits,
// 5.0 -> 3.1 at 3, 6.0 -> 3.0 at 8 (weights alone 0.5 to 1.2 at the copy rate); 16 tokens 8.5 -> 3.8, 32 tokens 9.0 -> 5.2.
// Of that, with 4 bits and one token: the loads of a token all at once 4.7 -> 3.7 (load_token), blocks dealt out
// to all SMs before a second warp of one takes any 3.7 -> 2.8; with 8 bits, one copy to a stage instead of 24
// short ones 4.0 -> 3.0. Short code matters as well: a CTA runs it once, from a cold instruction cache (see
// simt_linear_kernel).
#include <cuda_bf16.h>

#include <algorithm>
#include <type_traits>
#include <utility>

#include "daq_device.cuh"

namespace dp {

constexpr int kSimtRows = 8;        // tokens per CTA
constexpr int kSimtWarps = 8;
constexpr int kSimtLanesPerCh = 8;  // lanes sharing one output channel
constexpr int kSimtChPerCta = kSimtWarps * (32 / kSimtLanesPerCh);
constexpr int kSimtSlots = 5;       // units a lane holds per pass (K = 1152: 36 units / 8 lanes)
// Matrix-instruction form (K <= kMmaMaxK).
constexpr int kMmaMaxK = 1152;         // a token is kTokVec vectors a lane or fewer
constexpr int kMmaWarps = 8;
constexpr int kMmaRows = 16;          // tokens per CTA (the M of m16n8k32)
constexpr int kMmaCh = 8;             // output channels per block (the N of m16n8k32)
constexpr int kMmaMaxStages = 8;
constexpr int kMmaRingBytes = 9600;   // per warp
constexpr int kMmaCtasPerSm = 2;      // by registers (launch bounds) and by the rings, for every K
constexpr int kMmaUnits = kMmaMaxK / 128;  // 32-code units of a row per lane, at most

// Like daq_begin: the first launch of a plan run (hold) lets its dependents start only once everything before the call
// has finished, since they read the layers' constants ahead of their own wait. Other launches let them start at once
// (held back too, a single layer in a chain takes 2.83 us instead of 2.76: K = 1152, N = 6912, 4-bit, one token).
__device__ __forceinline__ void simt_begin(const int early, const int hold) {
  if (hold) pdl_wait();
  pdl_launch_dependents();
  if (!early) pdl_wait();
}

// Packed form of one unit (32 consecutive k of one weight row): BITS words.
template <int BITS>
__device__ __forceinline__ void fetch_unit(const uint32_t* __restrict__ row, int unit, uint32_t (&pk)[BITS]) {
  if constexpr (BITS == 8) {
    const uint4* p = reinterpret_cast<const uint4*>(row) + unit * 2;
    uint4 a, b;
    asm volatile("ld.global.nc.L1::no_allocate.v4.u32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(a.x), "=r"(a.y), "=r"(a.z), "=r"(a.w) : "l"(p));
    asm volatile("ld.global.nc.L1::no_allocate.v4.u32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(b.x), "=r"(b.y), "=r"(b.z), "=r"(b.w) : "l"(p + 1));
    pk[0] = a.x; pk[1] = a.y; pk[2] = a.z; pk[3] = a.w;
    pk[4] = b.x; pk[5] = b.y; pk[6] = b.z; pk[7] = b.w;
  } else if constexpr (BITS == 4) {
    const uint4* p = reinterpret_cast<const uint4*>(row) + unit;
    asm volatile("ld.global.nc.L1::no_allocate.v4.u32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(pk[0]), "=r"(pk[1]), "=r"(pk[2]), "=r"(pk[3]) : "l"(p));
  } else {
    const uint32_t* p = row + unit * 3;
#pragma unroll
    for (int i = 0; i < 3; ++i)
      asm volatile("ld.global.nc.L1::no_allocate.u32 %0, [%1];" : "=r"(pk[i]) : "l"(p + i));
  }
}

// Order in which a token's codes are laid out in shared memory for the matrix-instruction form. The
// contraction may visit k in any order as long as both operands agree, so the activations take the
// order in which cheap mask operations leave the weight codes of a packed unit:
//   ORDER_NATURAL  k ascending (8-bit weights, and the CUDA-core form);
//   ORDER_NIBBLE   within every 8 codes the even positions first, then the odd ones (4-bit: the low
//                  and the high nibbles of a packed word);
//   ORDER_PERIOD   within every 32 codes, word c (c = 0..7) holds positions c, 8 + c, 16 + c, 24 + c
//                  (3-bit: the fields at the same place of the four 3-byte periods of a packed unit).
enum { ORDER_NATURAL = 0, ORDER_NIBBLE = 1, ORDER_PERIOD = 2 };

// Codes 8i .. 8i + 7 of a token, put in that order: the eight bytes to store at 8i. Every lane takes part, lane l
// with an i of l (mod 4): ORDER_PERIOD transposes bytes among the four lanes of a unit (codes 8p .. 8p + 7 go to
// byte p of its eight words; byte stores in place of the two shuffles ran into two-way bank conflicts, 80 cycles
// of the store port for a token of 1152).
template <int ORDER>
__device__ __forceinline__ uint2 arrange_codes(const uint2 v, const int lane) {
  if constexpr (ORDER == ORDER_NATURAL) {
    return v;
  } else if constexpr (ORDER == ORDER_NIBBLE) {
    return make_uint2(__byte_perm(v.x, v.y, 0x6420), __byte_perm(v.x, v.y, 0x7531));
  } else {
    const bool up = (lane & 2) != 0, odd = (lane & 1) != 0;
    // lanes 0, 1 of the unit collect the first words of all four lanes, 2, 3 the second words
    const uint32_t own = up ? v.y : v.x, got = __shfl_xor_sync(0xFFFFFFFFu, up ? v.x : v.y, 2);
    const uint32_t lo = up ? got : own, hi = up ? own : got;  // of lanes (lane & 1) and (lane & 1) + 2
    // even lanes the lower halves, odd lanes the upper ones
    const uint32_t keep = __byte_perm(lo, hi, odd ? 0x7632 : 0x5410);
    const uint32_t other = __shfl_xor_sync(0xFFFFFFFFu, __byte_perm(lo, hi, odd ? 0x5410 : 0x7632), 1);
    const uint32_t e = odd ? other : keep, o = odd ? keep : other;  // lanes 0 and 2, lanes 1 and 3
    return make_uint2(__byte_perm(e, o, 0x6240), __byte_perm(e, o, 0x7351));
  }
}

// Vectors base + lane + 32 j (eight elements each) of a token, zeros beyond its end and for rows that are not
// there. The loads are predicated, not looped over the row: a loop leaves the lanes that have one vector fewer to a
// remainder of one load at a time, and for K = 1152 those four round trips through L2 were the longest phase of
// the kernel (K = 1152, N = 6912, 4-bit, a launch in a chain: M = 1 4.7 -> 3.7 us, M = 16 8.5 -> 5.8).
constexpr int kTokVec = 5;
__device__ __forceinline__ void load_token(const SimtArgs& a, const int64_t row, const int base,
                                           uint4 (&v)[kTokVec]) {
  const int first = base + (threadIdx.x & 31);
  const int left = row < a.M ? (a.K >> 3) - first : 0;
  if (a.s_a_in != nullptr) {
    const uint2* src = reinterpret_cast<const uint2*>(static_cast<const int8_t*>(a.x) + row * a.ldx) + first;
#pragma unroll
    for (int j = 0; j < kTokVec; ++j) {
      const uint2 c = 32 * j < left ? src[32 * j] : make_uint2(0, 0);
      v[j].x = c.x;
      v[j].y = c.y;
    }
  } else {
    const uint4* src = reinterpret_cast<const uint4*>(static_cast<const uint16_t*>(a.x) + row * a.ldx) + first;
#pragma unroll
    for (int j = 0; j < kTokVec; ++j) v[j] = 32 * j < left ? src[32 * j] : make_uint4(0, 0, 0, 0);
  }
}

// Token `slot` of this CTA (row m0 + slot) -> int8 in shared memory, by one warp (rows `pitch` bytes apart), its
// scale and (srs != nullptr) the sum of its codes: DAQ here (Step 3, Eq. "daq"), or the codes as they are when the
// caller passes quantized tokens. v: its first vectors (load_token), all there is of a token unless LONG.
template <int ORDER, bool LONG>
__device__ __forceinline__ void stage_token(const SimtArgs& a, const int64_t m0, const int block_x, int8_t* sq,
                                            const int pitch, float* ssa, const int slot, uint4 (&v)[kTokVec],
                                            int* srs = nullptr) {
  const int lane = threadIdx.x & 31;
  const int64_t row = m0 + slot;
  const int nvec = a.K >> 3;
  uint2* dst = reinterpret_cast<uint2*>(sq + slot * pitch);
  if (row >= a.M) {
    for (int i = lane; i < nvec; i += 32) dst[i] = make_uint2(0, 0);
    if (lane == 0) {
      ssa[slot] = 0.0f;
      if (srs != nullptr) srs[slot] = 0;
    }
    return;
  }
  const bool codes = a.s_a_in != nullptr;
  const bool tap_q = block_x == 0 && a.dbg_q != nullptr;  // optional taps, written once per token
  uint2* dq = tap_q ? reinterpret_cast<uint2*>(a.dbg_q + row * a.dbg_ldq) : nullptr;
  float sc, inv = 0.0f;
  if (codes) {
    sc = a.s_a_in[row];
  } else {
    uint32_t mx = 0;
#pragma unroll
    for (int j = 0; j < kTokVec; ++j)
      mx = absmax_bits2(absmax_bits2(absmax_bits2(absmax_bits2(mx, v[j].x), v[j].y), v[j].z), v[j].w);
    if constexpr (LONG) {
      for (int base = 32 * kTokVec; base < nvec; base += 32 * kTokVec) {
        uint4 u[kTokVec];
        load_token(a, row, base, u);
#pragma unroll
        for (int j = 0; j < kTokVec; ++j)
          mx = absmax_bits2(absmax_bits2(absmax_bits2(absmax_bits2(mx, u[j].x), u[j].y), u[j].z), u[j].w);
      }
    }
    token_scale(__reduce_max_sync(0xFFFFFFFFu, max(mx & 0xFFFFu, mx >> 16)), sc, inv);
  }
  int sum = 0;
  for (int base = 0;;) {
#pragma unroll
    for (int j = 0; j < kTokVec; ++j) {
      const int i = base + lane + 32 * j;
      const uint2 w = codes ? make_uint2(v[j].x, v[j].y) : quant_vec<false>(v[j], inv);
      sum = __dp4a(static_cast<int>(w.x), 0x01010101, __dp4a(static_cast<int>(w.y), 0x01010101, sum));
      const uint2 o = arrange_codes<ORDER>(w, lane);
      if (i < nvec) {
        dst[i] = o;
        if (tap_q) dq[i] = w;
      }
    }
    if constexpr (!LONG) break;
    base += 32 * kTokVec;
    if (base >= nvec) break;
    load_token(a, row, base, v);
  }
  if (srs != nullptr) sum = __reduce_add_sync(0xFFFFFFFFu, sum);
  if (lane == 0) {
    ssa[slot] = sc;
    if (srs != nullptr) srs[slot] = sum;
    if (block_x == 0 && a.dbg_sa != nullptr) a.dbg_sa[row] = sc;
  }
}

template <int BITS>
__device__ __forceinline__ void simt_linear_body(const SimtArgs& a, const int block_x, const int block_y) {
  extern __shared__ __align__(16) uint8_t smem[];
  int8_t* sq = reinterpret_cast<int8_t*>(smem);                       // [kSimtRows][K]
  float* ssa = reinterpret_cast<float*>(smem + kSimtRows * a.K);      // [kSimtRows]
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int sub = lane & (kSimtLanesPerCh - 1);
  const int64_t m0 = static_cast<int64_t>(block_y) * kSimtRows;
  const int K = a.K;
  const int units = K >> 5;
  const int n = block_x * kSimtChPerCta + warp * (32 / kSimtLanesPerCh) + (lane >> 3);
  const bool n_ok = n < a.N;
  const uint32_t* wrow = static_cast<const uint32_t*>(a.qweight) +
                         static_cast<int64_t>(n_ok ? n : 0) * ((K * BITS) >> 5);
  simt_begin(a.early_w, a.hold);

  // ---- first pass of this lane's weight units: in flight across the prologue ----
  uint32_t pk[kSimtSlots][BITS];
#pragma unroll
  for (int i = 0; i < kSimtSlots; ++i) {
    const int u = sub + kSimtLanesPerCh * i;
    if (n_ok && u < units) fetch_unit<BITS>(wrow, u, pk[i]);
  }
  if (a.early_w) pdl_wait();  // the tokens come from the preceding kernel on the stream

  uint4 tok[kTokVec];
  load_token(a, m0 + warp, 0, tok);
  stage_token<ORDER_NATURAL, true>(a, m0, block_x, sq, K, ssa, warp, tok);
  __syncthreads();

  // ---- contraction: passes of kSimtSlots units per lane ----
  int acc[kSimtRows];
#pragma unroll
  for (int m = 0; m < kSimtRows; ++m) acc[m] = 0;
  for (int base = 0; base < units; base += kSimtLanesPerCh * kSimtSlots) {
    if (base != 0) {
#pragma unroll
      for (int i = 0; i < kSimtSlots; ++i) {
        const int u = base + sub + kSimtLanesPerCh * i;
        if (n_ok && u < units) fetch_unit<BITS>(wrow, u, pk[i]);
      }
    }
#pragma unroll
    for (int i = 0; i < kSimtSlots; ++i) {
      const int u = base + sub + kSimtLanesPerCh * i;
      if (n_ok && u < units) {
        uint32_t w[8];
        expand_unit<BITS>(pk[i], w, 1u << (BITS - 1));
#pragma unroll
        for (int m = 0; m < kSimtRows; ++m) {
          const uint4* qp = reinterpret_cast<const uint4*>(sq + m * K + u * 32);
          const uint4 q0 = qp[0], q1 = qp[1];
          int s = acc[m];
          s = __dp4a(static_cast<int>(q0.x), static_cast<int>(w[0]), s);
          s = __dp4a(static_cast<int>(q0.y), static_cast<int>(w[1]), s);
          s = __dp4a(static_cast<int>(q0.z), static_cast<int>(w[2]), s);
          s = __dp4a(static_cast<int>(q0.w), static_cast<int>(w[3]), s);
          s = __dp4a(static_cast<int>(q1.x), static_cast<int>(w[4]), s);
          s = __dp4a(static_cast<int>(q1.y), static_cast<int>(w[5]), s);
          s = __dp4a(static_cast<int>(q1.z), static_cast<int>(w[6]), s);
          s = __dp4a(static_cast<int>(q1.w), static_cast<int>(w[7]), s);
          acc[m] = s;
        }
      }
    }
  }

  // ---- transpose-reduction over the 8 lanes of a channel: lane j ends with token j's sum ----
  {
    const bool hi4 = (sub & 4) != 0;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int send = hi4 ? acc[i] : acc[i + 4];
      const int keep = hi4 ? acc[i + 4] : acc[i];
      acc[i] = keep + __shfl_xor_sync(0xFFFFFFFFu, send, 4);
    }
    const bool hi2 = (sub & 2) != 0;
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const int send = hi2 ? acc[i] : acc[i + 2];
      const int keep = hi2 ? acc[i + 2] : acc[i];
      acc[i] = keep + __shfl_xor_sync(0xFFFFFFFFu, send, 2);
    }
    const bool hi1 = (sub & 1) != 0;
    const int send = hi1 ? acc[0] : acc[1];
    const int keep = hi1 ? acc[1] : acc[0];
    acc[0] = keep + __shfl_xor_sync(0xFFFFFFFFu, send, 1);
  }
  const int64_t row = m0 + sub;
  if (n_ok && row < a.M) {
    const int mine = acc[0];
    const float t = static_cast<float>(mine);
    const float sc = __fmul_rn(ssa[sub], a.s_w[n]);
    const float b = a.bias != nullptr ? __uint_as_float(static_cast<uint32_t>(a.bias[n]) << 16) : 0.0f;
    const float y = __fmaf_rn(t, sc, b);
    a.y[row * a.ldy + n] = __bfloat16_as_ushort(__float2bfloat16_rn(y));
    if (a.dbg_acc != nullptr) a.dbg_acc[row * a.dbg_ldacc + n] = mine;
  }
}

__device__ __forceinline__ void mma_m16n8k32_s8(int (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3,
                                                uint32_t b0, uint32_t b1) {
  asm volatile("mma.sync.aligned.m16n8k32.row.col.s32.s8.s8.s32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
               "{%0, %1, %2, %3};"
               : "+r"(c[0]), "+r"(c[1]), "+r"(c[2]), "+r"(c[3])
               : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// The same with unsigned 8-bit B (weight) operands.
__device__ __forceinline__ void mma_m16n8k32_s8u8(int (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3,
                                                  uint32_t b0, uint32_t b1) {
  asm volatile("mma.sync.aligned.m16n8k32.row.col.s32.s8.u8.s32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
               "{%0, %1, %2, %3};"
               : "+r"(c[0]), "+r"(c[1]), "+r"(c[2]), "+r"(c[3])
               : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// Packed unit `unit` of a staged weight row. 8-bit rows are a multiple of 128 bytes apart, so the lanes of an odd
// row take the two halves of a unit in the other order: every eight lanes then cover all banks.
template <int BITS>
__device__ __forceinline__ void stage_unit(const uint8_t* row, int unit, const bool odd, uint32_t (&pk)[BITS]) {
  if constexpr (BITS == 8) {
    const uint4* p = reinterpret_cast<const uint4*>(row) + unit * 2;
    const uint4 u = p[odd ? 1 : 0], v = p[odd ? 0 : 1];
    pk[0] = odd ? v.x : u.x; pk[1] = odd ? v.y : u.y; pk[2] = odd ? v.z : u.z; pk[3] = odd ? v.w : u.w;
    pk[4] = odd ? u.x : v.x; pk[5] = odd ? u.y : v.y; pk[6] = odd ? u.z : v.z; pk[7] = odd ? u.w : v.w;
  } else if constexpr (BITS == 4) {
    const uint4 u = reinterpret_cast<const uint4*>(row)[unit];
    pk[0] = u.x; pk[1] = u.y; pk[2] = u.z; pk[3] = u.w;
  } else {
    const uint32_t* p = reinterpret_cast<const uint32_t*>(row) + unit * 3;
    pk[0] = p[0]; pk[1] = p[1]; pk[2] = p[2];
  }
}

// Bounded wait without the abort shortcut: lets copies already issued land before a warp that gave
// up leaves its ring.
__device__ __forceinline__ void mbar_drain(uint64_t* bar, uint32_t parity) {
  const long long t0 = clock64();
  while (!mbar_try_wait(bar, parity)) {
    if (clock64() - t0 > (1ll << 26)) return;
  }
}

// Matrix-instruction form (K <= kMmaMaxK). Fragment roles of m16n8k32: A row = token (g and g + 8),
// B column = channel g of the block, D element (token g or g + 8, channels 2t and 2t + 1). The
// instruction's k index of a register is immaterial here: lane (g, t) supplies, for step s of its
// unit, words 2s and 2s + 1 of the unit as the (k-low, k-high) registers of BOTH operands, so every
// k meets its partner exactly once.
// KJ: K / 128 as a constant of the code, or 0 (then it is read from the arguments).
template <int BITS, int KJ>
__device__ __forceinline__ void simt_mma_body(const SimtArgs& a, const int block_x, const int block_y,
                                              const int grid_x) {
  extern __shared__ __align__(16) uint8_t smem[];
  const int K = KJ > 0 ? 128 * KJ : a.K, qpitch = K + 16;
  int8_t* sq = reinterpret_cast<int8_t*>(smem);                             // [kMmaRows][qpitch]
  float* ssa = reinterpret_cast<float*>(smem + kMmaRows * qpitch);          // [kMmaRows]
  volatile int* abort_flag = reinterpret_cast<volatile int*>(ssa + kMmaRows);
  int* srs = reinterpret_cast<int*>(ssa + kMmaRows + 4);                    // [kMmaRows] sums of the tokens' codes
  uint64_t* bars = reinterpret_cast<uint64_t*>(srs + kMmaRows);             // [kMmaWarps][kMmaMaxStages]
  uint8_t* ring = reinterpret_cast<uint8_t*>(bars + kMmaWarps * kMmaMaxStages);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int g = lane >> 2, t = lane & 3;
  const int64_t m0 = static_cast<int64_t>(block_y) * a.rows;
  const bool two = a.rows > 8 && a.M - m0 > 8;  // tokens g + 8 exist
  const int rowbytes = (K * BITS) >> 3;
  const int stage = kMmaCh * rowbytes;
  const int S = min(kMmaMaxStages, kMmaRingBytes / stage);
  uint64_t* bar = bars + warp * kMmaMaxStages;
  uint8_t* myring = ring + warp * kMmaRingBytes;
  const uint8_t* wbase = static_cast<const uint8_t*>(a.qweight);
  const int kj = K >> 7;
  // 8-channel blocks of this warp: blk0, blk0 + stride, ... Every CTA's first warp has one before any CTA's
  // second warp, so that a layer of few blocks is spread over all SMs.
  const int nblocks = a.N / kMmaCh;
  const int stride = grid_x * kMmaWarps;
  const int blk0 = warp * grid_x + block_x;
  const int total = blk0 < nblocks ? (nblocks - blk0 + stride - 1) / stride : 0;

  if (threadIdx.x == 0) *abort_flag = 0;
  if (lane == 0) {
    for (int s = 0; s < S; ++s) mbar_init(&bar[s], 1);
    fence_barrier_init();
  }
  __syncwarp();
  simt_begin(a.early_w, a.hold);

  // Producer side of the ring (lane 0): block i of this warp lands in stage i % S.
  int f_it = 0, f_blk = blk0, f_s = 0;
  auto issue = [&]() {
    if (f_it < total) {
      if (lane == 0) {
        mbar_arrive_expect_tx(&bar[f_s], static_cast<uint32_t>(stage));
        bulk_load_1d(myring + f_s * stage, wbase + static_cast<int64_t>(f_blk) * stage, static_cast<uint32_t>(stage),
                     &bar[f_s]);
      }
      ++f_it;
      if (++f_s == S) f_s = 0;
      f_blk += stride;
    }
  };
  // Weights and tokens are both in flight before either is waited for; the tokens first where they may be read at
  // once (theirs is the longer way: DAQ follows).
  uint4 tok[kMmaRows / kMmaWarps][kTokVec];
  auto load_tokens = [&]() {
    load_token(a, m0 + warp, 0, tok[0]);
    if (two) load_token(a, m0 + warp + kMmaWarps, 0, tok[1]);
  };
  if (!a.early_w) load_tokens();
#pragma unroll 1
  for (int s = 0; s < S; ++s) issue();
  if (a.early_w) {
    pdl_wait();
    load_tokens();
  }
  // Scale and bias of channels 2t, 2t + 1: of the current block, and fetched one block ahead for the
  // next (a load issued at the top of the block it is needed in came back, under a saturated memory
  // system, a couple of thousand cycles later, and its first use stalled the warp for that long).
  float sw[2] = {0.0f, 0.0f}, bs[2] = {0.0f, 0.0f};
  float nsw[2] = {0.0f, 0.0f};
  uint32_t nbs[2] = {0u, 0u};
  auto fetch_scales = [&](const int blk) {
    if (blk < nblocks) {
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        const int n = blk * kMmaCh + 2 * t + e;
        nsw[e] = a.s_w[n];
        nbs[e] = a.bias != nullptr ? static_cast<uint32_t>(a.bias[n]) : 0u;
      }
    }
  };
  auto take_scales = [&]() {
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      sw[e] = nsw[e];
      bs[e] = __uint_as_float(nbs[e] << 16);
    }
  };
  constexpr int ORDER = BITS == 4 ? ORDER_NIBBLE : BITS == 3 ? ORDER_PERIOD : ORDER_NATURAL;
  fetch_scales(blk0);  // of the first block: back by the time the tokens are staged
#pragma unroll 1
  for (int slot = warp; slot < (two ? kMmaRows : kMmaRows / 2); slot += kMmaWarps) {
    stage_token<ORDER, false>(a, m0, block_x, sq, qpitch, ssa, slot, tok[0], srs);
#pragma unroll
    for (int j = 0; j < kTokVec; ++j) tok[0][j] = tok[1][j];  // (one copy of the code: it is executed once)
  }
  __syncthreads();

  // One accumulator set per matrix instruction of a unit: consecutive instructions never wait on each
  // other's results. For packed weights the sets also differ in the power of two their operands
  // carry (see unit_step).
  constexpr int NC = 4;
  int c[NC][4];
#pragma unroll
  for (int i = 0; i < NC; ++i) c[i][0] = c[i][1] = c[i][2] = c[i][3] = 0;
  int c_blk = blk0, st = 0;
  uint32_t ph = 0;
  const int8_t* qrow = sq + g * qpitch + t * 32;
  auto epilogue = [&]() {
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      const int n = c_blk * kMmaCh + 2 * t + e;
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int tok = g + 8 * h;
        const int64_t row = m0 + tok;
        if (row < a.M && (h == 0 || two)) {
          const int i = 2 * h + e;
          // Packed weights enter as unsigned fields u = w + 2^(BITS-1), each set carrying its power of
          // two (the shifts are exact), so the sum of the tokens' codes comes off at the end.
          int mine;
          if constexpr (BITS == 8) mine = c[0][i] + c[1][i] + c[2][i] + c[3][i];
          else if constexpr (BITS == 4) mine = c[0][i] + c[1][i] + ((c[2][i] + c[3][i]) >> 4) - 8 * srs[tok];
          else mine = c[0][i] + c[1][i] + (c[2][i] >> 2) + (c[3][i] >> 4) - 4 * srs[tok];
          const float y = __fmaf_rn(static_cast<float>(mine), __fmul_rn(ssa[tok], sw[e]), bs[e]);
          a.y[row * a.ldy + n] = __bfloat16_as_ushort(__float2bfloat16_rn(y));
          if (a.dbg_acc != nullptr) a.dbg_acc[row * a.dbg_ldacc + n] = mine;
        }
      }
    }
  };
  // One unit (32 codes of this lane's channel) of the staged chunk against tokens g (and g + 8 when
  // TWO). qu: the unit's 32 activation codes of token g in the k order of this bit width.
  auto unit_step = [&](const uint8_t* srow, const int8_t* qu, const int u, auto two_tag) {
    constexpr bool TWO = decltype(two_tag)::value;
    const uint4 l0 = *reinterpret_cast<const uint4*>(qu), l1 = *reinterpret_cast<const uint4*>(qu + 16);
    uint4 h0 = make_uint4(0u, 0u, 0u, 0u), h1 = h0;
    if constexpr (TWO) {
      h0 = *reinterpret_cast<const uint4*>(qu + 8 * qpitch);
      h1 = *reinterpret_cast<const uint4*>(qu + 8 * qpitch + 16);
    }
    uint32_t pk[BITS];
    stage_unit<BITS>(srow, u, (g & 1) != 0, pk);
    if constexpr (BITS == 8) {
      mma_m16n8k32_s8(c[0], l0.x, h0.x, l0.y, h0.y, pk[0], pk[1]);
      mma_m16n8k32_s8(c[1], l0.z, h0.z, l0.w, h0.w, pk[2], pk[3]);
      mma_m16n8k32_s8(c[2], l1.x, h1.x, l1.y, h1.y, pk[4], pk[5]);
      mma_m16n8k32_s8(c[3], l1.z, h1.z, l1.w, h1.w, pk[6], pk[7]);
    } else if constexpr (BITS == 4) {
      // A packed word's low nibbles are its even codes, its high nibbles its odd codes times 16: one
      // mask each, no shifts. Activation words (ORDER_NIBBLE): even, odd codes of word 0, of word 1, ...
      constexpr uint32_t LO = 0x0F0F0F0Fu, HI = 0xF0F0F0F0u;
      mma_m16n8k32_s8u8(c[0], l0.x, h0.x, l0.z, h0.z, pk[0] & LO, pk[1] & LO);
      mma_m16n8k32_s8u8(c[1], l1.x, h1.x, l1.z, h1.z, pk[2] & LO, pk[3] & LO);
      mma_m16n8k32_s8u8(c[2], l0.y, h0.y, l0.w, h0.w, pk[0] & HI, pk[1] & HI);
      mma_m16n8k32_s8u8(c[3], l1.y, h1.y, l1.w, h1.w, pk[2] & HI, pk[3] & HI);
    } else {
      // The 96-bit unit is four periods of three bytes, eight codes each. r0, r1, r2 collect the
      // periods' first, second, third bytes; then the field of code class j (codes j, 8 + j, 16 + j,
      // 24 + j: activation word j under ORDER_PERIOD) sits at the same bits of every byte:
      //   r0: class 0 bits 0-2, class 1 bits 3-5, class 2 (low two bits) bits 6-7
      //   r1: class 2 (high bit) bit 0, class 3 bits 1-3, class 4 bits 4-6, class 5 (low bit) bit 7
      //   r2: class 5 (high two bits) bits 0-1, class 6 bits 2-4, class 7 bits 5-7
      // Masked (and moved by a few bits where that makes two fields carry the same power of two),
      // each field is an unsigned operand byte worth its true value times 1, 4 or 16; the two parts of
      // the straddling classes 2 and 5 are put together first. The contraction is bound by the rate of
      // the matrix instructions, so the few extra logic operations that save a fifth instruction pay.
      const uint32_t x0 = __byte_perm(pk[0], pk[1], 0x0630), x1 = __byte_perm(pk[0], pk[1], 0x0741),
                     x2 = __byte_perm(pk[0], pk[1], 0x0052);
      const uint32_t r0 = __byte_perm(x0, pk[2], 0x5210), r1 = __byte_perm(x1, pk[2], 0x6210),
                     r2 = __byte_perm(x2, pk[2], 0x7410);
      const uint32_t f2 = ((r0 >> 6) & 0x03030303u) | ((r1 & 0x01010101u) << 2);
      const uint32_t f5 = ((r1 >> 7) & 0x01010101u) | ((r2 & 0x03030303u) << 1);
      // times 1: class 0 | class 2;  class 5 | class 7 (moved down)
      mma_m16n8k32_s8u8(c[0], l0.x, h0.x, l0.z, h0.z, r0 & 0x07070707u, f2);
      mma_m16n8k32_s8u8(c[1], l1.y, h1.y, l1.w, h1.w, f5, (r2 >> 5) & 0x07070707u);
      // times 4: class 3 (moved up one bit) | class 6
      mma_m16n8k32_s8u8(c[2], l0.w, h0.w, l1.z, h1.z, (r1 & 0x0E0E0E0Eu) << 1, r2 & 0x1C1C1C1Cu);
      // times 16: class 1 (moved up one bit) | class 4
      mma_m16n8k32_s8u8(c[3], l0.y, h0.y, l1.x, h1.x, (r0 & 0x38383838u) << 1, r1 & 0x70707070u);
    }
  };
  int it = 0;
  for (; it < total; ++it) {
    take_scales();
    fetch_scales(c_blk + stride);
    if (!mbar_wait(&bar[st], ph, abort_flag)) break;
    const uint8_t* srow = myring + st * stage + g * rowbytes;
    auto contract = [&](auto two_tag) {
      int jj = 0;
#pragma unroll 1
      for (; jj + 3 <= kj; jj += 3) {
#pragma unroll
        for (int e = 0; e < 3; ++e) unit_step(srow, qrow + (jj + e) * 128, 4 * (jj + e) + t, two_tag);
      }
#pragma unroll 1
      for (; jj < kj; ++jj) unit_step(srow, qrow + jj * 128, 4 * jj + t, two_tag);
    };
    if (two) {
      contract(std::true_type{});
    } else if constexpr (KJ > 0) {  // up to 8 tokens: written out
#pragma unroll
      for (int jj = 0; jj < KJ; ++jj) unit_step(srow, qrow + jj * 128, 4 * jj + t, std::false_type{});
    } else {
      contract(std::false_type{});
    }
    __syncwarp();  // every lane has consumed the stage: refill it
    issue();
    epilogue();
#pragma unroll
    for (int i = 0; i < NC; ++i) c[i][0] = c[i][1] = c[i][2] = c[i][3] = 0;
    c_blk += stride;
    if (++st == S) { st = 0; ph ^= 1u; }
  }
  // A warp that gave up lets the copies it still has in flight land before the CTA may exit.
  for (; it < f_it; ++it) {
    mbar_drain(&bar[st], ph);
    if (++st == S) { st = 0; ph ^= 1u; }
  }
  __syncthreads();
  if (threadIdx.x == 0 && *abort_flag && a.status != nullptr) atomicExch(a.status, DP_ERR_TIMEOUT);
}

// KJ = K / 128 of the matrix-instruction form, 0: the other form, any K. A kernel for each row length of the first (nine):
// with K a constant the contraction of up to 8 tokens is written out and nothing else is in the code that a launch
// brings in cold. N = 6 K, 8 tokens, K = 384 / 768 / 1024 / 1152 against one kernel with a loop of three units: 4-bit 2.40 /
// 2.51 / 2.86 / 2.97 -> 2.39 / 2.49 / 2.79 / 2.91 us, 8-bit 2.32 / 2.56 / 3.09 / 3.56 -> 2.31 / 2.46 / 2.88 / 3.38.
template <int BITS, int KJ>
__global__ void __launch_bounds__(kSimtWarps * 32, KJ > 0 ? kMmaCtasPerSm : 0)
simt_linear_kernel(SimtArgs a) {
  if constexpr (KJ > 0) simt_mma_body<BITS, KJ>(a, blockIdx.x, blockIdx.y, gridDim.x);
  else simt_linear_body<BITS>(a, blockIdx.x, blockIdx.y);
}

// Several layers of one shape (M, K, N) in one launch: blockIdx.z picks the layer. Used for the
// adaLN modulation linears of a timestep, which are mutually independent and, one at a time, far
// too small (3..8 MB of weights) to fill the GPU for longer than a launch takes.
// DAQ of every token of a group under a policy (percentile clip, a-bit codes; one warp per token, grid = (ceil(M / 8),
// layers)): rows of up to 1280 elements in registers.
__global__ void __launch_bounds__(kSimtWarps * 32)
daq_group_robust_kernel(SimtGroupArgs g) {
  simt_begin(0, g.hold);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t row = static_cast<int64_t>(blockIdx.x) * kSimtWarps + warp;
  if (row >= g.M) return;
  const int layer = blockIdx.y;
  const uint16_t* x = static_cast<const uint16_t*>(g.layer[layer].x) + row * g.K;
  const QRow qr(g.q_scratch + static_cast<int64_t>(layer) * g.M * g.K, row, g.K, 0);
  float sc;
  int sum;
  robust_row<1, 5>(x, g.K, lane, g.daq_rank, static_cast<float>((1 << (g.daq_bits - 1)) - 1), qr, sc, sum);
  if (lane == 0) g.sa_scratch[static_cast<int64_t>(layer) * g.M + row] = sc;
}

template <bool MMA>
__global__ void __launch_bounds__(kSimtWarps * 32, MMA ? kMmaCtasPerSm : 0)
simt_group_kernel(SimtGroupArgs g) {
  SimtArgs a;
  int layer = blockIdx.z, block_x = blockIdx.x, grid_x = gridDim.x;
  if constexpr (MMA) {  // grid.x enumerates (layer, CTA of the layer)
    layer = 0;
    while (static_cast<int>(blockIdx.x) >= g.cta_begin[layer + 1]) ++layer;
    block_x = blockIdx.x - g.cta_begin[layer];
    grid_x = g.cta_begin[layer + 1] - g.cta_begin[layer];
  }
  const SimtGroupArgs::Layer& L = g.layer[layer];
  a.x = L.x;
  a.ldx = g.K;
  a.s_a_in = nullptr;
  if (g.q_scratch != nullptr) {  // tokens already quantized by daq_group_robust_kernel
    a.x = g.q_scratch + static_cast<int64_t>(layer) * g.M * g.K;
    a.s_a_in = g.sa_scratch + static_cast<int64_t>(layer) * g.M;
  }
  a.M = g.M;
  a.rows = kMmaRows;
  a.N = g.N;
  a.K = g.K;
  a.bits = L.bits;
  a.qweight = L.qweight;
  a.s_w = L.s_w;
  a.bias = L.bias;
  a.y = L.y;
  a.ldy = g.N;
  a.dbg_q = nullptr;
  a.dbg_ldq = 0;
  a.dbg_sa = nullptr;
  a.dbg_acc = nullptr;
  a.dbg_ldacc = 0;
  a.early_w = g.early_w;
  a.hold = g.hold;
  a.status = g.status;
  if constexpr (MMA) {
    if (L.bits == 8) simt_mma_body<8, 0>(a, block_x, blockIdx.y, grid_x);
    else if (L.bits == 4) simt_mma_body<4, 0>(a, block_x, blockIdx.y, grid_x);
    else simt_mma_body<3, 0>(a, block_x, blockIdx.y, grid_x);
  } else {
    if (L.bits == 8) simt_linear_body<8>(a, blockIdx.x, blockIdx.y);
    else if (L.bits == 4) simt_linear_body<4>(a, blockIdx.x, blockIdx.y);
    else simt_linear_body<3>(a, blockIdx.x, blockIdx.y);
  }
}

static bool simt_use_mma(int32_t K) { return K <= kMmaMaxK; }
static size_t simt_smem_bytes(int32_t K) {
  if (!simt_use_mma(K)) return static_cast<size_t>(kSimtRows) * K + kSimtRows * sizeof(float);
  return static_cast<size_t>(kMmaRows) * (K + 16) + kMmaRows * sizeof(float) + 16 + kMmaRows * sizeof(int) +
         sizeof(uint64_t) * kMmaWarps * kMmaMaxStages + static_cast<size_t>(kMmaWarps) * kMmaRingBytes;
}

// grid.x of the matrix-instruction form: one CTA per SM while that gives every block a warp of its own, else all
// CTAs that are resident at once (one wave), each warp walking its strided share of the blocks.
static int mma_grid_x(int32_t N, int64_t other_ctas) {
  const int64_t sms = num_sms();
  const int64_t blocks = N / kMmaCh;
  const int64_t room = std::max<int64_t>(1, (blocks * other_ctas <= sms * kMmaWarps ? sms : sms * kMmaCtasPerSm) /
                                                std::max<int64_t>(1, other_ctas));
  return static_cast<int>(std::max<int64_t>(1, std::min(blocks, room)));
}

static_assert(kMmaRingBytes >= kMmaCh * kMmaMaxK, "a stage holds eight whole rows of any bit width");
static_assert(kMmaCtasPerSm * (kMmaWarps * kMmaRingBytes + kMmaRows * (kMmaMaxK + 16) + 2048) <= 227 * 1024,
              "kMmaCtasPerSm CTAs fit an SM's shared memory");
static_assert(kMmaRows == 2 * kMmaWarps && kMmaMaxK <= 256 * kTokVec, "a warp holds its two tokens in registers");

size_t simt_max_k() { return 16384; }

using SimtKernel = void (*)(SimtArgs);
template <int BITS, int... KJ>
static SimtKernel simt_kernel(int kj, std::integer_sequence<int, KJ...>) {
  static constexpr SimtKernel kernels[] = {simt_linear_kernel<BITS, KJ>...};
  return kernels[kj];
}
// The kernel of a bit width, kj = K / 128 of the matrix-instruction form or 0.
static SimtKernel simt_kernel(int bits, int kj) {
  constexpr std::make_integer_sequence<int, kMmaUnits + 1> all;
  return bits == 8 ? simt_kernel<8>(kj, all) : bits == 4 ? simt_kernel<4>(kj, all) : simt_kernel<3>(kj, all);
}

// Once per device: the shared-memory limits of the kernels (a launch that set its own, and asked for the
// occupancy, spent 0.24 us of host time on it: 3.72 -> 3.48 us a call).
int simt_init_device() {
  const int mma = static_cast<int>(simt_smem_bytes(kMmaMaxK)), dp4a = 227 * 1024;
  const auto attr = cudaFuncAttributeMaxDynamicSharedMemorySize;
  for (int bits : {3, 4, 8})
    for (int kj = 0; kj <= kMmaUnits; ++kj) DP_CUDA_OK(cudaFuncSetAttribute(simt_kernel(bits, kj), attr, kj > 0 ? mma : dp4a));
  DP_CUDA_OK(cudaFuncSetAttribute(simt_group_kernel<true>, attr, mma));
  DP_CUDA_OK(cudaFuncSetAttribute(simt_group_kernel<false>, attr, dp4a));
  return DP_OK;
}

size_t simt_group_scratch_bytes(int64_t M, int32_t K, int32_t n_layers) {
  const size_t q = (static_cast<size_t>(n_layers) * M * K + 255) & ~static_cast<size_t>(255);
  return q + ((sizeof(float) * n_layers * M + 255) & ~static_cast<size_t>(255));
}

int launch_simt_group(const SimtGroupArgs& g, cudaStream_t stream, bool pdl) {
  if (g.M == 0 || g.n_layers == 0) return DP_OK;
  if (g.q_scratch != nullptr) {
    const dim3 dgrid(static_cast<unsigned>((g.M + kSimtWarps - 1) / kSimtWarps), static_cast<unsigned>(g.n_layers));
    if (g.K > 1280) return fail(DP_ERR_SHAPE, "grouped DAQ policy: K=%d above 1280", g.K);
    const cudaError_t e = launch(daq_group_robust_kernel, dgrid, dim3(kSimtWarps * 32), 0, stream, pdl, g);
    if (e != cudaSuccess) return fail(DP_ERR_CUDA, "grouped DAQ launch failed: %s", cudaGetErrorString(e));
  }
  const size_t smem = simt_smem_bytes(g.K);
  const bool mma = simt_use_mma(g.K);
  const int rows = mma ? kMmaRows : kSimtRows;
  const int64_t m_groups = (g.M + rows - 1) / rows;
  dim3 grid((g.N + kSimtChPerCta - 1) / kSimtChPerCta, static_cast<unsigned>(m_groups),
            static_cast<unsigned>(g.n_layers));
  const dim3 block(kSimtWarps * 32);
  void (*kern)(SimtGroupArgs) = mma ? simt_group_kernel<true> : simt_group_kernel<false>;
  SimtGroupArgs args = g;
  if (mma) {
    // One wave: the resident-CTA slots are shared out in proportion to the time a CTA of each
    // bit-width needs per channel block, every layer getting at least one CTA (8-bit between 1.4 and
    // 1.75 measures the same, 2.0 and above slower: plan of 64 tokens 829 -> 833 us).
    const int64_t slots = std::max<int64_t>(g.n_layers, static_cast<int64_t>(num_sms()) * kMmaCtasPerSm / m_groups);
    const int full = (g.N / kMmaCh + kMmaWarps - 1) / kMmaWarps;
    double cost[kSimtGroupMax], total = 0.0;
    for (int l = 0; l < g.n_layers; ++l) {
      cost[l] = g.layer[l].bits == 8 ? 1.75 : g.layer[l].bits == 4 ? 1.0 : 1.1;
      total += cost[l];
    }
    int begin = 0;
    double acc = 0.0;
    for (int l = 0; l < g.n_layers; ++l) {  // cumulative rounding: the counts sum to `slots`
      args.cta_begin[l] = begin;
      acc += cost[l];
      const int end = static_cast<int>(acc / total * static_cast<double>(slots) + 0.5);
      begin = std::min(begin + full, std::max(begin + 1, end));
    }
    args.cta_begin[g.n_layers] = begin;
    grid = dim3(static_cast<unsigned>(begin), static_cast<unsigned>(m_groups), 1);
  }
  if (!pdl) args.early_w = 0;
  if (g.q_scratch != nullptr && pdl) args.early_w = 1;  // the preceding kernel is the group's own DAQ
  cudaError_t e = launch(kern, grid, block, smem, stream, pdl, args);
  if (e != cudaSuccess) return fail(DP_ERR_CUDA, "grouped simt launch failed: %s", cudaGetErrorString(e));
  return DP_OK;
}

int launch_simt_linear(const SimtArgs& a, cudaStream_t stream, bool pdl) {
  if (a.M == 0) return DP_OK;
  const size_t smem = simt_smem_bytes(a.K);
  const bool mma = simt_use_mma(a.K);
  // Tokens per CTA: 8 (one to a warp) while that leaves a warp for each (block, token group), else 16, so that the
  // weights are read once for twice the tokens. N = K = 1152, 4-bit: M = 9 3.6 -> 2.4 us, M = 32 3.4 -> 2.5 with
  // groups of 8; N = 6912 M = 16 3.8 either way, and above it the second reading of the weights shows.
  const int rows = mma && a.N / kMmaCh * ((a.M + 7) / 8) > static_cast<int64_t>(num_sms()) * kMmaWarps ? kMmaRows : kSimtRows;
  const int64_t m_groups = (a.M + rows - 1) / rows;
  dim3 grid((a.N + kSimtChPerCta - 1) / kSimtChPerCta, static_cast<unsigned>(m_groups));
  const dim3 block(kSimtWarps * 32);
  const SimtKernel kern = simt_kernel(a.bits, mma ? a.K / 128 : 0);
  if (mma) grid.x = mma_grid_x(a.N, m_groups);
  SimtArgs args = a;
  args.rows = rows;
  if (!pdl) args.early_w = 0;
  cudaError_t e = launch(kern, grid, block, smem, stream, pdl, args);
  if (e != cudaSuccess) return fail(DP_ERR_CUDA, "simt launch failed: %s", cudaGetErrorString(e));
  return DP_OK;
}

}  // namespace dp
