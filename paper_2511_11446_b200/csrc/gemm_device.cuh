// Device-side pieces shared by the tensor-core GEMM kernels of libdiffpro: tile constants, kernel
// parameters, the in-shared-memory expansion of packed 3/4-bit weight tiles, and the dequant
// epilogue of one warp (tcgen05.ld -> fp32 sequence -> bf16 -> 16-byte stores).
#pragma once

#include <cuda_bf16.h>

#include "daq_device.cuh"

namespace dp {

constexpr int BM = 128;
constexpr int BK = 128;  // int8 elements = bytes = one 128-byte swizzle row
constexpr int kEpiWarp0 = 2, kEpiWarps = 8, kUnpackWarp0 = kEpiWarp0 + kEpiWarps, kUnpackWarps = 8;
constexpr int kUnpackThreads = kUnpackWarps * 32;
__host__ __device__ constexpr int gemm_threads(int bits) {
  return (kUnpackWarp0 + (bits == 8 ? 0 : kUnpackWarps)) * 32;
}
constexpr int kSmemBudget = 200 * 1024;
constexpr int kPStages = 3;

// bn below is the number of weight rows ONE CTA holds (BN for CG = 1, BN / 2 for a pair).
__host__ __device__ constexpr int p_stage_bytes(int bn, int bits) {
  return bits == 8 ? 0 : bn * (BK * bits / 8);
}
__host__ __device__ constexpr int ab_stage_bytes(int bn) { return BM * BK + bn * BK; }
__host__ __device__ constexpr int num_stages(int bn, int bits) {
  int n = (kSmemBudget - kPStages * p_stage_bytes(bn, bits)) / ab_stage_bytes(bn);
  return n > 8 ? 8 : n;
}
__host__ __device__ constexpr int tmem_cols(int bn) { return bn <= 64 ? 128 : bn <= 128 ? 256 : 512; }

// Two ranges a later launch will read soon (a plan's next layer's packed weights and its bf16 input):
// each CTA sends its slices on the way into L2 while this kernel, which leaves HBM mostly idle at a
// few thousand tokens, runs. Hints only (L2 is the point of coherence: a range rewritten after the
// hint is simply current when it is read); nullptr: none.
struct NextReads {
  const uint8_t* ptr[2] = {nullptr, nullptr};
  uint32_t bytes[2] = {0, 0}, slice[2] = {0, 0};
};
// One thread of each CTA.
__device__ __forceinline__ void prefetch_next_reads(const NextReads& n) {
#pragma unroll
  for (int r = 0; r < 2; ++r) {
    const uint32_t off = blockIdx.x * n.slice[r];
    if (n.ptr[r] != nullptr && off < n.bytes[r]) {
      const uint32_t len = min(n.slice[r], n.bytes[r] - off);
      for (uint32_t o = 0; o < len; o += 32768u) bulk_prefetch_l2(n.ptr[r] + off + o, min(32768u, len - o));
    }
  }
}
// The ranges given to gemm_set_next_reads by the calling thread, cut into slices for `ctas` CTAs; consumed.
NextReads take_next_reads(unsigned ctas);

struct GemmParams {
  const float* s_a;
  const float* s_w;
  const uint16_t* bias;
  uint16_t* y;
  int64_t ldy;
  int32_t* dbg_acc;
  int64_t dbg_ldacc;
  // Residual taken into the epilogue (res != nullptr): y = bf16(gate ? fma(gate, lin, res) : lin + res)
  // in fp32, lin the value otherwise rounded to bf16. res [M][ldr] bf16 (may be y itself); gate
  // [ceil(M / rows_per_gate)][N] bf16 or nullptr.
  const uint16_t* res;
  int64_t ldr;
  const uint16_t* gate;
  int64_t rows_per_gate;
  int64_t M;
  int32_t N, K;
  int32_t m_tiles, n_tiles;  // m_tiles counts row tiles of 128 * CG tokens
  // In-kernel DAQ (x != nullptr): the kernel quantizes the bf16 activations itself, into the tiled
  // scratch q_out / s_a_out that tmap_a and s_a refer to, and its CTAs tell each other through
  // sync[] (one counter per 128-token tile, then one exit counter; all zero between kernels) which
  // tiles are complete.
  const uint16_t* x;
  int64_t ldx;
  int8_t* q_out;
  float* s_a_out;
  int32_t* sync;
  int32_t sync_tiles;
  int32_t a_tiled;  // activations are stored as contiguous 128 x 128 tiles
  int32_t early_w;  // weights may be fetched before the preceding kernel on the stream has finished
  int32_t a_ready = 0;  // (with early_w) and activations
  int32_t* status;
  NextReads next;
  int32_t dbg_skip_kb = -1;  // test hook (dp_debug_skip_stage_load): k-block whose loads are left out, or -1
};

// TMA coordinates of the activation tile (token row m_row, a multiple of 128; k block kb).
__device__ __forceinline__ void a_tile_coords(const GemmParams& p, int m_row, int kb, int& c0, int& c1) {
  if (p.a_tiled) {
    c0 = 0;
    c1 = ((m_row >> 7) * (p.K / BK) + kb) * BM;
  } else {
    c0 = kb * BK;
    c1 = m_row;
  }
}

// ---- in-kernel DAQ -------------------------------------------------------------------------------
// Every CTA of the grid quantizes an equal share of the tokens (its 8 epilogue warps, one token per
// warp at a time), publishes each finished token on the counter of its 128-token tile, and only
// then turns to its GEMM tiles; the TMA producer of a tile first waits for that tile's counter.
template <bool EO>
__device__ __forceinline__ void daq_phase(const GemmParams& p, int epi_warp, int lane) {
  const int64_t per_cta = (p.M + gridDim.x - 1) / gridDim.x;
  const int64_t r0 = static_cast<int64_t>(blockIdx.x) * per_cta;
  const int64_t r1 = r0 + per_cta < p.M ? r0 + per_cta : p.M;
  const int kb = p.K / BK;
  for (int64_t row = r0 + epi_warp; row < r1; row += 2 * kEpiWarps) {  // two tokens per round
    const int64_t row_b = row + kEpiWarps;
    const bool has_b = row_b < r1;
    const QRow qa(p.q_out, row, 0, kb), qb(p.q_out, has_b ? row_b : row, 0, kb);
    float sc_a, sc_b;
    daq_two_rows_2pass<EO>(p.x + row * p.ldx, p.x + row_b * p.ldx, has_b, p.K, qa, qb, lane, sc_a, sc_b);
    if (lane == 0) {
      p.s_a_out[row] = sc_a;
      if (has_b) p.s_a_out[row_b] = sc_b;
    }
    __syncwarp();
    if (lane == 0) {
      __threadfence();  // the tokens' codes and scales are visible device-wide before they are counted
      if (has_b && (row_b >> 7) == (row >> 7)) {
        atomicAdd(p.sync + (row >> 7), 2);
      } else {
        atomicAdd(p.sync + (row >> 7), 1);
        if (has_b) atomicAdd(p.sync + (row_b >> 7), 1);
      }
    }
  }
}
// One thread: until every token of 128-token tile `t` has been quantized (bounded).
__device__ __forceinline__ bool wait_tile_quantized(const GemmParams& p, int t, volatile int* abort_flag) {
  const int64_t left = p.M - static_cast<int64_t>(t) * BM;
  const int expect = left >= BM ? BM : static_cast<int>(left);
  if (expect <= 0) return true;  // a tile wholly past M: the loads read the fill value
  const long long t0 = clock64();
  uint32_t polls = 0;
  while (ld_acquire_gpu(p.sync + t) < expect) {
    if ((++polls & 15u) == 0) {
      if (*abort_flag) return false;
      if (clock64() - t0 > kWaitBudgetCycles) {
        *abort_flag = 1;
        return false;
      }
    }
  }
  fence_proxy_async_all();  // the codes were written with ordinary stores and are read by TMA next
  return true;
}
// Last thing a CTA does (one thread, after all its roles have finished): count itself out; the last
// CTA of the grid returns every counter to zero for the next kernel.
__device__ __forceinline__ void daq_sync_exit(const GemmParams& p) {
  __threadfence();
  if (atomicAdd(p.sync + p.sync_tiles, 1) == static_cast<int>(gridDim.x) - 1) {
    for (int i = 0; i <= p.sync_tiles; ++i) p.sync[i] = 0;
    __threadfence();
  }
}

int launch_gemm_split(const CUtensorMap& tmap_a, const CUtensorMap& tmap_w, GemmParams& p, bool f16, int splits,
                      cudaStream_t stream, bool pdl);

// A producer that gave up: copies still in flight get a bounded time to land before the CTA exits.
__device__ __forceinline__ void producer_drain() {
  const long long t0 = clock64();
  while (clock64() - t0 < (1ll << 22)) {
  }
}

struct Ring {  // stage index + phase bit of a circular buffer
  int s = 0;
  uint32_t ph = 0;
  __device__ __forceinline__ void next(int n) {
    if (++s == n) {
      s = 0;
      ph ^= 1u;
    }
  }
};

// ---- in-smem weight expansion ------------------------------------------------------------------
// 4-bit: tile P is [BN][64 bytes]; each thread expands 8 bytes (16 codes) into one 16-byte chunk of
// the operand tile B = [BN][128 bytes], chunk position XOR-swizzled by (row & 7).
template <int BN, bool PERM>
__device__ __forceinline__ void unpack4_tile(const uint8_t* P, uint8_t* B, int tid) {
#pragma unroll
  for (int i = 0; i < (BN * 8 + kUnpackThreads - 1) / kUnpackThreads; ++i) {
    const int idx = tid + i * kUnpackThreads;
    if (BN * 8 % kUnpackThreads != 0 && idx >= BN * 8) break;
    const int row = idx >> 3, kc = idx & 7;
    const uint2 in = *reinterpret_cast<const uint2*>(P + row * 64 + kc * 8);
    uint4 o;
    const uint32_t lo0 = ((in.x << 4) & 0xF0F0F0F0u) ^ 0x80808080u;  // even fields
    const uint32_t hi0 = (in.x & 0xF0F0F0F0u) ^ 0x80808080u;         // odd fields
    const uint32_t lo1 = ((in.y << 4) & 0xF0F0F0F0u) ^ 0x80808080u;
    const uint32_t hi1 = (in.y & 0xF0F0F0F0u) ^ 0x80808080u;
    if constexpr (PERM) {
      o = make_uint4(lo0, hi0, lo1, hi1);
    } else {
      o.x = __byte_perm(lo0, hi0, 0x5140);
      o.y = __byte_perm(lo0, hi0, 0x7362);
      o.z = __byte_perm(lo1, hi1, 0x5140);
      o.w = __byte_perm(lo1, hi1, 0x7362);
    }
    *reinterpret_cast<uint4*>(B + row * 128 + ((kc ^ (row & 7)) << 4)) = o;
  }
}

// 3-bit: tile P is [BN][48 bytes]; each thread expands 3 words (32 codes) into two 16-byte chunks.
template <int BN>
__device__ __forceinline__ void unpack3_tile(const uint8_t* P, uint8_t* B, int tid) {
#pragma unroll
  for (int i = 0; i < (BN * 4 + kUnpackThreads - 1) / kUnpackThreads; ++i) {
    const int idx = tid + i * kUnpackThreads;
    if (BN * 4 % kUnpackThreads != 0 && idx >= BN * 4) break;
    const int row = idx >> 2, g = idx & 3;
    const uint32_t* src = reinterpret_cast<const uint32_t*>(P + row * 48 + g * 12);
    uint32_t w[8];
    expand3(src[0], src[1], src[2], 0xE0C0A080u, 0x60402000u, w);  // (u - 4) * 32
    uint8_t* brow = B + row * 128;
    const int sw = row & 7;
    *reinterpret_cast<uint4*>(brow + (((2 * g) ^ sw) << 4)) = make_uint4(w[0], w[1], w[2], w[3]);
    *reinterpret_cast<uint4*>(brow + (((2 * g + 1) ^ sw) << 4)) = make_uint4(w[4], w[5], w[6], w[7]);
  }
}

// ---- epilogue ---------------------------------------------------------------------------------------
// A warp serves its tensor-memory quadrant (32 tokens) over a range of accumulator columns in rounds of 32
// columns x 16 tokens: tcgen05.ld.16x256b.x4 leaves lane (r, t) = (lane / 4, lane % 4) the tokens r and
// r + 8 at columns 8j + 2t + e (j < 4, e < 2), which are the channels 8t .. 8t + 7 of the round, because the
// weight rows were brought in in that order (gemm_encode_w_rows). The next round's read is in flight while
// this one is converted: the fp32 sequence of Step 5 on packed pairs (two independent IEEE operations per
// instruction: int32 -> fp32, sc = s_a * s_w[n], fma(t, sc, bias[n]), bf16 round-to-nearest-even) and one
// 16-byte store per token, a quad covering 64 contiguous bytes of the token's row. Nothing is staged in
// shared memory.
// Why fragments and not one token per thread: a lane needs 8 scales and 8 biases per 4 tokens, four 16-byte
// shared-memory reads, where one token per thread needs sixteen. Such a read, even a broadcast, takes four
// clocks of the 128-byte port that the tensor core's operand reads (and TMA's writes) already keep busy:
// whole 8-bit layers, K = 1152, N = 4608, M = 4096 / 8192: 23.1 / 43.8 us with one token per thread, 20.9 /
// 39.8 this way; K = 384, N = 1536, M = 32768: 44.7 -> 38.0; K = 1152, N = 1152, M = 64: 6.8 -> 6.3.
template <int SHIFT>
struct RowEpilogue {
  static constexpr int CW = 32;         // columns per round
  static constexpr int kMaxCols = 128;  // columns a warp may own (its private copy of scales and biases)
  static constexpr int kScaleBytes = 2 * kMaxCols * 4;
  int qd, lane, staged_col;
  float *tsw, *tbias;
  uint32_t acc_empty_addr0, acc_empty_addr1;

  __device__ __forceinline__ void init(int warp, int lane_, float* scale_copy, uint32_t acc_empty0,
                                       uint32_t acc_empty1) {
    lane = lane_;
    qd = warp & 3;
    tsw = scale_copy;
    tbias = scale_copy + kMaxCols;
    acc_empty_addr0 = acc_empty0;
    acc_empty_addr1 = acc_empty1;
    staged_col = -1;
  }

  // Output columns col .. col + ncols - 1 (col and ncols multiples of 32, ncols at most 128), this
  // CTA's tokens cta_row0 .. +127; their accumulators start at tensor-memory column t_col (buffer
  // `buf`, published on acc_full with phase aph). False if the wait was aborted.
  // reused: another tile will be accumulated in the buffer. Only then is it handed back: the arrival may be a
  // write into the other CTA of a pair, and one that no tile waits for could land after that CTA has exited, on a
  // barrier of the next CTA there.
  // RES: the kernel takes the residual (and gate) of GemmParams into the output; without it those
  // members are ignored.
  template <bool RES = false>
  __device__ __forceinline__ bool tile(const GemmParams& p, int col, int ncols, int cta_row0, uint32_t tmem_base,
                                       uint32_t t_col, uint64_t* acc_full, uint32_t aph, int buf, bool reused,
                                       volatile int* abort_flag) {
    // this lane's tokens: row0 + 8 * i, i < 4; its channels of a round: col + 32 * round + tc .. + 7
    const int64_t row0 = static_cast<int64_t>(cta_row0) + qd * 32 + (lane >> 2);
    const int tc = (lane & 3) * 8;
    const int live = row0 >= p.M ? 0 : static_cast<int>(p.M - row0 > 24 ? 4 : (p.M - row0 + 7) >> 3);  // tokens inside M
    float sa[4];
#pragma unroll
    for (int i = 0; i < 4; ++i)  // from an earlier kernel: fetched while waiting
      sa[i] = (p.x == nullptr && i < live) ? ld_global_f32(p.s_a + row0 + 8 * i) : 0.0f;
    if (col != staged_col) {
      float sv[4], bv[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int c = lane + 32 * j;
        sv[j] = c < ncols ? __ldg(p.s_w + col + c) : 0.0f;
        bv[j] = (c < ncols && p.bias != nullptr)
                    ? __uint_as_float(static_cast<uint32_t>(__ldg(p.bias + col + c)) << 16)
                    : 0.0f;
      }
      __syncwarp();  // the previous sub-block's reads of the copy are done
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        tsw[lane + 32 * j] = sv[j];
        tbias[lane + 32 * j] = bv[j];
      }
      __syncwarp();
      staged_col = col;
    }
    // Residual and gate of this lane's tokens, fetched one round of 32 columns ahead of their use (plain loads:
    // the residual may be the output buffer, whose bytes this thread reads before it overwrites them).
    const bool has_res = RES && p.res != nullptr;
    const bool has_gate = has_res && p.gate != nullptr;
    const uint16_t* rrow = has_res ? p.res + row0 * p.ldr + col + tc : nullptr;
    // The gate rows of the four tokens, once per tile (a 64-bit division each).
    const uint16_t* grow[4] = {nullptr, nullptr, nullptr, nullptr};
    if constexpr (RES) {
#pragma unroll
      for (int i = 0; i < 4; ++i)
        if (has_gate && i < live) grow[i] = p.gate + ((row0 + 8 * i) / p.rows_per_gate) * p.N + col + tc;
    }
    uint4 rn[4], gn[4];
    auto fetch_res = [&](int c) {
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        rn[i] = gn[i] = make_uint4(0, 0, 0, 0);
        if (has_res && i < live) rn[i] = ld_global_v4(rrow + 8 * i * p.ldr + c * CW);
        if (has_gate && i < live) gn[i] = ld_global_v4(grow[i] + c * CW);
      }
    };
    if constexpr (RES) {
      // the later rounds' lines on their way into L2 while the accumulators are still being summed
      const int64_t prow = static_cast<int64_t>(cta_row0) + qd * 32 + lane;
      if (has_res && prow < p.M)
        for (int b = 128; b < ncols * 2; b += 128)
          prefetch_l2(reinterpret_cast<const uint8_t*>(p.res + prow * p.ldr + col) + b);
      fetch_res(0);
    }
    bool ok = mbar_wait(acc_full, aph, abort_flag);
    ok = __all_sync(0xFFFFFFFFu, ok);
    if (!ok) return false;
    tc_fence_after();
    if (p.x != nullptr) {  // scales written by other CTAs of this kernel: their tile is complete by now
      (void)ld_acquire_gpu(p.sync + (cta_row0 >> 7));
#pragma unroll
      for (int i = 0; i < 4; ++i)
        if (i < live) sa[i] = *reinterpret_cast<const volatile float*>(p.s_a + row0 + 8 * i);
    }
    const uint32_t t_addr = tmem_base + (static_cast<uint32_t>(qd * 32) << 16) + t_col;
    uint16_t* yrow = p.y + row0 * p.ldy + col + tc;
    const int rounds = ncols / CW;
    uint32_t lo[16], hi[16];  // tokens 0, 1 and 2, 3 of a round
    float s[8], b[8];
    auto emit = [&](const uint32_t (&a)[16], int c, int i0, const uint4* rr4, const uint4* gg4) {
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        const int i = i0 + k;
        const uint64_t sa2 = f32x2_pack(sa[i], sa[i]);
        uint32_t w[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {  // channels tc + 2j, tc + 2j + 1
          uint64_t t = f32x2_pack(__int2float_rn(static_cast<int>(a[4 * j + 2 * k])),
                                  __int2float_rn(static_cast<int>(a[4 * j + 2 * k + 1])));
          if constexpr (SHIFT != 0)  // exact: the accumulator is a multiple of 2^SHIFT
            t = f32x2_mul(t, f32x2_pack(1.0f / (1 << SHIFT), 1.0f / (1 << SHIFT)));
          float y0, y1;
          f32x2_unpack(f32x2_fma(t, f32x2_mul(sa2, f32x2_pack(s[2 * j], s[2 * j + 1])), f32x2_pack(b[2 * j], b[2 * j + 1])),
                       y0, y1);
          if (RES && has_res) {  // uniform over the grid
            const uint32_t r = reinterpret_cast<const uint32_t*>(&rr4[i])[j];
            const float r0 = __uint_as_float(r << 16), r1 = __uint_as_float(r & 0xFFFF0000u);
            if (has_gate) {
              const uint32_t g = reinterpret_cast<const uint32_t*>(&gg4[i])[j];
              y0 = fmaf(__uint_as_float(g << 16), y0, r0);
              y1 = fmaf(__uint_as_float(g & 0xFFFF0000u), y1, r1);
            } else {
              y0 = __fadd_rn(y0, r0);
              y1 = __fadd_rn(y1, r1);
            }
          }
          const __nv_bfloat162 v = __floats2bfloat162_rn(y0, y1);
          w[j] = *reinterpret_cast<const uint32_t*>(&v);
        }
        if (i < live) {
          if (p.dbg_acc != nullptr) {
            int32_t* arow = p.dbg_acc + (row0 + 8 * i) * p.dbg_ldacc + col + c * CW + tc;
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              arow[2 * j] = static_cast<int>(a[4 * j + 2 * k]) >> SHIFT;
              arow[2 * j + 1] = static_cast<int>(a[4 * j + 2 * k + 1]) >> SHIFT;
            }
          }
          st_global_v4(yrow + 8 * i * p.ldy + c * CW, w);
        }
      }
    };
    tmem_ld_16x256b_x4(t_addr, lo);
    for (int c = 0; c < rounds; ++c) {
      const float4* s4 = reinterpret_cast<const float4*>(tsw + c * CW + tc);
      const float4* b4 = reinterpret_cast<const float4*>(tbias + c * CW + tc);
      *reinterpret_cast<float4*>(s) = s4[0];
      *reinterpret_cast<float4*>(s + 4) = s4[1];
      *reinterpret_cast<float4*>(b) = b4[0];
      *reinterpret_cast<float4*>(b + 4) = b4[1];
      uint4 rr[4], gg[4];
      if constexpr (RES) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          rr[i] = rn[i];
          gg[i] = gn[i];
        }
        if (c + 1 < rounds) fetch_res(c + 1);
      }
      tmem_ld_wait();
      tmem_ld_16x256b_x4(t_addr + (16u << 16) + c * CW, hi);
      emit(lo, c, 0, rr, gg);
      tmem_ld_wait();
      if (c + 1 < rounds) {
        tmem_ld_16x256b_x4(t_addr + (c + 1) * CW, lo);
      } else {  // this warp's last accumulators are in registers: hand the buffer back
        tc_fence_before();
        __syncwarp();
        if (lane == 0 && reused) mbar_arrive_cluster(buf ? acc_empty_addr1 : acc_empty_addr0);
      }
      emit(hi, c, 2, rr, gg);
    }
    return true;
  }
};

}  // namespace dp
