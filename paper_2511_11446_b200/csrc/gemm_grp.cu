// Quantized linear with GROUP-WISE weight scales (and optional zero-points).
//
//   Step 2 of the paper: the GPTQ storage format of its plans keeps one scale and one zero-point per
//   output channel and group of g input channels (g in 32 .. 288), not one scale per channel. With
//   them the int32 accumulator can no longer be dequantized once at the end: every group's partial
//   sum has its own scale. Sequence (the oracle's, bit for bit):
//       acc_G = sum_{k in G} q[m,k] * (u[n,k] - z[n,G])                exact int32
//       t = 0;  for G in order:  t = fma((float)acc_G, s_w[n][G], t)    fp32
//       y = bf16_rne(fma(t, s_a[m], bias[n]))
//
// One persistent CTA per SM walks 128 x 128 output tiles. Warp 0: TMA producer (int8 activation and
// weight tiles, 128 bytes of K per stage). Warps 1 and 2: MMA issuers, which take groups in turn: tcgen05.mma kind::i8 in steps of 32
// bytes of K; the steps of one group accumulate in one of FOUR 128-column tensor-memory buffers, the
// next group starts in the next buffer (group boundaries need not fall on stage boundaries: g = 192
// or 288 span one and a half or two and a quarter stages). Warp 3 brings each group's 128 scales
// into the buffer's slot in shared memory, four groups ahead in registers (they lie ng apart in memory, a
// trip to L2 each; fetched by the folding warps one group ahead they set the pace). Warps 4-11: fold and
// epilogue, 32 tokens and 64 columns per warp in two blocks of 32, read as accumulator fragments (four tokens and eight
// channels of a block to a lane, see RowEpilogue): per block two tcgen05.ld, int32 -> fp32 and fma into 64 fp32 partial
// outputs held in registers, one block read while the other is folded; then the buffer goes back to the issuers; after the
// last group the token scale, bias, bf16 rounding and 16-byte stores.
// Zero-points of 3- and 4-bit layers are taken off when the packed weights are expanded to int8, up to 128 of
// them: u - 128 is the least an int8 holds. Zero-points are bytes, though no quantizer writes one above 2^bits: the
// expansion notes where it met one above 127, the fold warps read the notes while they wait for their first
// accumulators, and if there is one they leave the accumulators alone and sum the codes themselves, (128 - z) *
// rowsum_G[m] included (grp_fold_wide: exact, several times slower, and short of registers on purpose, so that the
// usual fold keeps its own: as a second copy of the fold it cost layers with zero-points up to 7 %). For 8-bit
// codes u - z does not fit a byte at all: the tensor core multiplies by u - 128 and (128 - z[n,G]) * rowsum_G[m] is
// added in int32 before the conversion (form ZP_8BIT, with rowsum from a kernel of its own).
// The fold is what bounds this kernel: the waits of a fold warp for the tensor core are a tenth of its time. 32 values a
// lane and warp, conversion and fma, take a scheduler 104 clocks in a loop of nothing else (packed fma 113, fma without
// the conversion 69), so a 128 x 128 group costs 420 clocks, with the loop around it 680 (g = 128, M = 64), against 560
// for a k-block of the plain kernel with this tile when all SMs load. Counters (K = 1152, N = 3456, g = 128, 4 bits with zero-points,
// M = 8192): issue slots 60 %, ALU pipe 52 %, FMA pipe 22 %, tensor pipe 30 %, DRAM 4 %. Eight warps of 64 columns take
// fewer instructions a value than sixteen of 32 and leave each 168 registers; packed fma needs its operands moved into pairs.
// K = 1152, N = 3456, M = 2048, sixteen warps, packed, one issuer -> this: 4 bits with zero-points, g = 128 19.2 -> 18.8 us, g = 32
// 45.6 -> 44.2; 8 bits, g = 64 27.5 -> 27.0, with zero-points, g = 128, 33.5 -> 29.8; K = 4608, N = 1152, M = 64, 3 bits, g = 32
// 54.0 -> 51.4, 8 bits with zero-points, g = 64, 64.0 -> 55.0; but K = 4608, N = 1152, M = 2048, 4 bits, g = 128 23.1 -> 23.3. Block of
// 4-bit layers with zero-points, g = 128, M = 2048: 91.0 -> 89.9. Over 210 layers (five shapes, 16 to 8192 tokens, 3, 4 and 8 bits, g of 32
// to 128) 1.05 times as fast in the mean, 1.10 to 1.19 with 8 bits and zero-points, 0.98 to 1.02 with g = 128 otherwise. (Tried: accumulators that start at the word of the float
// 1.5 * 2^23, so that an addition in place of the conversion makes the float: the tensor-memory stores cost more, g = 32
// 44 -> 58 us.)
#include "gemm_device.cuh"

namespace dp {

constexpr int kGrpBN = 128;
constexpr int kGrpBufs = 4;
constexpr int kGrpStages = 6;
constexpr int kGrpFoldWarp0 = 4, kGrpFoldWarps = 8;  // (warp & 3) is the tensor-memory quadrant
constexpr int kGrpIssuers = 2, kGrpScaleWarp = 3;  // warps 1 and 2 issue MMAs
constexpr int kGrpCols = kGrpBN / (kGrpFoldWarps / 4);  // columns of a fold warp
constexpr int kGrpThreads = (kGrpFoldWarp0 + kGrpFoldWarps) * 32;
constexpr int kGrpScaleWords = 2 * kGrpBufs * kGrpBN + kGrpFoldWarps * kGrpCols;  // scales, zero-point terms, biases

// Zero-points: none; of 8-bit codes; of packed codes.
enum { ZP_NONE, ZP_8BIT, ZP_PACKED };

struct GrpParams {
  const float* s_a;       // [M]
  const float* s_w;       // [N][ng]
  const uint8_t* zeros;   // [N][ng] (unless ZP_NONE)
  const int32_t* rowsum;  // [M][ng] (ZP_8BIT)
  const int8_t *q, *w8;   // ZP_PACKED: what tmap_a (tiled) and tmap_w read,
  const int32_t* wide;    // and the expansion's notes, n_wide words: nonzero for a zero-point above 127
  int32_t n_wide;
  const uint16_t* bias;
  uint16_t* y;
  int64_t ldy;
  int64_t M;
  int32_t N, K, g, ng, half;  // half = 2^(bits-1)
  int32_t m_tiles, n_tiles, a_tiled;
  int32_t* status;
};

// An MMA issuer's whole run over this CTA's tiles (one thread). The issuers take groups in turn.
template <int U>
__device__ __forceinline__ void grp_issue(const GrpParams& p, const uint8_t* sA, const uint8_t* sB, uint64_t* full,
                                          uint64_t* empty, uint64_t* grp_full, uint64_t* grp_empty, uint32_t tmem_base,
                                          int issuer, volatile int* abort_flag) {
  constexpr uint32_t idesc = idesc_i8(BM, kGrpBN);
  constexpr int NS = kGrpStages;
  const uint64_t adesc0 = smem_desc_sw128(smem_u32(sA)), bdesc0 = smem_desc_sw128(smem_u32(sB));
  const int KB = p.K / BK, total_tiles = p.m_tiles * p.n_tiles;
  const int rpg = (p.g >> 5) / U;  // runs per group
  Ring st, gb;                     // operand stage; group buffer
  bool mine = issuer == 0;         // this issuer takes the current group
  int pos = 0;                     // run inside the current group
  bool full_next = mbar_test_wait(&full[0], 0u);  // polled ahead
  for (int tile = blockIdx.x; tile < total_tiles; tile += gridDim.x) {
    for (int kb = 0; kb < KB; ++kb) {
      if (!full_next && !mbar_spin_wait(&full[st.s], st.ph, abort_flag)) return;
      tc_fence_after();
      Ring nx = st;
      nx.next(NS);
      full_next = mbar_test_wait(&full[nx.s], nx.ph);
      const uint64_t adesc = adesc0 + static_cast<uint64_t>(st.s * ((BM * BK) >> 4));
      const uint64_t bdesc = bdesc0 + static_cast<uint64_t>(st.s * ((kGrpBN * BK) >> 4));
      bool used = false;
#pragma unroll
      for (int u = 0; u < BK / 32 / U; ++u) {
        if (mine) {
          if (pos == 0) {  // a new group: its buffer must have been folded
            if (!mbar_spin_wait(&grp_empty[gb.s], gb.ph ^ 1u, abort_flag)) return;
            tc_fence_after();
          }
          const uint32_t d_tmem = tmem_base + gb.s * kGrpBN;
#pragma unroll
          for (int j = 0; j < U; ++j)
            mma_i8_ss(d_tmem, adesc + 2 * (u * U + j), bdesc + 2 * (u * U + j), idesc, (pos | j) != 0 ? 1u : 0u);
          used = true;
        }
        if (++pos == rpg) {
          if (mine) mma_commit(&grp_full[gb.s]);
          pos = 0;
          mine = !mine;
          gb.next(kGrpBufs);
        }
      }
      if (used) mma_commit(&empty[st.s]);
      else mbar_arrive(&empty[st.s]);  // (the other issuer's alone)
      st = nx;
    }
  }
}

// Shared memory of a CTA.
struct GrpSmem {
  uint8_t *a, *b;  // operand stages
  float* scale;    // [buffer][column] of the group in it
  int32_t* dz;     // the same, 2^(b-1) - z
  float* bias;     // per fold warp: its columns'
  uint64_t *full, *empty, *grp_full, *grp_empty;
  uint32_t* tmem_slot;
  volatile int* abort_flag;
  __device__ __forceinline__ GrpSmem() {
    extern __shared__ uint8_t smem_raw[];
    a = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    b = a + kGrpStages * BM * BK;
    scale = reinterpret_cast<float*>(b + kGrpStages * kGrpBN * BK);
    dz = reinterpret_cast<int32_t*>(scale + kGrpBufs * kGrpBN);
    bias = reinterpret_cast<float*>(dz + kGrpBufs * kGrpBN);
    full = reinterpret_cast<uint64_t*>(scale + kGrpScaleWords);
    empty = full + kGrpStages;
    grp_full = empty + kGrpStages;
    grp_empty = grp_full + kGrpBufs;
    tmem_slot = reinterpret_cast<uint32_t*>(grp_empty + kGrpBufs);
    abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  }
};

// Whether the expansion met a zero-point above 127 (a warp together).
__device__ __forceinline__ bool grp_wide_zeros(const GrpParams& p, int lane) {
  int any = 0;
  for (int i = lane; i < p.n_wide; i += 32 * 8) {  // eight loads in flight, predicated: a loop's remainder goes one by one
    int v[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) v[j] = i + 32 * j < p.n_wide ? ld_global_s32(p.wide + i + 32 * j) : 0;
#pragma unroll
    for (int j = 0; j < 8; ++j) any |= v[j];
  }
  return __any_sync(0xFFFFFFFFu, any != 0);
}

// A fold warp's whole run over this CTA's tiles: quadrant (warp & 3), column half (fw >> 2). A lane folds four tokens and
// eight channels of each of the warp's two 32-column blocks.
template <int ZP>
__device__ __forceinline__ void grp_fold(const GrpParams& p) {
  const GrpSmem sm;
  const float* s_scale = sm.scale;
  const int32_t* s_dz = sm.dz;
  uint64_t *grp_full = sm.grp_full, *grp_empty = sm.grp_empty;
  volatile int* abort_flag = sm.abort_flag;
  const uint32_t tmem_base = *sm.tmem_slot;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int total_tiles = p.m_tiles * p.n_tiles;
  const int fw = warp - kGrpFoldWarp0, qd = warp & 3;
  const int col0 = (fw >> 2) * kGrpCols;
  const int tc = (lane & 3) * 8;  // this lane's channels of a block of 32 (see RowEpilogue)
  float* wb = sm.bias + fw * kGrpCols;
  bool ok = true;
  uint32_t gcount = 0;
  for (int tile = blockIdx.x; tile < total_tiles && ok; tile += gridDim.x) {
    const int n0 = (tile % p.n_tiles) * kGrpBN + col0;
    const int64_t row0 = static_cast<int64_t>(tile / p.n_tiles) * BM + qd * 32 + (lane >> 2);
    bool live[4];
    float sa[4];
    int rs[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      live[i] = row0 + 8 * i < p.M;
      sa[i] = live[i] ? ld_global_f32(p.s_a + row0 + 8 * i) : 0.0f;
      rs[i] = (ZP == ZP_8BIT && live[i]) ? ld_global_s32(p.rowsum + (row0 + 8 * i) * p.ng) : 0;
    }
    __syncwarp();
#pragma unroll
    for (int c = lane; c < kGrpCols; c += 32)
      wb[c] = p.bias != nullptr ? __uint_as_float(static_cast<uint32_t>(__ldg(p.bias + n0 + c)) << 16) : 0.0f;
    float t[2][4][8];  // fp32 partial outputs: block, token row0 + 8 * i, channel tc + j
#pragma unroll
    for (int i = 0; i < 64; ++i) t[i >> 5][(i >> 3) & 3][i & 7] = 0.0f;
    const uint32_t t_row = tmem_base + (static_cast<uint32_t>(qd * 32) << 16) + col0;
    auto wait_group = [&](uint32_t g) {
      ok = mbar_wait(&grp_full[g % kGrpBufs], (g / kGrpBufs) & 1u, abort_flag);
      ok = __all_sync(0xFFFFFFFFu, ok);
      tc_fence_after();
    };
    auto load = [&](uint32_t (&lo)[16], uint32_t (&hi)[16], uint32_t at) {
      tmem_ld_16x256b_x4(at, lo);
      tmem_ld_16x256b_x4(at + (16u << 16), hi);
    };
    auto fold = [&](const uint32_t (&lo)[16], const uint32_t (&hi)[16], int b, uint32_t buf, const int* rs_g) {
      float sc[8];
      int dz[8];
      const float4* s4 = reinterpret_cast<const float4*>(s_scale + buf * kGrpBN + col0 + 32 * b + tc);
      *reinterpret_cast<float4*>(sc) = s4[0];
      *reinterpret_cast<float4*>(sc + 4) = s4[1];
      if constexpr (ZP == ZP_8BIT) {
        const int4* d4 = reinterpret_cast<const int4*>(s_dz + buf * kGrpBN + col0 + 32 * b + tc);
        *reinterpret_cast<int4*>(dz) = d4[0];
        *reinterpret_cast<int4*>(dz + 4) = d4[1];
      }
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const uint32_t(&a)[16] = i < 2 ? lo : hi;
          int a0 = static_cast<int>(a[4 * j + 2 * (i & 1)]), a1 = static_cast<int>(a[4 * j + 2 * (i & 1) + 1]);
          if constexpr (ZP == ZP_8BIT) {
            a0 += dz[2 * j] * rs_g[i];
            a1 += dz[2 * j + 1] * rs_g[i];
          }
          t[b][i][2 * j] = __fmaf_rn(__int2float_rn(a0), sc[2 * j], t[b][i][2 * j]);
          t[b][i][2 * j + 1] = __fmaf_rn(__int2float_rn(a1), sc[2 * j + 1], t[b][i][2 * j + 1]);
        }
    };
    // One block is folded while the next is read, the first of the next group under the second of this one.
    uint32_t lo0[16], hi0[16], lo1[16], hi1[16];
    wait_group(gcount);
    if (!ok) break;
    load(lo0, hi0, t_row + (gcount % kGrpBufs) * kGrpBN);
    for (int G = 0; G < p.ng; ++G, ++gcount) {
      const uint32_t buf = gcount % kGrpBufs;
      int rs_g[4];
      if constexpr (ZP == ZP_8BIT) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          rs_g[i] = rs[i];
          if (live[i] && G + 1 < p.ng) rs[i] = ld_global_s32(p.rowsum + (row0 + 8 * i) * p.ng + G + 1);
        }
      }
      tmem_ld_wait();
      load(lo1, hi1, t_row + buf * kGrpBN + 32);
      fold(lo0, hi0, 0, buf, rs_g);
      tmem_ld_wait();
      tc_fence_before();
      if (G + 1 < p.ng) {
        wait_group(gcount + 1);
        if (!ok) break;
        load(lo0, hi0, t_row + ((gcount + 1) % kGrpBufs) * kGrpBN);
      }
      fold(lo1, hi1, 1, buf, rs_g);
      __syncwarp();  // accumulators and scales have been read: the buffer may take another group
      if (lane == 0) mbar_arrive(&grp_empty[buf]);
    }
    if (!ok) break;
#pragma unroll
    for (int b = 0; b < 2; ++b) {
      float bb[8];
      *reinterpret_cast<float4*>(bb) = *reinterpret_cast<const float4*>(wb + 32 * b + tc);
      *reinterpret_cast<float4*>(bb + 4) = *reinterpret_cast<const float4*>(wb + 32 * b + tc + 4);
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        uint32_t w[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          float y0, y1;
          y0 = __fmaf_rn(t[b][i][2 * j], sa[i], bb[2 * j]);
          y1 = __fmaf_rn(t[b][i][2 * j + 1], sa[i], bb[2 * j + 1]);
          const __nv_bfloat162 v = __floats2bfloat162_rn(y0, y1);
          w[j] = *reinterpret_cast<const uint32_t*>(&v);
        }
        if (live[i]) st_global_v4(p.y + (row0 + 8 * i) * p.ldy + n0 + 32 * b + tc, w);
      }
    }
  }
}
// The same without the accumulators: a lane takes one token, eight channels at a time.
__device__ __forceinline__ void grp_fold_wide(const GrpParams& p) {
  const GrpSmem sm;
  const int fw = (threadIdx.x >> 5) - kGrpFoldWarp0, qd = (threadIdx.x >> 5) & 3, lane = threadIdx.x & 31;
  uint32_t gcount = 0;
  for (int tile = blockIdx.x; tile < p.m_tiles * p.n_tiles; tile += gridDim.x) {
#pragma unroll 1
    for (int G = 0; G < p.ng; ++G, ++gcount) {  // hand the buffers back as they come
      const bool ok = mbar_wait(&sm.grp_full[gcount % kGrpBufs], (gcount / kGrpBufs) & 1u, sm.abort_flag);
      if (!__all_sync(0xFFFFFFFFu, ok)) return;
      if (lane == 0) mbar_arrive(&sm.grp_empty[gcount % kGrpBufs]);
    }
    const int64_t m = static_cast<int64_t>(tile / p.n_tiles) * BM + qd * 32 + lane;
    if (m >= p.M) continue;
    const int8_t* q = p.q + (m >> 7) * (p.K >> 7) * 16384 + (m & 127) * 128;
#pragma unroll 1
    for (int c = 0; c < kGrpCols; c += 8) {
      const int n0 = (tile % p.n_tiles) * kGrpBN + (fw >> 2) * kGrpCols + c;
      float t[8] = {0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll 1
      for (int G = 0; G < p.ng; ++G) {
        int acc[8] = {0, 0, 0, 0, 0, 0, 0, 0}, rs = 0;
#pragma unroll 1
        for (int k = G * p.g; k < (G + 1) * p.g; k += 16) {
          const int4 a = *reinterpret_cast<const int4*>(q + (k >> 7) * 16384 + (k & 127));
          rs = __dp4a(a.x, 0x01010101, __dp4a(a.y, 0x01010101, __dp4a(a.z, 0x01010101, __dp4a(a.w, 0x01010101, rs))));
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            const int4 b = *reinterpret_cast<const int4*>(p.w8 + static_cast<int64_t>(n0 + j) * p.K + k);
            acc[j] = __dp4a(a.x, b.x, __dp4a(a.y, b.y, __dp4a(a.z, b.z, __dp4a(a.w, b.w, acc[j]))));
          }
        }
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          const int64_t at = static_cast<int64_t>(n0 + j) * p.ng + G;
          const int z = p.zeros[at];
          if (z > 128) acc[j] += (128 - z) * rs;
          t[j] = __fmaf_rn(__int2float_rn(acc[j]), p.s_w[at], t[j]);
        }
      }
      uint32_t w[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        float y[2];
#pragma unroll
        for (int e = 0; e < 2; ++e)
          y[e] = __fmaf_rn(t[2 * j + e], p.s_a[m], p.bias != nullptr
                                                       ? __uint_as_float(static_cast<uint32_t>(p.bias[n0 + 2 * j + e]) << 16) : 0.0f);
        const __nv_bfloat162 v = __floats2bfloat162_rn(y[0], y[1]);
        w[j] = *reinterpret_cast<const uint32_t*>(&v);
      }
      st_global_v4(p.y + m * p.ldy + n0, w);
    }
  }
}

template <int ZP>
__global__ void __launch_bounds__(kGrpThreads, 1)
gemm_grp_kernel(const __grid_constant__ CUtensorMap tmap_a, const __grid_constant__ CUtensorMap tmap_w,
                const __grid_constant__ GrpParams p) {
  constexpr int NS = kGrpStages, A_BYTES = BM * BK, B_BYTES = kGrpBN * BK;
  const GrpSmem sm;
  uint8_t *sA = sm.a, *sB = sm.b;
  float* s_scale = sm.scale;
  int32_t* s_dz = sm.dz;
  uint64_t *full = sm.full, *empty = sm.empty, *grp_full = sm.grp_full, *grp_empty = sm.grp_empty;
  uint32_t* tmem_slot = sm.tmem_slot;
  volatile int* abort_flag = sm.abort_flag;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int KB = p.K / BK;
  const int total_tiles = p.m_tiles * p.n_tiles;
  const int spg = p.g >> 5;  // MMA steps (32 bytes of K) per group

  if (threadIdx.x == 0) {
    for (int i = 0; i < NS; ++i) {
      mbar_init(&full[i], 1);
      mbar_init(&empty[i], kGrpIssuers);
    }
    for (int i = 0; i < kGrpBufs; ++i) {
      mbar_init(&grp_full[i], 2);  // the group's MMAs, its scales
      mbar_init(&grp_empty[i], kGrpFoldWarps);
    }
    *abort_flag = 0;
    fence_barrier_init();
    tma_prefetch_desc(&tmap_a);
    tma_prefetch_desc(&tmap_w);
  }
  if (warp == 1) {
    tmem_alloc(tmem_slot, 512);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;

  pdl_launch_dependents();
  pdl_wait();  // activations, scales and the int8 weight copy come from the preceding kernels on the stream

  if (warp == 0) {
    if (elect_one()) {  // see gemm_tc.cu: uniform registers for the single-thread roles
      Ring st;
      bool ok = true, free_next = mbar_test_wait(&empty[0], 1u);
      for (int tile = blockIdx.x; tile < total_tiles && ok; tile += gridDim.x) {
        const int w_row = (tile % p.n_tiles) * kGrpBN, m_row = (tile / p.n_tiles) * BM;
        int c0 = 0, c1 = p.a_tiled ? (m_row >> 7) * KB * BM : m_row;
        const int c0_step = p.a_tiled ? 0 : BK, c1_step = p.a_tiled ? BM : 0;
        for (int kb = 0; kb < KB; ++kb, c0 += c0_step, c1 += c1_step) {
          if (!free_next && !(ok = mbar_spin_wait(&empty[st.s], st.ph ^ 1u, abort_flag))) break;
          Ring nx = st;
          nx.next(NS);
          free_next = mbar_test_wait(&empty[nx.s], nx.ph ^ 1u);  // one k-block ahead
          mbar_arrive_expect_tx(&full[st.s], A_BYTES + B_BYTES);
          tma_load_2d(sA + st.s * A_BYTES, &tmap_a, c0, c1, &full[st.s]);
          tma_load_w(sB + st.s * B_BYTES, &tmap_w, kb * BK, w_row, &full[st.s]);
          st = nx;
        }
      }
      if (!ok) producer_drain();
    }
  } else if (warp < kGrpScaleWarp) {
    if (elect_one()) {
      // Steps are issued in straight-line runs of U, the largest power of two up to a stage's four that divides a group.
      const int issuer = warp - 1;
      if (spg % 4 == 0) grp_issue<4>(p, sA, sB, full, empty, grp_full, grp_empty, tmem_base, issuer, abort_flag);
      else if (spg % 2 == 0) grp_issue<2>(p, sA, sB, full, empty, grp_full, grp_empty, tmem_base, issuer, abort_flag);
      else grp_issue<1>(p, sA, sB, full, empty, grp_full, grp_empty, tmem_base, issuer, abort_flag);
    }
  } else if (warp == kGrpScaleWarp) {
    // ================= scales of each group, columns lane + 32 c =================
    constexpr int AHEAD = 4, C = kGrpBN / 32;
    const int c0 = lane;
    bool ok = true;
    uint32_t gcount = 0;
    for (int tile = blockIdx.x; tile < total_tiles && ok; tile += gridDim.x) {
      const int64_t n0 = (tile % p.n_tiles) * kGrpBN + c0;
      float nx[AHEAD][C];
      int nz[AHEAD][C];
      auto fetch = [&](int G0) {
#pragma unroll
        for (int i = 0; i < AHEAD; ++i)
#pragma unroll
          for (int c = 0; c < C; ++c) {
            const int64_t at = (n0 + 32 * c) * p.ng + G0 + i;
            if (G0 + i < p.ng) {
              nx[i][c] = __ldg(p.s_w + at);
              if constexpr (ZP == ZP_8BIT) nz[i][c] = __ldg(p.zeros + at);
            }
          }
      };
      fetch(0);
      for (int G0 = 0; G0 < p.ng && ok; G0 += AHEAD) {
        float sc[AHEAD][C];
        int dz[AHEAD][C];
#pragma unroll
        for (int i = 0; i < AHEAD; ++i)
#pragma unroll
          for (int c = 0; c < C; ++c) {
            sc[i][c] = nx[i][c];
            if constexpr (ZP == ZP_8BIT) dz[i][c] = p.half - nz[i][c];
          }
        fetch(G0 + AHEAD);
#pragma unroll
        for (int i = 0; i < AHEAD; ++i) {
          if (G0 + i >= p.ng) break;
          const uint32_t buf = gcount % kGrpBufs;
          ok = mbar_wait(&grp_empty[buf], ((gcount / kGrpBufs) & 1u) ^ 1u, abort_flag);
          ok = __all_sync(0xFFFFFFFFu, ok);
          if (!ok) break;
#pragma unroll
          for (int c = 0; c < C; ++c) {
            s_scale[buf * kGrpBN + c0 + 32 * c] = sc[i][c];
            if constexpr (ZP == ZP_8BIT) s_dz[buf * kGrpBN + c0 + 32 * c] = dz[i][c];
          }
          __syncwarp();
          if (lane == 0) mbar_arrive(&grp_full[buf]);
          ++gcount;
        }
      }
    }
  } else {
    // ================= fold + epilogue =================
    if (ZP == ZP_PACKED && grp_wide_zeros(p, lane)) grp_fold_wide(p);
    else grp_fold<ZP == ZP_8BIT ? ZP_8BIT : ZP_NONE>(p);
  }

  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem_base, 512);
  }
  if (threadIdx.x == 0 && *abort_flag && p.status != nullptr) atomicExch(p.status, DP_ERR_TIMEOUT);
}

// Per-group sums of a token's int8 codes, rowsum[m][G] = sum_{k in G} q[m,k] (the zero-point term of the
// fold), from the tiled scratch the DAQ launch wrote ([row tile][k block][128][128]) or a row-major q.
// One warp per token: a lane sums 16 consecutive codes per load (a group is a multiple of 32 codes,
// so the 16 belong to one group) and adds the partial sum to the group's counter in shared memory.
constexpr int kRowsumWarps = 8;
__global__ void __launch_bounds__(kRowsumWarps * 32)
group_rowsum_kernel(const int8_t* __restrict__ q, int64_t M, int K, int64_t ldq, int tiled, int g, int ng,
                    int32_t* __restrict__ rowsum) {
  __shared__ int sums[kRowsumWarps][kGrpZeroMaxGroups];
  pdl_launch_dependents();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t m = static_cast<int64_t>(blockIdx.x) * kRowsumWarps + warp;
  for (int G = lane; G < ng; G += 32) sums[warp][G] = 0;
  __syncwarp();
  pdl_wait();
  if (m >= M) return;
  for (int k = lane * 16; k < K; k += 32 * 16) {
    const int8_t* src = tiled ? q + ((m >> 7) * (K >> 7) + (k >> 7)) * 16384 + (m & 127) * 128 + (k & 127)
                              : q + m * ldq + k;
    const uint4 v = ld_global_v4(src);
    int s = __dp4a(static_cast<int>(v.x), 0x01010101, 0);
    s = __dp4a(static_cast<int>(v.y), 0x01010101, s);
    s = __dp4a(static_cast<int>(v.z), 0x01010101, s);
    s = __dp4a(static_cast<int>(v.w), 0x01010101, s);
    atomicAdd(&sums[warp][k / g], s);
  }
  __syncwarp();
  for (int G = lane; G < ng; G += 32) rowsum[m * ng + G] = sums[warp][G];
}

// ---- host side -------------------------------------------------------------------------------------
constexpr size_t grp_smem_bytes() {
  return 1024 + static_cast<size_t>(kGrpStages) * (BM + kGrpBN) * BK + kGrpScaleWords * 4 +
         (2 * kGrpStages + 2 * kGrpBufs + 1) * 8 + 64;
}

int gemm_grp_init_device() {
  for (auto kernel : {gemm_grp_kernel<ZP_NONE>, gemm_grp_kernel<ZP_8BIT>, gemm_grp_kernel<ZP_PACKED>})
    DP_CUDA_OK(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(grp_smem_bytes())));
  return DP_OK;
}

// q / s_a: the quantized activations (tiled scratch when a_tiled, as packed layers with zero-points need it); w8:
// int8 [N][K], u - 2^(bits-1) of 8-bit codes and of layers without zero-points, else u - min(z, 128); rowsum: scratch
// int32 [M][K/g], used (and filled here) only for 8-bit codes with zero-points. wide: the expansion's notes (packed
// layers with zero-points).
int launch_gemm_grp(const int8_t* q, int64_t ldq, bool a_tiled, const float* s_a, const int8_t* w8, int32_t bits,
                    int32_t g, const float* s_w, const uint8_t* zeros, const uint8_t* wide, const uint16_t* bias,
                    int32_t* rowsum, int64_t M, int32_t N, int32_t K, uint16_t* y, int64_t ldy, int32_t* status, cudaStream_t stream, bool pdl) {
  if (M == 0) return DP_OK;
  if (N % kGrpBN || g <= 0 || g % 32 || K % g)
    return fail(DP_ERR_SHAPE, "group-wise layer: need N %% 128 == 0, g %% 32 == 0, K %% g == 0 (N=%d K=%d g=%d)", N, K, g);
  const int ng = K / g;
  const int form = zeros == nullptr ? ZP_NONE : bits == 8 ? ZP_8BIT : ZP_PACKED;
  if (form == ZP_PACKED && !a_tiled) return fail(DP_ERR_INVALID_ARG, "packed group-wise layer: the codes are not tiled");
  if (form == ZP_8BIT) {
    const cudaError_t e = launch(group_rowsum_kernel, dim3(static_cast<unsigned>((M + kRowsumWarps - 1) / kRowsumWarps)),
                                 dim3(kRowsumWarps * 32), 0, stream, pdl, q, M, static_cast<int>(K), ldq,
                                 a_tiled ? 1 : 0, static_cast<int>(g), ng, rowsum);
    if (e != cudaSuccess) return fail(DP_ERR_CUDA, "group row-sum launch failed: %s", cudaGetErrorString(e));
  }
  CUtensorMap ta, tw;
  int st = a_tiled ? gemm_encode_a_tiled(&ta, q, M, K) : gemm_encode_a(&ta, q, M, K, ldq);
  if (st != DP_OK) return st;
  st = gemm_encode_w(&tw, w8, N, K, 8, kGrpBN, 1);
  if (st != DP_OK) return st;
  GrpParams p;
  p.s_a = s_a;
  p.s_w = s_w;
  p.zeros = zeros;
  p.rowsum = rowsum;
  p.q = q;
  p.w8 = w8;
  p.wide = reinterpret_cast<const int32_t*>(wide);
  p.n_wide = static_cast<int32_t>(unpack_notes(static_cast<int64_t>(N) * K / 32) / 4);
  p.bias = bias;
  p.y = y;
  p.ldy = ldy;
  p.M = M;
  p.N = N;
  p.K = K;
  p.g = g;
  p.ng = ng;
  p.half = 1 << (bits - 1);
  p.m_tiles = static_cast<int32_t>((M + BM - 1) / BM);
  p.n_tiles = N / kGrpBN;
  p.a_tiled = a_tiled ? 1 : 0;
  p.status = status;
  const int64_t tiles = static_cast<int64_t>(p.m_tiles) * p.n_tiles;
  const int sms = num_sms() > 0 ? num_sms() : 148;
  const auto kernel = form == ZP_NONE ? gemm_grp_kernel<ZP_NONE> : form == ZP_8BIT ? gemm_grp_kernel<ZP_8BIT>
                                                                                  : gemm_grp_kernel<ZP_PACKED>;
  const cudaError_t e = launch(kernel, dim3(static_cast<unsigned>(tiles < sms ? tiles : sms)), dim3(kGrpThreads),
                               grp_smem_bytes(), stream, pdl, ta, tw, p);
  if (e != cudaSuccess) return fail(DP_ERR_CUDA, "group-wise GEMM launch failed: %s", cudaGetErrorString(e));
  return DP_OK;
}

}  // namespace dp
