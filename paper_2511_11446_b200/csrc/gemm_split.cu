// Split-K form of the streaming kernels for layers with fewer output tiles than SMs.
//
// At up to a few hundred tokens a layer has tens of 128 x 64 tiles: most SMs idle while a tile's CTA
// walks all of K, 36 k-blocks for an MLP output layer. Here a cluster of S CTAs shares one tile, each summing its
// share of the k-blocks into its own tensor memory; each CTA finishes an S-th of the outputs and
// is sent the other CTAs' sums of it (stores into its shared memory: pulling them cost a round trip per load). int32 partial sums add up to the same integer whatever the split; the
// bf16 form adds fp32 partial sums in rank order.
// Bound by latency: one tile per cluster, so prologue, first loads, cluster barrier, exchange and stores are all
// exposed (2 us more than an unsplit tile), against the k-blocks saved: K = 4608, N = 1152, M = 48 / 128: 8-bit 9.5 /
// 9.8 -> 7.4 / 7.8 us, 16-bit 11.1 / 12.2 -> 6.9 / 7.5.
//
// Warps: 0 TMA producer of activations, 1 MMA issuer, 2 TMA producer of weights, 4-11 partial sums and outputs.
#include "gemm_device.cuh"

namespace dp {

constexpr int kSplitEpiWarp0 = 4, kSplitThreads = (kSplitEpiWarp0 + kEpiWarps) * 32;
constexpr int kSplitEpiThreads = kEpiWarps * 32;
constexpr int kSplitBN = 64;
// What a CTA receives: all S partial sums of its S-th of the tile, in blocks of 256 pieces of 8 channels (8 KB).
// Of a tile's four blocks a CTA has one (S = 4) or up to two: three CTAs need the most, 3 x 2 blocks.
constexpr int kSplitPartBytes = 3 * 2 * 8192;
constexpr int kSplitStages = (kSmemBudget - kSplitPartBytes) / ab_stage_bytes(kSplitBN);
constexpr size_t kSplitSmemBytes = 1024 + static_cast<size_t>(kSplitStages) * ab_stage_bytes(kSplitBN) + kSplitPartBytes +
                                   (2 * kSplitBN + BM) * 4 + (2 * kSplitStages + 1) * 8 + 16;

__device__ __forceinline__ void st_cluster_v4(uint32_t addr, uint32_t x, uint32_t y, uint32_t z, uint32_t w) {
  asm volatile("st.shared::cluster.v4.u32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(x), "r"(y), "r"(z), "r"(w) : "memory");
}

// F16: bf16 operands and fp32 sums (s_a and s_w unused); else int8 operands.
template <bool F16>
__global__ void __launch_bounds__(kSplitThreads, 1)
gemm_split_kernel(const __grid_constant__ CUtensorMap tmap_a, const __grid_constant__ CUtensorMap tmap_w,
                  const GemmParams p, const int splits) {
  constexpr int BN = kSplitBN, NS = kSplitStages, A_BYTES = BM * BK, B_BYTES = BN * BK;
  constexpr int CH = BN / 8;  // pieces of 8 channels in a token's part of the tile
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* sA = smem;
  uint8_t* sB = sA + NS * A_BYTES;
  // Piece (token r, channels 8c ..) has the number i = r * CH + c and belongs to CTA (i / 256) % S, which holds
  // the S CTAs' sums of its j-th 256 pieces at part[(from * per_cta + j) * 256 + i % 256].
  uint4* part = reinterpret_cast<uint4*>(sB + NS * B_BYTES);
  const int per_cta = (BM * CH / kSplitEpiThreads + splits - 1) / splits;
  float* s_sw = reinterpret_cast<float*>(sB + NS * B_BYTES + kSplitPartBytes);
  float* s_bias = s_sw + BN;
  float* s_sa = s_bias + BN;
  uint64_t* full = reinterpret_cast<uint64_t*>(s_sa + BM);
  uint64_t* empty = full + NS;
  uint64_t* acc_full = empty + NS;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(acc_full + 1);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int rank = static_cast<int>(cluster_ctarank());
  const int tile = blockIdx.x / splits;
  const int n0 = (tile % p.n_tiles) * BN, m_row = (tile / p.n_tiles) * BM;
  const int KB = (F16 ? 2 * p.K : p.K) / BK;
  const int kb0 = rank * KB / splits, kb1 = (rank + 1) * KB / splits;

  if (threadIdx.x == 0) {
    for (int i = 0; i < NS; ++i) {
      mbar_init(&full[i], 2);  // one arrival per producer
      mbar_init(&empty[i], 1);
    }
    mbar_init(acc_full, 1);
    *abort_flag = 0;
    fence_barrier_init();
    tma_prefetch_desc(&tmap_a);
    tma_prefetch_desc(&tmap_w);
  }
  if (warp == 1) {
    tmem_alloc(tmem_slot, BN);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  cluster_arrive_relaxed();  // this CTA has started; waited for before its shared memory is written from outside

  if (threadIdx.x == 96) prefetch_next_reads(p.next);
  if (!p.early_w) pdl_wait();

  if (warp == 0) {
    if (elect_one()) {
      Ring st;
      bool ok = true;
      if (p.early_w && !p.a_ready) pdl_wait();
      for (int kb = kb0; kb < kb1; ++kb) {
        if (!(ok = mbar_spin_wait(&empty[st.s], st.ph ^ 1u, abort_flag))) break;
        mbar_arrive_expect_tx(&full[st.s], A_BYTES);
        int c0 = kb * BK, c1 = m_row;
        if constexpr (!F16) a_tile_coords(p, m_row, kb, c0, c1);
        tma_load_2d(sA + st.s * A_BYTES, &tmap_a, c0, c1, &full[st.s]);
        st.next(NS);
      }
      if (!ok) producer_drain();
    }
  } else if (warp == 1) {
    if (elect_one()) {
      constexpr uint32_t idesc = F16 ? idesc_bf16(BM, BN) : idesc_i8(BM, BN);
      const uint64_t adesc0 = smem_desc_sw128(smem_u32(sA)), bdesc0 = smem_desc_sw128(smem_u32(sB));
      Ring st;
      bool ok = true, full_next = mbar_test_wait(&full[0], 0u);
      for (int kb = kb0; kb < kb1; ++kb) {
        if (!full_next && !(ok = mbar_spin_wait(&full[st.s], st.ph, abort_flag))) break;
        tc_fence_after();
        Ring nx = st;
        nx.next(NS);
        full_next = mbar_test_wait(&full[nx.s], nx.ph);
        const uint64_t adesc = adesc0 + static_cast<uint64_t>(st.s * (A_BYTES >> 4));
        const uint64_t bdesc = bdesc0 + static_cast<uint64_t>(st.s * (B_BYTES >> 4));
#pragma unroll
        for (int k4 = 0; k4 < BK / 32; ++k4) {
          if constexpr (F16)
            mma_bf16_ss(tmem_base, adesc + 2 * k4, bdesc + 2 * k4, idesc, (kb != kb0 || k4 != 0) ? 1u : 0u);
          else
            mma_i8_ss(tmem_base, adesc + 2 * k4, bdesc + 2 * k4, idesc, (kb != kb0 || k4 != 0) ? 1u : 0u);
        }
        mma_commit(&empty[st.s]);
        st = nx;
      }
      if (ok) mma_commit(acc_full);
    }
  } else if (warp == 2) {
    if (elect_one()) {
      Ring st;
      bool ok = true;
      for (int kb = kb0; kb < kb1; ++kb) {
        if (!(ok = mbar_spin_wait(&empty[st.s], st.ph ^ 1u, abort_flag))) break;
        mbar_arrive_expect_tx(&full[st.s], B_BYTES);
        tma_load_w(sB + st.s * B_BYTES, &tmap_w, kb * BK, n0, &full[st.s]);
        st.next(NS);
      }
      if (!ok) producer_drain();
    }
  } else if (warp >= kSplitEpiWarp0) {
    // ================= partial sums: tensor memory -> shared memory, rows of channels in order =================
    const int et = threadIdx.x - kSplitEpiWarp0 * 32, ew = et >> 5, qd = warp & 3;
    if (et < BN) {
      if constexpr (!F16) s_sw[et] = __ldg(p.s_w + n0 + et);
      s_bias[et] = p.bias != nullptr ? __uint_as_float(static_cast<uint32_t>(__ldg(p.bias + n0 + et)) << 16) : 0.0f;
    }
    if (p.early_w) pdl_wait();  // s_a is written by the preceding kernel
    pdl_launch_dependents();  // as in gemm_tc.cu
    if constexpr (!F16) {
      if (et >= 128) s_sa[et - 128] = m_row + et - 128 < p.M ? ld_global_f32(p.s_a + m_row + et - 128) : 0.0f;
    }
    bool ok = mbar_wait(acc_full, 0u, abort_flag);
    ok = __all_sync(0xFFFFFFFFu, ok);
    cluster_wait();
    if (ok) {
      tc_fence_after();
      constexpr int NCOLS = BN / 2;
      const int col0 = (ew >> 2) * NCOLS;
      const uint32_t t_addr = tmem_base + (static_cast<uint32_t>(qd * 32) << 16) + col0;
#pragma unroll
      for (int c = 0; c < NCOLS / 32; ++c)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          uint32_t a[16];
          tmem_ld_16x256b_x4(t_addr + (static_cast<uint32_t>(16 * h) << 16) + c * 32, a);
          tmem_ld_wait();
#pragma unroll
          for (int k = 0; k < 2; ++k) {  // see RowEpilogue for what a lane holds
            const int i = (qd * 32 + 16 * h + 8 * k + (lane >> 2)) * CH + (col0 >> 3) + 4 * c + (lane & 3);
            const int blk = i / kSplitEpiThreads;
            const uint32_t dst = map_to_cta(part + 2 * ((rank * per_cta + blk / splits) * kSplitEpiThreads + i % kSplitEpiThreads),
                                            static_cast<uint32_t>(blk % splits));
            st_cluster_v4(dst, a[2 * k], a[2 * k + 1], a[4 + 2 * k], a[4 + 2 * k + 1]);
            st_cluster_v4(dst + 16, a[8 + 2 * k], a[8 + 2 * k + 1], a[12 + 2 * k], a[12 + 2 * k + 1]);
          }
        }
    }
    tc_fence_before();
  }
  if (warp < kSplitEpiWarp0) {
    __syncwarp();
    cluster_wait();
  }
  __syncwarp();
  cluster_sync();  // every CTA has received its sums (and nothing reaches into another CTA after this)

  if (warp >= kSplitEpiWarp0 && !*abort_flag) {
    // ================= outputs: this CTA's pieces =================
    const int et = threadIdx.x - kSplitEpiWarp0 * 32;
    for (int j = 0; j < per_cta; ++j) {
      const int it = (j * splits + rank) * kSplitEpiThreads + et;
      if (it >= BM * CH) break;
      const int r = it / CH, c = (it % CH) * 8;
      const int64_t row = static_cast<int64_t>(m_row) + r;
      if (row >= p.M) continue;
      const uint16_t* rp = p.res != nullptr ? p.res + row * p.ldr + n0 + c : nullptr;
      uint4 rr = make_uint4(0, 0, 0, 0), gg = rr;
      if (rp != nullptr) rr = ld_global_v4(rp);
      if (rp != nullptr && p.gate != nullptr) gg = ld_global_v4(p.gate + (row / p.rows_per_gate) * p.N + n0 + c);
      uint32_t a[8] = {0, 0, 0, 0, 0, 0, 0, 0};  // (fp32 0 is all zero bits too)
      for (int s = 0; s < splits; ++s) {
        const uint4* src = part + 2 * ((s * per_cta + j) * kSplitEpiThreads + et);
        const uint4 u = src[0], v = src[1];
        const uint32_t x[8] = {u.x, u.y, u.z, u.w, v.x, v.y, v.z, v.w};
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          if constexpr (F16) a[i] = __float_as_uint(__fadd_rn(__uint_as_float(a[i]), __uint_as_float(x[i])));
          else a[i] += x[i];
        }
      }
      uint32_t w[4];
#pragma unroll
      for (int jj = 0; jj < 4; ++jj) {
        float y[2];
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          const int i = 2 * jj + e;
          if constexpr (F16) {
            y[e] = __fadd_rn(__uint_as_float(a[i]), s_bias[c + i]);
          } else {
            y[e] = __fmaf_rn(__int2float_rn(static_cast<int>(a[i])), __fmul_rn(s_sa[r], s_sw[c + i]), s_bias[c + i]);
            if (rp != nullptr) {
              const uint32_t rw = reinterpret_cast<const uint32_t*>(&rr)[jj], gw = reinterpret_cast<const uint32_t*>(&gg)[jj];
              const float rv = __uint_as_float(e ? rw & 0xFFFF0000u : rw << 16);
              y[e] = p.gate != nullptr ? __fmaf_rn(__uint_as_float(e ? gw & 0xFFFF0000u : gw << 16), y[e], rv)
                                       : __fadd_rn(y[e], rv);
            }
          }
        }
        const __nv_bfloat162 v = __floats2bfloat162_rn(y[0], y[1]);
        w[jj] = *reinterpret_cast<const uint32_t*>(&v);
      }
      st_global_v4(p.y + row * p.ldy + n0 + c, w);
    }
  }
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem_base, BN);
  }
  if (threadIdx.x == 0 && *abort_flag && p.status != nullptr) atomicExch(p.status, DP_ERR_TIMEOUT);
}

// ---- host side -------------------------------------------------------------------------------------
// max_clusters[s]: clusters of s CTAs that are resident at once (current device), s = 2 .. kMaxSplits
int gemm_split_init_device(int* max_clusters) {
  DP_CUDA_OK(cudaFuncSetAttribute(gemm_split_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  static_cast<int>(kSplitSmemBytes)));
  DP_CUDA_OK(cudaFuncSetAttribute(gemm_split_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  static_cast<int>(kSplitSmemBytes)));
  for (int s = 0; s <= kMaxSplits; ++s) {
    max_clusters[s] = 0;
    if (s < 2) continue;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(static_cast<unsigned>(s * 64));
    cfg.blockDim = dim3(kSplitThreads);
    cfg.dynamicSmemBytes = kSplitSmemBytes;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = static_cast<unsigned>(s);
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    DP_CUDA_OK(cudaOccupancyMaxActiveClusters(&max_clusters[s], gemm_split_kernel<false>, &cfg));
  }
  return DP_OK;
}

// CTAs to a tile for `tiles` 64-wide tiles of kb k-blocks at per_kb us each (1: not split), and the time saved.
// What the exchange and the wider launch cost, fitted to measurements: 0.9 us and 19 ns per CTA (a launch that
// fills the SMs cannot set up beside its predecessor), 2.1 us at least. 8-bit K = 4608, N = 1152: M = 128, 18 tiles, four CTAs
// 9.7 -> 7.8 us, two 9.0; M = 512, 72 tiles, two 11.2 -> 11.4: not split. 16-bit (twice the k-blocks): M = 256
// three 12.7 -> 9.5, M = 512 two 13.0 -> 11.4. (128-wide tiles, with twice the sums to exchange, only lose.)
int gemm_split_factor(const GemmLimits& lim, int64_t tiles, int kb, double per_kb, double* saved_us) {
  int best = 1;
  *saved_us = 0.0;
  for (int s = 2; s <= kMaxSplits; ++s) {
    const double cost = fmax(2.1, 0.9 + 0.019 * static_cast<double>(tiles * s));
    const double saved = (kb - (kb + s - 1) / s) * per_kb - cost;
    if (tiles <= lim.clusters[s] && saved > *saved_us) {
      best = s;
      *saved_us = saved;
    }
  }
  return best;
}

int launch_gemm_split(const CUtensorMap& tmap_a, const CUtensorMap& tmap_w, GemmParams& p, bool f16, int splits,
                      cudaStream_t stream, bool pdl) {
  const dim3 grid(static_cast<unsigned>(p.m_tiles * p.n_tiles * splits)), block(kSplitThreads);
  p.next = take_next_reads(grid.x);
  const cudaError_t e = launch_cluster(f16 ? gemm_split_kernel<true> : gemm_split_kernel<false>, grid, block,
                                       kSplitSmemBytes, stream, pdl, static_cast<unsigned>(splits), tmap_a, tmap_w, p, splits);
  if (e != cudaSuccess) return fail(DP_ERR_CUDA, "split-K GEMM launch failed: %s", cudaGetErrorString(e));
  return DP_OK;
}

}  // namespace dp
