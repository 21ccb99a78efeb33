// Pass-through linear for layers the plan keeps in 16-bit precision: Y = X . W^T + bias, bf16 inputs
// and weights, fp32 accumulation on the tensor cores, bf16 output.
//
//   Step 1 tiering / Step 2 results of the paper: the most sensitive layers are frozen in FP16 (22 of
//   113 in its best plan) and run beside the INT8 ones, so a deployed plan (Algorithm 2, Phase B) must
//   be able to run them in the same call sequence. No DAQ, no weight scales.
//
// One persistent CTA per SM walks 128 x BN output tiles (column tiles of a row strip together). Warp 0:
// TMA producer (activation tiles, the last warp: weight tiles, of 64 bf16 = 128-byte rows, 128-byte swizzle, straight
// from the caller's row-major matrices); warp 1: MMA issuer (tcgen05.mma kind::f16 with bf16 operands,
// fp32 accumulators in tensor memory, two buffers); warps 2-9: epilogue:
// tcgen05.ld -> + bias -> bf16 -> 16-byte stores.
#include "gemm_device.cuh"

namespace dp {

constexpr int kBfWeightWarp = kUnpackWarp0;  // the warp after the epilogue's
constexpr int kBfThreads = (kBfWeightWarp + 1) * 32;
constexpr int kBfBK = 128;  // bytes of K per k-block = 64 bf16

struct BfParams {
  const uint16_t* bias;
  uint16_t* y;
  int64_t ldy;
  int64_t M;
  int32_t N, K;
  int32_t m_tiles, n_tiles;
  int32_t* status;
  NextReads next;
};

__host__ __device__ constexpr int bf_stages(int bn) { return (200 * 1024) / ((BM + bn) * kBfBK); }

template <int BN>
__global__ void __launch_bounds__(kBfThreads, 1)
gemm_bf16_kernel(const __grid_constant__ CUtensorMap tmap_a, const __grid_constant__ CUtensorMap tmap_w,
                 const BfParams p) {
  constexpr int NS = bf_stages(BN) > 8 ? 8 : bf_stages(BN);
  constexpr int A_BYTES = BM * kBfBK, B_BYTES = BN * kBfBK;
  constexpr int TCOLS = tmem_cols(BN);

  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* sA = smem;
  uint8_t* sB = sA + NS * A_BYTES;
  float* s_bias = reinterpret_cast<float*>(sB + NS * B_BYTES);  // per epilogue warp: fp32 copy of its columns' biases
  uint64_t* full = reinterpret_cast<uint64_t*>(s_bias + kEpiWarps * 128);
  uint64_t* empty = full + NS;
  uint64_t* acc_full = empty + NS;
  uint64_t* acc_empty = acc_full + 2;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(acc_empty + 2);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int KB = (p.K * 2) / kBfBK;
  const int total_tiles = p.m_tiles * p.n_tiles;

  if (threadIdx.x == 0) {
    for (int i = 0; i < NS; ++i) {
      mbar_init(&full[i], 2);
      mbar_init(&empty[i], 1);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(&acc_full[i], 1);
      mbar_init(&acc_empty[i], kEpiWarps);
    }
    *abort_flag = 0;
    fence_barrier_init();
    tma_prefetch_desc(&tmap_a);
    tma_prefetch_desc(&tmap_w);
  }
  if (warp == 1) {
    tmem_alloc(tmem_slot, TCOLS);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;

  if (threadIdx.x == kEpiWarp0 * 32) prefetch_next_reads(p.next);
  pdl_wait();  // the activations may come from the preceding kernel on the stream
  pdl_launch_dependents();  // as in gemm_tc.cu

  if (warp == 0) {
    if (elect_one()) {  // see gemm_tc.cu: single-thread roles, activations and weights by a thread each
      Ring st;
      bool ok = true, free_next = mbar_test_wait(&empty[0], 1u);
      for (int tile = blockIdx.x; tile < total_tiles && ok; tile += gridDim.x) {
        const int m_row = (tile / p.n_tiles) * BM;
        for (int kb = 0; kb < KB; ++kb) {
          if (!free_next && !(ok = mbar_spin_wait(&empty[st.s], st.ph ^ 1u, abort_flag))) break;
          Ring nx = st;
          nx.next(NS);
          free_next = mbar_test_wait(&empty[nx.s], nx.ph ^ 1u);  // one k-block ahead
          mbar_arrive_expect_tx(&full[st.s], A_BYTES);
          tma_load_2d(sA + st.s * A_BYTES, &tmap_a, kb * kBfBK, m_row, &full[st.s]);
          st = nx;
        }
      }
      if (!ok) producer_drain();
    }
  } else if (warp == kBfWeightWarp) {
    if (elect_one()) {
      Ring st;
      bool ok = true, free_next = mbar_test_wait(&empty[0], 1u);
      for (int tile = blockIdx.x; tile < total_tiles && ok; tile += gridDim.x) {
        const int w_row = (tile % p.n_tiles) * BN;
        for (int kb = 0; kb < KB; ++kb) {
          if (!free_next && !(ok = mbar_spin_wait(&empty[st.s], st.ph ^ 1u, abort_flag))) break;
          Ring nx = st;
          nx.next(NS);
          free_next = mbar_test_wait(&empty[nx.s], nx.ph ^ 1u);
          mbar_arrive_expect_tx(&full[st.s], B_BYTES);
          tma_load_w(sB + st.s * B_BYTES, &tmap_w, kb * kBfBK, w_row, &full[st.s]);
          st = nx;
        }
      }
      if (!ok) producer_drain();
    }
  } else if (warp == 1) {
    if (elect_one()) {  // see gemm_tc.cu: uniform registers for the single-thread roles
      constexpr uint32_t idesc = idesc_bf16(BM, BN);
      const uint64_t adesc0 = smem_desc_sw128(smem_u32(sA)), bdesc0 = smem_desc_sw128(smem_u32(sB));
      Ring st;
      bool ok = true, full_next = mbar_test_wait(&full[0], 0u);
      int tcount = 0;
      for (int tile = blockIdx.x; tile < total_tiles && ok; tile += gridDim.x, ++tcount) {
        const int buf = tcount & 1;
        if (!(ok = mbar_wait(&acc_empty[buf], ((tcount >> 1) & 1u) ^ 1u, abort_flag))) break;
        tc_fence_after();
        const uint32_t d_tmem = tmem_base + buf * (TCOLS / 2);
        for (int kb = 0; kb < KB; ++kb) {
          if (!full_next && !(ok = mbar_spin_wait(&full[st.s], st.ph, abort_flag))) break;
          tc_fence_after();
          Ring nx = st;
          nx.next(NS);
          full_next = mbar_test_wait(&full[nx.s], nx.ph);
          const uint64_t adesc = adesc0 + static_cast<uint64_t>(st.s * (A_BYTES >> 4));
          const uint64_t bdesc = bdesc0 + static_cast<uint64_t>(st.s * (B_BYTES >> 4));
#pragma unroll
          for (int k4 = 0; k4 < kBfBK / 32; ++k4)  // 16 bf16 = 32 bytes of K per instruction
            mma_bf16_ss(d_tmem, adesc + 2 * k4, bdesc + 2 * k4, idesc, (kb | k4) != 0 ? 1u : 0u);
          mma_commit(&empty[st.s]);
          st = nx;
        }
        if (ok) mma_commit(&acc_full[buf]);
      }
    }
  } else {
    // ================= epilogue: quadrant (warp & 3), column half (ew >> 2) =================
    const int ew = warp - kEpiWarp0, qd = warp & 3;
    constexpr int NCOLS = BN >= 64 ? BN / 2 : BN;  // columns per warp
    const int col0 = (ew >> 2) * NCOLS;
    float* tb = s_bias + ew * 128;
    const int tc = (lane & 3) * 8;  // this lane's channels of a round of 32 (see RowEpilogue)
    bool ok = true;
    int tcount = 0, staged = -1;
    for (int tile = blockIdx.x; tile < total_tiles && ok; tile += gridDim.x, ++tcount) {
      const int buf = tcount & 1;
      const int n0 = (tile % p.n_tiles) * BN + col0;
      const int64_t row0 = static_cast<int64_t>(tile / p.n_tiles) * BM + qd * 32 + (lane >> 2);
      if (n0 != staged) {
        __syncwarp();
        for (int c = lane; c < NCOLS; c += 32)
          tb[c] = p.bias != nullptr ? __uint_as_float(static_cast<uint32_t>(__ldg(p.bias + n0 + c)) << 16) : 0.0f;
        __syncwarp();
        staged = n0;
      }
      ok = mbar_wait(&acc_full[buf], (tcount >> 1) & 1u, abort_flag);
      ok = __all_sync(0xFFFFFFFFu, ok);
      if (!ok) break;
      tc_fence_after();
      const uint32_t t_addr = tmem_base + (static_cast<uint32_t>(qd * 32) << 16) + buf * (TCOLS / 2) + col0;
      uint16_t* yrow = p.y + row0 * p.ldy + n0 + tc;
      uint32_t lo[16], hi[16];
      float bb[8];
      auto emit = [&](const uint32_t (&a)[16], int c, int i0) {  // tokens row0 + 8 * i0, + 8 more
#pragma unroll
        for (int k = 0; k < 2; ++k) {
          uint32_t w[4];
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            const __nv_bfloat162 v = __floats2bfloat162_rn(__fadd_rn(__uint_as_float(a[4 * j + 2 * k]), bb[2 * j]),
                                                           __fadd_rn(__uint_as_float(a[4 * j + 2 * k + 1]), bb[2 * j + 1]));
            w[j] = *reinterpret_cast<const uint32_t*>(&v);
          }
          if (row0 + 8 * (i0 + k) < p.M) st_global_v4(yrow + 8 * (i0 + k) * p.ldy + c * 32, w);
        }
      };
      tmem_ld_16x256b_x4(t_addr, lo);
      for (int c = 0; c < NCOLS / 32; ++c) {
        *reinterpret_cast<float4*>(bb) = *reinterpret_cast<const float4*>(tb + c * 32 + tc);
        *reinterpret_cast<float4*>(bb + 4) = *reinterpret_cast<const float4*>(tb + c * 32 + tc + 4);
        tmem_ld_wait();
        tmem_ld_16x256b_x4(t_addr + (16u << 16) + c * 32, hi);
        emit(lo, c, 0);
        tmem_ld_wait();
        if (c + 1 < NCOLS / 32) {
          tmem_ld_16x256b_x4(t_addr + (c + 1) * 32, lo);
        } else {
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(&acc_empty[buf]);
        }
        emit(hi, c, 2);
      }
    }
  }

  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem_base, TCOLS);
  }
  if (threadIdx.x == 0 && *abort_flag && p.status != nullptr) atomicExch(p.status, DP_ERR_TIMEOUT);
}

// ---- host side -------------------------------------------------------------------------------------
template <int BN>
constexpr size_t bf_smem_bytes() {
  return 1024 + static_cast<size_t>(bf_stages(BN) > 8 ? 8 : bf_stages(BN)) * (BM + BN) * kBfBK + kEpiWarps * 128 * 4 +
         (2 * 8 + 4) * 8 + 64;
}

int gemm_bf16_init_device() {
  DP_CUDA_OK(cudaFuncSetAttribute(gemm_bf16_kernel<64>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  static_cast<int>(bf_smem_bytes<64>())));
  DP_CUDA_OK(cudaFuncSetAttribute(gemm_bf16_kernel<128>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  static_cast<int>(bf_smem_bytes<128>())));
  DP_CUDA_OK(cudaFuncSetAttribute(gemm_bf16_kernel<256>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  static_cast<int>(bf_smem_bytes<256>())));
  return DP_OK;
}

// x bf16 [M][ldx], w bf16 [N][K] (row-major, K contiguous), bias bf16 [N] or null, y bf16 [M][ldy].
// N % 64 == 0, K % 128 == 0 (checked by the caller), pointers 16-byte aligned.
int launch_gemm_bf16(const void* x, int64_t ldx, const void* w, const uint16_t* bias, int64_t M, int32_t N, int32_t K,
                     uint16_t* y, int64_t ldy, int32_t* status, cudaStream_t stream, bool pdl) {
  if (M == 0) return DP_OK;
  int bn = 0, cg = 1, splits = 1;
  gemm_pick_tile(M, N, 2 * K, 16, 0xA, 0, &bn, &cg, &splits);  // a k-block is 128 bytes here too
  CUtensorMap ta, tw;
  int st = gemm_encode_bytes_2d(&ta, x, static_cast<uint64_t>(K) * 2, static_cast<uint64_t>(M),
                                static_cast<uint64_t>(ldx) * 2, kBfBK, BM);
  if (st != DP_OK) return st;
  st = gemm_encode_w_rows(&tw, w, static_cast<uint64_t>(K) * 2, static_cast<uint64_t>(N), kBfBK, bn, true);
  if (st != DP_OK) return st;
  const int32_t m_tiles = static_cast<int32_t>((M + BM - 1) / BM), n_tiles = N / bn;
  if (splits > 1) {
    GemmParams g{};
    g.bias = bias;
    g.y = y;
    g.ldy = ldy;
    g.M = M;
    g.N = N;
    g.K = K;
    g.m_tiles = m_tiles;
    g.n_tiles = n_tiles;
    g.status = status;
    return launch_gemm_split(ta, tw, g, true, splits, stream, pdl);
  }
  BfParams p;
  p.bias = bias;
  p.y = y;
  p.ldy = ldy;
  p.M = M;
  p.N = N;
  p.K = K;
  p.m_tiles = m_tiles;
  p.n_tiles = n_tiles;
  p.status = status;
  const int64_t tiles = static_cast<int64_t>(p.m_tiles) * p.n_tiles;
  const int sms = num_sms() > 0 ? num_sms() : 148;
  const dim3 grid(static_cast<unsigned>(tiles < sms ? tiles : sms)), block(kBfThreads);
  p.next = take_next_reads(grid.x);
  cudaError_t e;
  if (bn == 256) e = launch(gemm_bf16_kernel<256>, grid, block, bf_smem_bytes<256>(), stream, pdl, ta, tw, p);
  else if (bn == 128) e = launch(gemm_bf16_kernel<128>, grid, block, bf_smem_bytes<128>(), stream, pdl, ta, tw, p);
  else e = launch(gemm_bf16_kernel<64>, grid, block, bf_smem_bytes<64>(), stream, pdl, ta, tw, p);
  if (e != cudaSuccess) return fail(DP_ERR_CUDA, "bf16 GEMM launch failed: %s", cudaGetErrorString(e));
  return DP_OK;
}

}  // namespace dp
