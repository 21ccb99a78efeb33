// GEMMs of several layers of a plan in one launch, over one list of tiles.
//
// A layer of a few hundred or thousand tokens is one or two waves of tiles, and a launch of its own pays for the
// hand-over from the kernel before, the first stages' loads, a last wave that is partly empty and the last epilogues:
// at 256 tokens most of its 5.9 us, at 2048 about 4 of 12. Layers that do not read each other's outputs need none of
// that between them. Here a CTA pair walks a run of 256 x bn tiles of each layer in turn (bn 128, 192 or 256 by layer),
// the operand ring and the two accumulator buffers running on across layers; the runs are levelled by the host with the
// tiles' expected times, long contractions first (gemm_plan_schedule).
//
// Operands are int8 (the unit's packed weights have been expanded and its activations quantized by launch_plan_prep,
// kind::i8) or, for layers kept in 16 bits, the caller's bf16 matrices (kind::f16); a k-block is 128 bytes of either.
// A CTA is held to 96 registers a thread: that leaves an SM room for six CTAs of the next unit's preparation (40 registers, 128
// threads), which runs beside this kernel; with 130 and 56 it had room for two and ran after it (28 blocks, mixed
// bits, 2048 tokens: 1050 -> 985 us a step; 1024 tokens with 16-bit layers and the percentile rule 752 -> 700).
// A step of 28 blocks of width 1152, a launch or two a layer -> two a unit of up to 64 MB of operands, the first pass on new inputs /
// passes one behind the other over the same: 256 tokens 715 -> 308 / 659 -> 267 us, 2048 1330 -> 951 / 1363 -> 1086, 1024 (policy, 16-bit
// layers) 1329 -> 648 / 1268 -> 708. Units of 24 / 48 / 64 / 72 MB, two sets of inputs in turn: 256 tokens 287 / 256 / 246 / 246, 2048
// 1100 / 991 / 986 / 998, 1024 663 / 654 / 637 / 637, 4096 (12 blocks) 918 / 827 / 789 / 805. One block on its own (one unit, nothing
// beside its preparation): 256 tokens 32.9 -> 19.9, 4096 77.7 -> 70.4. 16-bit layers take no scratch, so units of any token count:
// four blocks of them, 32768 tokens, 4150 -> 3900.
// What bounds it, by counters of the two kernels launched alone: at 2048 tokens the MMAs (tensor pipe busy 74 % of this kernel's time,
// 54 us to the preparation's 23), at 256 bringing operands in (43 %, 23 us to 17). Through DRAM go 1.5 times the
// bytes that the method must move: of the codes and expanded weights a part leaves L2 before it is read.
// Starting a unit's GEMMs on a count of finished preparation CTAs, ahead of the end of the unit before, was
// tried and left out: it once hung, and why was not found.
// Roles as in gemm_tc.cu: warps 0 and 10 bring in activations and weights, warp 1 of the pair's leader issues the MMAs,
// warps 2-9 convert and store.
#include <algorithm>
#include <iterator>
#include <utility>
#include <vector>

#include "gemm_device.cuh"

namespace dp {

constexpr int kPlanStages = 6, kPlanMaxBN = 256;
constexpr int kPlanStageA = BM * BK, kPlanStageB = kPlanMaxBN / 2 * BK;
constexpr int kPlanWeightWarp = kUnpackWarp0;
constexpr int kPlanThreads = (kPlanWeightWarp + 1) * 32;

// Epilogue of a 16-bit layer's tile: columns col .. col + ncols - 1, tokens cta_row0 .. (see RowEpilogue, whose fragment
// layout and buffer hand-back these are).
__device__ __forceinline__ bool plan_tile_f16(const GemmPlanLayer& L, int col, int ncols, int cta_row0, uint32_t t_addr,
                                              float* tb, bool stage_bias, uint64_t* acc_full, uint32_t aph,
                                              uint32_t acc_empty, bool reused, int lane, int qd, volatile int* abort_flag) {
  const int tc = (lane & 3) * 8;
  const int64_t row0 = static_cast<int64_t>(cta_row0) + qd * 32 + (lane >> 2);
  if (stage_bias) {
    __syncwarp();
    for (int c = lane; c < ncols; c += 32)
      tb[c] = L.bias != nullptr ? __uint_as_float(static_cast<uint32_t>(__ldg(L.bias + col + c)) << 16) : 0.0f;
    __syncwarp();
  }
  bool ok = mbar_wait(acc_full, aph, abort_flag);
  ok = __all_sync(0xFFFFFFFFu, ok);
  if (!ok) return false;
  tc_fence_after();
  uint16_t* yrow = L.y + row0 * L.N + col + tc;
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
      if (row0 + 8 * (i0 + k) < L.M) st_global_v4(yrow + static_cast<int64_t>(8 * (i0 + k)) * L.N + c * 32, w);
    }
  };
  const int rounds = ncols / 32;
  tmem_ld_16x256b_x4(t_addr, lo);
  for (int c = 0; c < rounds; ++c) {
    *reinterpret_cast<float4*>(bb) = *reinterpret_cast<const float4*>(tb + c * 32 + tc);
    *reinterpret_cast<float4*>(bb + 4) = *reinterpret_cast<const float4*>(tb + c * 32 + tc + 4);
    tmem_ld_wait();
    tmem_ld_16x256b_x4(t_addr + (16u << 16) + c * 32, hi);
    emit(lo, c, 0);
    tmem_ld_wait();
    if (c + 1 < rounds) {
      tmem_ld_16x256b_x4(t_addr + (c + 1) * 32, lo);
    } else {
      tc_fence_before();
      __syncwarp();
      if (lane == 0 && reused) mbar_arrive_cluster(acc_empty);
    }
    emit(hi, c, 2);
  }
  return true;
}

__global__ void __maxnreg__(96)
gemm_plan_kernel(const __grid_constant__ GemmPlanParams p) {
  constexpr int NS = kPlanStages;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* sA = smem;
  uint8_t* sB = sA + NS * kPlanStageA;
  float* s_scale = reinterpret_cast<float*>(sB + NS * kPlanStageB);
  uint64_t* full = reinterpret_cast<uint64_t*>(s_scale + kEpiWarps * (RowEpilogue<0>::kScaleBytes / 4));
  uint64_t* empty = full + NS;
  uint64_t* acc_full = empty + NS;
  uint64_t* acc_empty = acc_full + 2;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(acc_empty + 2);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  // The pair's runs and the layers, out of the constant bank: every role reads them at every change of layer, and a miss
  // there is a trip to L2 (left where they are, four or five of them one behind the other kept the MMA issuer waiting).
  GemmPlanRuns* s_runs = reinterpret_cast<GemmPlanRuns*>(tmem_slot + 2);
  GemmPlanLayer* s_layer = reinterpret_cast<GemmPlanLayer*>(s_runs + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = cluster_ctarank();  // 0 = leader of the pair
  {
    const uint32_t* runs = reinterpret_cast<const uint32_t*>(&p.runs[blockIdx.x >> 1]);
    const uint32_t* layers = reinterpret_cast<const uint32_t*>(&p.layer[0]);
    constexpr int kRunWords = sizeof(GemmPlanRuns) / 4, kLayerWords = sizeof(GemmPlanLayer) / 4;
    const int words = kRunWords + kLayerWords * p.n_layers;
    for (int i = threadIdx.x; i < words; i += kPlanThreads)
      reinterpret_cast<uint32_t*>(s_runs)[i] = i < kRunWords ? runs[i] : layers[i - kRunWords];
    if (threadIdx.x >= 64 && threadIdx.x < 64 + 2 * p.n_layers) {
      const int i = threadIdx.x - 64;
      tma_prefetch_desc(i < p.n_layers ? &p.tmap_a[i] : &p.tmap_w[i - p.n_layers]);
    }
  }
  if (threadIdx.x == 0) {
    for (int i = 0; i < NS; ++i) {
      mbar_init(&full[i], 4);  // two producers of each CTA
      mbar_init(&empty[i], 1);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(&acc_full[i], 1);
      mbar_init(&acc_empty[i], 2 * kEpiWarps);
    }
    *abort_flag = 0;
    fence_barrier_init();
  }
  if (warp == 1) {
    tmem_alloc_pair(tmem_slot, 512);
    tmem_relinquish_pair();
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync();  // both CTAs' barriers exist before either signals the other
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;

  pdl_wait();  // codes, scales and expanded weights come from the kernel before

  if (warp == 0 || warp == kPlanWeightWarp) {
    // ================= TMA producers: activations, weights =================
    if (elect_one()) {
      const bool acts = warp == 0;
      Ring st;
      bool ok = true, free_next = mbar_test_wait(&empty[0], 1u);
      const uint32_t full0 = map_to_cta(&full[0], 0);  // both CTAs' bytes are counted on the leader's barrier
      for (int li = 0; li < p.n_layers && ok; ++li) {
        const GemmPlanLayer L = s_layer[li];
        const int kbs = L.kb, n_tiles = L.n_tiles, end = s_runs->end[li];
        for (int tile = s_runs->begin[li]; tile < end && ok; ++tile) {
          if (acts) {
            const int m_row = (tile / n_tiles) * (2 * BM) + static_cast<int>(rank) * BM;
            int a0 = 0, a1 = L.f16 ? m_row : (m_row >> 7) * kbs * BM;
            const int a0_step = L.f16 ? BK : 0, a1_step = L.f16 ? 0 : BM;
            for (int kb = 0; kb < kbs; ++kb, a0 += a0_step, a1 += a1_step) {
              if (!free_next && !(ok = mbar_spin_wait(&empty[st.s], st.ph ^ 1u, abort_flag))) break;
              Ring nx = st;
              nx.next(NS);
              free_next = mbar_test_wait(&empty[nx.s], nx.ph ^ 1u);
              mbar_arrive_expect_tx_cluster(full0 + 8u * st.s, kPlanStageA);
              tma_load_2d_pair(sA + st.s * kPlanStageA, &p.tmap_a[li], a0, a1, full0 + 8u * st.s);
              st = nx;
            }
          } else {
            const int bnl = L.bn >> 1;
            const uint32_t bytes = static_cast<uint32_t>(bnl * BK);
            const int w_row = (tile % n_tiles) * L.bn + static_cast<int>(rank) * bnl;
            for (int kb = 0; kb < kbs; ++kb) {
              if (!free_next && !(ok = mbar_spin_wait(&empty[st.s], st.ph ^ 1u, abort_flag))) break;
              Ring nx = st;
              nx.next(NS);
              free_next = mbar_test_wait(&empty[nx.s], nx.ph ^ 1u);
              mbar_arrive_expect_tx_cluster(full0 + 8u * st.s, bytes);
              tma_load_w_pair(sB + st.s * kPlanStageB, &p.tmap_w[li], kb * BK, w_row, full0 + 8u * st.s);
              st = nx;
            }
          }
        }
      }
      // The last stages' hand-backs are arrivals from the pair's leader that no load waits for: they must have landed before
      // this CTA may exit and another set up its barriers at the same place.
      if (acts)
        for (int i = 0; i < NS && ok; ++i) {
          ok = mbar_spin_wait(&empty[st.s], st.ph ^ 1u, abort_flag);
          st.next(NS);
        }
      if (!ok) producer_drain();
    }
  } else if (warp == 1) {
    // ================= MMA issuer (the pair's leader) =================
    if (rank == 0 && elect_one()) {
      const uint64_t adesc0 = smem_desc_sw128(smem_u32(sA)), bdesc0 = smem_desc_sw128(smem_u32(sB));
      Ring st;
      bool ok = true, full_next = mbar_test_wait(&full[0], 0u);
      int tcount = 0;
      for (int li = 0; li < p.n_layers && ok; ++li) {
        const GemmPlanLayer L = s_layer[li];
        const int kbs = L.kb, end = s_runs->end[li];
        const uint32_t idesc = (L.f16 ? idesc_bf16(2 * BM, 0) : idesc_i8(2 * BM, 0)) | (static_cast<uint32_t>(L.bn >> 3) << 17);
        const bool f16 = L.f16 != 0;
        for (int tile = s_runs->begin[li]; tile < end && ok; ++tile, ++tcount) {
          const int buf = tcount & 1;
          if (!(ok = mbar_spin_wait(&acc_empty[buf], ((tcount >> 1) & 1u) ^ 1u, abort_flag))) break;
          tc_fence_after();
          const uint32_t d_tmem = tmem_base + buf * 256;
          for (int kb = 0; kb < kbs; ++kb) {
            if (!full_next && !(ok = mbar_spin_wait(&full[st.s], st.ph, abort_flag))) break;
            tc_fence_after();
            Ring nx = st;
            nx.next(NS);
            full_next = mbar_test_wait(&full[nx.s], nx.ph);
            const uint64_t adesc = adesc0 + static_cast<uint64_t>(st.s * (kPlanStageA >> 4));
            const uint64_t bdesc = bdesc0 + static_cast<uint64_t>(st.s * (kPlanStageB >> 4));
            if (f16) {
#pragma unroll
              for (int k4 = 0; k4 < BK / 32; ++k4)
                mma_bf16_ss_pair(d_tmem, adesc + 2 * k4, bdesc + 2 * k4, idesc, (kb | k4) != 0 ? 1u : 0u);
            } else {
#pragma unroll
              for (int k4 = 0; k4 < BK / 32; ++k4)
                mma_i8_ss_pair(d_tmem, adesc + 2 * k4, bdesc + 2 * k4, idesc, (kb | k4) != 0 ? 1u : 0u);
            }
            mma_commit_pair(&empty[st.s]);
            st = nx;
          }
          if (ok) mma_commit_pair(&acc_full[buf]);
        }
      }
    }
  } else {
    // ================= epilogue: quadrant (warp & 3), column half (ew >> 2) =================
    const int ew = warp - kEpiWarp0;
    float* copy = s_scale + ew * (RowEpilogue<0>::kScaleBytes / 4);
    RowEpilogue<0> epi;
    const uint32_t empty0 = map_to_cta(&acc_empty[0], 0), empty1 = map_to_cta(&acc_empty[1], 0);
    epi.init(warp, lane, copy, empty0, empty1);
    int total = 0;
    for (int li = 0; li < p.n_layers; ++li) total += s_runs->end[li] - s_runs->begin[li];
    pdl_launch_dependents();  // only now that everything before this launch has finished: see plan_run_step
    bool ok = true;
    int tcount = 0;
    for (int li = 0; li < p.n_layers && ok; ++li) {
      const GemmPlanLayer L = s_layer[li];
      const int n_tiles = L.n_tiles, bn = L.bn, ncols = bn >> 1, col0 = (ew >> 2) * ncols;
      const int begin = s_runs->begin[li], end = s_runs->end[li];
      GemmParams g;
      g.s_a = L.s_a;
      g.s_w = L.s_w;
      g.bias = L.bias;
      g.y = L.y;
      g.ldy = L.N;
      g.dbg_acc = nullptr;
      g.x = nullptr;
      g.M = L.M;
      epi.staged_col = -1;
      int staged = -1;
      for (int tile = begin; tile < end && ok; ++tile, ++tcount) {
        const int buf = tcount & 1, col = (tile % n_tiles) * bn + col0;
        const int cta_row0 = (tile / n_tiles) * (2 * BM) + static_cast<int>(rank) * BM;
        const bool reused = tcount + 2 < total;
        if (L.f16) {
          ok = plan_tile_f16(L, col, ncols, cta_row0, tmem_base + (static_cast<uint32_t>((warp & 3) * 32) << 16) + buf * 256 + col0,
                             copy, col != staged, &acc_full[buf], (tcount >> 1) & 1, buf ? empty1 : empty0, reused, lane,
                             warp & 3, abort_flag);
          staged = col;
        } else {
          ok = epi.tile<false>(g, col, ncols, cta_row0, tmem_base, buf * 256 + col0, &acc_full[buf], (tcount >> 1) & 1, buf,
                               reused, abort_flag);
        }
      }
    }
  }

  tc_fence_before();
  __syncthreads();
  cluster_sync_relaxed();  // neither CTA frees tensor memory or exits while the other may still touch it
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc_pair(tmem_base, 512);
  }
  if (threadIdx.x == 0 && *abort_flag && p.status != nullptr) atomicExch(p.status, DP_ERR_TIMEOUT);
}

// ---- host side -------------------------------------------------------------------------------------
constexpr size_t plan_smem_bytes() {
  return 1024 + static_cast<size_t>(kPlanStages) * (kPlanStageA + kPlanStageB) + kEpiWarps * RowEpilogue<0>::kScaleBytes +
         (2 * kPlanStages + 4) * 8 + 16 + sizeof(GemmPlanRuns) + kPlanGroupMax * sizeof(GemmPlanLayer);
}

int gemm_plan_init_device() {
  DP_CUDA_OK(cudaFuncSetAttribute(gemm_plan_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  static_cast<int>(plan_smem_bytes())));
  return DP_OK;
}

// Tile width of each layer and, per layer, the run of its tiles (row-major, columns fastest) that each pair takes.
// Layers stand in the order of their tiles' expected times, longest first, and every tile goes to the pair with the least
// so far; the widths tried are the widest of up to 256, 192 and 128 that divide each N, and the set that ends first is
// taken. False: a layer that the kernel does not take (or more tiles than the table counts).
bool gemm_plan_schedule(const GemmPlanShape* shape, int n, GemmPlanSchedule* out) {
  if (n < 1 || n > kPlanGroupMax) return false;
  const int pairs_max = std::min(gemm_max_pairs() > 0 ? gemm_max_pairs() : 74, kPlanMaxPairs);
  double best = 1e30;
  for (const int widest : {256, 192, 128}) {
    int bn[kPlanGroupMax], order[kPlanGroupMax];
    double us[kPlanGroupMax];
    for (int l = 0; l < n; ++l) {
      bn[l] = 0;
      for (const int w : {256, 192, 128})
        if (w <= widest && shape[l].N % w == 0 && bn[l] == 0) bn[l] = w;
      if (bn[l] == 0 && shape[l].N % 192 == 0) bn[l] = 192;
      if (bn[l] == 0 || (shape[l].M + 2 * BM - 1) / (2 * BM) * (shape[l].N / bn[l]) > 65535) return false;
      us[l] = gemm_pair_tile_us(bn[l], shape[l].kb);
      order[l] = l;
    }
    std::stable_sort(order, order + n, [&](int a, int b) { return us[a] > us[b]; });
    // Pairs by their load so far, least first. All tiles of a layer take as long, so the pairs that have taken one are in
    // order too, behind each other: the least of all is the first of one queue or of the other.
    using Load = std::pair<double, int>;
    std::vector<Load> loads, taken;
    for (int i = 0; i < pairs_max; ++i) loads.push_back({0.0, i});
    std::vector<int> count(static_cast<size_t>(n) * kPlanMaxPairs, 0);
    double end = 0.0;
    int used = 0;
    for (int o = 0; o < n; ++o) {
      const GemmPlanShape& s = shape[order[o]];
      const int64_t tiles = (s.M + 2 * BM - 1) / (2 * BM) * (s.N / bn[order[o]]);
      taken.clear();
      size_t first = 0, first_taken = 0;
      for (int64_t t = 0; t < tiles; ++t) {
        const bool again = first == loads.size() || (first_taken < taken.size() && taken[first_taken] < loads[first]);
        Load least = again ? taken[first_taken++] : loads[first++];
        least.first += us[order[o]];
        end = std::max(end, least.first);
        used = std::max(used, least.second + 1);
        ++count[o * kPlanMaxPairs + least.second];
        taken.push_back(least);
      }
      std::vector<Load> next;
      std::merge(loads.begin() + first, loads.end(), taken.begin() + first_taken, taken.end(), std::back_inserter(next));
      loads.swap(next);
    }
    if (end >= best) continue;
    best = end;
    out->n = n;
    out->pairs = used;
    for (int o = 0; o < n; ++o) {
      out->order[o] = order[o];
      out->bn[o] = bn[order[o]];
      int at = 0;
      for (int i = 0; i < kPlanMaxPairs; ++i) {
        out->runs[i].begin[o] = static_cast<uint16_t>(at);
        at += count[o * kPlanMaxPairs + i];
        out->runs[i].end[o] = static_cast<uint16_t>(at);
      }
    }
  }
  return best < 1e30;
}

int launch_gemm_plan(const GemmPlanParams& p, cudaStream_t stream, bool pdl) {
  const cudaError_t e = launch_cluster(gemm_plan_kernel, dim3(static_cast<unsigned>(2 * p.pairs)), dim3(kPlanThreads),
                                       plan_smem_bytes(), stream, pdl, 2, p);
  if (e != cudaSuccess) return fail(DP_ERR_CUDA, "plan GEMM launch failed: %s", cudaGetErrorString(e));
  return DP_OK;
}

}  // namespace dp
