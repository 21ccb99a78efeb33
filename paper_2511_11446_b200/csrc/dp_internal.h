// Internal interfaces between the translation units of libdiffpro (host side).
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/diffpro.h"

namespace dp {

// Order in which the int8 codes of a token are stored along K in the activation scratch.
enum KOrder {
  KORDER_NATURAL = 0,   // q[k] at byte k
  KORDER_EVEN_ODD = 1   // every group of 8 codes stored as k = 0,2,4,6,1,3,5,7 (4-bit weight path)
};
// The order the tensor-core path wants for weights of this width when it runs DAQ itself.
int gemm_korder(int32_t bits);

// daq.cu
// Expansion of a packed weight matrix to int8 [N][K] (codes less their zero-point, or 128 of it, k ascending) in global scratch,
// run by extra CTAs of a DAQ launch or on its own: `units` = N * K / 32 units of 32 codes.
struct UnpackJob {
  const uint32_t* packed = nullptr;
  int8_t* out = nullptr;
  int64_t units = 0;
  int32_t bits = 0;         // 3 or 4
  int32_t first_block = 0;  // filled by the launcher: CTAs from here on unpack
  int32_t early = 0;        // the preceding kernel on the stream is of the same call, so it cannot be writing
                            // `packed` or `zeros`: they are read before it has finished
  int32_t ahead = 0;        // (with early) nor x, nor reading the destinations: the whole launch runs beside it. One CTA
                            // stays until it has finished, so that whatever waits for this launch waits for both
  const uint8_t* zeros = nullptr;  // group-wise zero-points [N][row_units / group_units], or null (symmetric)
  uint32_t row_units = 0, group_units = 0;
  // With zeros: a byte for every 128 units, nonzero where a zero-point above 127 was among them (128 of it are taken
  // off; the fold that reads `out` has to know).
  uint8_t* wide = nullptr;
};
// Notes of a matrix of `units` units (a multiple of 512: N and K are multiples of 128).
inline int64_t unpack_notes(int64_t units) { return units / 128; }
int launch_daq(const void* x, int64_t M, int64_t K, int64_t ldx, int8_t* q, int64_t ldq,
               float* s_a, int32_t* rowsum, int korder, bool tiled, cudaStream_t stream, bool pdl,
               const UnpackJob* unpack = nullptr);
int launch_unpack(const UnpackJob& job, cudaStream_t stream, bool pdl);
// ln.cu -- LayerNorm + adaLN modulation + DAQ in one pass (K a multiple of 8, at most 4608)
int launch_ln_modulate_daq(const void* x, int64_t M, int64_t K, int64_t ldx, const void* shift, const void* scale,
                           int64_t rows_per_sample, float eps, int8_t* q, int64_t ldq, float* s_a,
                           cudaStream_t stream, bool pdl);
int launch_daq_robust(const void* x, int64_t M, int64_t K, int64_t ldx, int8_t* q, int64_t ldq, float* s_a,
                      int32_t* rowsum, int clip_rank, int act_bits, bool tiled, cudaStream_t stream, bool pdl,
                      const UnpackJob* unpack);

// simt.cu — CUDA-core weight-streaming linear for small M (DAQ fused in the CTA prologue).
struct SimtArgs {
  const void* x;        // bf16 [M][ldx] or int8 [M][ldx] when s_a_in != nullptr
  int64_t ldx;
  const float* s_a_in;  // nullptr -> DAQ inside the kernel
  int rows;  // tokens per CTA of the matrix-instruction form, 8 or 16 (set by the launch)
  int64_t M;
  int32_t N, K, bits;
  const void* qweight;
  const float* s_w;
  const uint16_t* bias;
  uint16_t* y;
  int64_t ldy;
  int8_t* dbg_q;
  int64_t dbg_ldq;
  float* dbg_sa;
  int32_t* dbg_acc;
  int64_t dbg_ldacc;
  int32_t early_w;  // weights may be fetched before the preceding kernel on the stream has finished
  int32_t hold;     // first launch of a plan run: dependents start only once what precedes it has finished
  int32_t* status;  // device word raised to DP_ERR_TIMEOUT when a bounded wait expires (may be null)
};
int launch_simt_linear(const SimtArgs& a, cudaStream_t stream, bool pdl);
// Up to kSimtGroupMax layers of one shape (bf16 inputs [M][K], outputs [M][N], both contiguous).
constexpr int kSimtGroupMax = 32;
struct SimtGroupArgs {
  struct Layer {
    const void* x;
    uint16_t* y;
    const void* qweight;
    const float* s_w;
    const uint16_t* bias;
    int32_t bits;
  } layer[kSimtGroupMax];
  int64_t M;
  int32_t N, K, n_layers;
  int32_t early_w, hold;  // as in SimtArgs
  // Scratch for the group's int8 tokens [n_layers][M][K] and scales [n_layers][M]: when given (a DAQ rule other
  // than the plain one), one small kernel quantizes all tokens of the group first and the main kernel's CTAs only
  // fetch the codes; when null every CTA quantizes its tokens itself.
  int8_t* q_scratch;
  float* sa_scratch;
  int32_t* status;  // as SimtArgs::status
  int32_t daq_rank, daq_bits;  // the group's DAQ rule: (1, 8) = absmax, 8 bits; else percentile clip / a-bit codes
  // Matrix-instruction form: CTAs [cta_begin[l], cta_begin[l + 1]) of grid.x work on layer l (filled
  // by launch_simt_group: more CTAs for the layers that take longer).
  int32_t cta_begin[kSimtGroupMax + 1];
};
size_t simt_group_scratch_bytes(int64_t M, int32_t K, int32_t n_layers);
int launch_simt_group(const SimtGroupArgs& g, cudaStream_t stream, bool pdl);
size_t simt_max_k();

// gemm_tc.cu — tcgen05 kind::i8 GEMM with in-smem weight unpack and fused dequant epilogue.
struct GemmProblem {
  CUtensorMap tmap_a;  // int8 activations [M][K]
  CUtensorMap tmap_w;  // packed weights, byte view [N][K*bits/8]
  const float* s_a;    // [M]
  const float* s_w;    // [N]
  const uint16_t* bias;
  uint16_t* y;
  int64_t ldy;
  int32_t* dbg_acc;
  int64_t dbg_ldacc;
  const uint16_t* res = nullptr;  // residual (and gate) taken into the epilogue, see dp_wq_linear_residual
  int64_t ldr = 0;
  const uint16_t* gate = nullptr;
  int64_t rows_per_gate = 1;
  int64_t M;
  int32_t N, K, bits, bn;
  int32_t cg;       // 1: one CTA per 128-row tile; 2: a CTA pair per 256-row tile
  int32_t ws;       // 1: weight-stationary pair kernel (cg == 2, bn in {192, 256}); 2: activation-stationary
                    // pair kernel (bn = width of its column sub-blocks)
  int32_t korder;   // KOrder of the activations behind tmap_a
  int32_t a_tiled;  // the activations behind tmap_a are stored as 128 x 128 tiles (see gemm_encode_a_tiled)
  int32_t early_w;  // the preceding kernel on the stream is this call's own DAQ: weights may be
                    // fetched before it has finished
  int32_t a_ready = 0;  // (with early_w) nor is it writing the activations or the int8 copy of the weights: only
                        // the epilogue waits for it
  int32_t* status;
  // In-kernel DAQ (x != nullptr): the GEMM kernel quantizes x into q_out / s_a_out (the buffers
  // behind tmap_a and s_a) itself; sync = zeroed counters, one per 128-token tile plus one.
  const uint16_t* x;
  int64_t ldx;
  int8_t* q_out;
  float* s_a_out;
  int32_t* sync;
};
// allow: bit 1 = single-CTA tiles permitted, bit 2 = CTA-pair tiles permitted, bit 3 = no 192-wide ones, bit 4 = no
// tile shared along K (a kernel that quantizes its own activations)
// forced_bn: 0, or the width to take; *splits_out: CTAs that share a tile along K (1: not split).
void gemm_pick_tile(int64_t M, int32_t N, int32_t K, int32_t bits, uint32_t allow, int forced_bn, int* bn_out, int* cg_out,
                    int* splits_out);
// The model's estimate (us) for one width and CTA count of an 8-bit layer's GEMM.
double gemm_tile_cost(int64_t M, int32_t N, int32_t K, int bn, int cg, bool may_split);
int gemm_max_pairs();
// gemm_split.cu -- split-K form of the single-CTA streaming kernel and of the 16-bit kernel (64-wide tiles).
constexpr int kMaxSplits = 4;
struct GemmLimits {  // of the current device: SMs, resident CTA pairs, resident clusters of s split-K CTAs
  int sms, pairs, clusters[kMaxSplits + 1];
};
GemmLimits gemm_limits();
int gemm_split_init_device(int* max_clusters);
int gemm_split_factor(const GemmLimits& lim, int64_t tiles, int kb, double per_kb, double* saved_us);
int gemm_encode_a(CUtensorMap* out, const int8_t* q, int64_t M, int64_t K, int64_t ldq);
// int8 activations stored as [ceil(M/128)][K/128] tiles of 128 tokens x 128 codes (16 KB each).
int gemm_encode_a_tiled(CUtensorMap* out, const int8_t* q, int64_t M, int64_t K);
int gemm_encode_w(CUtensorMap* out, const void* qweight, int32_t N, int32_t K, int32_t bits,
                  int32_t bn, int32_t cg);
int launch_gemm(const GemmProblem& p, cudaStream_t stream, bool pdl);
void gemm_debug_skip_stage_load(int32_t kb);  // see dp_debug_skip_stage_load
// Two ranges (a plan's next layer's packed weights and its bf16 input) that the calling thread's next
// tensor-core launch sends on their way into L2 while it runs; cleared by that launch. Hints: any valid
// device ranges of the caller's, or nullptr.
void gemm_set_next_reads(const void* w, size_t w_bytes, const void* x, size_t x_bytes);

// gemm_plan.cu -- the GEMMs of several layers of a plan in one launch.
constexpr int kPlanGroupMax = 16, kPlanMaxPairs = 80;
struct GemmPlanLayer {  // of a layer, copied into shared memory by each CTA
  const float* s_a;
  const float* s_w;
  const uint16_t* bias;
  uint16_t* y;  // [M][N]
  int64_t M;
  int32_t N, kb;  // kb: 128-byte k-blocks
  int32_t bn, n_tiles;
  int32_t f16, pad;
};
struct GemmPlanRuns {  // of a pair: tiles [begin[l], end[l]) of layer l
  uint16_t begin[kPlanGroupMax], end[kPlanGroupMax];
};
struct GemmPlanParams {
  CUtensorMap tmap_a[kPlanGroupMax];  // int8 codes as 128 x 128 tiles, or (f16) bf16 [M][K]
  CUtensorMap tmap_w[kPlanGroupMax];  // int8 or bf16 weights, boxes of bn / 2 rows x 128 bytes
  GemmPlanRuns runs[kPlanMaxPairs];
  GemmPlanLayer layer[kPlanGroupMax];
  int32_t n_layers, pairs;
  int32_t* status;
};
struct GemmPlanShape {
  int64_t M;
  int32_t N, kb;
};
struct GemmPlanSchedule {  // by place in the launch: which layer, its tile width, its tiles' runs
  int n, pairs;
  int order[kPlanGroupMax], bn[kPlanGroupMax];
  GemmPlanRuns runs[kPlanMaxPairs];
};
bool gemm_plan_schedule(const GemmPlanShape* shape, int n, GemmPlanSchedule* out);
int launch_gemm_plan(const GemmPlanParams& p, cudaStream_t stream, bool pdl);
int gemm_plan_init_device();
double gemm_pair_tile_us(int bn, int kb);  // expected time of a pair's tile

// daq.cu -- what those GEMMs read, prepared in one launch: activations quantized, packed weights expanded, weights that
// are read as they are sent on their way into L2.
struct PlanPrepSeg {
  enum Kind { ROWS, EXPAND, FETCH };
  const void* src;      // bf16 [M][K]; packed codes; weights
  int8_t* dst;          // codes as 128 x 128 tiles; int8 [N][K]
  float* s_a;
  int64_t count;        // rows; units of 32 codes; bytes
  int16_t kind, arg;    // arg: K / 8; bits
  int32_t rank;         // ROWS under a clip policy: rank of the threshold from the top
};
constexpr int kPlanPrepSegs = 2 * kPlanGroupMax;
struct PlanPrepParams {
  int32_t first_block[kPlanPrepSegs];  // filled by the launch (INT_MAX beyond the last segment)
  PlanPrepSeg seg[kPlanPrepSegs];
  int32_t n_seg;
  int32_t early;  // the preceding kernel on the stream is of the same call: it does not write packed weights
  int32_t ahead;  // (with early) nor x, nor does it read what this launch writes: see UnpackJob::ahead
  float qmax;
};
int launch_plan_prep(PlanPrepParams& p, bool robust, cudaStream_t stream, bool pdl);
constexpr int kPlanMaxK = 4608;  // rows that every form of the preparation holds in registers

// gemm_ws.cu -- weight-stationary CTA-pair kernel (K <= 1152, N a multiple of 192 or 256).
bool gemm_ws_supported(int32_t N, int32_t K);
int gemm_ws_pick_bn(int32_t N);
int launch_gemm_ws(const GemmProblem& p, cudaStream_t stream, bool pdl);
// Per-device set-up (kernel attributes, tensor-map encoder, SM and CTA-pair counts), called once per
// device by check_device() with that device current.
int gemm_init_device(int dev, int* num_sms_out, int* max_pairs_out, int* max_clusters_out);
int gemm_ws_init_device();
int simt_init_device();
int gemm_as_init_device();
int gemm_bf16_init_device();
int gemm_grp_init_device();

// gemm_grp.cu -- layers with group-wise weight scales (and zero-points): folding tensor-core kernel.
constexpr int kGrpZeroMaxGroups = 160;  // per row, of a layer with zero-points (K <= 5120 at g = 32)
// (for packed weights the expansion has taken the zero-points up to 128 off already)
int launch_gemm_grp(const int8_t* q, int64_t ldq, bool a_tiled, const float* s_a, const int8_t* w8, int32_t bits,
                    int32_t g, const float* s_w, const uint8_t* zeros, const uint8_t* wide, const uint16_t* bias,
                    int32_t* rowsum, int64_t M, int32_t N, int32_t K, uint16_t* y, int64_t ldy, int32_t* status, cudaStream_t stream, bool pdl);

// gemm_bf16.cu -- pass-through linear of 16-bit layers (bf16 x bf16 -> fp32 -> bf16, tcgen05 kind::f16).
int launch_gemm_bf16(const void* x, int64_t ldx, const void* w, const uint16_t* bias, int64_t M, int32_t N, int32_t K,
                     uint16_t* y, int64_t ldy, int32_t* status, cudaStream_t stream, bool pdl);
int gemm_encode_w_rows(CUtensorMap* out, const void* base, uint64_t row_bytes, uint64_t rows, uint32_t box_inner,
                       uint32_t box_rows, bool swizzle128);
int gemm_encode_bytes_2d(CUtensorMap* out, const void* base, uint64_t inner_bytes, uint64_t rows, uint64_t pitch_bytes,
                         uint32_t box_inner, uint32_t box_rows);

// gemm_as.cu -- activation-stationary CTA-pair kernel (K <= 1152, 8-bit weights, tiled activations).
bool gemm_as_supported(int32_t N, int32_t K);
// Sub-block width (forced_bns, or the model's choice when 0) and sub-blocks per slice; *bns_out = 0 if none fits.
void gemm_as_config(int64_t M, int32_t N, int32_t K, int forced_bns, int* bns_out, int* nsub_out);
int launch_gemm_as(const GemmProblem& p, cudaStream_t stream, bool pdl);

int num_sms();

}  // namespace dp
