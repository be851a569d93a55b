// Internal declarations shared by the translation units of liboscars.
#pragma once

#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace oscars {

// Lets `kernel` take `bytes` of dynamic shared memory.  The limit belongs to the
// kernel in the process, not to a launch: set to each launch's own size, a host
// thread could lower it between another one's setting and its launch, which then
// fails.  So every launch sets the same limit, all of an SM's shared memory but
// room for static variables (only kernels that always pass one constant take more).
constexpr size_t kSmemLimit = 225 * 1024;
template <typename F>
cudaError_t allow_smem(F* kernel, size_t bytes) {
  return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              static_cast<int>(bytes > kSmemLimit ? bytes : kSmemLimit));
}

// Two kernels on clusters that together want more than an SM's tensor memory must
// not meet on an SM: a tcgen05.alloc waits without a limit, and two clusters of
// different streams, each with one CTA that has its columns and one that waits
// for the other's, would wait for ever.  Every kernel on clusters that allocates
// tensor memory takes at least kLeastClusterSmem of dynamic shared memory, and one
// that allocates all of it leaves less on its SM.  (The others wait for nobody, so
// a wait for their columns ends.)
constexpr size_t kLeastClusterSmem = 64 * 1024;
constexpr size_t kSmSmem = 228 * 1024, kCtaSmem = 1024;   // shared memory of an SM; taken by each CTA beside its own
constexpr bool no_cluster_beside(size_t smem) { return smem + kCtaSmem + kLeastClusterSmem + kCtaSmem > kSmSmem; }

constexpr int kMaxMergeWorkers = 256;   // pointer table of the merge kernel
constexpr int kMaxWorkersMLP = 64;
constexpr int kMaxClasses = 32;
constexpr int kRowsPerLossChunk = 16;   // rows per loss partial in the head kernel

// ---------------------------------------------------------------- merge
struct MergeArgs {
  const float* src[kMaxMergeWorkers];  // delta_k, or replica x^k
  float w[kMaxMergeWorkers];
  int W;
};

// x_g <- x_g + eta * sum_k w_k * (replica ? src_k - x_g : src_k), p < P;
// shadow (optional): shadow[p] = bf16(new x_g[p]) in the same pass.
cudaError_t launch_merge(const MergeArgs& a, float* x_g, int64_t P, float eta, bool replica,
                         cudaStream_t s, __nv_bfloat16* shadow = nullptr);

// The same over pieces of the vector, in one launch: elements [dst, dst + n)
// of x_g (and shadow) take [src, src + n) of every pushed buffer (head and n4
// are filled in by the launcher).
constexpr int kMaxMergeSegs = 32;   // two tensors per layer
struct MergeSeg {
  int64_t dst, src, n;
  int head;                         // single elements before the first 16-byte chunk
  int64_t n4;                       // 16-byte chunks
};
cudaError_t launch_merge_segs(const MergeArgs& a, const MergeSeg* seg, int nseg, float* x_g, float eta, bool replica,
                              cudaStream_t s, __nv_bfloat16* shadow = nullptr);

// Copy between a padded slot and a canonical vector on the device: piece i is
// `rows` rows of `len` floats, `pitch` apart in the slot and contiguous in
// the canonical vector.
constexpr int kMaxCopySegs = 40;
struct CopySeg {
  int64_t slot, canon;
  int64_t len;
  int rows, pitch;
};
cudaError_t launch_unpad(const float* slot, float* canon, const CopySeg* seg, int nseg, cudaStream_t s);

// one thread waits `polls` polls on an mbarrier nothing completes, then
// records its timeout code in *err (the bounded-wait failure path)
cudaError_t launch_wait_selfcheck(int* err, uint32_t polls, cudaStream_t s);

// ---------------------------------------------------------------- scheduler (host)
int iteration_ticks(const double* speed, int n, int64_t Q, int64_t* t, const char** why);
int schedule_solve(const int64_t* t, int n, int64_t M, int mode, int64_t* T_star,
                   int64_t* max_wait, int32_t* tau, const char** why);
void merge_weights(int rule, const int32_t* tau, int n, float* w);

// ---------------------------------------------------------------- softmax regression (fp32)
struct SoftregArgs {
  const float* master;          // slab base (slots of P_pad floats)
  float* master_out;
  int64_t slot_stride;          // P_pad
  int global_slot;              // W
  int64_t offW, offB;           // element offsets inside a slot
  int D, C, B;
  float lr;
  const int32_t* tau = nullptr; // [W]; null (cluster kernel, one worker): the values below
  const float* const* shard_x = nullptr;  // [W] device pointers
  const int32_t* const* shard_y = nullptr;
  const int64_t* shard_n = nullptr;       // [W]
  const int64_t* cursor = nullptr;        // [W]
  int tau1 = 0;                 // one worker's step count, shard and cursor
  const float* x1 = nullptr;
  const int32_t* y1 = nullptr;
  int64_t n1 = 0, cursor1 = 0;
  float* loss_part = nullptr;   // single-CTA kernel: [W][max_tau] (sum of per-sample losses of one step)
  int max_tau = 0;
  int* err = nullptr;           // cluster kernel: device error word of the bounded waits, or null
  // round bookkeeping in the same launch (null: not done): the worker's mean
  // loss over its steps, and its cursor advanced by tau * B (mod the shard)
  float* loss_out = nullptr;    // [W]
  int64_t* cursor_next = nullptr;   // [W], may be `cursor` itself
};
cudaError_t launch_softreg_round(const SoftregArgs& a, int W, cudaStream_t s);
size_t softreg_smem_bytes(int D, int C, int B);
// the round kernel gives each mini-batch row one thread for its row offset,
// label and softmax: B must not exceed its block size
constexpr int kSoftregMaxBatch = 512;
// the same round with each worker on a cluster of 8 CTAs splitting the input
// columns (a column slice of the weights, two of the mini-batch and the
// exchange buffers in shared memory); writes loss_out, which must be set
bool softreg_cluster_supported(int D, int C, int B);
cudaError_t launch_softreg_cluster_round(const SoftregArgs& a, int W, cudaStream_t s);

struct SoftregEvalArgs {
  const float* master;  // global slot
  int64_t offW, offB;
  int D, C;
  const float* x;
  const int32_t* y;
  int64_t n;
  float* loss_sum;      // [blocks] partial sums
};
int softreg_eval_blocks(int64_t n, int sms);   // loss_sum entries
cudaError_t launch_softreg_eval(const SoftregEvalArgs& a, int blocks, cudaStream_t s);

// ---------------------------------------------------------------- MLP (bf16 GEMMs)
// In the step kernels below active lane i uses activation buffers of lane
// `wid[i]` and reads parameters from slot `src[i]` (the global slot on the
// first local step: the fused pull), writing them to slot `wid[i]`.

// Staging of a round's mini-batches: fp32 rows to bf16, both layouts
struct StageArgs {
  const float* const* x;   // [lanes] sample matrix per lane (device pointers)
  const int32_t* const* y;
  const int64_t* n;        // [lanes] rows available
  const int64_t* start;    // [lanes] first row (cursor)
  int D, B;
  __nv_bfloat16* A0;       // [lanes][B][D]
  __nv_bfloat16* A0T;      // [lanes][D][B]
  int32_t* labels;         // [lanes][B]
  const int32_t* ahead;    // stage_round: null, or tau (the next round: rows from start + tau * B)
  const int32_t* slots;    // stage_round: the n_slots active slots s * W + w (s < tau[w]), or null (all)
  int n_slots;
};
// out[i] = bf16(x[i]), count a multiple of 8
cudaError_t launch_cast_rows(const float* x, __nv_bfloat16* out, int64_t count, int sms, cudaStream_t s);
// all mini-batches of a round: step s of worker w (s < tau[w]) at slot s * W + w
// (grid z over a.slots when given, else over all max_tau * W slots)
cudaError_t launch_stage_round(const StageArgs& a, const int32_t* tau, int W, int max_tau, cudaStream_t s);
// the same staging from `blocks` blocks striding over the tiles (bounded footprint beside other kernels)
cudaError_t launch_stage_round_strided(const StageArgs& a, const int32_t* tau, int W, int max_tau, int blocks,
                                       int priority, cudaStream_t s);
// the first form with a launch priority (cudaLaunchAttributePriority)
cudaError_t launch_stage_round_priority(const StageArgs& a, const int32_t* tau, int W, int max_tau, int priority,
                                        cudaStream_t s);

enum GemmEpi { kEpiFwd = 0, kEpiDh = 1 };

struct GemmArgs {
  const int* wid;     // [n_active]
  const int* src;     // [n_active]
  int M, N, K;
  int a_z_src, b_z_src;  // TMA z coordinate of A / B: 1 = src slot, 0 = lane id
  int b_mn;              // B read MN-major (its transpose [lane][K][N] in boxes of 64 N x 64 K; N % 64 == 0)
  int pdl;               // launch as a programmatic dependent of the previous kernel on the stream
  int* err;
  // kEpiFwd: relu(acc + bias[m]) -> H [lane][N][M], H^T [lane][M][N]
  // kEpiDh : acc * (h > 0) -> G [lane][N][M], G^T [lane][M][N], gb[lane][m]
  // With out null (N = 64 or 128) only the transposes are written.
  const float* master;      // fp32 slab base
  int64_t slot_stride;      // P_pad
  int64_t offB;             // element offset of b_l in a slot
  const __nv_bfloat16* hmask;  // kEpiDh: h [lanes][N][M]; h^T [lanes][M][N] with out null
  __nv_bfloat16* out;       // [lanes][N][M], or null
  __nv_bfloat16* outT;      // [lanes][M][N]
  float* gb_out;            // [lanes][M] (kEpiDh)
};
struct GemmMaps {
  const CUtensorMap *a, *b;
  const CUtensorMap* t;     // outT [lane][M][N], box {64, 32}: used when out is null
  const CUtensorMap* mask;  // hmask [lane][M][N], box {64, 128}: kEpiDh, used when out is null
};
cudaError_t launch_gemm(int epi, const GemmMaps& m, const GemmArgs& a, int n_active, cudaStream_t s);

// One large product D[m][n] = sum_k A[m][k] B[n][k] (csrc/gemm_rows.cu).
enum RowsEpi { kRowsStore = 0, kRowsRelu = 1, kRowsLoss = 2, kRowsNarrow = 3 };
struct RowsPlan {
  int BN, cl;              // columns per tile, CTAs per tile (row tiles of 128 each)
};
struct RowsArgs {
  int M, N, K;
  int BN, stages, mt, nt;  // set by the launcher
  float* C;                // kRowsStore (when tma_store is 0), kRowsNarrow: [M][N]
  int tma_store;           // kRowsStore: 1 = through mD (N % 4 == 0 and C 16-byte aligned)
  const float* bias;       // kRowsRelu, kRowsLoss: [N]
  const int32_t* labels;   // kRowsLoss: [M]
  float* loss_part;        // kRowsLoss: [4 ceil(M / 128)] sums over 32 rows
  int* err;
  int pdl;                 // launch as a programmatic dependent of the previous kernel on the stream
};
// kRowsRelu: N a multiple of 64, bias 16-byte aligned; kRowsLoss, kRowsNarrow: N <= 32
RowsPlan gemm_rows_plan(int epi, int M, int N, int K);
// mA: [M][K] bf16, box {64, 128}; mB: [N][K] bf16, box {64, BN / cl}; mD: the
// result, boxes of 32 rows x 128 bytes (kRowsStore fp32, kRowsRelu bf16); all
// with 128-byte swizzle
cudaError_t launch_gemm_rows(int epi, const RowsPlan& p, const CUtensorMap& mA, const CUtensorMap& mB,
                             const CUtensorMap& mD, RowsArgs a, cudaStream_t s);

// Weight gradient + SGD of up to kDwMaxLayers hidden layers, persistent
// (csrc/gemm_dw.cu): W[wid] = W[src] - lr * G^T X over the batch, its bf16
// copy, and the bias b[wid] = b[src] - lr * gb[wid] (outputs m < M, inputs n <
// N, batch K; M a multiple of 128, N of 8).
constexpr int kDwMaxLayers = 4;
struct DwLayer {
  int M, N;
  int64_t offB;             // element offset of b_l in a slot
  const float* gb;          // [W][M] bias gradient
};
struct DwArgs {
  const int* wid;           // [n_active] destination slots (device), or null = lane id
  const int* src;           // [n_active] source slots (device), or null = lane id
  int n_active, n_layers;
  int K;
  float lr;
  const float* master;      // fp32 slab (bias read)
  float* master_w;          // fp32 slab (bias written)
  int64_t slot_stride;      // P_pad
  DwLayer layer[kDwMaxLayers];
  int first_tile[kDwMaxLayers + 1];   // set by the launcher
  int* err;
  int pdl;                  // launch as a programmatic dependent of the previous kernel on the stream
};
// gt: G^T [lane][M][K] bf16, box {64, 128}; xt: X^T [lane][N][K] bf16, box
// {64, 128}; master: W_l fp32 [slot][M][N], box {32, 128} (loads); master_st:
// the same with box {32, 32} (stores); shadow_st: W_l bf16 [slot][M][N], box
// {64, 32} (stores); all with 128-byte swizzle
struct DwMaps {
  struct Layer {
    CUtensorMap gt, xt, master, master_st, shadow_st;
  } l[kDwMaxLayers];
};
// `sms`: the device's multiprocessors (one CTA each at most)
cudaError_t launch_gemm_dw(const DwMaps& maps, DwArgs a, int sms, cudaStream_t s);

struct HeadArgs {
  const int* wid;
  const int* src;
  int H, C, B;
  const __nv_bfloat16* Ain;   // [lanes][B][H] input of the last layer
  const int32_t* labels;      // [lanes][B]
  const __nv_bfloat16* shadow;
  const float* master;
  float* master_w;
  __nv_bfloat16* shadow_w;
  int64_t slot_stride;
  int64_t offW, offB;
  float lr;
  float* dlog;                // [lanes][B][C]
  float* loss_part;           // rows of (B/16) partial sums
  int part_mul, part_add;     // row = wid * part_mul + part_add
  __nv_bfloat16* G;           // [lanes][B][H] (head_bwd)
  __nv_bfloat16* GT;          // [lanes][H][B]
  float* gb;                  // [lanes][H]
  int* err;                   // device error word (bounded waits of the tensor-core head)
  int pdl;                    // tensor-core head: launch as a programmatic dependent
};
cudaError_t launch_head_fwd(const HeadArgs& a, int n_active, cudaStream_t s);
// forward + backward of the last layer on the tensor cores (csrc/head_tc.cu):
// one cluster of H/128 CTAs per active lane; 2 <= C <= 32, 32 <= B <= 128.
// mH: the layer input [lane][B][H] bf16 (its transpose [lane][H][B] when a.G
// is null), box {64, 128}; mW2: the head weights
// of every slot [slot][C][H] bf16, box {64, head_tc_class_rows(C)}; mGT: the
// input gradient^T [lane][H][B] bf16 (a.GT), box {64, 128}, written through
// when a.G is null (B a multiple of 64); all with 128-byte swizzle.
int head_tc_class_rows(int C);
bool head_tc_supported(int H, int B, int C);
cudaError_t launch_head_tc(const CUtensorMap& mH, const CUtensorMap& mW2, const CUtensorMap& mGT,
                           const HeadArgs& a, int n_active, cudaStream_t s);
// forward + backward of the last layer in one launch: one cluster of H/128
// CTAs per active lane (H <= 1024); false if the shape needs the two-kernel path
bool head_fused_supported(int H, int B, int C);
cudaError_t launch_head_fused(const HeadArgs& a, int n_active, cudaStream_t s);
cudaError_t launch_head_bwd(const HeadArgs& a, int n_active, cudaStream_t s);

// ---------------------------------------------------------------- fused round (2-layer MLP)
struct FusedRoundArgs {
  const int32_t* tau;
  const int32_t* order;           // [W] workers, cluster by cluster (longest first)
  const int32_t* cl_first;        // [n_clusters + 1] cluster k runs order[cl_first[k] .. cl_first[k + 1])
  int W, n_clusters, D, H, B;
  int global_slot;
  float lr;
  const float* master;
  float* master_w;
  int64_t slot_stride;
  int64_t offW0, offB0, offW1, offB1;
  const int32_t* labels;
  int max_tau;
  int* err;
  unsigned long long* phase_ts;   // [max_tau][4] phase stamps of worker 0, or null
  float* loss_out;                // [W] mean mini-batch loss of the round (written at the end)
  int64_t* cursor;                // [W] advanced by tau * B modulo n at the end, or null
  const int64_t* shard_n;         // [W]
  int priority;                   // launch priority (cudaLaunchAttributePriority); 0: the stream's
};
// whole-round kernel for input -> H ReLU -> 10 classes (one cluster per
// worker, the worker's model resident on chip for the round)
bool fused_round_supported(int L, int D, int H, int C, int B);
int fused_round_xt_rows(int B);   // rows of the X^T box the kernel loads
// clusters of the round kernel that fit on the device at once (0 if unknown)
int fused_round_max_clusters(int D, int H, int B);
// mX: staged inputs {D, B, W, steps} box {64, B}; mXT: staged transposed
// inputs {B, D, W, steps} box {64, fused_round_xt_rows(B)}; both bf16,
// 128-byte swizzle.  mW0f: the global slot's W0 {D, H, 1} fp32, box
// {32, 128}, 128-byte swizzle (the kernel rounds its own bf16 operand).
// mRep32 / mRep16: W0 of every replica slot {D, H, slots} fp32, box
// {32, 32} with 128-byte swizzle / {16, 32} without (the last step's stores)
cudaError_t launch_fused_round(const CUtensorMap& mX, const CUtensorMap& mXT, const CUtensorMap& mW0f,
                               const CUtensorMap& mRep32, const CUtensorMap& mRep16, const FusedRoundArgs& a,
                               cudaStream_t s);

// loss[w] = sum_{s < tau[w]} sum_c part[(w*max_tau + s)*nc + c] / (B * tau[w])
cudaError_t launch_loss_finalize(const float* part, const int32_t* tau, int W, int max_tau,
                                 int nc, int B, float* loss, cudaStream_t s);
// the result of an evaluation: loss = scale * sum_i part[i] (fixed order), err
// = the device error word, which is cleared; `out` in mapped host memory.
// pdl: as a programmatic dependent of the launch before it.
struct EvalResult {
  float loss;
  int err;
};
cudaError_t launch_eval_result(const float* part, int64_t count, double scale, int* err, EvalResult* out, int pdl,
                               cudaStream_t s);
// cursor[w] = (cursor[w] + tau[w] * B) % n[w]
cudaError_t launch_cursor_advance(int64_t* cursor, const int32_t* tau, const int64_t* n, int B,
                                  int W, cudaStream_t s);
// shadow[p] = bf16(master[p]) for one slot
cudaError_t launch_shadow_refresh(const float* master, __nv_bfloat16* shadow, int64_t count,
                                  cudaStream_t s);
// replicas[k] = x_g for k < W (fp32 and bf16 shadows)
cudaError_t launch_broadcast(const float* xg, float* slab, int64_t stride, int W, int64_t count,
                             cudaStream_t s);

// ---------------------------------------------------------------- convolutional worker
// 32 x 32 images, 64 channels, 3x3 convolutions (csrc/cnn.cu)

struct ConvArgs {
  const int* wid;              // [n_active] lane of each active entry
  const int* src;              // [n_active] slot whose weights the step reads
  int B;                       // images per lane
  const float* bias;           // forward: fp32 slab; bias of slot s at bias + s * slot_stride + off_bias
  int64_t slot_stride, off_bias;
  int has_add;                 // a tensor is added before the activation / mask (ConvMaps::add4)
  float* pool_part;            // forward: [lane * B + image][32 image rows][64] channel sums of the output, or null
  float* bias_part;            // input gradient: [lane][cpw][64] per-CTA channel sums, or null
  int* err;
  int im2col;                  // forward only: 1 = the stem as one 64 x 64 product over the im2col input
};
// tensors an implicit GEMM's epilogue reads and writes, [lane * B + image][32][32][64] bf16
struct ConvMaps {
  CUtensorMap add4;            // added before the activation / mask, box of 4 image rows (has_add)
  CUtensorMap mask4;           // input gradient: stored activation of the layer input (> 0 keeps), 4 image rows
  CUtensorMap out1;            // the output, box of one image row
};
struct WgradArgs {
  const int* wid;
  int B, n_chunks;             // chunk c: K-blocks (2 image rows) [c n / n_chunks, (c + 1) n / n_chunks) of n = 16 B
  float* part;                 // [lane][n_chunks][9][64 in][64 out]
  int* err;
  int im2col;                  // 1 = the stem over the im2col input: tap 0 of `part` only
};
constexpr int kMaxConvLayers = 9;
struct ConvSgdArgs {
  const int* wid;
  const int* src;
  int n_chunks, layers;
  int n_tiles[kMaxConvLayers];             // per layer: bias partials per lane
  const float* part[kMaxConvLayers];       // per layer, as WgradArgs::part
  const float* bias_part[kMaxConvLayers];  // per layer: [lane][n_tiles][64]
  __nv_bfloat16* wt[kMaxConvLayers];       // per layer: transposed bf16 copy in slot 0, or null
  int im2col[kMaxConvLayers];              // per layer: 1 = weights [64 out][64 k] (one tap)
  int64_t offW[kMaxConvLayers], offB[kMaxConvLayers];
  const float* master;
  float* master_w;
  __nv_bfloat16* shadow;
  int64_t slot_stride, wt_slot_stride;
  float lr;
};
struct CnnStageArgs {
  const float* const* x;       // [W] fp32 NHWC shards; null: the evaluation set below
  const int32_t* const* y;
  const int64_t* n;
  const int64_t* start;        // [W] cursors
  const float* x1;             // evaluation: images from eval_base + lane * B (mod n1)
  const int32_t* y1;
  int64_t n1, eval_base;
  const int* wid;
  int step, B, Cin;
  int im2col;                  // 1: channel k = tap * Cin + i holds x[y + dy - 1][x + dx - 1][i], tap = 3 dy + dx
  __nv_bfloat16* out;          // [lane][B][1024][64]
  int32_t* labels;             // [lane][B] or null
};
struct CnnHeadArgs {
  const int* wid;
  const int* src;
  int B, K, step, max_tau, n_loss_chunks;
  const float* pool_part;      // [lane * B + image][32][64] channel sums of the image rows
  const int32_t* labels;       // [lane][B]
  float* dg;                   // [lane][B][64]
  float* loss_part;            // [(lane * max_tau + step) * n_loss_chunks + chunk]
  const float* master;
  float* master_w;
  __nv_bfloat16* shadow;
  int64_t slot_stride, offWf, offBf;
  float lr;
};
int cnn_tiles_per_image();
// split-K chunks of the weight gradient per worker (one wave of CTAs over the active workers, at most B)
int conv_wgrad_chunks(int B, int n_active, int sms);
// CTAs per worker of the implicit-GEMM kernel (one per SM over the active workers)
int conv_ctas_per_worker(int B, int n_active, int sms);
cudaError_t launch_conv_igemm(int mode, const CUtensorMap& mIn, const CUtensorMap& mW, const ConvMaps& mm,
                              const ConvArgs& a, int n_active, int cpw, cudaStream_t s);
cudaError_t launch_conv_wgrad(const CUtensorMap& mIn, const CUtensorMap& mDz, const WgradArgs& a, int n_active,
                              cudaStream_t s);
cudaError_t launch_conv_sgd(const ConvSgdArgs& a, int n_active, cudaStream_t s);
cudaError_t launch_conv_refresh_wt(const float* master, __nv_bfloat16* wt, int64_t offW, cudaStream_t s);
cudaError_t launch_cnn_stage(const CnnStageArgs& a, int n_active, cudaStream_t s);
cudaError_t launch_cnn_head(const CnnHeadArgs& a, int n_active, cudaStream_t s);
// out[lane] = loss sum of the lane's first min(B, n_img - lane * B) images, lane < lanes
cudaError_t launch_cnn_head_loss(const float* pool_part, const int32_t* labels, int lanes, int B, int64_t n_img, int K,
                                 const float* master, int64_t offWf, int64_t offBf, float* out, cudaStream_t s);
cudaError_t launch_cnn_dzb(const __nv_bfloat16* v, const float* dg, const int* wid, int B, __nv_bfloat16* dz,
                           float* bias_part, int n_active, cudaStream_t s);

}  // namespace oscars
