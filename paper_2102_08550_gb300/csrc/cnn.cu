// The convolutional worker: local SGD steps of a CIFAR-shaped residual
// network (Eq. 4, "otherwise" branch, for the paper's kind of workload:
// ResNet on CIFAR-10, Section "Dataset and DL Models").
//
//   s = relu(conv(x) + b0);  per block u = relu(conv(h) + b_a),
//   v = relu(conv(u) + b_b + h);  g = mean_{y,x} v;  logits = g W_f^T + b_f
//
// Every convolution is 3x3, stride 1, zero padding 1, on 32 x 32 images with
// 64 channels (the input's channels are zero-padded to 64).  Activations are
// bf16 NHWC [lane][image][32][32][64]; a lane is one worker's batch.
//
// Kernels (all workers of a local step in one launch, grid y = active worker):
//  * conv_igemm_kernel: implicit GEMM on tcgen05.  An output tile is 128
//    pixels (4 image rows) x 64 channels, the sum over the 9 taps of
//    [128 pixels x 64 in-channels] x [64 x 64] products; one TMA box of 6 rows
//    serves the three y-offsets (the zero padding is TMA's out-of-bounds
//    fill), the three x-offsets are 192 columns of one product whose sum is
//    taken in the epilogue, and a CTA keeps its worker's weights resident across its
//    tiles.  Forward epilogue: bias, optional residual, ReLU, bf16.
//    Input-gradient mode: the boxes are shifted the other way and the weights
//    are the transposed copy; epilogue: optional skip-path gradient, the ReLU
//    mask of the layer input, bf16, and per-CTA channel sums for the bias
//    gradient.
//  * conv_wgrad_kernel: dW[o][tap][i] = sum_p dz[p][o] x[p + off(tap)][i] on
//    tcgen05 with both operands MN-major straight from the NHWC tensors: the
//    K dimension is the pixels, M = 128 (in-channels of two taps), N = 192
//    (out-channels of three x-offsets).  Split over chunks of the worker's
//    pixels (one wave of CTAs); partial sums go to global memory.
//  * conv_sgd_kernel: sums the chunks in order, SGD of the fp32 master and
//    its bf16 copies (the forward layout and the transposed one), bias from
//    the per-tile sums.
//  * head (pooling of the last convolution's row sums, FC, softmax) and
//    output-gradient kernels on CUDA cores; input staging.
#include "common.cuh"
#include "internal.h"

namespace oscars {
namespace {

constexpr int kCC = 64;                     // channels
constexpr int kImg = 32;                    // image height and width
constexpr int kPix = kImg * kImg;
constexpr int kTileRows = 4;                // image rows per 128-pixel tile
constexpr int kTilePix = kTileRows * kImg;  // 128
constexpr int kTilesPerImg = kImg / kTileRows;
constexpr int kTaps = 9;
constexpr int kCT = 128;                    // threads of the implicit-GEMM and pixel kernels
constexpr int kCB = kCC * kCC * 2;          // 8 KB: one tap of the weights
// weight gradient
constexpr int kWT = 128;
constexpr int kWTile = 2 * kImg * kCC * 2;  // 8 KB: 64 pixels (2 rows) x 64 channels

__device__ __forceinline__ uint8_t* align1024(uint8_t* p) {
  return reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(p) + 1023) & ~uintptr_t(1023));
}

// ------------------------------------------------------------------ implicit GEMM (forward / input gradient)
// A CTA works through tiles c, c + cpw, c + 2 cpw, ... of one worker (grid x
// = c < cpw, grid y = active worker) with that worker's 9 weight taps resident
// in shared memory.  Per tile TMA loads one box of 6 image rows (y0 - 1 .. y0
// + 4); the three y-offsets are its 4-row sub-tiles at row offsets 0, 1, 2
// (multiples of 8 pixel rows of 128 bytes, so the 128-byte swizzle phase is
// unchanged).  The x-offsets are not shifts of the input but columns of the
// product: with N = 192 the three taps of one dy multiply the same sub-tile,
//   E[q][dx][o] = sum_dy x[q + (dy - 1, 0)] W[dy][dx][o],
//   out[p][o] = sum_dx E[p + (0, dx - 1)][dx][o],
// and a row of the image is the 32 lanes of a warp, so the sum over dx is two
// shuffles a channel with zero at the image's edges.  What bounds the kernel
// is the shared memory bandwidth (128 bytes a clock): operands 120 KB, TMA
// writes 24 KB, shuffles and epilogue about 100 KB a tile; with three shifted
// boxes and N = 64 it was 216 + 72 KB and 2900 to 3400 clocks a tile (36 us a
// forward launch of up to 16 workers, 48 an input gradient), 33 and 49:
// at 16 workers a launch moves 128 to 256 MB of activations, 19 to 38 us of HBM.
//
// Two TMEM accumulators and two epilogue warpgroups, tile k with accumulator
// and group k % 2: the epilogues of two tiles overlap the MMAs of a third.
// What an epilogue reads beside the accumulator (the residual, the mask, the
// skip gradient) comes by TMA into a tile buffer of its group, laid out like
// the output; a thread (one pixel) updates its 128-byte row there in place,
// and a warp (one image row) sends it out with one TMA store.  Loads and
// stores of a pixel's row by its thread touched 32 lines an instruction: they
// took the load/store unit about 2000 clocks a tile, four times the MMAs, and
// the kernels ran at 41 us (forward) and 60 us (input gradient) a launch of
// up to 16 workers; 36 and 48 us with this epilogue.  In the input gradient a
// thread also keeps 64 channel sums over its tiles: 168 registers at 320 threads,
// and 52 bytes spilled.
constexpr int kGT = 320;                    // warp 0 TMA, warp 1 MMA, warps 2-5 and 6-9 epilogue
constexpr int kGSlots = 4;                  // input boxes in flight (one a tile)
constexpr int kGAcc = 256;                  // TMEM columns of an accumulator (192 used)
constexpr int kGBox = 6 * kImg * kCC * 2;   // 24 KB: 6 rows x 32 pixels x 64 channels
constexpr int kGW = kTaps * kCB;            // 72 KB of resident weights
constexpr int kGTile = kTilePix * kCC * 2;  // 16 KB: an output tile
constexpr int kGOffE = kGW + kGSlots * kGBox;      // [2] tile buffer of a group: residual or mask, then the output
constexpr int kGOffS = kGOffE + 2 * kGTile;        // skip gradient (input gradient)
constexpr int kGOffBar = kGOffS + kGTile;
constexpr int kGSmem = kGOffBar + 512 + 1024;      // + barriers, TMEM slot, bias
static_assert(2 * kTilePix * (kCC + 1) * 4 <= kGSlots * kGBox, "the bias reduction reuses the input slots");

template <int MODE>   // 0 forward, 1 input gradient
__global__ void __launch_bounds__(kGT, 1) conv_igemm_kernel(const __grid_constant__ CUtensorMap mIn,
                                                            const __grid_constant__ CUtensorMap mW,
                                                            const __grid_constant__ ConvMaps mm,
                                                            const __grid_constant__ ConvArgs a) {
  extern __shared__ uint8_t cs_raw[];
  uint8_t* sm = align1024(cs_raw);
  uint8_t* wts = sm;                 // [9][64][64] bf16, 128-byte swizzled K-major
  uint8_t* slots = sm + kGW;         // [kGSlots][6 rows][32][64]
  uint64_t* wfull = reinterpret_cast<uint64_t*>(sm + kGOffBar);
  uint64_t* full = wfull + 1;
  uint64_t* empty = full + kGSlots;
  uint64_t* accf = empty + kGSlots;  // [2]
  uint64_t* acce = accf + 2;         // [2] 128 arrivals
  uint64_t* auxf = acce + 2;         // [2] the tile buffer (and skip gradient) has landed
  uint64_t* auxe = auxf + 2;         // [2] the tile buffer has been stored: 4 arrivals
  uint64_t* skipe = auxe + 2;        // the skip gradient has been read: 4 arrivals
  uint32_t* tslot = reinterpret_cast<uint32_t*>(skipe + 1);
  float* bias_s = reinterpret_cast<float*>(tslot + 4);   // [64] this worker's bias (forward)
  const int t = threadIdx.x, warp = __shfl_sync(0xffffffffu, t >> 5, 0), lane_id = t & 31;
  const int c0 = blockIdx.x, cpw = gridDim.x, e = blockIdx.y;
  const int lane = a.wid[e], slot = a.src[e];
  const int ntiles = a.B * kTilesPerImg;
  const int my_tiles = (ntiles - c0 + cpw - 1) / cpw;
  if (t == 0) {
    prefetch_tmap(&mIn);
    prefetch_tmap(&mW);
    prefetch_tmap(&mm.out1);
    mbar_init(wfull, 1);
    for (int i = 0; i < kGSlots; ++i) {
      mbar_init(&full[i], 1);
      mbar_init(&empty[i], 1);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(&accf[i], 1);
      mbar_init(&acce[i], 128);
      mbar_init(&auxf[i], 1);
      mbar_init(&auxe[i], 4);
    }
    mbar_init(skipe, 4);
    fence_barrier_init();
  }
  if (warp == 0) {
    tmem_alloc(tslot, 512);
    tmem_relinquish();
  }
  if (MODE == 0 && t >= 64 && t < 64 + kCC)
    bias_s[t - 64] = a.bias[static_cast<int64_t>(slot) * a.slot_stride + a.off_bias + (t - 64)];
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tslot;
  // im2col stem (forward): one tap of weights, one 4-row box per tile (mIn's
  // box is {64, 32, 4, 1}), four MMAs
  const bool one_tap = MODE == 0 && a.im2col;
  // forward: the residual (if any) in the tile buffer; input gradient: the
  // mask there and the skip gradient (if any) in its own buffer
  const bool aux = MODE == 1 || a.has_add, skip = MODE == 1 && a.has_add;
  if (t == 0) {
    mbar_arrive_expect_tx(wfull, one_tap ? kCB : kGW);
    for (int tap = 0; tap < (one_tap ? 1 : kTaps); ++tap) {
      if (MODE == 0) tma_load_4d(wts + tap * kCB, &mW, 0, tap, 0, slot, wfull);   // {in, tap, out, slot}
      else tma_load_4d(wts + tap * kCB, &mW, 0, 0, tap, slot, wfull);             // {out, in, tap, slot}
    }
    for (int k = 0; k < my_tiles; ++k) {
      const int tile = c0 + k * cpw;
      const int img = lane * a.B + tile / kTilesPerImg, y0 = (tile % kTilesPerImg) * kTileRows;
      const int sl = k % kGSlots;
      if (k >= kGSlots && !mbar_wait(&empty[sl], ((k / kGSlots) + 1) & 1, a.err, kDevTimeoutEmpty)) break;
      mbar_arrive_expect_tx(&full[sl], one_tap ? kGTile : kGBox);
      tma_load_4d(slots + sl * kGBox, &mIn, 0, 0, one_tap ? y0 : y0 - 1, img, &full[sl]);
      if (aux) {
        const int p = k & 1, use = k >> 1;
        // the group's previous output has left the tile buffer; the previous tile has read the skip gradient
        if (use >= 1 && !mbar_wait(&auxe[p], (use - 1) & 1, a.err, kDevTimeoutEmpty)) break;
        if (skip && k >= 1 && !mbar_wait(skipe, (k - 1) & 1, a.err, kDevTimeoutEmpty)) break;
        mbar_arrive_expect_tx(&auxf[p], skip ? 2 * kGTile : kGTile);
        tma_load_4d(sm + kGOffE + p * kGTile, MODE == 1 ? &mm.mask4 : &mm.add4, 0, 0, y0, img, &auxf[p]);
        if (skip) tma_load_4d(sm + kGOffS, &mm.add4, 0, 0, y0, img, &auxf[p]);
      }
    }
  } else if (warp == 1) {   // converged, one elected lane issues: see elect_one
    constexpr uint32_t idesc = idesc_bf16_f32(128, kCC), idesc3 = idesc_bf16_f32(128, 3 * kCC);
    uint32_t limit = kSpinLimit;
    mbar_wait_keep(limit, wfull, 0, a.err, kDevTimeoutFull);
    tc_fence_after();
    const uint64_t wb = smem_desc_k128(smem_u32(wts));
    for (int k = 0; k < my_tiles; ++k) {
      const int buf = k & 1, use = k >> 1, sl = k % kGSlots;
      if (use >= 1) mbar_wait_keep(limit, &acce[buf], (use - 1) & 1, a.err, kDevTimeoutAccum);
      mbar_wait_keep(limit, &full[sl], (k / kGSlots) & 1, a.err, kDevTimeoutFull);
      tc_fence_after();
      // descriptors count 16 bytes: 2 for the 32 bytes of a K slice
      const uint64_t sa = smem_desc_k128(smem_u32(slots + sl * kGBox));
      const uint32_t acc = tmem + buf * kGAcc;
      if (elect_one() && limit > 1) {
        if (one_tap) {
#pragma unroll
          for (int j = 0; j < kCC / 16; ++j) umma_bf16(acc, sa + 2 * j, wb + 2 * j, idesc, j != 0 ? 1u : 0u);
        } else {
#pragma unroll
          for (int dy = 0; dy < 3; ++dy) {
            // sub-tile of the 6-row box; the input gradient reads the output gradient at p - off(tap)
            const int rowoff = MODE == 0 ? dy : 2 - dy;
            const uint64_t aa = sa + rowoff * (kImg * kCC * 2 / 16), bb = wb + dy * (3 * kCB / 16);
#pragma unroll
            for (int j = 0; j < kCC / 16; ++j)
              umma_bf16(acc, aa + 2 * j, bb + 2 * j, idesc3, (dy | j) != 0 ? 1u : 0u);
          }
        }
        umma_commit(&empty[sl]);
        umma_commit(&accf[buf]);
      }
      __syncwarp();
    }
  } else if (warp >= 2) {
    // epilogue: thread = output pixel (TMEM lane of its warp's quarter), 64
    // channels; warp = image row y0 + quarter
    const int grp = (warp - 2) >> 2, quarter = warp & 3;
    const int p = quarter * 32 + lane_id;
    const uint32_t trow = tmem + (static_cast<uint32_t>(quarter * 32) << 16) + grp * kGAcc;
    uint8_t* row = sm + kGOffE + grp * kGTile + p * 128;          // 16-byte chunk q at (q ^ (p & 7))
    const uint8_t* srow = sm + kGOffS + p * 128;
    const uint32_t sw = static_cast<uint32_t>(p & 7);
    float bsum[kCC];
#pragma unroll
    for (int c = 0; c < kCC; ++c) bsum[c] = 0.f;
    for (int k = grp; k < my_tiles; k += 2) {
      const int tile = c0 + k * cpw;
      const int img = lane * a.B + tile / kTilesPerImg, y0 = (tile % kTilesPerImg) * kTileRows;
      const int use = k >> 1;
      int ok = mbar_wait(&accf[grp], use & 1, a.err, kDevTimeoutAccum) ? 1 : 0;
      ok = __all_sync(0xffffffffu, ok);
      tc_fence_after();
      if (aux) {
        mbar_wait(&auxf[grp], use & 1, a.err, kDevTimeoutFull);
      } else {   // this warp's previous output has left its rows
        if (lane_id == 0) bulk_wait_read_all();
        __syncwarp();
      }
#pragma unroll
      for (int h = 0; h < 2; ++h) {   // 32 channels at a time
        float v[32];
        // forward: dx 0 from the pixel before, dx 2 from the one after; the input gradient the other way round
        const uint32_t before = trow + (MODE == 0 ? 0 : 2 * kCC) + 32 * h, after = trow + (MODE == 0 ? 2 * kCC : 0) + 32 * h;
        if (one_tap) {
          tmem_ld_32x32b_x32(trow + 32 * h, v);
        } else {
          float l[32];
          tmem_ld_32x32b_x32_pair(trow + kCC + 32 * h, v, before, l);
#pragma unroll
          for (int c = 0; c < 32; ++c) {
            const float x = __shfl_up_sync(0xffffffffu, l[c], 1);
            v[c] += lane_id == 0 ? 0.f : x;
          }
          tmem_ld_32x32b_x32(after, l);
#pragma unroll
          for (int c = 0; c < 32; ++c) {
            const float x = __shfl_down_sync(0xffffffffu, l[c], 1);
            v[c] += lane_id == 31 ? 0.f : x;
          }
        }
        if (h == 1) {
          tc_fence_before();
          mbar_arrive(&acce[grp]);   // the accumulator has been read: the next tile may use it
        }
#pragma unroll
        for (int c = 0; c < 32; ++c) v[c] = ok ? v[c] + (MODE == 0 ? bias_s[32 * h + c] : 0.f) : 0.f;
        if (a.has_add) {
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            const uint4 r = *reinterpret_cast<const uint4*>((MODE == 0 ? row : srow) + (((4 * h + q) ^ sw) << 4));
            const __nv_bfloat162* r2 = reinterpret_cast<const __nv_bfloat162*>(&r);
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              const float2 f = __bfloat1622float2(r2[j]);
              v[8 * q + 2 * j] += f.x;
              v[8 * q + 2 * j + 1] += f.y;
            }
          }
          if (skip && h == 1) {
            __syncwarp();
            if (lane_id == 0) mbar_arrive(skipe);
          }
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          uint4* chunk = reinterpret_cast<uint4*>(row + (((4 * h + q) ^ sw) << 4));
          if (MODE == 0) {
#pragma unroll
            for (int j = 0; j < 8; ++j) v[8 * q + j] = fmaxf(v[8 * q + j], 0.f);
          } else {
            const uint4 r = *chunk;   // the mask
            const __nv_bfloat162* r2 = reinterpret_cast<const __nv_bfloat162*>(&r);
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              const float2 f = __bfloat1622float2(r2[j]);
              if (!(f.x > 0.f)) v[8 * q + 2 * j] = 0.f;
              if (!(f.y > 0.f)) v[8 * q + 2 * j + 1] = 0.f;
            }
#pragma unroll
            for (int j = 0; j < 8; ++j) bsum[32 * h + 8 * q + j] += v[8 * q + j];
          }
          const uint4 o = make_uint4(pack_bf16x2(v[8 * q], v[8 * q + 1]), pack_bf16x2(v[8 * q + 2], v[8 * q + 3]),
                                     pack_bf16x2(v[8 * q + 4], v[8 * q + 5]), pack_bf16x2(v[8 * q + 6], v[8 * q + 7]));
          *chunk = o;
          if (MODE == 0) {   // the pooling sums the stored values
            const __nv_bfloat162* o2 = reinterpret_cast<const __nv_bfloat162*>(&o);
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              const float2 f = __bfloat1622float2(o2[j]);
              v[8 * q + 2 * j] = f.x;
              v[8 * q + 2 * j + 1] = f.y;
            }
          }
        }
        if (MODE == 0 && a.pool_part) {
          // channel sums over the image row's 32 pixels: halves exchanged over
          // the lanes until a lane holds one channel (its own index of the 32)
#pragma unroll
          for (int w = 16; w > 0; w >>= 1) {
            const bool up = lane_id & w;
#pragma unroll
            for (int c = 0; c < 16; ++c)
              if (c < w) {
                const float keep = up ? v[c + w] : v[c], give = up ? v[c] : v[c + w];
                v[c] = keep + __shfl_xor_sync(0xffffffffu, give, w);
              }
          }
          a.pool_part[(static_cast<int64_t>(img) * kImg + y0 + quarter) * kCC + 32 * h + lane_id] = v[0];
        }
      }
      fence_proxy_async_smem();   // the rows are read by the TMA store
      __syncwarp();
      if (lane_id == 0) {
        tma_store_4d(&mm.out1, sm + kGOffE + grp * kGTile + quarter * 32 * 128, 0, 0, y0 + quarter, img);
        bulk_commit_group();
      }
      if (aux && lane_id == 0) {   // the tile buffer may take the next tile's inputs
        bulk_wait_read_all();
        mbar_arrive(&auxe[grp]);
      }
    }
    if (lane_id == 0) bulk_wait_all();
    if (MODE == 1 && a.bias_part) {
      bar_named(1, 256);   // both groups have seen their last product: the input slots are idle
      // this CTA's channel sums: per thread over its tiles in order, then over
      // the two groups' 128 pixels in order
      float* T = reinterpret_cast<float*>(slots);
#pragma unroll
      for (int c = 0; c < kCC; ++c) T[(grp * kTilePix + p) * (kCC + 1) + c] = bsum[c];
    }
  }
  if (MODE == 1 && a.bias_part) {
    __syncthreads();
    float* T = reinterpret_cast<float*>(slots);
    float* part = reinterpret_cast<float*>(sm + kGOffE);   // [4][64]: every store has left the tile buffers
    if (t < 256) {
      float s = 0.f;
      for (int q = (t >> 6) * 64; q < (t >> 6) * 64 + 64; ++q) s += T[q * (kCC + 1) + (t & 63)];
      part[t] = s;
    }
    __syncthreads();
    if (t < kCC)
      a.bias_part[(static_cast<int64_t>(lane) * cpw + c0) * kCC + t] = part[t] + part[64 + t] + part[128 + t] + part[192 + t];
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    tc_fence_after();
    tmem_dealloc(tmem, 512);
  }
}

// ------------------------------------------------------------------ weight gradient
// K-block = 64 pixels (2 image rows yr, yr + 1).  Per K-block TMA loads one
// 4-row box of the input (rows yr - 1 .. yr + 2) and the two output-gradient
// rows three times, shifted by 1 - dx pixels: sum_p dz[p] x[p + off] over the
// pixels p equals the sum over q = p + (0, dx - 1) of dz[q - (0, dx - 1)]
// x[q + (dy - 1, 0)], and TMA's zero fill drops the terms outside the image.
// So every tap of one dx has the same B, and one MMA covers
//   M = 128: two 64-channel atoms of the input 4 KB apart (dy 0 and dy 1; for
//            dy 2 the upper half is not used)
//   N = 192: the three shifted output gradients, 64 channels each, 8 KB apart
// - 8 MMAs a K-block for the nine taps.  What bounds the kernel is the shared
// memory that the operands are read from (about 128 bytes a clock) and TMA
// writes: 80 + 40 KB a K-block; with the input shifted instead (three boxes,
// 20 MMAs of N = 64) it was 120 + 56 KB and 1350 clocks a K-block: 43 us a
// launch of up to 16 workers, 32 now (nine chunks a worker instead of eight
// whole-image ones and coalesced partial rows included).
constexpr int kWRow = kImg * kCC * 2;           // 4 KB: one image row, 64 channels
constexpr int kWBox = 4 * kWRow;                // 16 KB
constexpr int kWStage2 = kWBox + 3 * kWTile;    // 40 KB: the input box and three output-gradient tiles
constexpr int kWStages2 = 5;
constexpr int kWSmem2 = kWStages2 * kWStage2 + 256 + 1024;
constexpr int kWLd = kCC + 4;                   // row stride of the epilogue's staging (floats): conflict-free both ways
static_assert(kWT / 32 * 32 * kWLd * 4 <= kWStages2 * kWStage2, "the epilogue stages in the operand ring");

__global__ void __launch_bounds__(kWT, 1) conv_wgrad_kernel(const __grid_constant__ CUtensorMap mIn,
                                                            const __grid_constant__ CUtensorMap mDz,
                                                            const __grid_constant__ WgradArgs a) {
  extern __shared__ uint8_t ws_raw[];
  uint8_t* sm = align1024(ws_raw);
  uint64_t* full = reinterpret_cast<uint64_t*>(sm + kWStages2 * kWStage2);
  uint64_t* empty = full + kWStages2;
  uint64_t* accb = empty + kWStages2;
  uint32_t* tslot = reinterpret_cast<uint32_t*>(accb + 1);
  const int t = threadIdx.x, warp = __shfl_sync(0xffffffffu, t >> 5, 0), lane_id = t & 31;
  const int chunk = blockIdx.x, e = blockIdx.y;
  const int lane = a.wid[e];
  const int all = a.B * (kImg / 2);              // the worker's K-blocks; this chunk's [kb0, kb0 + nk)
  const int kb0 = static_cast<int>(static_cast<int64_t>(chunk) * all / a.n_chunks);
  const int nk = static_cast<int>(static_cast<int64_t>(chunk + 1) * all / a.n_chunks) - kb0;
  if (t == 0) {
    prefetch_tmap(&mIn);
    prefetch_tmap(&mDz);
    for (int i = 0; i < kWStages2; ++i) {
      mbar_init(&full[i], 1);
      mbar_init(&empty[i], 1);
    }
    mbar_init(accb, 1);
    fence_barrier_init();
  }
  if (warp == 0) {
    tmem_alloc(tslot, 512);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tslot;
  // im2col stem: one 2-row input box per K-block (mIn's box is {64, 32, 2, 1}),
  // one unshifted output-gradient tile and one accumulator, tap 0 in its lower half
  if (t == 0) {
    for (int kb = 0; kb < nk; ++kb) {
      const int st = kb % kWStages2;
      if (kb >= kWStages2 && !mbar_wait(&empty[st], ((kb / kWStages2) + 1) & 1, a.err, kDevTimeoutEmpty)) break;
      uint8_t* sa = sm + st * kWStage2;
      const int img = lane * a.B + (kb0 + kb) / (kImg / 2), yr = ((kb0 + kb) % (kImg / 2)) * 2;
      if (a.im2col) {
        mbar_arrive_expect_tx(&full[st], 2 * kWRow + kWTile);
        tma_load_4d(sa, &mIn, 0, 0, yr, img, &full[st]);
        tma_load_4d(sa + kWBox, &mDz, 0, 0, yr, img, &full[st]);
      } else {
        mbar_arrive_expect_tx(&full[st], kWStage2);
        tma_load_4d(sa, &mIn, 0, 0, yr - 1, img, &full[st]);
        for (int dx = 0; dx < 3; ++dx) tma_load_4d(sa + kWBox + dx * kWTile, &mDz, 0, 1 - dx, yr, img, &full[st]);
      }
    }
  } else if (warp == 1) {   // converged, one elected lane issues: see elect_one
    constexpr uint32_t idesc1 = idesc_bf16_f32_mn(128, kCC), idesc3 = idesc_bf16_f32_mn(128, 3 * kCC);
    uint32_t limit = kSpinLimit;
    for (int kb = 0; kb < nk; ++kb) {
      const int st = kb % kWStages2;
      mbar_wait_keep(limit, &full[st], (kb / kWStages2) & 1, a.err, kDevTimeoutFull);
      tc_fence_after();
      const uint32_t sa = smem_u32(sm + st * kWStage2);
      const uint64_t ad = smem_desc_mn128(sa, kWRow), bd = smem_desc_mn128(sa + kWBox, kWTile);
      if (elect_one() && limit > 1) {
        // K = 16 pixels per MMA: two 8-row groups, 2048 bytes (descriptors count 16)
        if (a.im2col) {   // A's upper atom (the next row) is not read back
#pragma unroll
          for (int j = 0; j < 4; ++j) umma_bf16(tmem, ad + 128 * j, bd + 128 * j, idesc1, (kb | j) != 0 ? 1u : 0u);
        } else {
#pragma unroll
          for (int j = 0; j < 4; ++j) umma_bf16(tmem, ad + 128 * j, bd + 128 * j, idesc3, (kb | j) != 0 ? 1u : 0u);
#pragma unroll
          for (int j = 0; j < 4; ++j)   // dy 2: two image rows further
            umma_bf16(tmem + 3 * kCC, ad + 2 * kWRow / 16 + 128 * j, bd + 128 * j, idesc3, (kb | j) != 0 ? 1u : 0u);
        }
        umma_commit(&empty[st]);
      }
      __syncwarp();
    }
    if (elect_one()) umma_commit(accb);
    __syncwarp();
  }
  int ok = mbar_wait(accb, 0, a.err, kDevTimeoutAccum) ? 1 : 0;
  ok = __all_sync(0xffffffffu, ok);
  tc_fence_after();
  // TMEM lane r: in-channel r % 64 of dy 0 (r < 64) and dy 1 in columns [0,
  // 192), of dy 2 (r < 64) in [192, 384); columns dx * 64 + out-channel.  Rows
  // of 64 go through shared memory (the ring is idle: every product is done)
  // so that a warp writes whole 256-byte rows, two an instruction.
  float* T = reinterpret_cast<float*>(sm) + warp * 32 * kWLd;
  const uint32_t trow = tmem + (static_cast<uint32_t>(warp * 32) << 16);
  const int ci0 = (warp & 1) * 32;
  float* part = a.part + (static_cast<int64_t>(lane) * a.n_chunks + chunk) * kTaps * kCC * kCC;
  for (int i = 0; i < 6; ++i) {
    const int dy = i < 3 ? warp >> 1 : 2, dx = i % 3;
    if (i >= 3 && warp >= 2) break;            // dy 2: lanes 0..63
    if (a.im2col && (i > 0 || warp >= 2)) break;
    float lo[32], hi[32];
    tmem_ld_32x32b_x32_pair(trow + i * kCC, lo, trow + i * kCC + 32, hi);
    if (!ok) continue;
    __syncwarp();
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      *reinterpret_cast<float4*>(T + lane_id * kWLd + 4 * q) = make_float4(lo[4 * q], lo[4 * q + 1], lo[4 * q + 2], lo[4 * q + 3]);
      *reinterpret_cast<float4*>(T + lane_id * kWLd + 32 + 4 * q) = make_float4(hi[4 * q], hi[4 * q + 1], hi[4 * q + 2], hi[4 * q + 3]);
    }
    __syncwarp();
    float* dst = part + ((a.im2col ? 0 : dy * 3 + dx) * kCC + ci0) * kCC;
#pragma unroll 4
    for (int r = 0; r < 32; r += 2) {
      const int rr = r + (lane_id >> 4), q = lane_id & 15;
      *reinterpret_cast<float4*>(dst + rr * kCC + 4 * q) = *reinterpret_cast<const float4*>(T + rr * kWLd + 4 * q);
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    tc_fence_after();
    tmem_dealloc(tmem, 512);
  }
}

// ------------------------------------------------------------------ reduce + SGD of the convolution layers
// grid (taps * 4, active workers, layers), 256 threads: one tap's 16 in-channel
// rows x 64 out-channels of one layer; the chunks are summed in chunk order.
// Latency of the loads is what bounds it: 56 MB for 16 workers took 33 us a
// launch with one load after the other in the bias sums (256 of them), 21
// now.
// The im2col stem has one tap (its blocks of taps 1..8 return at once).
constexpr int kSgdRows = 16;
__global__ void __launch_bounds__(256) conv_sgd_kernel(const __grid_constant__ ConvSgdArgs a) {
  __shared__ float T[kSgdRows][kCC + 1];   // [in][out]
  const int tap = blockIdx.x / (kCC / kSgdRows), r0 = (blockIdx.x % (kCC / kSgdRows)) * kSgdRows;
  const int e = blockIdx.y, layer = blockIdx.z;
  const int lane = a.wid[e], src = a.src[e];
  const int t = threadIdx.x;
  const int ntap = a.im2col[layer] ? 1 : kTaps;   // the im2col stem: [out][k], one tap
  if (tap >= ntap) return;
  const float* part = a.part[layer] + (static_cast<int64_t>(lane) * a.n_chunks * kTaps + tap) * kCC * kCC + r0 * kCC;
  const int64_t chunk_stride = static_cast<int64_t>(kTaps) * kCC * kCC;
  static_assert(kSgdRows * kCC == 4 * 256, "four values a thread");
  {   // eight 16-byte loads in flight a thread
    float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 8
    for (int c = 0; c < a.n_chunks; ++c) {
      const float4 v = *reinterpret_cast<const float4*>(part + c * chunk_stride + 4 * t);
      s.x += v.x;
      s.y += v.y;
      s.z += v.z;
      s.w += v.w;
    }
    float* d = &T[t / (kCC / 4)][t % (kCC / 4) * 4];
    d[0] = s.x;
    d[1] = s.y;
    d[2] = s.z;
    d[3] = s.w;
  }
  __syncthreads();
  const int64_t so = static_cast<int64_t>(src) * a.slot_stride, dof = static_cast<int64_t>(lane) * a.slot_stride;
  const int64_t offW = a.offW[layer];
  // master / forward copy: [out][tap][in], in fastest
  for (int q = t; q < kSgdRows * kCC; q += 256) {
    const int co = q / kSgdRows, ci = q % kSgdRows;
    const int64_t off = offW + (static_cast<int64_t>(co) * ntap + tap) * kCC + r0 + ci;
    const float nw = fmaf(-a.lr, T[ci][co], a.master[so + off]);
    a.master_w[dof + off] = nw;
    a.shadow[dof + off] = __float2bfloat16_rn(nw);
    T[ci][co] = nw;   // in this loop every element is read and rewritten by one thread
  }
  if (a.wt[layer]) {
    __syncthreads();
    // transposed copy [tap][in][out], out fastest
    __nv_bfloat16* wt = a.wt[layer] + static_cast<int64_t>(lane) * a.wt_slot_stride +
                        (static_cast<int64_t>(tap) * kCC + r0) * kCC;
    for (int q = t; q < kSgdRows * kCC; q += 256) wt[q] = __float2bfloat16_rn(T[q / kCC][q % kCC]);
  }
  if (blockIdx.x == 0) {   // bias: four threads a channel over the per-tile sums, 16 loads in flight each
    __syncthreads();
    float* P = &T[0][0];   // [4][64]
    const int n = a.n_tiles[layer], c = t & (kCC - 1), g = t / kCC;
    const float* bp = a.bias_part[layer] + static_cast<int64_t>(lane) * n * kCC + c;
    float s = 0.f;
#pragma unroll 16
    for (int i = g; i < n; i += 4) s += bp[static_cast<int64_t>(i) * kCC];
    P[t] = s;
    __syncthreads();
    if (t < kCC) {
      s = P[t] + P[kCC + t] + P[2 * kCC + t] + P[3 * kCC + t];
      a.master_w[dof + a.offB[layer] + t] = fmaf(-a.lr, s, a.master[so + a.offB[layer] + t]);
    }
  }
}

// bf16 transposed weight copies of one slot from its fp32 master (after a merge)
__global__ void conv_refresh_wt_kernel(const float* master, __nv_bfloat16* wt, int64_t offW) {
  const int tap = blockIdx.x;
  for (int q = threadIdx.x; q < kCC * kCC; q += blockDim.x) {
    const int ci = q / kCC, co = q % kCC;
    wt[static_cast<int64_t>(tap) * kCC * kCC + q] =
        __float2bfloat16_rn(master[offW + (static_cast<int64_t>(co) * kTaps + tap) * kCC + ci]);
  }
}

// ------------------------------------------------------------------ input staging
// grid (B * 8 tiles, active), 128 threads: the image row of sample b is
// (start[lane] + s * B + b) mod n[lane] of the lane's shard (fp32 NHWC, Cin
// channels).  Channels >= Cin stay zero: the buffer is cleared once when the
// context is built, so only the 16-byte chunks that hold input channels are
// written (one chunk for Cin <= 8), item = (pixel, chunk) with consecutive
// threads on consecutive chunks.  With im2col (9 Cin <= 64) channel
// k = tap * Cin + i of pixel (y, x) is x[y + dy - 1][x + dx - 1][i] for
// tap = 3 dy + dx (zero outside the image): the stem becomes one 64 x 64
// product per pixel.
// im2col: the tile's 6 source rows (y0 - 1 .. y0 + 4) are first copied to
// shared memory with coalesced loads, with a zero pixel on either side; a
// thread always has the same 16-byte chunk, so that its 8 channels' offsets
// from the centre pixel stay in registers.
constexpr int kStageMaxCin = kCC / kTaps;   // 7: the largest input with an im2col stem
__global__ void __launch_bounds__(kCT) cnn_stage_kernel(const __grid_constant__ CnnStageArgs a) {
  __shared__ float rows[(kTileRows + 2) * (kImg + 2) * kStageMaxCin + 1];
  __shared__ int koff_s[kCC];
  const int tile = blockIdx.x, e = blockIdx.y;
  const int lane = a.wid[e];
  const int b = tile / kTilesPerImg, pix0 = (tile % kTilesPerImg) * kTilePix;
  const bool eval = a.x == nullptr;
  const int64_t n = eval ? a.n1 : a.n[lane];
  const int64_t row = (eval ? a.eval_base + static_cast<int64_t>(lane) * a.B + b
                            : a.start[lane] + static_cast<int64_t>(a.step) * a.B + b) % n;
  const float* src = (eval ? a.x1 : a.x[lane]) + row * static_cast<int64_t>(kPix) * a.Cin;
  __nv_bfloat16* dst = a.out + ((static_cast<int64_t>(lane) * a.B + b) * kPix + pix0) * kCC;
  const int K = a.im2col ? kTaps * a.Cin : a.Cin;
  const int chunks = (K + 7) / 8;
  if (a.labels && tile % kTilesPerImg == 0 && threadIdx.x == 0)
    a.labels[static_cast<int64_t>(lane) * a.B + b] = (eval ? a.y1 : a.y[lane])[row];
  if (a.im2col) {
    const int Cin = a.Cin, rowel = kImg * Cin, pitch = rowel + 2 * Cin, y0 = pix0 / kImg;
    // chunk of this thread: chunks rounded up to a power of two lanes a pixel
    const int csh = chunks <= 1 ? 0 : 32 - __clz(chunks - 1);
    const int q = threadIdx.x & ((1 << csh) - 1);
    const int zero = (kTileRows + 2) * pitch;   // an element that stays zero: channels past K
    if (threadIdx.x < kCC) {
      const int k = threadIdx.x, tap = k / Cin, i = k - tap * Cin;
      koff_s[k] = k < K ? (tap / 3) * pitch + (tap % 3) * Cin + i : -1;
    }
    for (int i = threadIdx.x; i < (kTileRows + 2) * rowel; i += kCT) {
      const int r = i / rowel, x = i - r * rowel, yy = y0 - 1 + r;
      rows[r * pitch + Cin + x] = yy >= 0 && yy < kImg ? src[static_cast<int64_t>(y0 - 1) * rowel + i] : 0.f;
    }
    for (int i = threadIdx.x; i < (kTileRows + 2) * 2 * Cin; i += kCT) {   // the pixels beside the image
      const int r = i / (2 * Cin), x = i - r * 2 * Cin;
      rows[r * pitch + (x < Cin ? x : rowel + x)] = 0.f;
    }
    if (threadIdx.x == 0) rows[zero] = 0.f;
    __syncthreads();
    int koff[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) koff[j] = koff_s[8 * q + j];
    if (q < chunks)
      for (int px = threadIdx.x >> csh; px < kTilePix; px += kCT >> csh) {
        const int centre = (px / kImg) * pitch + (px % kImg) * Cin;   // its upper left neighbour
        float v[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) v[j] = rows[koff[j] >= 0 ? centre + koff[j] : zero];
        *reinterpret_cast<uint4*>(dst + static_cast<int64_t>(px) * kCC + 8 * q) =
            make_uint4(pack_bf16x2(v[0], v[1]), pack_bf16x2(v[2], v[3]), pack_bf16x2(v[4], v[5]), pack_bf16x2(v[6], v[7]));
      }
    return;
  }
  for (int it = threadIdx.x; it < kTilePix * chunks; it += kCT) {
    const int px = it / chunks, q = it - px * chunks;
    float v[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const int c = 8 * q + j;
      v[j] = c < K ? src[static_cast<int64_t>(pix0 + px) * a.Cin + c] : 0.f;
    }
    *reinterpret_cast<uint4*>(dst + static_cast<int64_t>(px) * kCC + 8 * q) =
        make_uint4(pack_bf16x2(v[0], v[1]), pack_bf16x2(v[2], v[3]), pack_bf16x2(v[4], v[5]), pack_bf16x2(v[6], v[7]));
  }
}

// ------------------------------------------------------------------ head: pooling, FC, softmax CE, backward, SGD of the FC
// The last convolution leaves the channel sums of every image row
// (pool_part [image][32 rows][64]); g[b][c] = their sum / 1024.  A row of 64
// features is kept kGld floats apart in shared memory: with 64 the threads of
// a warp, one sample each, all read one bank (the logits then took 10 us).
constexpr int kGld = kCC + 1;

// rounded pooled features of `n` images of a lane into gb [n][kGld]
__device__ __forceinline__ void gather_pooled(const float* pool, int n, float* gb, int threads) {
  for (int i = threadIdx.x; i < n * (kCC / 4); i += threads) {
    const int b = i >> 4, c = (i & 15) * 4;
    const float4* src = reinterpret_cast<const float4*>(pool + static_cast<int64_t>(b) * kImg * kCC + c);
    float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 16
    for (int y = 0; y < kImg; ++y) {
      const float4 v = src[y * (kCC / 4)];
      s.x += v.x;
      s.y += v.y;
      s.z += v.z;
      s.w += v.w;
    }
    float* d = gb + b * kGld + c;
    d[0] = bf16_round(s.x / static_cast<float>(kPix));
    d[1] = bf16_round(s.y / static_cast<float>(kPix));
    d[2] = bf16_round(s.z / static_cast<float>(kPix));
    d[3] = bf16_round(s.w / static_cast<float>(kPix));
  }
}

// grid (active), 512 threads; B <= 256, K <= 32
constexpr int kHeadT = 512;
__global__ void __launch_bounds__(kHeadT) cnn_head_kernel(const __grid_constant__ CnnHeadArgs a) {
  extern __shared__ float hsm[];
  const int K = a.K, B = a.B;
  float* gb = hsm;                    // [B][kGld] bf16-rounded pooled features
  float* wf = gb + B * kGld;          // [K][64] bf16-rounded head weights
  float* wm = wf + K * kCC;           // [K][64] fp32 master
  float* dl = wm + K * kCC;           // [B][K] logits, then their fp32 gradient
  float* dlb = dl + B * K;            // [B][K] bf16-rounded
  float* rl = dlb + B * K;            // [B] per-sample loss
  float* bfm = rl + B;                // [32]
  const int e = blockIdx.x, lane = a.wid[e], src = a.src[e];
  const int t = threadIdx.x;
  const int64_t so = static_cast<int64_t>(src) * a.slot_stride, dof = static_cast<int64_t>(lane) * a.slot_stride;
  gather_pooled(a.pool_part + static_cast<int64_t>(lane) * B * kImg * kCC, B, gb, kHeadT);
  for (int q = t; q < K * kCC; q += kHeadT) {
    const float m = a.master[so + a.offWf + q];
    wm[q] = m;
    wf[q] = bf16_round(m);
  }
  if (t < K) bfm[t] = a.master[so + a.offBf + t];
  __syncthreads();
  // logits: item = (class, sample), samples fastest (the class weights broadcast)
  for (int q = t; q < B * K; q += kHeadT) {
    const int k = q / B, b = q - k * B;
    float acc = 0.f;
#pragma unroll 16
    for (int c = 0; c < kCC; ++c) acc = fmaf(gb[b * kGld + c], wf[k * kCC + c], acc);
    dl[b * K + k] = acc + bfm[k];
  }
  __syncthreads();
  for (int b = t; b < B; b += kHeadT) {
    const int y = a.labels[static_cast<int64_t>(lane) * B + b];
    float* z = dl + b * K;
    float mx = -INFINITY;
    for (int k = 0; k < K; ++k) mx = fmaxf(mx, z[k]);
    float se = 0.f, so_ = 0.f;
    const float zy = z[y];
    for (int k = 0; k < K; ++k) {
      const float ev = expf(z[k] - mx);
      z[k] = ev;
      se += ev;
      if (k != y) so_ += ev;
    }
    rl[b] = mx + logf(se) - zy;
    const float inv = 1.0f / static_cast<float>(B);
    for (int k = 0; k < K; ++k) {
      const float gk = (k == y ? -so_ : z[k]) / se * inv;
      z[k] = gk;
      dlb[b * K + k] = bf16_round(gk);
    }
  }
  __syncthreads();
  if (a.loss_part && t < (B + kRowsPerLossChunk - 1) / kRowsPerLossChunk) {
    float l = 0.f;
    for (int r = t * kRowsPerLossChunk; r < min(B, (t + 1) * kRowsPerLossChunk); ++r) l += rl[r];
    a.loss_part[(static_cast<int64_t>(lane) * a.max_tau + a.step) * a.n_loss_chunks + t] = l;
  }
  // dg[b][c] = sum_k dlb[b][k] wf[k][c] (old weights)
  for (int q = t; q < B * kCC; q += kHeadT) {
    const int b = q / kCC, c = q % kCC;
    float acc = 0.f;
    for (int k = 0; k < K; ++k) acc = fmaf(dlb[b * K + k], wf[k * kCC + c], acc);
    a.dg[static_cast<int64_t>(lane) * B * kCC + q] = acc;
  }
  // head weights and bias
  for (int q = t; q < K * kCC; q += kHeadT) {
    const int k = q / kCC, c = q % kCC;
    float acc = 0.f;
#pragma unroll 4
    for (int b = 0; b < B; ++b) acc = fmaf(dlb[b * K + k], gb[b * kGld + c], acc);
    const float nw = fmaf(-a.lr, acc, wm[q]);
    a.master_w[dof + a.offWf + q] = nw;
    a.shadow[dof + a.offWf + q] = __float2bfloat16_rn(nw);
  }
  if (t < K) {
    float acc = 0.f;
    for (int b = 0; b < B; ++b) acc += dl[b * K + t];
    const float nb = fmaf(-a.lr, acc, bfm[t]);
    a.master_w[dof + a.offBf + t] = nb;
    a.shadow[dof + a.offBf + t] = __float2bfloat16_rn(nb);
  }
}

// loss of the global model on labelled images (evaluation): grid = lanes, 256
// threads, one image of the lane's (B <= 256) per thread
__global__ void __launch_bounds__(256) cnn_head_loss_kernel(const float* pool, const int32_t* labels, int B, int64_t n_img,
                                                            int K, const float* master, int64_t offWf, int64_t offBf,
                                                            float* out) {
  extern __shared__ float hsm[];
  float* gb = hsm;                    // [B][kGld]
  float* wf = gb + B * kGld;          // [K][64]
  __shared__ float bfm[32];
  __shared__ float rl[8];
  const int t = threadIdx.x, lane = blockIdx.x;
  const int64_t left = n_img - static_cast<int64_t>(lane) * B;
  const int mine = left < B ? static_cast<int>(left) : B;
  gather_pooled(pool + static_cast<int64_t>(lane) * B * kImg * kCC, mine, gb, 256);
  for (int q = t; q < K * kCC; q += 256) wf[q] = bf16_round(master[offWf + q]);
  if (t < K) bfm[t] = master[offBf + t];
  __syncthreads();
  float l = 0.f;
  if (t < mine) {
    const int y = labels[static_cast<int64_t>(lane) * B + t];
    float z[32], mx = -INFINITY, zy = 0.f;
#pragma unroll
    for (int k = 0; k < 32; ++k) {
      if (k >= K) continue;
      float acc = 0.f;
#pragma unroll 16
      for (int c = 0; c < kCC; ++c) acc = fmaf(gb[t * kGld + c], wf[k * kCC + c], acc);
      z[k] = acc + bfm[k];
      mx = fmaxf(mx, z[k]);
      if (k == y) zy = z[k];
    }
    float se = 0.f;
#pragma unroll
    for (int k = 0; k < 32; ++k)
      if (k < K) se += expf(z[k] - mx);
    l = mx + logf(se) - zy;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) l += __shfl_xor_sync(0xffffffffu, l, o);
  if ((t & 31) == 0) rl[t >> 5] = l;
  __syncthreads();
  if (t == 0) {
    float s = 0.f;
    for (int i = 0; i < 8; ++i) s += rl[i];
    out[lane] = s;
  }
}

// ------------------------------------------------------------------ output gradient of the last block
// grid (B * 8 tiles, active), 128 threads: dz = v > 0 ? dg / 1024 : 0, bf16,
// and per-tile channel sums of the fp32 values.  Item = (pixel, 16-byte
// chunk of 8 channels): thread t always has chunk t % 8 (pixels t / 8 + 16 i),
// so its 8 channel sums stay in registers; the 16 threads of a chunk add
// theirs in order through shared memory.  dg / 1024 is exact as dg * 2^-10.
__global__ void __launch_bounds__(kCT) cnn_dzb_kernel(const __nv_bfloat16* v, const float* dg, const int* wid, int B,
                                                      __nv_bfloat16* dz, float* bias_part) {
  __shared__ float dgs[kCC];
  __shared__ float T[kCT / 8][kCC + 1];
  const int tile = blockIdx.x, lane = wid[blockIdx.y];
  const int b = tile / kTilesPerImg, pix0 = (tile % kTilesPerImg) * kTilePix;
  const int64_t base = ((static_cast<int64_t>(lane) * B + b) * kPix + pix0) * kCC;
  if (threadIdx.x < kCC) dgs[threadIdx.x] = dg[(static_cast<int64_t>(lane) * B + b) * kCC + threadIdx.x] / static_cast<float>(kPix);
  __syncthreads();
  const int q = threadIdx.x & 7, p0 = threadIdx.x >> 3;
  float d[8], sum[8];
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    d[j] = dgs[8 * q + j];
    sum[j] = 0.f;
  }
#pragma unroll 4
  for (int p = p0; p < kTilePix; p += kCT / 8) {
    const int64_t off = base + static_cast<int64_t>(p) * kCC + 8 * q;
    const uint4 r = *reinterpret_cast<const uint4*>(v + off);
    const __nv_bfloat162* r2 = reinterpret_cast<const __nv_bfloat162*>(&r);
    float o[8];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const float2 f = __bfloat1622float2(r2[j]);
      o[2 * j] = f.x > 0.f ? d[2 * j] : 0.f;
      o[2 * j + 1] = f.y > 0.f ? d[2 * j + 1] : 0.f;
    }
#pragma unroll
    for (int j = 0; j < 8; ++j) sum[j] += o[j];
    *reinterpret_cast<uint4*>(dz + off) = make_uint4(pack_bf16x2(o[0], o[1]), pack_bf16x2(o[2], o[3]),
                                                     pack_bf16x2(o[4], o[5]), pack_bf16x2(o[6], o[7]));
  }
#pragma unroll
  for (int j = 0; j < 8; ++j) T[p0][8 * q + j] = sum[j];
  __syncthreads();
  if (threadIdx.x < kCC) {
    float s = 0.f;
    for (int r = 0; r < kCT / 8; ++r) s += T[r][threadIdx.x];
    bias_part[(static_cast<int64_t>(lane) * B * kTilesPerImg + tile) * kCC + threadIdx.x] = s;
  }
}

}  // namespace

// ------------------------------------------------------------------ launchers
int cnn_tiles_per_image() { return kTilesPerImg; }

int conv_ctas_per_worker(int B, int n_active, int sms) {
  const int tiles = B * kTilesPerImg;
  int cpw = sms / (n_active > 0 ? n_active : 1);
  if (cpw < 1) cpw = 1;
  if (cpw > tiles) cpw = tiles;
  return cpw;
}

cudaError_t launch_conv_igemm(int mode, const CUtensorMap& mIn, const CUtensorMap& mW, const ConvMaps& mm,
                              const ConvArgs& a, int n_active, int cpw, cudaStream_t s) {
  const dim3 grid(cpw, n_active);
  if (mode == 0) {
    cudaError_t e = allow_smem(conv_igemm_kernel<0>, kGSmem);
    if (e != cudaSuccess) return e;
    conv_igemm_kernel<0><<<grid, kGT, kGSmem, s>>>(mIn, mW, mm, a);
  } else {
    cudaError_t e = allow_smem(conv_igemm_kernel<1>, kGSmem);
    if (e != cudaSuccess) return e;
    conv_igemm_kernel<1><<<grid, kGT, kGSmem, s>>>(mIn, mW, mm, a);
  }
  return cudaGetLastError();
}

int conv_wgrad_chunks(int B, int n_active, int sms) {
  int per_worker = sms / (n_active > 0 ? n_active : 1);   // CTAs per worker in one wave
  if (per_worker < 1) per_worker = 1;
  return per_worker < B ? per_worker : B;
}

cudaError_t launch_conv_wgrad(const CUtensorMap& mIn, const CUtensorMap& mDz, const WgradArgs& a, int n_active,
                              cudaStream_t s) {
  cudaError_t e = allow_smem(conv_wgrad_kernel, kWSmem2);
  if (e != cudaSuccess) return e;
  conv_wgrad_kernel<<<dim3(a.n_chunks, n_active), kWT, kWSmem2, s>>>(mIn, mDz, a);
  return cudaGetLastError();
}

cudaError_t launch_conv_sgd(const ConvSgdArgs& a, int n_active, cudaStream_t s) {
  if (a.layers < 1 || a.layers > kMaxConvLayers) return cudaErrorInvalidValue;
  conv_sgd_kernel<<<dim3(kTaps * (kCC / kSgdRows), n_active, a.layers), 256, 0, s>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_conv_refresh_wt(const float* master, __nv_bfloat16* wt, int64_t offW, cudaStream_t s) {
  conv_refresh_wt_kernel<<<kTaps, 256, 0, s>>>(master, wt, offW);
  return cudaGetLastError();
}

cudaError_t launch_cnn_stage(const CnnStageArgs& a, int n_active, cudaStream_t s) {
  cnn_stage_kernel<<<dim3(a.B * kTilesPerImg, n_active), kCT, 0, s>>>(a);
  return cudaGetLastError();
}

static size_t cnn_head_smem(int B, int K) {
  return sizeof(float) * (static_cast<size_t>(B) * kGld + 2 * K * kCC + 2 * B * K + B + 32);
}

cudaError_t launch_cnn_head(const CnnHeadArgs& a, int n_active, cudaStream_t s) {
  const size_t smem = cnn_head_smem(a.B, a.K);
  cudaError_t e = allow_smem(cnn_head_kernel, smem);
  if (e != cudaSuccess) return e;
  cnn_head_kernel<<<n_active, kHeadT, smem, s>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_cnn_head_loss(const float* pool_part, const int32_t* labels, int lanes, int B, int64_t n_img, int K,
                                 const float* master, int64_t offWf, int64_t offBf, float* out, cudaStream_t s) {
  const size_t smem = sizeof(float) * (static_cast<size_t>(B) * kGld + K * kCC);
  cudaError_t e = allow_smem(cnn_head_loss_kernel, smem);
  if (e != cudaSuccess) return e;
  cnn_head_loss_kernel<<<lanes, 256, smem, s>>>(pool_part, labels, B, n_img, K, master, offWf, offBf, out);
  return cudaGetLastError();
}

cudaError_t launch_cnn_dzb(const __nv_bfloat16* v, const float* dg, const int* wid, int B, __nv_bfloat16* dz,
                           float* bias_part, int n_active, cudaStream_t s) {
  cnn_dzb_kernel<<<dim3(B * kTilesPerImg, n_active), kCT, 0, s>>>(v, dg, wid, B, dz, bias_part);
  return cudaGetLastError();
}

}  // namespace oscars
