// Grouped bf16 GEMM on the 5th-generation tensor cores (tcgen05, sm_103a)
// for the workers' dense layers (Eq. 4, "otherwise" branch: the forward and
// backward passes of x - lr * g(x)), with the step's elementwise work fused
// into the epilogue.
//
//   D[m][n] = sum_k A[m][k] * B[n][k]     A, B bf16 K-major, D fp32 in TMEM
//
// One CTA computes one 128 x BN tile of one active worker (grid z = worker).
// Warp 0 lane 0 streams K-blocks of 64 with TMA (128-byte swizzle, 3-D
// tensor maps whose z coordinate selects the worker's buffer or the
// parameter slot), warp 1 (an elected lane) issues tcgen05.mma (M=128, N=BN, K=16) into
// a TMEM accumulator and frees each stage with tcgen05.commit, warp 2 owns
// the TMEM allocation; then all four warps read their 32 TMEM lanes
// (one output row per thread) and run the epilogue:
//
// Where the samples come in boxes of 64 and the head reads H^T (out null; TT
// below), only the transposes H^T and G^T are kept: the next layer's forward
// and the input gradient read them MN-major, the ReLU mask comes by TMA as one
// ring entry more, and each warp stores its rows of a tile by TMA.  With both
// layouts written, and the mask read, by the threads of a row, the epilogue
// took 5000 to 9500 clocks of a forward (main loop 12000 for K = 1024) and
// 7400 to 15000 of an input gradient (12000 to 16000): a round of
// 3072-1024-1024-10, batch 128, 32 workers, 1576 -> 1524 us.
//
//  kEpiFwd  hidden layer forward, m = output feature, n = sample:
//           h = relu(acc + bias[m]) -> bf16 H[n][m] and H^T[m][n].
//  kEpiDh   input gradient of a hidden layer, m = input feature, n = sample:
//           g = acc * (Hmask[n][m] > 0) -> bf16 G[n][m], G^T[m][n] and the
//           bias gradient gb[m] = sum_n g (fp32, whole batch in one tile).
//
// All waits are bounded (see common.cuh) and report through a device word.
#include <cstdio>

#include "common.cuh"
#include "internal.h"

namespace oscars {

namespace {

constexpr int BM = 128;
constexpr int BK = 64;
constexpr int kABytes = BM * BK * 2;
constexpr int kBarrierBytes = 256;          // mbarriers + TMEM address slot
constexpr int kWarps = 4;

template <int BN>
struct TileCfg {
  static constexpr int kBBytes = BN * BK * 2;
  static constexpr int kStageBytes = kABytes + kBBytes;
  static constexpr uint32_t kTmemCols = BN <= 32 ? 32 : BN <= 64 ? 64 : BN <= 128 ? 128 : 256;
};

// 32 samples of a forward row: relu(acc + bias) as bf16 pairs
__device__ __forceinline__ void fwd_pack(const float (&v)[32], float bias, uint32_t (&pk)[16]) {
#pragma unroll
  for (int c = 0; c < 32; c += 2) pk[c >> 1] = pack_bf16x2(fmaxf(v[c] + bias, 0.f), fmaxf(v[c + 1] + bias, 0.f));
}

// 32 samples of an input-gradient row, masked by h > 0 (pk: bf16 pairs of h,
// replaced by the gradient's); returns their sum in sample order
__device__ __forceinline__ float dh_mask_pack(const float (&v)[32], uint32_t (&pk)[16]) {
  float gsum = 0.f;
#pragma unroll
  for (int c = 0; c < 32; c += 2) {
    const uint32_t h = pk[c >> 1];
    const float g0 = __uint_as_float(h << 16) > 0.f ? v[c] : 0.f;
    const float g1 = __uint_as_float(h & 0xffff0000u) > 0.f ? v[c + 1] : 0.f;
    gsum += g0;
    gsum += g1;
    pk[c >> 1] = pack_bf16x2(g0, g1);
  }
  return gsum;
}

__device__ __forceinline__ void lds128(uint32_t addr, uint32_t* r) {
  asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}
__device__ __forceinline__ void sts128(uint32_t addr, const uint32_t* r) {
  asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]) : "memory");
}

__device__ __forceinline__ void epi_fwd(const GemmArgs& a, int wid, int src, int m, int n0,
                                        const float (&v)[32]) {
  const float bias = a.master[static_cast<int64_t>(src) * a.slot_stride + a.offB + m];
  __nv_bfloat16* out = a.out + static_cast<int64_t>(wid) * a.N * a.M;
  uint32_t pk[16];
#pragma unroll
  for (int c = 0; c < 32; c += 2) {
    const float h0 = fmaxf(v[c] + bias, 0.f);
    const float h1 = fmaxf(v[c + 1] + bias, 0.f);
    const __nv_bfloat162 p = __floats2bfloat162_rn(h0, h1);
    out[static_cast<int64_t>(n0 + c) * a.M + m] = p.x;
    out[static_cast<int64_t>(n0 + c + 1) * a.M + m] = p.y;
    pk[c >> 1] = *reinterpret_cast<const uint32_t*>(&p);
  }
  uint4* outT = reinterpret_cast<uint4*>(a.outT + (static_cast<int64_t>(wid) * a.M + m) * a.N + n0);
#pragma unroll
  for (int q = 0; q < 4; ++q) outT[q] = make_uint4(pk[4 * q], pk[4 * q + 1], pk[4 * q + 2], pk[4 * q + 3]);
}

// The input-gradient epilogue's ReLU mask for 32 columns: mk[c] = the raw
// bf16 bits of Hmask[n0 + c][m].  All 32 loads are issued before any is
// used, and the caller issues the next chunk's loads before it stores the
// current one, so the mask reads of a thread overlap instead of waiting
// one by one behind its stores.
__device__ __forceinline__ void epi_dh_mask(const GemmArgs& a, int wid, int m, int n0, unsigned short (&mk)[32]) {
  const unsigned short* hm = reinterpret_cast<const unsigned short*>(a.hmask) +
                             static_cast<int64_t>(wid) * a.N * a.M + static_cast<int64_t>(n0) * a.M + m;
#pragma unroll
  for (int c = 0; c < 32; ++c) mk[c] = __ldg(hm + static_cast<int64_t>(c) * a.M);
}

template <bool kTest>
__device__ __forceinline__ float epi_dh(const GemmArgs& a, int wid, int m, int n0, const float (&v)[32],
                                        const unsigned short (&mk)[32]) {
  // the row-major copy: always written here, but with eight chunks a thread
  // (kTest) a test around its stores keeps the compiler from weaving them into
  // the next chunk's mask loads (64 registers and few loads in flight instead of
  // 144: 1024 x 1024, 256 samples, 32 workers: 43 us so, 31 with the test); with
  // one it costs (17-class round, batch 32: 315.8 us without, 319.3 with)
  __nv_bfloat16* out = a.out + static_cast<int64_t>(wid) * a.N * a.M;
  uint32_t pk[16];
  float gsum = 0.f;
#pragma unroll
  for (int c = 0; c < 32; c += 2) {
    const int64_t e0 = static_cast<int64_t>(n0 + c) * a.M + m;
    const int64_t e1 = e0 + a.M;
    const float g0 = __bfloat162float(__ushort_as_bfloat16(mk[c])) > 0.f ? v[c] : 0.f;
    const float g1 = __bfloat162float(__ushort_as_bfloat16(mk[c + 1])) > 0.f ? v[c + 1] : 0.f;
    gsum += g0;
    gsum += g1;
    const __nv_bfloat162 p = __floats2bfloat162_rn(g0, g1);
    if (!kTest || a.out) {
      out[e0] = p.x;
      out[e1] = p.y;
    }
    pk[c >> 1] = *reinterpret_cast<const uint32_t*>(&p);
  }
  uint4* outT = reinterpret_cast<uint4*>(a.outT + (static_cast<int64_t>(wid) * a.M + m) * a.N + n0);
#pragma unroll
  for (int q = 0; q < 4; ++q) outT[q] = make_uint4(pk[4 * q], pk[4 * q + 1], pk[4 * q + 2], pk[4 * q + 3]);
  return gsum;
}

// Split-K (SPLIT > 1, forward and input-gradient epilogues): a cluster of
// SPLIT CTAs shares one output tile, CTA r multiplying K-blocks [r nk / SPLIT,
// (r + 1) nk / SPLIT).  Each CTA pushes its fp32 partial rows into the CTA
// that owns them (rows [r 128 / SPLIT, (r + 1) 128 / SPLIT) belong to CTA r)
// through distributed shared memory, between two cluster barriers (every CTA
// has started before the first store, arrived on in the prologue and so free;
// every partial has landed before the first is read), and each
// owner sums the SPLIT partials in rank order and runs the epilogue on its
// rows.  Used when a launch has too few tiles to fill the GPU: small layers,
// and the tail of a round, where one worker with many local steps runs alone
// (split_for).
constexpr int kRedLd = 4;   // padding of a partial row (floats)

__device__ __forceinline__ void st_dsmem_f32x4(float* local, uint32_t rank, float4 v) {
  uint32_t remote;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(remote) : "r"(smem_u32(local)), "r"(rank));
  asm volatile("st.shared::cluster.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(remote), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w)
               : "memory");
}

template <int BN, int EPI, int SPLIT, bool TT>
__global__ void __launch_bounds__(kWarps * 32) gemm_tc_kernel(const __grid_constant__ CUtensorMap mapA,
                                                           const __grid_constant__ CUtensorMap mapB,
                                                           const __grid_constant__ CUtensorMap mapT,
                                                           const __grid_constant__ CUtensorMap mapM,
                                                           const __grid_constant__ GemmArgs a,
                                                           int stages) {
  static_assert(!TT || BN == 64 || BN == 128, "transposed results are stored in boxes of 64 samples");
  using Cfg = TileCfg<BN>;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* sA = smem;
  uint8_t* sB = smem + stages * kABytes;
  uint64_t* full = reinterpret_cast<uint64_t*>(sB + stages * Cfg::kBBytes);
  uint64_t* empty = full + stages;
  uint64_t* accum = empty + stages;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(accum + 1);
  float* epi_tiles = reinterpret_cast<float*>(reinterpret_cast<uint8_t*>(full) + kBarrierBytes);

  const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
  const int li = blockIdx.z / SPLIT;
  const int rank = SPLIT > 1 ? static_cast<int>(cluster_ctarank()) : 0;
  const int wid = a.wid ? a.wid[li] : li, src = a.src ? a.src[li] : li;
  const int m0 = blockIdx.x * BM, n0 = blockIdx.y * BN;
  const int nk_all = (a.K + BK - 1) / BK;
  const int kb0 = rank * nk_all / SPLIT;                 // this CTA's K-blocks [kb0, kb0 + nk)
  const int nk = (rank + 1) * nk_all / SPLIT - kb0;

  if (threadIdx.x == 0) {
    prefetch_tmap(&mapA);
    prefetch_tmap(&mapB);
    if (TT && SPLIT == 1) prefetch_tmap(&mapT);
    for (int s = 0; s < stages; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    mbar_init(accum, 1);
    fence_barrier_init();
    fence_proxy_async_smem();
  }
  if (warp == 2) {
    tmem_alloc(tmem_slot, Cfg::kTmemCols);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (SPLIT > 1) cluster_arrive();   // this CTA has started; the wait stands before the first store into a peer
  const uint32_t tmem = *tmem_slot;
  pdl_wait();      // the previous kernel's outputs (operands, masks, biases) are complete
  pdl_trigger();

  if (warp == 0 && lane == 0) {
    // TMA producer
    const int za = a.a_z_src ? src : wid;
    const int zb = a.b_z_src ? src : wid;
    for (int kb = 0; kb < nk; ++kb) {
      const int s = kb % stages;
      if (kb >= stages && !mbar_wait(&empty[s], ((kb / stages) + 1) & 1, a.err, kDevTimeoutEmpty)) break;
      mbar_arrive_expect_tx(&full[s], kABytes + Cfg::kBBytes);
      const int k = (kb0 + kb) * BK;   // global K coordinate
      if constexpr (EPI == kEpiDh) {
        // A = W^T read MN-major from W [K = out][M = in]: two boxes of 64 M x
        // 64 K, the second 64 M-elements further along (8 KB in shared memory)
        tma_load_3d(sA + s * kABytes, &mapA, m0, k, za, &full[s]);
        tma_load_3d(sA + s * kABytes + kABytes / 2, &mapA, m0 + 64, k, za, &full[s]);
      } else {
        tma_load_3d(sA + s * kABytes, &mapA, k, m0, za, &full[s]);
      }
      if (a.b_mn) {
        // B (G, H) read MN-major from its transpose [K][N = batch]: boxes of 64 N x 64 K, 8 KB apart
        for (int nb = 0; nb < BN / 64; ++nb)
          tma_load_3d(sB + s * Cfg::kBBytes + nb * 8192, &mapB, n0 + 64 * nb, k, zb, &full[s]);
      } else {
        tma_load_3d(sB + s * Cfg::kBBytes, &mapB, k, n0, zb, &full[s]);
      }
    }
    if constexpr (TT && SPLIT == 1 && EPI == kEpiDh) {
      // the ReLU mask, one entry of the ring more: h^T tiles of 64 samples
      const int s = nk % stages;
      if (nk < stages || mbar_wait(&empty[s], ((nk / stages) + 1) & 1, a.err, kDevTimeoutEmpty)) {
        mbar_arrive_expect_tx(&full[s], BN / 64 * kABytes);
        tma_load_3d(sA + s * kABytes, &mapM, n0, m0, wid, &full[s]);
        if (BN == 128) tma_load_3d(sB + s * Cfg::kBBytes, &mapM, n0 + 64, m0, wid, &full[s]);
      }
    }
  } else if (warp == 1) {
    // MMA issuer: the warp converged, one elected lane issues (see elect_one)
    // A MN-major (transpose-A bit 15) for the input gradient, K-major otherwise;
    // B MN-major (bit 16) when it is read from its transpose
    const bool bmn = a.b_mn;
    const uint32_t idesc = idesc_bf16_f32(BM, BN) | (EPI == kEpiDh ? (1u << 15) : 0u) | (bmn ? (1u << 16) : 0u);
    uint32_t limit = kSpinLimit;
    for (int kb = 0; kb < nk; ++kb) {
      const int s = kb % stages;
      mbar_wait_keep(limit, &full[s], (kb / stages) & 1, a.err, kDevTimeoutFull);
      tc_fence_after();
      const uint32_t a_base = smem_u32(sA + s * kABytes);
      const uint32_t b_base = smem_u32(sB + s * Cfg::kBBytes);
      // K-major: 16 K-elements are 32 bytes along a row; MN-major: 16 rows of
      // 128 bytes (the descriptor's address field counts 16 bytes)
      const uint64_t ad = EPI == kEpiDh ? smem_desc_mn128(a_base, kABytes / 2) : smem_desc_k128(a_base);
      const uint64_t bd = bmn ? smem_desc_mn128(b_base, 8192) : smem_desc_k128(b_base);
      const uint32_t astep = EPI == kEpiDh ? 128 : 2, bstep = bmn ? 128 : 2;
      if (elect_one() && limit > 1) {
#pragma unroll
        for (int j = 0; j < BK / 16; ++j)
          umma_bf16(tmem, ad + j * astep, bd + j * bstep, idesc, (kb | j) != 0 ? 1u : 0u);
        umma_commit(&empty[s]);
      }
      __syncwarp();
    }
    if (elect_one()) umma_commit(accum);  // arrives once every issued MMA has completed
    __syncwarp();
  }
  __syncwarp();

  if constexpr (SPLIT > 1) {
    // ---- split-K epilogue (4 warps): push the partial rows to their owners
    constexpr int R = BM / SPLIT;                   // rows owned per CTA
    constexpr int ld = BN + kRedLd;
    float* red = epi_tiles;                         // [SPLIT][R][ld] fp32: the partials of this CTA's rows
    int acc_ok = mbar_wait(accum, 0, a.err, kDevTimeoutAccum) ? 1 : 0;
    acc_ok = __all_sync(0xffffffffu, acc_ok);
    tc_fence_after();
    const int row = (warp & 3) * 32 + lane;        // accumulator row of this thread
    const int owner = row / R;
    float* dst = red + (rank * R + (row - owner * R)) * ld;
    const uint32_t trow = tmem + (static_cast<uint32_t>((warp & 3) * 32) << 16);
    cluster_wait();   // every CTA of the cluster has started: its shared memory may be written
#pragma unroll 1
    for (int c0 = 0; c0 < BN; c0 += 32) {
      float v[32];
      if (acc_ok) tmem_ld_32x32b_x32(trow + c0, v);
      else
#pragma unroll
        for (int j = 0; j < 32; ++j) v[j] = 0.f;
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        const float4 p4 = make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
        if (owner == rank) *reinterpret_cast<float4*>(dst + c0 + 4 * q) = p4;
        else st_dsmem_f32x4(dst + c0 + 4 * q, owner, p4);
      }
    }
    tc_fence_before();
    // TT: the mask bits of this thread's (one) item, while the partials land
    uint4 hm[4];
    if constexpr (TT && EPI == kEpiDh) {
      const int it = threadIdx.x < R * (BN / 32) ? threadIdx.x : 0;
      const uint4* hrow = reinterpret_cast<const uint4*>(
          a.hmask + (static_cast<int64_t>(wid) * a.M + m0 + rank * R + it / (BN / 32)) * a.N + n0 + it % (BN / 32) * 32);
#pragma unroll
      for (int q = 0; q < 4; ++q) hm[q] = __ldg(hrow + q);
    }
    cluster_sync();   // every partial has landed in its owner
    // own rows: item = (row, 32-column chunk); partials summed in rank order
    float* gpart = red + SPLIT * R * ld;            // [R][BN / 32] bias-gradient partials (input gradient)
    for (int it = threadIdx.x; it < R * (BN / 32); it += kWarps * 32) {
      const int rl = it / (BN / 32), c0 = (it % (BN / 32)) * 32;
      float v[32];
#pragma unroll
      for (int j = 0; j < 32; ++j) v[j] = 0.f;
#pragma unroll
      for (int p = 0; p < SPLIT; ++p) {
        const float* src_row = red + (p * R + rl) * ld + c0;
#pragma unroll
        for (int q = 0; q < 8; ++q) {
          const float4 x = *reinterpret_cast<const float4*>(src_row + 4 * q);
          v[4 * q] += x.x;
          v[4 * q + 1] += x.y;
          v[4 * q + 2] += x.z;
          v[4 * q + 3] += x.w;
        }
      }
      const int m = m0 + rank * R + rl;
      if constexpr (TT) {
        uint32_t pk[16];
        if constexpr (EPI == kEpiFwd) {
          fwd_pack(v, a.master[static_cast<int64_t>(src) * a.slot_stride + a.offB + m], pk);
        } else {
          if (it != threadIdx.x) {   // SPLIT = 2 at 128 samples: a thread's second item
            const uint4* hrow =
                reinterpret_cast<const uint4*>(a.hmask + (static_cast<int64_t>(wid) * a.M + m) * a.N + n0 + c0);
#pragma unroll
            for (int q = 0; q < 4; ++q) hm[q] = __ldg(hrow + q);
          }
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            pk[4 * q] = hm[q].x;
            pk[4 * q + 1] = hm[q].y;
            pk[4 * q + 2] = hm[q].z;
            pk[4 * q + 3] = hm[q].w;
          }
          gpart[rl * (BN / 32) + c0 / 32] = dh_mask_pack(v, pk);
        }
        uint4* outT = reinterpret_cast<uint4*>(a.outT + (static_cast<int64_t>(wid) * a.M + m) * a.N + n0 + c0);
#pragma unroll
        for (int q = 0; q < 4; ++q) outT[q] = make_uint4(pk[4 * q], pk[4 * q + 1], pk[4 * q + 2], pk[4 * q + 3]);
      } else if constexpr (EPI == kEpiFwd) {
        epi_fwd(a, wid, src, m, n0 + c0, v);
      } else {
        unsigned short mk[32];
        epi_dh_mask(a, wid, m, n0 + c0, mk);
        gpart[rl * (BN / 32) + c0 / 32] = epi_dh<false>(a, wid, m, n0 + c0, v, mk);
      }
    }
    if constexpr (EPI == kEpiDh) {
      __syncthreads();
      for (int rl = threadIdx.x; rl < R; rl += kWarps * 32) {
        float g = 0.f;
        for (int c = 0; c < BN / 32; ++c) g += gpart[rl * (BN / 32) + c];
        a.gb_out[static_cast<int64_t>(wid) * a.M + m0 + rank * R + rl] = g;
      }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 2) {
      tc_fence_after();
      tmem_dealloc(tmem, Cfg::kTmemCols);
    }
    return;
  }

  if constexpr (TT) {
    // ---- epilogue with H^T / G^T alone: thread = one accumulator row, its
    // 64-sample halves in tiles [128][64] (128-byte swizzle) in the ring: the
    // mask's entry, overwritten in place, or the first one; each warp stores
    // its 32 rows of a tile with one TMA store
    const int m = m0 + 32 * warp + lane, row = 32 * warp + lane;
    const float bias = EPI == kEpiFwd ? a.master[static_cast<int64_t>(src) * a.slot_stride + a.offB + m] : 0.f;
    const int st = EPI == kEpiDh ? nk % stages : 0;
    bool ok = mbar_wait(accum, 0, a.err, kDevTimeoutAccum);
    if constexpr (EPI == kEpiDh) ok = mbar_wait(&full[st], (nk / stages) & 1, a.err, kDevTimeoutFull) && ok;
    const int all_ok = __all_sync(0xffffffffu, ok);
    tc_fence_after();
    if (all_ok) {
      const uint32_t trow = tmem + (static_cast<uint32_t>(warp * 32) << 16);
      float gsum = 0.f;
#pragma unroll 1
      for (int c0 = 0; c0 < BN; c0 += 32) {
        float v[32];
        tmem_ld_32x32b_x32(trow + c0, v);
        uint8_t* tile = c0 < 64 ? sA + st * kABytes : sB + st * Cfg::kBBytes;
        const uint32_t at = smem_u32(tile) + row * 128, ch = (c0 & 63) >> 3;
        uint32_t pk[16];
        if constexpr (EPI == kEpiFwd) {
          fwd_pack(v, bias, pk);
        } else {
#pragma unroll
          for (int q = 0; q < 4; ++q) lds128(at + (((ch + q) ^ (row & 7)) << 4), pk + 4 * q);
          gsum += dh_mask_pack(v, pk);
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) sts128(at + (((ch + q) ^ (row & 7)) << 4), pk + 4 * q);
        if (c0 & 32) {
          fence_proxy_async_smem();
          __syncwarp();
          if (lane == 0) {
            tma_store_3d(&mapT, tile + 32 * warp * 128, n0 + (c0 & 64), m0 + 32 * warp, wid);
            bulk_commit_group();
          }
        }
      }
      if constexpr (EPI == kEpiDh) a.gb_out[static_cast<int64_t>(wid) * a.M + m] = gsum;
      if (lane == 0) bulk_wait_all();
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 2) {
      tc_fence_after();
      tmem_dealloc(tmem, Cfg::kTmemCols);
    }
    return;
  }

  // epilogue: thread = one accumulator row
  unsigned short mk[32];   // input-gradient mask of the next 32 columns, read while the MMAs run
  if constexpr (EPI == kEpiDh) epi_dh_mask(a, wid, m0 + (warp & 3) * 32 + lane, n0, mk);
  int acc_ok = mbar_wait(accum, 0, a.err, kDevTimeoutAccum) ? 1 : 0;
  acc_ok = __all_sync(0xffffffffu, acc_ok);
  tc_fence_after();
  if (acc_ok) {
    const int quarter = warp & 3;
    const int m = m0 + quarter * 32 + lane;
    const uint32_t trow = tmem + (static_cast<uint32_t>(quarter * 32) << 16);
    if constexpr (EPI == kEpiDh) {
      float gsum = 0.f;
#pragma unroll
      for (int c0 = 0; c0 < BN; c0 += 32) {
        float v[32];
        tmem_ld_32x32b_x32(trow + c0, v);
        unsigned short cur[32];
#pragma unroll
        for (int c = 0; c < 32; ++c) cur[c] = mk[c];
        if (c0 + 32 < BN) epi_dh_mask(a, wid, m, n0 + c0 + 32, mk);
        gsum += epi_dh<BN == 256>(a, wid, m, n0 + c0, v, cur);
      }
      a.gb_out[static_cast<int64_t>(wid) * a.M + m] = gsum;
    } else {
#pragma unroll 1
      for (int c0 = 0; c0 < BN; c0 += 32) {
        float v[32];
        tmem_ld_32x32b_x32(trow + c0, v);
        epi_fwd(a, wid, src, m, n0 + c0, v);
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 2) {
    tc_fence_after();
    tmem_dealloc(tmem, Cfg::kTmemCols);
  }
}

// Shared memory that keeps the number of resident CTAs per SM at or below
// 512 / (TMEM columns per CTA), so a tcgen05.alloc never has to wait.
size_t smem_floor_for_tmem(uint32_t cols) {
  const size_t per_sm = 233472;  // 228 KB
  const size_t max_ctas = 512 / cols;
  return per_sm / (max_ctas + 1) - 1024 + 16;
}

int device_sms() {
  static int sms = 0;
  if (sms == 0) {
    int dev = 0;
    cudaGetDevice(&dev);
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms < 1) sms = 1;
  }
  return sms;
}

template <int BN, int EPI, int SPLIT, bool TT>
cudaError_t launch_tile(const GemmMaps& m, const GemmArgs& a, int n_active, cudaStream_t s) {
  using Cfg = TileCfg<BN>;
  // ring entries of the CTA with the most K-blocks, and the mask's
  const int nk = ((a.K + BK - 1) / BK + SPLIT - 1) / SPLIT + (TT && SPLIT == 1 && EPI == kEpiDh ? 1 : 0);
  dim3 grid(a.M / BM, (a.N + BN - 1) / BN, n_active * SPLIT);
  // A grid that fits one CTA per SM gets as many stages as K-blocks, within
  // ~200 KB of shared memory: the whole K extent of these skinny GEMMs is
  // then in flight at once.  A larger grid gets stages for ~100 KB, so two
  // CTAs share each SM and the grid runs in one wave instead of two (the
  // bytes in flight per SM stay the same).  A split grid keeps room for the
  // partial rows its CTAs exchange.
  const int sms = device_sms();
  const long long ctas = static_cast<long long>(grid.x) * grid.y * grid.z;
  const size_t red_bytes = SPLIT > 1 ? sizeof(float) * (static_cast<size_t>(BM) * (BN + kRedLd) + BM / SPLIT * (BN / 32))
                                     : 0;
  const int budget = SPLIT > 1 ? 150 * 1024 : ctas > sms ? 100 * 1024 : 200 * 1024;
  const int max_stages = budget / Cfg::kStageBytes;
  int stages = nk < max_stages ? nk : (max_stages < 8 ? max_stages : 8);
  static_assert(SPLIT == 1 || (4 * Cfg::kStageBytes >= kLeastClusterSmem && 4 * Cfg::kStageBytes <= 150 * 1024),
                "at least 4 K-blocks a CTA (split_for), so 4 stages: see kLeastClusterSmem");
  if (stages < 2) stages = nk < 2 ? nk : 2;
  size_t smem = 1024 + static_cast<size_t>(stages) * Cfg::kStageBytes + kBarrierBytes + red_bytes;
  const size_t floor_b = smem_floor_for_tmem(Cfg::kTmemCols);
  if (smem < floor_b) smem = floor_b;
  cudaError_t e = allow_smem(gemm_tc_kernel<BN, EPI, SPLIT, TT>, smem);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(kWarps * 32, 1, 1);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[2];
  int n = 0;
  if (SPLIT > 1) {
    attr[n].id = cudaLaunchAttributeClusterDimension;
    attr[n].val.clusterDim.x = 1;
    attr[n].val.clusterDim.y = 1;
    attr[n].val.clusterDim.z = SPLIT;
    ++n;
  }
  if (a.pdl) {
    attr[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[n].val.programmaticStreamSerializationAllowed = 1;
    ++n;
  }
  cfg.attrs = attr;
  cfg.numAttrs = n;
  return cudaLaunchKernelEx(&cfg, gemm_tc_kernel<BN, EPI, SPLIT, TT>, *m.a, *m.b, TT ? *m.t : *m.a, TT && EPI == kEpiDh ? *m.mask : *m.a, a, stages);
}

// K split of a forward or input-gradient launch of up to 128 samples: 4 or 2
// CTAs per tile when the unsplit grid would leave most of the GPU idle (one SM
// takes in about 60 bytes a clock: by that, K = 1000 at 32 samples is 5000
// clocks) and each CTA keeps at least 4 K-blocks.  Rounds of
// 1000-384-256-17, batch 32, 5 workers, and 3072-1024-1024-10, batch 128, 32
// workers: 336.7 and 1574 us without a split below 128 samples, 316.9 and 1573
// with this rule (one run); 318.5 and 1580 with this rule, 328.3 and 1581 with
// 2 K-blocks a CTA, 327.4 and 1592 with that and 8 CTAs from 16 K-blocks
// (another).
int split_for(int M, int N, int BN, int K, int n_active) {
  const long long tiles = static_cast<long long>(M / BM) * ((N + BN - 1) / BN) * n_active;
  const int nk = (K + BK - 1) / BK;
  const int sms = device_sms();
  if (tiles * 4 <= sms && nk >= 16) return 4;
  if (tiles * 2 <= sms && nk >= 8) return 2;
  return 1;
}

template <int BN, int EPI, bool TT>
cudaError_t launch_split(const GemmMaps& m, const GemmArgs& a, int n_active, cudaStream_t s) {
  switch (split_for(a.M, a.N, BN, a.K, n_active)) {
    case 4: return launch_tile<BN, EPI, 4, TT>(m, a, n_active, s);
    case 2: return launch_tile<BN, EPI, 2, TT>(m, a, n_active, s);
    default: return launch_tile<BN, EPI, 1, TT>(m, a, n_active, s);
  }
}

template <int EPI>
cudaError_t launch_epi(int bn, const GemmMaps& m, const GemmArgs& a, int n_active, cudaStream_t s) {
  const bool tt = a.out == nullptr;
  switch (bn) {
    case 32: return tt ? cudaErrorInvalidValue : launch_split<32, EPI, false>(m, a, n_active, s);
    case 64: return tt ? launch_split<64, EPI, true>(m, a, n_active, s) : launch_split<64, EPI, false>(m, a, n_active, s);
    case 128: return tt ? launch_split<128, EPI, true>(m, a, n_active, s) : launch_split<128, EPI, false>(m, a, n_active, s);
    case 256: return tt ? cudaErrorInvalidValue : launch_tile<256, EPI, 1, false>(m, a, n_active, s);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace

cudaError_t launch_gemm(int epi, const GemmMaps& m, const GemmArgs& a, int n_active, cudaStream_t s) {
  if (a.M % BM != 0) return cudaErrorInvalidValue;
  const int bn = a.N;   // the whole batch in one tile
  return epi == kEpiFwd ? launch_epi<kEpiFwd>(bn, m, a, n_active, s) : launch_epi<kEpiDh>(bn, m, a, n_active, s);
}

}  // namespace oscars
