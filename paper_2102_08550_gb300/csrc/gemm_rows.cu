// D[m][n] = sum_k A[m][k] B[n][k] for one large bf16 problem on the
// 5th-generation tensor cores (tcgen05, sm_103a): the library GEMM of the
// ABI, and the forward layers of the evaluation (Eq. 4's worker model on a
// held-out set), where m is a sample and all samples go in one launch.
//
//  kRowsStore  C[m][n] fp32 row-major
//  kRowsNarrow the same for at most 32 columns whose rows are not 16-byte aligned
//  kRowsRelu   out[m][n] = bf16(relu(D + bias[n])) row-major
//  kRowsLoss   n = class: softmax cross-entropy of row m against its label,
//              summed over the 32 rows of a warp into loss_part
//
// Persistent: one CTA per SM strides over tiles of 128 x BN.  Warp 0 lane 0
// streams K-blocks of 64 (TMA, 128-byte swizzle) through a ring of stages,
// warp 1 (an elected lane) issues tcgen05.mma (M = 128, N = BN, K = 16) into one of two
// TMEM accumulators, warps 4-7 (one accumulator row per thread) run the
// epilogue of a tile under the products of the next; fp32 and bf16 rows go
// out as TMA stores from per-warp staging boxes (plain coalesced stores where
// C's rows are not 16-byte aligned).
//
// With an even number of row tiles the two CTAs of a cluster work on one tile
// of 256 x BN (cta_group::2): each loads its 128 rows of A and half of the B
// tile, the leader (rank 0) issues the products of both, and each keeps its
// 128 accumulator rows.  A k-block then brings 16 KB + 64 BN bytes into an
// SM instead of 16 KB + 128 BN, and the bytes an SM takes in (about 60 a
// clock) are what bounds a big product: with 128 x 256 tiles, each CTA alone or
// with the B tile multicast, a k-block took 800 clocks, its products 256.  In
// pairs, 1024 x 8192 x 3072 reads 438 MB through L2, 39 bytes a clock and SM over
// the whole launch, and keeps the tensor pipe 70% busy.
//
// BN (a multiple of the 32 or 64 columns of a staging box, up to 256) is the width with the least estimated time:
// waves of tiles times the longer of a tile's products and loads.  For
// 1024 x 8192 x 3072 on 152 SMs: BN 224, two full waves (296 tiles); 256 has
// two waves as well, the second of 104 tiles, and each 14% longer.
// Measured, 1024 x 8192 x 3072, a call: 55.7 us with one 128 x 128 tile a CTA
// and no overlap of the epilogue; 46 with this kernel on CTAs alone, B
// multicast; 43.5 with the issuing warp converged (elect.sync: the descriptors
// stay in uniform registers); 38 with pairs.  4096 x 8192 x 3072: 185 -> 118 us
// (1.74 PFLOP/s).
#include <atomic>

#include "common.cuh"
#include "internal.h"

namespace oscars {

namespace {

constexpr int kRM = 128, kRK = 64;
constexpr int kRThreads = 256;
constexpr int kRMaxBN = 256;
constexpr int kRABytes = kRM * kRK * 2;
constexpr int kRMaxStages = 8;
constexpr int kRStg = 4096;                       // one staging box: 32 rows x 128 bytes
constexpr int kRStgBytes = 4 * 2 * kRStg;         // two per epilogue warp
constexpr int kRBarBytes = 256;
constexpr int kRSmem = 227 * 1024;                // at most
constexpr int kRRing = kRSmem - 1024 - kRBarBytes - kRStgBytes;

struct RowsBars {
  uint64_t full[kRMaxStages], empty[kRMaxStages], accf[2], acce[2];
  uint32_t tmem;
};
static_assert(sizeof(RowsBars) <= kRBarBytes, "barriers fit");

// ---- the cta_group::2 forms: the pair's CTAs hold the same offsets, and a
// shared::cluster address without the peer bit is the leader's
constexpr uint32_t kLeaderMask = 0xFEFFFFFFu;
__device__ __forceinline__ void tma_load_3d_pair(void* smem_dst, const CUtensorMap* map, int c0, int c1, int c2,
                                                 uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.tensor.3d.cta_group::2.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%2, %3, %4}], [%5];" ::"r"(smem_u32(smem_dst)),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(c2), "r"(smem_u32(bar) & kLeaderMask)
      : "memory");
}
__device__ __forceinline__ void umma_bf16_pair(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc,
                                               uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
      "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate)
      : "memory");
}
// the commit arrives on the barrier at this offset in both CTAs
__device__ __forceinline__ void umma_commit_pair(uint64_t* bar) {
  asm volatile(
      "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(
          smem_u32(bar)),
      "h"(static_cast<uint16_t>(0x3))
      : "memory");
}
__device__ __forceinline__ void mbar_arrive_at(uint32_t cluster_bar) {
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(cluster_bar) : "memory");
}
template <int CL>
__device__ __forceinline__ void tmem_alloc_cl(uint32_t* dst) {
  if (CL == 1) {
    tmem_alloc(dst, 512);
    tmem_relinquish();
  } else {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(dst)), "r"(512)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  }
}
template <int CL>
__device__ __forceinline__ void tmem_dealloc_cl(uint32_t taddr) {
  if (CL == 1) tmem_dealloc(taddr, 512);
  else asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(512) : "memory");
}

template <int EPI, int CL>
__global__ void __launch_bounds__(kRThreads, 1) gemm_rows_kernel(const __grid_constant__ CUtensorMap mapA,
                                                                 const __grid_constant__ CUtensorMap mapB,
                                                                 const __grid_constant__ CUtensorMap mapD,
                                                                 const __grid_constant__ RowsArgs a) {
  extern __shared__ uint8_t rs_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(rs_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* stg = smem;                              // [4 warps][2][32 rows][128 bytes]
  uint8_t* ring = smem + kRStgBytes;                // [stages][A 16 KB | B BN / CL x 128 bytes]
  const int stage_bytes = kRABytes + a.BN / CL * 128;
  RowsBars* bars = reinterpret_cast<RowsBars*>(ring + a.stages * stage_bytes);
  const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
  const int rank = CL > 1 ? static_cast<int>(cluster_ctarank()) : 0;
  const int nk = (a.K + kRK - 1) / kRK;
  // work unit = CL row tiles of the same columns, one per CTA of the cluster; rows fastest
  const int mu = a.mt / CL, units = mu * a.nt;
  const int u0 = blockIdx.x / CL, ustep = gridDim.x / CL;

  if (threadIdx.x == 0) {
    prefetch_tmap(&mapA);
    prefetch_tmap(&mapB);
    if (EPI == kRowsStore || EPI == kRowsRelu) prefetch_tmap(&mapD);
    for (int i = 0; i < a.stages; ++i) {
      mbar_init(&bars->full[i], 1);
      mbar_init(&bars->empty[i], 1);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(&bars->accf[i], 1);
      mbar_init(&bars->acce[i], 4 * CL);
    }
    fence_barrier_init();
    fence_proxy_async_smem();
  }
  if (warp == 2) {
    tmem_alloc_cl<CL>(&bars->tmem);
  }
  tc_fence_before();
  if (CL > 1) cluster_sync();   // the peer's barriers are initialised before anything arrives on them
  else __syncthreads();
  tc_fence_after();
  const uint32_t tmem = bars->tmem;
  pdl_wait();
  pdl_trigger();

  if (warp == 0 && lane == 0) {
    // ---- TMA producer
    int it = 0, s = 0, ph = 1;   // ph: the parity that a freed slot shows
    bool ok = true;
    int armed = 0;
    for (int u = u0; ok && u < units; u += ustep) {
      const int m0 = ((u % mu) * CL + rank) * kRM, n0 = (u / mu) * a.BN;
      for (int kb = 0; kb < nk; ++kb, ++it) {
        if (it >= a.stages && !(ok = mbar_wait(&bars->empty[s], ph, a.err, kDevTimeoutEmpty))) break;
        uint8_t* sa = ring + s * stage_bytes;
        // a pair's bytes all count on the leader's barrier
        if (rank == 0) mbar_arrive_expect_tx(&bars->full[s], CL * stage_bytes);
        armed = it + 1;
        if (CL > 1) {
          tma_load_3d_pair(sa, &mapA, kb * kRK, m0, 0, &bars->full[s]);
          tma_load_3d_pair(sa + kRABytes, &mapB, kb * kRK, n0 + rank * (a.BN / 2), 0, &bars->full[s]);
        } else {
          tma_load_3d(sa, &mapA, kb * kRK, m0, 0, &bars->full[s]);
          tma_load_3d(sa + kRABytes, &mapB, kb * kRK, n0, 0, &bars->full[s]);
        }
        if (++s == a.stages) {
          s = 0;
          ph ^= 1;
        }
      }
    }
    // no copy, and no commit of the leader, may still be on its way to this
    // CTA when it ends (all complete at once in a normal run; after a timeout
    // the waits are bounded).  A slot is freed after its copies have landed.
    for (int i = armed > a.stages ? armed - a.stages : 0; i < armed; ++i) {
      if (rank == 0) mbar_wait(&bars->full[i % a.stages], (i / a.stages) & 1, a.err, kDevTimeoutFull);
      if (!mbar_wait(&bars->empty[i % a.stages], (i / a.stages) & 1, a.err, kDevTimeoutEmpty)) break;
    }
  } else if (warp == 1 && rank == 0) {
    // ---- MMA issuer (of the pair: the leader's): the warp runs the loop together and one elected lane
    // issues, so that the descriptors stay in uniform registers
    const uint32_t idesc = idesc_bf16_f32(kRM * CL, a.BN);
    const uint32_t ring0 = smem_u32(ring);
    int s = 0, ph = 0, t = 0;
    uint32_t limit = kSpinLimit;
    for (int u = u0; u < units; u += ustep, ++t) {
      const int b = t & 1;
      if (t >= 2) mbar_wait_keep(limit, &bars->acce[b], ((t >> 1) + 1) & 1, a.err, kDevTimeoutAccum);
      tc_fence_after();
      const uint32_t acc = tmem + static_cast<uint32_t>(b * kRMaxBN);
      for (int kb = 0; kb < nk; ++kb) {
        mbar_wait_keep(limit, &bars->full[s], ph, a.err, kDevTimeoutFull);
        tc_fence_after();
        const uint64_t ad = smem_desc_k128(ring0 + s * stage_bytes);
        const uint64_t bd = smem_desc_k128(ring0 + s * stage_bytes + kRABytes);
        if (elect_one() && limit > 1) {
#pragma unroll
          for (int j = 0; j < kRK / 16; ++j) {   // 32 bytes along K: 2 in the descriptor's address field
            if (CL > 1) umma_bf16_pair(acc, ad + 2 * j, bd + 2 * j, idesc, (kb | j) != 0 ? 1u : 0u);
            else umma_bf16(acc, ad + 2 * j, bd + 2 * j, idesc, (kb | j) != 0 ? 1u : 0u);
          }
          if (CL > 1) umma_commit_pair(&bars->empty[s]);
          else umma_commit(&bars->empty[s]);
        }
        __syncwarp();
        if (++s == a.stages) {
          s = 0;
          ph ^= 1;
        }
      }
      if (elect_one() && limit > 1) {
        if (CL > 1) umma_commit_pair(&bars->accf[b]);
        else umma_commit(&bars->accf[b]);
      }
      __syncwarp();
    }
  } else if (warp >= 4) {
    // ---- epilogue: thread = one accumulator row
    const int quarter = warp & 3;
    uint8_t* my = stg + quarter * 2 * kRStg;
    int t = 0, nst = 0;
    for (int u = u0; u < units; u += ustep, ++t) {
      const int mtile = (u % mu) * CL + rank, m0 = mtile * kRM + 32 * quarter, n0 = (u / mu) * a.BN;
      const int b = t & 1;
      int ok = mbar_wait(&bars->accf[b], (t >> 1) & 1, a.err, kDevTimeoutAccum) ? 1 : 0;
      if (!__all_sync(0xffffffffu, ok)) break;
      tc_fence_after();
      const uint32_t row = tmem + (static_cast<uint32_t>(32 * quarter) << 16) + b * kRMaxBN;
      if constexpr (EPI == kRowsStore) {
        for (int c0 = 0; c0 < a.BN && n0 + c0 < a.N; c0 += 32) {
          float v[32];
          tmem_ld_32x32b_x32(row + c0, v);
          uint8_t* box = my + (nst & 1) * kRStg;
          if (a.tma_store) {   // the store of two boxes ago has read this one
            if (lane == 0 && nst >= 2) bulk_wait_read_but_one();
          }
          __syncwarp();
#pragma unroll
          for (int q = 0; q < 8; ++q)
            *reinterpret_cast<float4*>(box + lane * 128 + ((q ^ (lane & 7)) << 4)) =
                make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
          if (a.tma_store) {
            fence_proxy_async_smem();
            __syncwarp();
            if (lane == 0) {
              tma_store_3d(&mapD, box, n0 + c0, m0, 0);
              bulk_commit_group();
            }
          } else {
            __syncwarp();
            const int col = n0 + c0 + lane;
            const bool in = col < a.N;
            for (int r = 0; r < 32; ++r) {
              const float x = *reinterpret_cast<const float*>(box + r * 128 + (((lane >> 2) ^ (r & 7)) << 4) + (lane & 3) * 4);
              if (in && m0 + r < a.M) a.C[static_cast<int64_t>(m0 + r) * a.N + col] = x;
            }
            __syncwarp();
          }
          ++nst;
        }
      } else if constexpr (EPI == kRowsNarrow) {   // a thread's row as it is (staged as above it took a warp 32 turns)
        float v[32];
        tmem_ld_32x32b_x32(row, v);
        float* out = a.C + static_cast<int64_t>(m0 + lane) * a.N;
#pragma unroll
        for (int c = 0; c < 32; ++c)
          if (c < a.N && m0 + lane < a.M) out[c] = v[c];
      } else if constexpr (EPI == kRowsRelu) {
        for (int c0 = 0; c0 < a.BN && n0 + c0 < a.N; c0 += 64) {   // BN and N are multiples of 64
          float v0[32], v1[32];
          tmem_ld_32x32b_x32_pair(row + c0, v0, row + c0 + 32, v1);
          uint8_t* box = my + (nst & 1) * kRStg;
          if (lane == 0 && nst >= 2) bulk_wait_read_but_one();
          __syncwarp();
          const float4* bias = reinterpret_cast<const float4*>(a.bias + n0 + c0);
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            const float (&v)[32] = h ? v1 : v0;
#pragma unroll
            for (int q = 0; q < 4; ++q) {
              const float4 b0 = __ldg(bias + 8 * h + 2 * q), b1 = __ldg(bias + 8 * h + 2 * q + 1);
              *reinterpret_cast<uint4*>(box + lane * 128 + (((4 * h + q) ^ (lane & 7)) << 4)) =
                  make_uint4(pack_bf16x2(fmaxf(v[8 * q] + b0.x, 0.f), fmaxf(v[8 * q + 1] + b0.y, 0.f)),
                             pack_bf16x2(fmaxf(v[8 * q + 2] + b0.z, 0.f), fmaxf(v[8 * q + 3] + b0.w, 0.f)),
                             pack_bf16x2(fmaxf(v[8 * q + 4] + b1.x, 0.f), fmaxf(v[8 * q + 5] + b1.y, 0.f)),
                             pack_bf16x2(fmaxf(v[8 * q + 6] + b1.z, 0.f), fmaxf(v[8 * q + 7] + b1.w, 0.f)));
            }
          }
          fence_proxy_async_smem();
          __syncwarp();
          if (lane == 0) {
            tma_store_3d(&mapD, box, n0 + c0, m0, 0);
            bulk_commit_group();
          }
          ++nst;
        }
      } else {   // kRowsLoss: BN = 32, one column tile; classes in columns
        float z[32];
        tmem_ld_32x32b_x32(row, z);
        const int m = m0 + lane;
        float loss = 0.f;
        if (m < a.M) {
          const int y = a.labels[m];
          float mx = -INFINITY, zy = 0.f, se = 0.f;
#pragma unroll
          for (int c = 0; c < 32; ++c)
            if (c < a.N) {
              z[c] += __ldg(a.bias + c);
              mx = fmaxf(mx, z[c]);
              if (c == y) zy = z[c];
            }
#pragma unroll
          for (int c = 0; c < 32; ++c)
            if (c < a.N) se += expf(z[c] - mx);
          loss = mx + logf(se) - zy;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) loss += __shfl_xor_sync(0xffffffffu, loss, o);
        if (lane == 0) a.loss_part[mtile * 4 + quarter] = loss;
      }
      // the accumulator is free for tile t + 2
      tc_fence_before();
      __syncwarp();
      if (lane == 0) {
        if (CL > 1) mbar_arrive_at(cluster_addr(&bars->acce[b], 0));
        else mbar_arrive(&bars->acce[b]);
      }
    }
    if (lane == 0) bulk_wait_all();
  }
  tc_fence_before();
  if (CL > 1) cluster_sync();   // the pair's products and arrivals are done in both CTAs
  else __syncthreads();
  if (warp == 2) {
    tc_fence_after();
    tmem_dealloc_cl<CL>(tmem);
  }
}

constexpr int kMaxDevices = 64;
// SMs of the current device, and clusters of two of the kernel's CTAs that fit (queried once per device)
struct DevInfo {
  std::atomic<int> sms{0}, pairs{0};
};
DevInfo g_dev[kMaxDevices];

// at least 164 KB: one CTA per SM and none of another kernel's clusters beside it,
// so that a tcgen05.alloc of all 512 columns never waits for one
constexpr size_t kRLeastSmem = 164 * 1024;
static_assert(no_cluster_beside(kRLeastSmem), "the pair's CTAs meet no other cluster's");
size_t rows_smem(int stages, int BN, int cl) {
  const size_t b = 1024 + kRStgBytes + static_cast<size_t>(stages) * (kRABytes + BN / cl * 128) + kRBarBytes;
  return b < kRLeastSmem ? kRLeastSmem : b;
}
int rows_stages(int BN, int nk, int cl) {
  int st = kRRing / (kRABytes + BN / cl * 128);
  st = st > kRMaxStages ? kRMaxStages : st;
  return st > nk ? (nk < 2 ? 2 : nk) : st;
}

template <int EPI, int CL>
cudaLaunchConfig_t rows_config(cudaLaunchAttribute* attr, int grid, size_t smem, cudaStream_t s) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid, 1, 1);
  cfg.blockDim = dim3(kRThreads, 1, 1);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cfg.attrs = attr;
  cfg.numAttrs = 0;
  if (CL > 1) {
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = CL;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.numAttrs = 1;
  }
  return cfg;
}

// {SMs, resident clusters of two}
void device_room(int& sms, int& pairs) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) dev = 0;
  sms = g_dev[dev].sms.load(std::memory_order_relaxed);
  pairs = g_dev[dev].pairs.load(std::memory_order_relaxed);
  if (sms > 0 && pairs > 0) return;
  if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms < 1) sms = 1;
  cudaLaunchAttribute attr[1];
  const size_t smem = rows_smem(rows_stages(kRMaxBN, 64, 2), kRMaxBN, 2);
  pairs = 0;
  if (allow_smem(gemm_rows_kernel<kRowsStore, 2>, kRSmem) == cudaSuccess) {
    cudaLaunchConfig_t cfg = rows_config<kRowsStore, 2>(attr, 2, smem, nullptr);
    if (cudaOccupancyMaxActiveClusters(&pairs, gemm_rows_kernel<kRowsStore, 2>, &cfg) != cudaSuccess) pairs = 0;
  }
  cudaGetLastError();
  if (pairs < 1) pairs = 1;
  g_dev[dev].sms.store(sms, std::memory_order_relaxed);
  g_dev[dev].pairs.store(pairs, std::memory_order_relaxed);
}

// relative time of a launch with tiles of BN columns: waves x the longer of a
// k-block's products (BN cycles) and loads (bytes at 60 a cycle), plus a
// tile's fixed part, plus what a launch on clusters takes longer (start and end
// barriers, both SMs' tensor memory): 1500 cycles, so that products of few
// K-blocks run on CTAs alone.  Device time of a launch, one 128 x BN tile a CTA
// without clusters before this kernel / pairs wherever the row tiles are even /
// this rule, us: 1024 x 1 x 64: 3.0 / 4.5 / 2.8; 4096 x 64 x 64: 3.8 / 4.2 / 3.2;
// 1024 x 1 x 784: 7.4 / 8.4 / 7.1; 1024 x 1000 x 784: 9.9 / 8.5 / 7.4.
double rows_cost(int mt, int N, int nk, int BN, int CL, int room) {
  const int units = mt / CL * ((N + BN - 1) / BN);
  const int waves = (units + room - 1) / room;
  const double load = (kRABytes + BN * 128.0 / CL) / 60.0, mma = BN;
  return waves * (nk * (load > mma ? load : mma) + 4.0 * BN + 600.0) + (CL > 1 ? 1500.0 : 0.0);
}

template <int EPI, int CL>
cudaError_t launch_rows_t(const CUtensorMap& mA, const CUtensorMap& mB, const CUtensorMap& mD, const RowsArgs& a,
                          int grid, cudaStream_t s) {
  const size_t smem = rows_smem(a.stages, a.BN, CL);
  cudaError_t e = allow_smem(gemm_rows_kernel<EPI, CL>, kRSmem);
  if (e != cudaSuccess) return e;
  cudaLaunchAttribute attr[2];
  cudaLaunchConfig_t cfg = rows_config<EPI, CL>(attr, grid, smem, s);
  if (a.pdl) {
    attr[cfg.numAttrs].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[cfg.numAttrs].val.programmaticStreamSerializationAllowed = 1;
    ++cfg.numAttrs;
  }
  return cudaLaunchKernelEx(&cfg, gemm_rows_kernel<EPI, CL>, mA, mB, mD, a);
}

}  // namespace

RowsPlan gemm_rows_plan(int epi, int M, int N, int K) {
  RowsPlan p;
  int sms, pairs;
  device_room(sms, pairs);
  const int mt = (M + kRM - 1) / kRM, nk = (K + kRK - 1) / kRK;
  p.cl = 1;
  p.BN = 32;
  if (epi == kRowsLoss) return p;   // one column tile of 32 classes
  const int step = epi == kRowsRelu ? 64 : 32, most = (N + step - 1) / step * step;
  double best = 0.0;
  for (int cl = 1; cl <= 2; ++cl) {
    if (mt % cl != 0) continue;
    for (int bn = step; bn <= kRMaxBN && bn <= most; bn += step) {
      const double c = rows_cost(mt, N, nk, bn, cl, cl == 2 ? pairs : sms);
      if (best == 0.0 || c < best) {
        best = c;
        p.cl = cl;
        p.BN = bn;
      }
    }
  }
  return p;
}

cudaError_t launch_gemm_rows(int epi, const RowsPlan& p, const CUtensorMap& mA, const CUtensorMap& mB,
                             const CUtensorMap& mD, RowsArgs a, cudaStream_t s) {
  int sms, pairs;
  device_room(sms, pairs);
  a.BN = p.BN;
  a.mt = (a.M + kRM - 1) / kRM;
  a.nt = (a.N + p.BN - 1) / p.BN;
  a.stages = rows_stages(p.BN, (a.K + kRK - 1) / kRK, p.cl);
  const int64_t units = static_cast<int64_t>(a.mt / p.cl) * a.nt;
  const int room = p.cl == 2 ? pairs : sms;
  const int grid = static_cast<int>(units < room ? units : room) * p.cl;
  if (epi == kRowsStore)
    return p.cl == 2 ? launch_rows_t<kRowsStore, 2>(mA, mB, mD, a, grid, s) : launch_rows_t<kRowsStore, 1>(mA, mB, mD, a, grid, s);
  if (epi == kRowsNarrow)
    return p.cl == 2 ? launch_rows_t<kRowsNarrow, 2>(mA, mB, mD, a, grid, s) : launch_rows_t<kRowsNarrow, 1>(mA, mB, mD, a, grid, s);
  if (epi == kRowsRelu)
    return p.cl == 2 ? launch_rows_t<kRowsRelu, 2>(mA, mB, mD, a, grid, s) : launch_rows_t<kRowsRelu, 1>(mA, mB, mD, a, grid, s);
  return launch_rows_t<kRowsLoss, 1>(mA, mB, mD, a, grid, s);
}

}  // namespace oscars
