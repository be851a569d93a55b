// Forward and backward of the last layer (2 to 32 classes) of the per-layer path
// on the tensor cores (Eq. 4, "otherwise" branch: one SGD step of the
// worker's head).  A cluster of H/F CTAs serves one active worker; CTA r owns
// hidden features [F r, F r + F), F = 128 NH with NH = 1 or 2 halves of 128
// (NH = 2 keeps the cluster at 4 CTAs for H = 1024: only 15 clusters of 8
// are resident on the GPU at once).  With h = the layer input (bf16,
// [B][H]) and W2 the head weights ([C][H]):
//
//  1. partial logits of the CTA's features, P[b][c] = sum_f h[b][f] W2[c][f]:
//     tcgen05.mma M = 128 rows, N = NC = 16 or 32 classes (rows >= B and classes >= C
//     are zero-filled by the TMA loads), K = F features;
//  2. cluster barrier; the logits are the partials of ranks 0..n-1 summed in
//     that order from distributed shared memory, plus the bias; softmax
//     cross-entropy on 2, 4 or 8 threads per row, four classes at a time
//     (with one thread a row its divisions and bank conflicts took 8800 of
//     the kernel's 22500 clocks with 17 classes, 4500 with 10); dz (fp32) and
//     its bf16 copy, written into two shared tiles laid out as tensor-core
//     operands;
//  3. head weight gradient dW2^T[f][c] = sum_b h[b][f] dz[b][c] (per half
//     M = 128 features, N = NC, K = B: the h tile read MN-major) and SGD of
//     the CTA's head columns;
//  4. input gradient of the layer below, transposed: dh^T[f][b] = sum_c
//     W2[c][f] dz[b][c] (per half M = 128 features, N = B, K = NC: the W2
//     tile read MN-major); masked by h > 0; the fp32
//     bias gradient per feature, and the bf16 gradient.
// For B a multiple of 64, where the next kernels read only G^T, the tile in
// shared memory is h^T (as in memory, [H][B]): the products read it MN-major
// in 1 and K-major in 3, a thread finds the masks of 16 rows in two of its own
// 16-byte chunks and leaves the gradient there, and TMA stores write G^T (with
// the h tile, a thread reads 2-byte elements and stores 16-byte chunks of its
// own row, 32 lines an instruction; mask bits read beforehand from the h tile
// took 2700 clocks: 3072-1024-1024-10, a round: 1584 -> 1573 us).  For other B it is
// the h tile [B][H]; G^T rows are written from registers, G rows through the
// tile (overwritten in place, then written as full 16-byte chunks).
// Rank 0 also writes the loss partials and updates the head bias.  One
// thread issues the TMA loads and the MMAs; the accumulators share 128 NH
// TMEM columns (the phases run one after another).  All mbarrier waits are
// bounded; the cluster barriers are unconditional, so a timeout cannot leave
// a CTA of the cluster behind at one.
//
// NC is C rounded up to 16 or 32; C = 10 is also a template argument (CT), which
// keeps the row softmax in as few registers and instructions as it needs.
// Bound by latency and by instruction fetch: each launch runs its code once,
// so the phases are short loops, not unrolled ones (a first pass over 32 rows
// in phase 4 took 4500 clocks, the next ones 720), and one warp brings the
// code in early (below).  One launch replaces a forward and a backward launch
// on the CUDA cores for other class counts (17 and 12 us each with 17 classes,
// 256 features, batch 32).  A round of the 1000-384-256-17 model, 5 workers:
// 534 us with those, 440 with this kernel's first form, 335 now (374 before
// the loops, the early code and the h^T tile); 3072-1024-1024-10, 32 workers:
// 1579 -> 1573.  (Both models' rounds have become shorter by other kernels
// since.)
#include <atomic>

#include "common.cuh"
#include "internal.h"

namespace oscars {

namespace {

constexpr int kHT = 128;                 // hidden features per half (tensor-core rows)
constexpr int kHTThreads = 256;
constexpr int kHTMaxCluster = 8;
constexpr int kHTRows = 128;             // rows of the h tile (B <= 128; the rest zero)

// shared memory carve-up (bytes from a 1024-aligned base) for NH halves
template <int NH, int NC>
struct HTCfg {
  static constexpr int F = kHT * NH;                     // features per CTA
  static constexpr int oH = 0;                           // h tile: F/64 boxes [128 rows][64 features] bf16, 128-B swizzle
  static constexpr int oW2 = oH + (F / 64) * kHTRows * 128;   // W2 tile: F/64 boxes [NC classes][64 features]
  static constexpr int oDzT = oW2 + (F / 64) * NC * 128;    // dz^T: [16 classes][B rows] K-major (K = rows), 2 atoms
  static constexpr int oDzK = oDzT + 2 * NC * 128;       // dz: [B rows][NC classes] K-major, no swizzle
  static constexpr int oPl = oDzK + kHTRows * NC * 2;    // [128][NC] fp32 partial logits (read by the cluster)
  static constexpr int oDz = oPl + kHTRows * NC * 4;   // [128][kLdz] fp32 dlogits
  static constexpr int kLdz = NC + 4;                    // row stride of dz: rows of neighbouring threads in other banks
  static constexpr int oLoss = oDz + kHTRows * kLdz * 4; // [128]
  static constexpr int oGbp = oLoss + kHTRows * 4;       // [2][F]
  static constexpr int oLab = oGbp + 2 * F * 4;          // [128] int
  static constexpr int oB2 = oLab + kHTRows * 4;         // [16]
  static constexpr int oBar = oB2 + NC * 4;            // tma, mma barriers, TMEM slot
  static constexpr int kSmem = oBar + 64 + 1024;
  static constexpr uint32_t kTmemCols = 128 * NH;
  static_assert(kSmem >= kLeastClusterSmem, "a kernel on clusters with tensor memory");
};

// element (row b, feature f) of the h tile (K-major, 128-byte swizzle, one box per 64 features)
__device__ __forceinline__ uint32_t h_off(int b, int f) {
  return static_cast<uint32_t>((f >> 6) * (kHTRows * 128) + b * 128 + ((((f & 63) >> 3) ^ (b & 7)) << 4) + (f & 7) * 2);
}

// K-major no-swizzle descriptor: core matrices of 8 rows x 16 bytes, `lbo`
// bytes apart along K and `sbo` bytes apart along M/N.
__device__ __forceinline__ uint64_t smem_desc_none(uint32_t saddr, uint32_t lbo, uint32_t sbo) {
  uint64_t d = 0;
  d |= static_cast<uint64_t>((saddr & 0x3FFFFu) >> 4);
  d |= static_cast<uint64_t>((lbo >> 4) & 0x3FFFu) << 16;
  d |= static_cast<uint64_t>((sbo >> 4) & 0x3FFFu) << 32;
  d |= static_cast<uint64_t>(1) << 46;
  return d;
}

__device__ __forceinline__ float4 ld_dsmem_f32x4(const float* local, uint32_t rank) {
  uint32_t remote;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(remote) : "r"(smem_u32(local)), "r"(rank));
  float4 v;
  asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];"
               : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
               : "r"(remote)
               : "memory");
  return v;
}

__device__ __forceinline__ void tmem_ld_32x32b_x16(uint32_t taddr, float (&v)[16]) {
  uint32_t r[16];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
      "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];\n\t"
      "tcgen05.wait::ld.sync.aligned;"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr)
      : "memory");
#pragma unroll
  for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}

// Phase 2 with TPR = 1 << TSH threads per row (the whole block for B = 32, 64
// and 128): thread q takes the 4-class chunks q, q + TPR, ...
template <int NH, int NC, int CT, int TSH>
__device__ __forceinline__ void head_softmax(const HeadArgs& a, uint8_t* sm, int t, int ncl) {
  using Cfg = HTCfg<NH, NC>;
  const float* pl = reinterpret_cast<const float*>(sm + Cfg::oPl);
  const float* b2 = reinterpret_cast<const float*>(sm + Cfg::oB2);
  const int* labs = reinterpret_cast<const int*>(sm + Cfg::oLab);
  float* dz = reinterpret_cast<float*>(sm + Cfg::oDz);
  float* rowloss = reinterpret_cast<float*>(sm + Cfg::oLoss);
  uint8_t* dzT = sm + Cfg::oDzT;
  uint8_t* dzK = sm + Cfg::oDzK;
  const int B = a.B, C = CT > 0 ? CT : a.C;
  constexpr int CL = CT > 0 ? CT : NC;   // class loops: compile-time bound, `c < C` inside
  constexpr int tpr = 1 << TSH;
  const int b = t >> TSH, q = t & (tpr - 1);
  constexpr int QN = (CL + 3) / 4;      // chunks with classes
  constexpr int QT = (QN + tpr - 1) / tpr;   // chunks of a thread at most
  const bool row = b < B;
  float z[4 * QT];
#pragma unroll
  for (int i = 0; i < 4 * QT; ++i) z[i] = 0.f;
  if (row) {
    // four ranks' partials are requested before the first is added (a remote
    // load waits a round trip across the cluster); NH = 1 has at most four
#pragma unroll
    for (int r0 = 0; r0 < (NH == 1 ? 4 : kHTMaxCluster); r0 += 4) {
      float4 p[4][QT];
#pragma unroll
      for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int i = 0; i < QT; ++i)
          if (r0 + r < ncl && q + i * tpr < QN) p[r][i] = ld_dsmem_f32x4(pl + b * NC + 4 * (q + i * tpr), r0 + r);
#pragma unroll
      for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int i = 0; i < QT; ++i)
          if (r0 + r < ncl && q + i * tpr < QN) {
            z[4 * i] += p[r][i].x;
            z[4 * i + 1] += p[r][i].y;
            z[4 * i + 2] += p[r][i].z;
            z[4 * i + 3] += p[r][i].w;
          }
    }
  }
  const int y = row ? labs[b] : 0;
  float m = -INFINITY, zy = -INFINITY;
#pragma unroll
  for (int i = 0; i < 4 * QT; ++i) {
    const int c = 4 * (q + i / 4 * tpr) + i % 4;
    z[i] = c < C ? z[i] + b2[c < NC ? c : 0] : -INFINITY;
    m = fmaxf(m, z[i]);
    if (c == y) zy = z[i];
  }
  for (int o = tpr >> 1; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
  float s = 0.f, so_ = 0.f;
#pragma unroll
  for (int i = 0; i < 4 * QT; ++i) {
    const int c = 4 * (q + i / 4 * tpr) + i % 4;
    z[i] = c < C ? expf(z[i] - m) : 0.f;
    s += z[i];
    if (c != y) so_ += z[i];
  }
  for (int o = tpr >> 1; o > 0; o >>= 1) {
    s += __shfl_xor_sync(0xffffffffu, s, o);
    so_ += __shfl_xor_sync(0xffffffffu, so_, o);
  }
  const float inv = 1.0f / static_cast<float>(B);
  if (row) {
    if (q == ((y >> 2) & (tpr - 1))) rowloss[b] = m + logf(s) - zy;   // the thread that has class y
    uint8_t* ck = dzK + (b >> 3) * (NC / 8 * 128) + (b & 7) * 16;
    uint8_t* at = dzT + (b >> 6) * (NC * 128);
    const int e64 = b & 63;
#pragma unroll
    for (int i = 0; i < QT; ++i) {
      const int k = q + i * tpr;
      if (k >= QN) continue;
      float g[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int c = 4 * k + j;
        g[j] = c < C ? (c == y ? -so_ : z[4 * i + j]) / s * inv : 0.f;
      }
      *reinterpret_cast<float4*>(dz + b * Cfg::kLdz + 4 * k) = make_float4(g[0], g[1], g[2], g[3]);
      // dz as the K-major [rows][NC classes] operand: classes 8 j .. 8 j + 7
      // one 16-byte chunk of core matrix (b / 8, j)
      *reinterpret_cast<uint2*>(ck + 128 * (k >> 1) + 8 * (k & 1)) = make_uint2(pack_bf16x2(g[0], g[1]), pack_bf16x2(g[2], g[3]));
      // dz^T as the K-major [NC classes][rows] operand (K = rows, atoms of 64 rows)
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int c = 4 * k + j;
        *reinterpret_cast<__nv_bfloat16*>(at + c * 128 + ((((e64 >> 3) ^ (c & 7)) & 7) << 4) + (e64 & 7) * 2) =
            __float2bfloat16_rn(g[j]);
      }
    }
  }
}

// K CTAs share an SM (registers): see head_per_sm
template <int NH, int NC, int CT, int K>
__global__ void __launch_bounds__(kHTThreads, K) head_tc_kernel(const __grid_constant__ CUtensorMap mH,
                                                              const __grid_constant__ CUtensorMap mW2,
                                                              const __grid_constant__ CUtensorMap mGT,
                                                              const __grid_constant__ HeadArgs a) {
  using Cfg = HTCfg<NH, NC>;
  constexpr int F = Cfg::F;
  extern __shared__ uint8_t ht_raw[];
  uint8_t* sm = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(ht_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* hT = sm + Cfg::oH;
  uint8_t* w2 = sm + Cfg::oW2;
  uint8_t* dzT = sm + Cfg::oDzT;
  uint8_t* dzK = sm + Cfg::oDzK;
  float* pl = reinterpret_cast<float*>(sm + Cfg::oPl);
  float* dz = reinterpret_cast<float*>(sm + Cfg::oDz);
  float* rowloss = reinterpret_cast<float*>(sm + Cfg::oLoss);
  float* gbp = reinterpret_cast<float*>(sm + Cfg::oGbp);
  int* labs = reinterpret_cast<int*>(sm + Cfg::oLab);
  float* b2 = reinterpret_cast<float*>(sm + Cfg::oB2);
  uint64_t* tma_bar = reinterpret_cast<uint64_t*>(sm + Cfg::oBar);
  uint64_t* mma_bar = tma_bar + 1;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(mma_bar + 1);

  const int H = a.H, B = a.B, C = CT > 0 ? CT : a.C;
  constexpr int CL = CT > 0 ? CT : NC;   // class loops: compile-time bound, `c < C` inside
  const int i = blockIdx.x;
  const int w = a.wid[i], src = a.src[i];
  const uint32_t rank = cluster_ctarank();
  const int ncl = static_cast<int>(gridDim.y);
  const int k0 = blockIdx.y * F;
  const int t = threadIdx.x, warp = __shfl_sync(0xffffffffu, t >> 5, 0), lane = t & 31;
  const int64_t so = static_cast<int64_t>(src) * a.slot_stride;
  const int64_t dof = static_cast<int64_t>(w) * a.slot_stride;

  if (t == 0) {
    prefetch_tmap(&mH);
    prefetch_tmap(&mW2);
    mbar_init(tma_bar, 1);
    mbar_init(mma_bar, 1);
    fence_barrier_init();
  }
  // B a multiple of 64: the tile is h^T [features][rows], boxes (half, 64 rows)
  // of 128 features; otherwise h [rows][features], boxes of 64 features
  const bool ht = !a.G;
  const int hb = B >> 6;                 // h^T: boxes per half
  bool ok = false;
  uint32_t tmem = 0;
  float old[CL];
  const int e_mh = NH == 2 ? warp >> 2 : 0;                    // phases 3 and 4: this thread's half, feature and rows
  const int e_fl = 32 * (warp & 3) + lane, e_f = kHT * e_mh + e_fl;
  const int e_rows = NH == 2 ? B : B / 2, e_r0 = NH == 2 ? 0 : (warp >> 2) * e_rows;
  // rows e_r0, e_r0 + 1, ... of the h tile (e_r0 is a multiple of 16) at this feature: see h_off
  uint8_t* const h_col = hT + (e_f >> 6) * (kHTRows * 128) + e_r0 * 128 + (e_f & 7) * 2;
  const int h_chunk = (e_f & 63) >> 3;
  // While the previous kernel still runs, the last warp goes through the code
  // of phases 2 to 4 once on whatever shared memory holds, without touching
  // other memory, the cluster or the tensor core: it brings the instructions
  // to the SM.  Each launch runs them once, and the weights that stream
  // through L2 between two launches evict them (a round of
  // 1000-384-256-17, 5 workers: 346 -> 338 us; 3072-1024-1024-10, 32: 1592 -> 1584).
#pragma unroll 1
  for (int dry = a.pdl && warp == kHTThreads / 32 - 1 ? 1 : 0; dry >= 0; --dry) {
    if (!dry) {
      __syncthreads();   // the dry pass has left the tiles
      // what the previous kernel does not write is requested while it runs (the
      // weights of the previous step: every kernel of the chain waits for its
      // predecessor before it lets its successor start); rounds as above: 318.9
      // -> 313.9 us and 1526 -> 1521
      if (t == 0) {
        mbar_arrive_expect_tx(tma_bar, (ht ? NH * hb : F / 64) * (kHTRows * 128) + (F / 64) * (NC * 128));
#pragma unroll
        for (int q = 0; q < F / 64; ++q) tma_load_3d(w2 + q * NC * 128, &mW2, k0 + 64 * q, 0, src, tma_bar);
      }
      if (warp == 0) {
        tmem_alloc(tmem_slot, Cfg::kTmemCols);
        tmem_relinquish();
      }
      // the old master values of this thread's head column, requested long before
      // the update needs them (and before any new value is stored: source and
      // destination slots may be the same slab)
      if (warp < 4 * NH) {
        const int f = kHT * (warp >> 2) + 32 * (warp & 3) + lane;
#pragma unroll
        for (int c = 0; c < CL; ++c)
          if (c < C) old[c] = a.master[so + a.offW + static_cast<int64_t>(c) * H + k0 + f];
      }
      // the dz tiles' padding (classes >= C, rows >= B) stays zero
      for (int q = t; q < (2 * NC * 128 + kHTRows * NC * 2) / 16; q += kHTThreads)
        reinterpret_cast<uint4*>(dzT)[q] = make_uint4(0, 0, 0, 0);
      for (int b = t; b < B; b += kHTThreads) labs[b] = a.labels[static_cast<int64_t>(w) * B + b];
      if (t < NC) b2[t] = t < C ? a.master[so + a.offB + t] : 0.f;
      pdl_wait();      // the layer input (the previous kernel's output) is complete
      if (t == 0) {
        if (ht) {
          for (int q = 0; q < NH * hb; ++q)
            tma_load_3d(hT + q * (kHT * 128), &mH, 64 * (q & (hb - 1)), k0 + kHT * (q / hb), w, tma_bar);
        } else {
#pragma unroll
          for (int q = 0; q < F / 64; ++q) tma_load_3d(hT + q * kHTRows * 128, &mH, k0 + 64 * q, 0, w, tma_bar);
        }
      }
      tc_fence_before();
      __syncthreads();
      tc_fence_after();
      tmem = *tmem_slot;
      pdl_trigger();

      // ---- 1. partial logits
      if (warp == 0) {   // converged, one elected lane issues: see elect_one
        const bool landed = mbar_wait(tma_bar, 0, a.err, kDevTimeoutFull);
        tc_fence_after();
        // A = h: MN-major from the h^T tile (rows >= B are whatever follows it; their
        // logits are not used), K-major from the h tile
        const uint32_t idesc = idesc_bf16_f32(kHTRows, NC) | (ht ? 1u << 15 : 0u);
        const uint64_t hd = ht ? smem_desc_mn128(smem_u32(hT), kHT * 128) : smem_desc_k128(smem_u32(hT));
        const uint64_t wd = smem_desc_k128(smem_u32(w2));   // addresses in 16 bytes
        const uint32_t jstep = ht ? 128 : 2, ostep = ht ? 512 : kHTRows * 128 / 16, hstep = ht ? hb * 1024 : 2 * 1024;
        if (elect_one()) {
          if (landed)
#pragma unroll
            for (int kb = 0; kb < F / 64; ++kb)
#pragma unroll
              for (int j = 0; j < 4; ++j)
                umma_bf16(tmem, hd + (kb >> 1) * hstep + (kb & 1) * ostep + j * jstep, wd + kb * (NC * 128 / 16) + 2 * j,
                          idesc, (kb | j) != 0 ? 1u : 0u);
          umma_commit(mma_bar);   // arrives even with nothing issued, so the waits below end
        }
        __syncwarp();
      }
      ok = mbar_wait_warp(mma_bar, 0, a.err, kDevTimeoutAccum);
      tc_fence_after();
      if (warp < 4) {
        float v[NC];
        if constexpr (NC == 16) tmem_ld_32x32b_x16(tmem + (static_cast<uint32_t>(32 * warp) << 16), v);
        else tmem_ld_32x32b_x32(tmem + (static_cast<uint32_t>(32 * warp) << 16), v);
        float4* row = reinterpret_cast<float4*>(pl + (32 * warp + lane) * NC);
#pragma unroll
        for (int q = 0; q < NC / 4; ++q) row[q] = make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
      }
      tc_fence_before();
      cluster_sync();
      tc_fence_after();

    }

    // ---- 2. logits (cluster sum in rank order), softmax cross-entropy, dz tiles.
    // 8, 4 or 2 threads a row, each count its own code: chunks that no thread
    // of a count has cost their instructions' fetch (17 classes,
    // batch 32: this phase 5000 -> 2300 clocks)
    if (B <= 32) head_softmax<NH, NC, CT, 3>(a, sm, dry ? lane : t, dry ? 0 : ncl);
    else if (B <= 64) head_softmax<NH, NC, CT, 2>(a, sm, dry ? lane : t, dry ? 0 : ncl);
    else head_softmax<NH, NC, CT, 1>(a, sm, dry ? lane : t, dry ? 0 : ncl);
    if (!dry) {
      fence_proxy_async_smem();   // the dz tiles are read by the tensor core
      tc_fence_before();
      __syncthreads();
      tc_fence_after();

      // ---- 3. head weight gradient (M = features, N = classes, K = rows) + SGD
      if (warp == 0) {
        // A = h^T: K-major from the h^T tile, MN-major from the h tile
        const uint32_t idesc = idesc_bf16_f32(kHT, NC) | (ht ? 0u : 1u << 15);
        const uint64_t hd = ht ? smem_desc_k128(smem_u32(hT)) : smem_desc_mn128(smem_u32(hT), kHTRows * 128);
        const uint64_t zd = smem_desc_k128(smem_u32(dzT));
        const uint32_t jstep = ht ? 2 : 128, qstep = ht ? 1024 : 512, hstep = ht ? hb * 1024 : 2 * 1024;
        if (elect_one()) {
          if (ok)
#pragma unroll
            for (int mh = 0; mh < NH; ++mh)   // half mh: features [128 mh, 128 mh + 128) into columns [NC mh, NC mh + NC)
              for (int j = 0; j < B / 16; ++j)
                umma_bf16(tmem + NC * mh, hd + mh * hstep + (j >> 2) * qstep + (j & 3) * jstep,
                          zd + (j >> 2) * (NC * 128 / 16) + 2 * (j & 3), idesc, j != 0 ? 1u : 0u);
          umma_commit(mma_bar);
        }
        __syncwarp();
      }
      if (rank == 0 && warp >= 4) {   // loss partials and the head bias (CUDA cores, meanwhile)
        const int u = t - 128;
        if (u < B / kRowsPerLossChunk) {
          float l = 0.f;
          for (int r = 0; r < kRowsPerLossChunk; ++r) l += rowloss[u * kRowsPerLossChunk + r];
          const int64_t row = static_cast<int64_t>(w) * a.part_mul + a.part_add;
          a.loss_part[row * (B / kRowsPerLossChunk) + u] = l;
        }
        if (u >= 32) {   // warps 5-7: 8 lanes per class (12 classes a pass), then shuffles within each group of 8
          const int j = u & 7;
          for (int c0 = 0; c0 < C; c0 += 12) {
            const int c = c0 + ((u - 32) >> 3);
            float g = 0.f;
            if (c < C)
              for (int b = j; b < B; b += 8) g += dz[b * Cfg::kLdz + c];
#pragma unroll
            for (int o = 4; o > 0; o >>= 1) g += __shfl_xor_sync(0xffffffffu, g, o, 8);
            if (c < C && j == 0) a.master_w[dof + a.offB + c] = fmaf(-a.lr, g, a.master[so + a.offB + c]);
          }
        }
      }
      ok = mbar_wait_warp(mma_bar, 1, a.err, kDevTimeoutAccum) && ok;
      tc_fence_after();
      if (warp < 4 * NH && ok) {
        const int mh = warp >> 2, q = warp & 3;
        const int f = kHT * mh + 32 * q + lane;
        float v[NC];
        if constexpr (NC == 16) tmem_ld_32x32b_x16(tmem + NC * mh + (static_cast<uint32_t>(32 * q) << 16), v);
        else tmem_ld_32x32b_x32(tmem + NC * mh + (static_cast<uint32_t>(32 * q) << 16), v);
#pragma unroll
        for (int c = 0; c < CL; ++c) {
          if (c >= C) continue;
          const int64_t e = a.offW + static_cast<int64_t>(c) * H + k0 + f;
          const float nw = fmaf(-a.lr, v[c], old[c]);
          a.master_w[dof + e] = nw;
          a.shadow_w[dof + e] = __float2bfloat16_rn(nw);
        }
      }
      tc_fence_before();
      __syncthreads();
      tc_fence_after();

      // ---- 4. input gradient, transposed (M = features, N = rows, K = NC classes)
      if (warp == 0) {
        const uint32_t idesc = idesc_bf16_f32(kHT, B) | (1u << 15);   // A (W2^T) MN-major
        const uint64_t wd = smem_desc_mn128(smem_u32(w2), NC * 128), kd = smem_desc_none(smem_u32(dzK), 128, NC / 8 * 128);
        if (elect_one()) {
          if (ok)
#pragma unroll
            for (int mh = 0; mh < NH; ++mh)   // half mh into columns [B mh, B mh + B)
#pragma unroll
              for (int j = 0; j < NC / 16; ++j)   // 16 classes: 16 rows of the W2 tile, two core matrices of dz
                umma_bf16(tmem + B * mh, wd + mh * (2 * NC * 128 / 16) + 128 * j, kd + 16 * j, idesc, j != 0 ? 1u : 0u);
          umma_commit(mma_bar);
        }
        __syncwarp();
      }
      ok = mbar_wait_warp(mma_bar, 0, a.err, kDevTimeoutAccum) && ok;
      mbar_wait(tma_bar, 0, a.err, kDevTimeoutFull);   // completed long ago: orders the tile reads below
      tc_fence_after();
    }
    {
      // warp quarter q: features 32 q .. of its half; NH = 1: the two warp
      // groups split the rows; NH = 2: warp group g takes half g, all rows
      const int g = warp >> 2;
      const uint32_t tq = tmem + static_cast<uint32_t>(B * e_mh + e_r0) + (static_cast<uint32_t>(32 * (warp & 3)) << 16);
      const int together = NH == 1 && B == 64 ? 256 : 128;   // threads that fill one tile
      float gsum = 0.f;
#pragma unroll 1
      for (int r = 0; r < (dry ? 16 : e_rows); r += 16) {
        const int b0 = e_r0 + r;
        if (ok || dry) {
          float v[16];
          if (!dry) tmem_ld_32x32b_x16(tq + r, v);
          else
#pragma unroll
            for (int j = 0; j < 16; ++j) v[j] = 0.f;
          // the ReLU mask, and the bf16 gradient in its place: the thread's two
          // 16-byte chunks of the h^T tile, or its 16 elements of the h tile
          uint4* c0 = reinterpret_cast<uint4*>(hT + (e_mh * hb + (b0 >> 6)) * (kHT * 128) + e_fl * 128 +
                                               ((((b0 & 63) >> 3) ^ (e_fl & 7)) << 4));
          uint4* c1 = reinterpret_cast<uint4*>(reinterpret_cast<uintptr_t>(c0) ^ 16);
          uint32_t pk[8];
          if (ht) {
            const uint4 x = *c0, y = *c1;
            pk[0] = x.x; pk[1] = x.y; pk[2] = x.z; pk[3] = x.w;
            pk[4] = y.x; pk[5] = y.y; pk[6] = y.z; pk[7] = y.w;
          } else {
#pragma unroll
            for (int j = 0; j < 16; j += 2) {
              const uint32_t lo = *reinterpret_cast<const unsigned short*>(h_col + (r + j) * 128 + ((h_chunk ^ (j & 7)) << 4));
              const uint32_t hi =
                  *reinterpret_cast<const unsigned short*>(h_col + (r + j + 1) * 128 + ((h_chunk ^ ((j + 1) & 7)) << 4));
              pk[j >> 1] = lo | hi << 16;
            }
          }
#pragma unroll
          for (int j = 0; j < 16; j += 2) {
            const uint32_t h2 = pk[j >> 1];
            const float d0 = __uint_as_float(h2 << 16) > 0.f ? v[j] : 0.f;
            const float d1 = __uint_as_float(h2 & 0xffff0000u) > 0.f ? v[j + 1] : 0.f;
            gsum += d0;
            gsum += d1;
            pk[j >> 1] = pack_bf16x2(d0, d1);
          }
          if (ht) {
            *c0 = make_uint4(pk[0], pk[1], pk[2], pk[3]);
            *c1 = make_uint4(pk[4], pk[5], pk[6], pk[7]);
          } else {   // for the G rows below; the G^T rows from registers
#pragma unroll
            for (int j = 0; j < 16; ++j)
              *reinterpret_cast<unsigned short*>(h_col + (r + j) * 128 + ((h_chunk ^ (j & 7)) << 4)) =
                  static_cast<unsigned short>(pk[j >> 1] >> (16 * (j & 1)));
            if (dry) continue;
            uint4* gt = reinterpret_cast<uint4*>(a.GT + (static_cast<int64_t>(w) * H + k0 + e_f) * B + b0);
            gt[0] = make_uint4(pk[0], pk[1], pk[2], pk[3]);
            gt[1] = make_uint4(pk[4], pk[5], pk[6], pk[7]);
          }
        }
        if (!dry && ht && (together == 256 ? r + 16 == e_rows : (b0 & 48) == 48)) {   // 64 rows are complete: one TMA store
          fence_proxy_async_smem();
          if (together == 256) bar_named(1, 256);
          else if (g == 0) bar_named(1, 128);
          else bar_named(2, 128);
          if (ok && lane == 0 && warp == (together == 256 ? 0 : 4 * g)) {
            tma_store_3d(&mGT, hT + (e_mh * hb + (b0 >> 6)) * (kHT * 128), b0 & ~63, k0 + kHT * e_mh, w);
            bulk_commit_group();
          }
        }
      }
      gbp[(NH == 2 ? 0 : g) * F + e_f] = gsum;
    }
    if (dry) fence_proxy_async_smem();   // its writes of the h tile's place, before the TMA load
  }
  tc_fence_before();
  __syncthreads();
  if (t < F && ok) a.gb[static_cast<int64_t>(w) * H + k0 + t] = NH == 2 ? gbp[t] : gbp[t] + gbp[F + t];
  if (ok && a.G) {   // G rows: 16-byte chunks of 8 features (when a consumer reads G K-major)
    for (int q = t; q < B * (F / 8); q += kHTThreads) {
      const int b = q / (F / 8), j = q % (F / 8);
      *reinterpret_cast<uint4*>(a.G + (static_cast<int64_t>(w) * B + b) * H + k0 + 8 * j) =
          *reinterpret_cast<const uint4*>(hT + h_off(b, 8 * j));
    }
  }
  if (ht && lane == 0 && (warp & 3) == 0) bulk_wait_all();
  cluster_sync();   // no CTA leaves while another may still read its partial logits
  if (warp == 0) {
    tc_fence_after();
    tmem_dealloc(tmem, Cfg::kTmemCols);
  }
}

// halves per CTA: two when one half per CTA would need a cluster of more than 4
int head_tc_halves(int H) { return H / kHT > 4 ? 2 : 1; }

}  // namespace

bool head_tc_supported(int H, int B, int C) {
  if (C < 2 || C > 32 || B % 32 != 0 || B < 32 || B > kHTRows || H % kHT != 0) return false;
  const int F = kHT * head_tc_halves(H);
  return H % F == 0 && H / F <= kHTMaxCluster;
}

int head_tc_class_rows(int C) { return C <= 16 ? 16 : 32; }

namespace {
template <int NH, int NC, int CT, int K>
cudaLaunchConfig_t head_config(cudaLaunchAttribute* attr, int clusters, int size, int pdl, cudaStream_t s) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(clusters, size, 1);
  cfg.blockDim = dim3(kHTThreads, 1, 1);
  cfg.dynamicSmemBytes = HTCfg<NH, NC>::kSmem;
  cfg.stream = s;
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 1;
  attr[0].val.clusterDim.y = size;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = pdl ? 2 : 1;
  return cfg;
}

// CTAs an SM: one with all the registers it likes (175 to 246 a thread), or two
// with 128 where the workers' clusters are more than run at once with one
// (queried once per device).  2048 features, 10 classes, batch 32, 16 workers on
// clusters of 8: 25 us with one CTA an SM, two waves; 17.5 with two.  1024
// features, where one wave does: 15.7 and 16.4.  With more than 16 classes 128
// registers spill (2048 x 32, batch 32, a round of one worker 38 -> 44 us, of 64
// 308 -> 360): always one.
constexpr int kMaxDevices = 64;
std::atomic<int> g_head_room[kMaxDevices][kHTMaxCluster + 1];
template <int NH>
int head_per_sm(int size, int clusters) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) dev = 0;
  std::atomic<int>& r = g_head_room[dev][size];
  int room = r.load(std::memory_order_relaxed);
  if (room == 0) {
    cudaLaunchAttribute attr[2];
    const cudaLaunchConfig_t cfg = head_config<NH, 16, 10, 1>(attr, 1, size, 0, nullptr);
    if (allow_smem(head_tc_kernel<NH, 16, 10, 1>, HTCfg<NH, 16>::kSmem) != cudaSuccess ||
        cudaOccupancyMaxActiveClusters(&room, head_tc_kernel<NH, 16, 10, 1>, &cfg) != cudaSuccess || room < 1) {
      cudaGetLastError();
      room = 1;
    }
    r.store(room, std::memory_order_relaxed);
  }
  return clusters > room ? 2 : 1;
}

template <int NH, int NC, int CT, int K>
cudaError_t launch_head_tc_k(const CUtensorMap& mH, const CUtensorMap& mW2, const CUtensorMap& mGT,
                             const HeadArgs& a, int n_active, cudaStream_t s) {
  using Cfg = HTCfg<NH, NC>;
  cudaError_t e = allow_smem(head_tc_kernel<NH, NC, CT, K>, Cfg::kSmem);
  if (e != cudaSuccess) return e;
  cudaLaunchAttribute attr[2];
  const cudaLaunchConfig_t cfg = head_config<NH, NC, CT, K>(attr, n_active, a.H / Cfg::F, a.pdl, s);
  return cudaLaunchKernelEx(&cfg, head_tc_kernel<NH, NC, CT, K>, mH, mW2, mGT, a);
}

template <int NH>
cudaError_t launch_head_tc_c(const CUtensorMap& mH, const CUtensorMap& mW2, const CUtensorMap& mGT,
                             const HeadArgs& a, int n_active, cudaStream_t s) {
  if (a.C > 16) return launch_head_tc_k<NH, 32, 0, 1>(mH, mW2, mGT, a, n_active, s);
  const int k = head_per_sm<NH>(a.H / (kHT * NH), n_active);
  if (a.C == 10) return k == 2 ? launch_head_tc_k<NH, 16, 10, 2>(mH, mW2, mGT, a, n_active, s)
                               : launch_head_tc_k<NH, 16, 10, 1>(mH, mW2, mGT, a, n_active, s);
  return k == 2 ? launch_head_tc_k<NH, 16, 0, 2>(mH, mW2, mGT, a, n_active, s)
                : launch_head_tc_k<NH, 16, 0, 1>(mH, mW2, mGT, a, n_active, s);
}
}  // namespace

cudaError_t launch_head_tc(const CUtensorMap& mH, const CUtensorMap& mW2, const CUtensorMap& mGT,
                           const HeadArgs& a, int n_active, cudaStream_t s) {
  if (!head_tc_supported(a.H, a.B, a.C) || (!a.G && a.B % 64 != 0)) return cudaErrorInvalidValue;
  return head_tc_halves(a.H) == 2 ? launch_head_tc_c<2>(mH, mW2, mGT, a, n_active, s)
                                  : launch_head_tc_c<1>(mH, mW2, mGT, a, n_active, s);
}

}  // namespace oscars
