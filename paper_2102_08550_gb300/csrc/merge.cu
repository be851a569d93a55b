// Server merge and global update (Eq. 4, first branch; the parameter-server
// push / combine / pull of the Introduction), delta form:
//
//   x_g[p] <- x_g[p] + eta_s * sum_k w_k * delta_k[p],
//   delta_k = pushed delta, or x^k[p] - x_g[p] for pushed replicas.
//
// HBM-bound streaming kernel: every byte of the W pushed buffers is read
// once with 16-byte streaming loads (ld.global.cs: evict-first, they are
// never reused), the sum is kept in fp32 registers in worker order
// k = 0..W-1, and x_g is read and written once.  Algorithmic traffic:
// (W + 2) * P * 4 bytes.  The pointer table and weights travel in a
// __grid_constant__ parameter block, so each thread only loads data.
//
// In MLP mode the same pass also writes the bf16 operand copy of x_g.
//
// Grid: persistent, (SM count) x 3 blocks of 224 threads striding over
// 16-byte chunks; each thread keeps 16 independent 16-byte loads in flight
// per group of 16 workers (the rest in groups of 8, 4, 2 and 1), still
// summing in worker order.
//
// Segments: the vector of a call may come in up to kMaxMergeSegs pieces that
// lie at different offsets in x_g and in the pushed buffers (the tensors of a
// padded slot against a canonical delta); all run in one launch, each on its
// own range of blocks.  16 deltas of the 784-512-10 model (four tensors):
// four vector launches, a scalar one for a tail and a bf16 refresh of the
// whole slot took 42 us with the pull and their gaps, one
// launch (and a one-launch pull) 12 us.
//
// Alignment: the 16-byte path needs every buffer at the same offset modulo
// 16 bytes.  When they share one offset that is not 0, the first (up to 3)
// elements of a segment are peeled off; those and the tail are single
// elements that threads of the same launch take after their chunks.  Only
// buffers with different offsets take single elements throughout.
#include <atomic>

#include "common.cuh"
#include "internal.h"

namespace oscars {

namespace {

// 7 warps and 3 resident blocks per SM: the launch bounds cap a thread at 96
// registers, enough for 16 float4 loads in flight (without the cap the
// compiler picks 32 registers for full occupancy and the loads of a thread
// run one after the other); 672 threads per SM cover the 407 K-parameter
// model of the 784-512-10 MLP in one wave
constexpr int kThreads = 224;
constexpr int kMinBlocks = 3;
constexpr int kGroup = 16;   // replica loads in flight per thread before the first is used

__device__ __forceinline__ float4 ld_stream4(const float4* p) { return __ldcs(p); }

// Workers [k, k + G) of the 16-byte chunk at element p added to acc in worker order: all G
// loads are issued before the first is used, so a thread keeps G of them in
// flight (the kernel's launch bounds leave it the registers for 16).
template <int G, bool kReplica>
__device__ __forceinline__ void merge_group(const MergeArgs& a, int k, int64_t p, const float4& x, float4& acc) {
  float4 v[G];
#pragma unroll
  for (int j = 0; j < G; ++j) v[j] = ld_stream4(reinterpret_cast<const float4*>(a.src[k + j] + p));
#pragma unroll
  for (int j = 0; j < G; ++j) {
    const float w = a.w[k + j];
    if (kReplica) {
      acc.x = fmaf(w, v[j].x - x.x, acc.x);
      acc.y = fmaf(w, v[j].y - x.y, acc.y);
      acc.z = fmaf(w, v[j].z - x.z, acc.z);
      acc.w = fmaf(w, v[j].w - x.w, acc.w);
    } else {
      acc.x = fmaf(w, v[j].x, acc.x);
      acc.y = fmaf(w, v[j].y, acc.y);
      acc.z = fmaf(w, v[j].z, acc.z);
      acc.w = fmaf(w, v[j].w, acc.w);
    }
  }
}

// The same for single element p.
template <int G, bool kReplica>
__device__ __forceinline__ void merge_group1(const MergeArgs& a, int k, int64_t p, float x, float& acc) {
  float v[G];
#pragma unroll
  for (int j = 0; j < G; ++j) v[j] = __ldcs(a.src[k + j] + p);
#pragma unroll
  for (int j = 0; j < G; ++j) acc = fmaf(a.w[k + j], kReplica ? v[j] - x : v[j], acc);
}

struct MergeSegs {
  MergeSeg s[kMaxMergeSegs];
  int first_block[kMaxMergeSegs + 1];   // segment i runs on blocks [first_block[i], first_block[i + 1])
  int n;
};

template <bool kReplica>
__global__ void __launch_bounds__(kThreads, kMinBlocks) merge_vec4_kernel(const __grid_constant__ MergeArgs a,
                                                                     const __grid_constant__ MergeSegs segs,
                                                                     float* __restrict__ x_g, float eta,
                                                                     __nv_bfloat16* __restrict__ shadow) {
  int si = 0;
  while (si + 1 < segs.n && static_cast<int>(blockIdx.x) >= segs.first_block[si + 1]) ++si;
  const MergeSeg& sg = segs.s[si];
  const int64_t stride = static_cast<int64_t>(segs.first_block[si + 1] - segs.first_block[si]) * kThreads;
  const int64_t t0 = static_cast<int64_t>(blockIdx.x - segs.first_block[si]) * kThreads + threadIdx.x;
  // 16-byte chunks: [head, head + 4 n4) of the segment
  const int64_t so = sg.src + sg.head, go = sg.dst + sg.head;
  float4* xg4 = reinterpret_cast<float4*>(x_g + go);
  for (int64_t i = t0; i < sg.n4; i += stride) {
    const float4 x = __ldcs(xg4 + i);
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
    int k = 0;
    for (; k + kGroup <= a.W; k += kGroup) merge_group<kGroup, kReplica>(a, k, so + 4 * i, x, acc);
    // the rest in groups of 8, 4, 2 and 1, still in worker order
    if (k + 8 <= a.W) {
      merge_group<8, kReplica>(a, k, so + 4 * i, x, acc);
      k += 8;
    }
    if (k + 4 <= a.W) {
      merge_group<4, kReplica>(a, k, so + 4 * i, x, acc);
      k += 4;
    }
    if (k + 2 <= a.W) {
      merge_group<2, kReplica>(a, k, so + 4 * i, x, acc);
      k += 2;
    }
    if (k < a.W) merge_group<1, kReplica>(a, k, so + 4 * i, x, acc);
    float4 out;
    out.x = fmaf(eta, acc.x, x.x);
    out.y = fmaf(eta, acc.y, x.y);
    out.z = fmaf(eta, acc.z, x.z);
    out.w = fmaf(eta, acc.w, x.w);
    __stcs(xg4 + i, out);
    if (shadow)   // the bf16 operand copy of the new global model, same pass
      reinterpret_cast<uint2*>(shadow + go)[i] = make_uint2(pack_bf16x2(out.x, out.y), pack_bf16x2(out.z, out.w));
  }
  // single elements: [0, head) and [head + 4 n4, n), from the segment's last
  // threads (the ones with the fewest chunks)
  const int64_t tail = sg.head + 4 * sg.n4, count = sg.head + (sg.n - tail);
  for (int64_t q = stride - 1 - t0; q < count; q += stride) {
    const int64_t p = q < sg.head ? q : tail + (q - sg.head);
    const float x = x_g[sg.dst + p];
    float acc = 0.f;
    int k = 0;
    for (; k + 8 <= a.W; k += 8) merge_group1<8, kReplica>(a, k, sg.src + p, x, acc);
    for (; k < a.W; ++k) merge_group1<1, kReplica>(a, k, sg.src + p, x, acc);
    const float out = fmaf(eta, acc, x);
    x_g[sg.dst + p] = out;
    if (shadow) shadow[sg.dst + p] = __float2bfloat16_rn(out);
  }
}

constexpr int kMaxDevices = 64;
std::atomic<int> g_sm_count[kMaxDevices];

// SM count of the current device (queried once per device)
int sm_count() {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0) return 1;
  if (dev >= kMaxDevices) {
    int n = 0;
    return cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess && n > 0 ? n : 1;
  }
  int n = g_sm_count[dev].load(std::memory_order_relaxed);
  if (n == 0) {
    if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n <= 0) n = 1;
    g_sm_count[dev].store(n, std::memory_order_relaxed);
  }
  return n;
}

}  // namespace

cudaError_t launch_merge_segs(const MergeArgs& a, const MergeSeg* seg, int nseg, float* x_g, float eta, bool replica,
                              cudaStream_t s, __nv_bfloat16* shadow) {
  if (nseg < 0 || nseg > kMaxMergeSegs) return cudaErrorInvalidValue;
  MergeSegs m;
  m.n = 0;
  m.first_block[0] = 0;
  // every pushed buffer at the same offset modulo 16 bytes?
  const uintptr_t b0 = a.W > 0 ? reinterpret_cast<uintptr_t>(a.src[0]) & 15 : 0;
  bool same = true;
  for (int k = 1; k < a.W && same; ++k) same = (reinterpret_cast<uintptr_t>(a.src[k]) & 15) == b0;
  const int64_t most = static_cast<int64_t>(sm_count()) * kMinBlocks;
  for (int i = 0; i < nseg; ++i) {
    MergeSeg g = seg[i];
    if (g.n <= 0) continue;
    // elements before the first 16-byte boundary of x_g; 16-byte chunks run
    // from there when the pushed buffers have the same offset (and the bf16
    // copy, two bytes per element, is then 8-byte aligned)
    const uintptr_t off = reinterpret_cast<uintptr_t>(x_g + g.dst) & 15;
    const uintptr_t soff = (b0 + static_cast<uintptr_t>(g.src) * 4) & 15;
    g.head = 0;
    g.n4 = 0;
    if (same && (off & 3) == 0 && soff == off) {
      const int head = static_cast<int>((16 - off) & 15) / 4;
      if (head < g.n && (!shadow || (reinterpret_cast<uintptr_t>(shadow + g.dst + head) & 7) == 0)) {
        g.head = head;
        g.n4 = (g.n - head) / 4;
        if (g.n4 == 0) g.head = 0;
      }
    }
    const int64_t singles = g.n - 4 * g.n4, work = g.n4 > singles ? g.n4 : singles;
    int64_t blocks = (work + kThreads - 1) / kThreads;
    if (blocks > most) blocks = most;
    m.s[m.n] = g;
    m.first_block[m.n + 1] = m.first_block[m.n] + static_cast<int>(blocks);
    ++m.n;
  }
  if (m.n == 0) return cudaSuccess;
  const unsigned nb = static_cast<unsigned>(m.first_block[m.n]);
  if (replica) merge_vec4_kernel<true><<<nb, kThreads, 0, s>>>(a, m, x_g, eta, shadow);
  else merge_vec4_kernel<false><<<nb, kThreads, 0, s>>>(a, m, x_g, eta, shadow);
  return cudaGetLastError();
}

cudaError_t launch_merge(const MergeArgs& a, float* x_g, int64_t P, float eta, bool replica, cudaStream_t s,
                         __nv_bfloat16* shadow) {
  const MergeSeg g{0, 0, P, 0, 0};
  return launch_merge_segs(a, &g, 1, x_g, eta, replica, s, shadow);
}

}  // namespace oscars
