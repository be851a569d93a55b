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
// buffers with different offsets take single elements throughout, four a thread
// at a time: one at a time, 5 M elements of 1 and 3 workers took 23 and 45 us (19
// and 43 on a kernel of their own before), 12.5 and 20.8 now; of 16 workers 57
// (206), 52 now.
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

// The same for E single elements p.
template <int G, int E, bool kReplica>
__device__ __forceinline__ void merge_singles(const MergeArgs& a, int k, int64_t at, const int64_t (&p)[E],
                                              const float (&x)[E], float (&acc)[E]) {
  float v[G][E];
#pragma unroll
  for (int g = 0; g < G; ++g)
#pragma unroll
    for (int j = 0; j < E; ++j) v[g][j] = __ldcs(a.src[k + g] + at + p[j]);
#pragma unroll
  for (int g = 0; g < G; ++g)
#pragma unroll
    for (int j = 0; j < E; ++j) acc[j] = fmaf(a.w[k + g], kReplica ? v[g][j] - x[j] : v[g][j], acc[j]);
}

// E single elements q, q + stride, ... of a segment, G E loads in flight
template <int G, int E, bool kReplica>
__device__ __forceinline__ void merge_at(const MergeArgs& a, const MergeSeg& sg, float* __restrict__ x_g, float eta,
                                         __nv_bfloat16* __restrict__ shadow, int64_t q, int64_t stride) {
  int64_t p[E];
  float x[E], acc[E];
#pragma unroll
  for (int j = 0; j < E; ++j) {
    const int64_t at = q + j * stride;
    p[j] = at < sg.head ? at : at + 4 * sg.n4;
    x[j] = x_g[sg.dst + p[j]];
    acc[j] = 0.f;
  }
  int k = 0;
  for (; k + G <= a.W; k += G) merge_singles<G, E, kReplica>(a, k, sg.src, p, x, acc);
  for (; k < a.W; ++k) merge_singles<1, E, kReplica>(a, k, sg.src, p, x, acc);
#pragma unroll
  for (int j = 0; j < E; ++j) {
    const float out = fmaf(eta, acc[j], x[j]);
    x_g[sg.dst + p[j]] = out;
    if (shadow) shadow[sg.dst + p[j]] = __float2bfloat16_rn(out);
  }
}

// Up to N segments: 1, 8 or kMaxMergeSegs.  The pointer and weight tables are 3 KB;
// with a table of 32 segments beside them, and the code for single elements in a
// kernel that has none, a launch took 0.3 us longer (device time of 1000
// elements, 16 workers, us: 1.8, 2.1 with both, 1.9 now; 400 000: 2.9, 3.2, 2.9).
template <int N>
struct MergeSegs {
  MergeSeg s[N];
  int first_block[N + 1];   // segment i runs on blocks [first_block[i], first_block[i + 1])
  int n;
};

// kSingle: some segment has single elements (any may, with N > 1)
template <bool kReplica, int N, bool kSingle>
__global__ void __launch_bounds__(kThreads, kMinBlocks) merge_vec4_kernel(const __grid_constant__ MergeArgs a,
                                                                     const __grid_constant__ MergeSegs<N> segs,
                                                                     float* __restrict__ x_g, float eta,
                                                                     __nv_bfloat16* __restrict__ shadow) {
  int si = 0;
  while (N > 1 && si + 1 < segs.n && static_cast<int>(blockIdx.x) >= segs.first_block[si + 1]) ++si;
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
  if (!kSingle) return;
  // single elements: [0, head) and [head + 4 n4, n), from the segment's last
  // threads (the ones with the fewest chunks); four a thread at a time where
  // there are that many (buffers with different offsets)
  const int64_t count = sg.n - 4 * sg.n4;
  int64_t q = stride - 1 - t0;
  for (; q + 3 * stride < count; q += 4 * stride) merge_at<4, 4, kReplica>(a, sg, x_g, eta, shadow, q, stride);
  for (; q < count; q += stride) merge_at<8, 1, kReplica>(a, sg, x_g, eta, shadow, q, stride);
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

namespace {
template <int N>
cudaError_t launch_merge_n(const MergeArgs& a, const MergeSeg* seg, int nseg, float* x_g, float eta, bool replica,
                           cudaStream_t s, __nv_bfloat16* shadow) {
  MergeSegs<N> m;
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
  if constexpr (N == 1) {
    // no single elements, and less than a full grid: without their code (see
    // above; a full grid is bound by memory, and 25.6 M elements of 64 workers
    // took 955 us without that code, 943 with it)
    if (m.s[0].head == 0 && m.s[0].n == 4 * m.s[0].n4 && nb < static_cast<unsigned>(most)) {
      if (replica) merge_vec4_kernel<true, 1, false><<<nb, kThreads, 0, s>>>(a, m, x_g, eta, shadow);
      else merge_vec4_kernel<false, 1, false><<<nb, kThreads, 0, s>>>(a, m, x_g, eta, shadow);
      return cudaGetLastError();
    }
  }
  if (replica) merge_vec4_kernel<true, N, true><<<nb, kThreads, 0, s>>>(a, m, x_g, eta, shadow);
  else merge_vec4_kernel<false, N, true><<<nb, kThreads, 0, s>>>(a, m, x_g, eta, shadow);
  return cudaGetLastError();
}
}  // namespace

cudaError_t launch_merge_segs(const MergeArgs& a, const MergeSeg* seg, int nseg, float* x_g, float eta, bool replica,
                              cudaStream_t s, __nv_bfloat16* shadow) {
  if (nseg < 0 || nseg > kMaxMergeSegs) return cudaErrorInvalidValue;
  return nseg <= 1   ? launch_merge_n<1>(a, seg, nseg, x_g, eta, replica, s, shadow)
         : nseg <= 8 ? launch_merge_n<8>(a, seg, nseg, x_g, eta, replica, s, shadow)
                     : launch_merge_n<kMaxMergeSegs>(a, seg, nseg, x_g, eta, replica, s, shadow);
}

cudaError_t launch_merge(const MergeArgs& a, float* x_g, int64_t P, float eta, bool replica, cudaStream_t s,
                         __nv_bfloat16* shadow) {
  const MergeSeg g{0, 0, P, 0, 0};
  return launch_merge_segs(a, &g, 1, x_g, eta, replica, s, shadow);
}

}  // namespace oscars
