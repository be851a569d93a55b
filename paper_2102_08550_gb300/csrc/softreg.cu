// Local steps of softmax regression in fp32 (one linear layer + softmax
// cross-entropy): Eq. 4, "otherwise" branch, x <- x - lr * g(x) with g the
// mean mini-batch gradient.
//
// Each worker's whole round runs in one launch: the worker pulls the global
// model into shared memory (the pull of the parameter-server description,
// fused: nothing is copied through HBM), runs tau_i SGD steps on successive
// mini-batches of its shard with the weights resident in shared memory, and
// writes the result to the worker's replica (the push).  Workers never
// exchange data inside a round.  Two kernels: softreg_cluster_round_kernel
// puts each worker on a cluster of 8 CTAs that split the input columns;
// softreg_round_kernel puts each worker on one CTA (only where the cluster's
// exchange buffers do not fit: from about 390 rows with 17 classes and more, 470
// with 15; 241 us a step of 100 x 20 with 400 rows).
//
// Per step: logits z[b][c] = sum_k x[b][k] W[c][k] + bias[c] (warp-level dot
// products), p = softmax(z), loss_b = logsumexp(z_b) - z_b[y_b],
// dz = (p - onehot(y)) / B, dW[c][k] = sum_b dz[b][c] x[b][k],
// db[c] = sum_b dz[b][c], W <- W - lr dW (fmaf), all fp32.
#include <atomic>

#include "common.cuh"
#include "internal.h"

namespace oscars {

namespace {

constexpr int kThreads = 512;
constexpr int kWarps = kThreads / 32;
static_assert(kSoftregMaxBatch <= kThreads, "one thread per mini-batch row");

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// float4 items of one mini-batch a thread holds in registers while the
// previous step computes (the next step's rows are loaded ahead)
constexpr int kPrefetch = 16;

// Round bookkeeping of worker w at the end of its round: the mean loss over
// its tau steps (the step partials summed in step order in double, divided
// by B tau) and the data cursor advanced by tau mini-batches.
__device__ __forceinline__ void finish_worker(const SoftregArgs& a, int w, int tau, int64_t cur, int64_t n) {
  if (a.loss_out) {
    double sum = 0.0;
    for (int st = 0; st < tau; ++st) sum += a.loss_part[static_cast<int64_t>(w) * a.max_tau + st];
    a.loss_out[w] = static_cast<float>(sum / (static_cast<double>(a.B) * tau));
  }
  if (a.cursor_next) a.cursor_next[w] = (cur + static_cast<int64_t>(tau) * a.B) % n;
}

__global__ void __launch_bounds__(kThreads) softreg_round_kernel(const __grid_constant__ SoftregArgs a) {
  extern __shared__ __align__(16) float sm[];
  const int D = a.D, C = a.C, B = a.B;
  float* Wsm = sm;                 // [C][D]
  float* bsm = Wsm + C * D;        // [C] (padded to 32)
  float* Xsm = bsm + 32;           // [B][D]
  float* Zsm = Xsm + B * D;        // [B][C] logits, then dz
  float* Lsm = Zsm + B * C;        // [B] per-sample loss
  int* Ysm = reinterpret_cast<int*>(Lsm + B);  // [B]
  int64_t* Rsm = reinterpret_cast<int64_t*>((reinterpret_cast<uintptr_t>(Ysm + B) + 7) & ~uintptr_t(7));   // [B] row offsets

  const int w = blockIdx.x;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int tau = a.tau[w];
  const float* gsrc = a.master + static_cast<int64_t>(a.global_slot) * a.slot_stride;
  float* dst = a.master_out + static_cast<int64_t>(w) * a.slot_stride;

  // pull: global model -> shared memory
  for (int i = tid; i < C * D; i += kThreads) Wsm[i] = gsrc[a.offW + i];
  for (int i = tid; i < C; i += kThreads) bsm[i] = gsrc[a.offB + i];

  const float* X = a.shard_x[w];
  const int32_t* Y = a.shard_y[w];
  const int64_t n = a.shard_n[w];
  const int64_t cur = a.cursor[w];
  const float invB = 1.0f / static_cast<float>(B);
  // with D % 4 == 0, a 16-byte aligned shard and a mini-batch of at most
  // kPrefetch float4 per thread, step s + 1's rows are loaded into registers
  // while step s computes (otherwise rows are read one float at a time)
  const int D4 = D / 4;
  const bool vec = (D & 3) == 0 && (reinterpret_cast<uintptr_t>(X) & 15) == 0 && B * D4 <= kPrefetch * kThreads;
  float4 pf[kPrefetch];
  auto fetch = [&](int s) {   // rows of step s into registers (row offsets already in Rsm)
#pragma unroll
    for (int j = 0; j < kPrefetch; ++j) {
      const int i = tid + j * kThreads;
      if (i < B * D4) {
        const int b = i / D4, k4 = i - b * D4;
        pf[j] = *reinterpret_cast<const float4*>(X + Rsm[b] + 4 * k4);
      }
    }
  };
  auto row_offsets = [&](int s) {
    if (tid < B) {
      const int64_t r = (cur + static_cast<int64_t>(s) * B + tid) % n;
      Rsm[tid] = r * D;
      Ysm[tid] = Y[r];
    }
  };
  if (vec && tau > 0) {
    row_offsets(0);
    __syncthreads();
    fetch(0);
  }

  for (int s = 0; s < tau; ++s) {
    __syncthreads();   // the previous step is done with Xsm and Zsm
    int yl = 0;        // the label of row tid (tid < B) of this step
    if (vec) {
      // this step's rows, fetched during the previous step; then the next
      // step's row offsets and labels (thread tid rewrites only entry tid,
      // which it alone has read) and its rows, in flight during this step
      if (tid < B) yl = Ysm[tid];
#pragma unroll
      for (int j = 0; j < kPrefetch; ++j) {
        const int i = tid + j * kThreads;
        if (i < B * D4) reinterpret_cast<float4*>(Xsm)[i] = pf[j];
      }
      if (s + 1 < tau) row_offsets(s + 1);
      __syncthreads();
      if (s + 1 < tau) fetch(s + 1);
    } else {
      // mini-batch rows (cursor + s*B + b) mod n
      row_offsets(s);
      __syncthreads();
      for (int i = tid; i < B * D; i += kThreads) {
        const int b = i / D, k = i - b * D;
        Xsm[i] = X[Rsm[b] + k];
      }
      if (tid < B) yl = Ysm[tid];
      __syncthreads();
    }
    // logits: one warp per (b, c) dot product
    for (int q = warp; q < B * C; q += kWarps) {
      const int b = q / C, c = q - b * C;
      const float* xr = Xsm + b * D;
      const float* wr = Wsm + c * D;
      float acc = 0.f;
      if ((D & 3) == 0) {
        for (int k4 = lane; k4 < D4; k4 += 32) {
          const float4 xv = reinterpret_cast<const float4*>(xr)[k4];
          const float4 wv = reinterpret_cast<const float4*>(wr)[k4];
          acc = fmaf(xv.x, wv.x, acc);
          acc = fmaf(xv.y, wv.y, acc);
          acc = fmaf(xv.z, wv.z, acc);
          acc = fmaf(xv.w, wv.w, acc);
        }
      } else {
        for (int k = lane; k < D; k += 32) acc = fmaf(xr[k], wr[k], acc);
      }
      acc = warp_sum(acc);
      if (lane == 0) Zsm[q] = acc + bsm[c];
    }
    __syncthreads();
    // softmax cross-entropy, one thread per row
    if (tid < B) {
      const int b = tid;
      float* z = Zsm + b * C;
      float m = z[0];
      for (int c = 1; c < C; ++c) m = fmaxf(m, z[c]);
      // p_c = e_c / s; 1 - p_y = (sum_{c != y} e_c) / s (no cancellation)
      const int y = yl;
      float se = 0.f, so = 0.f;
      for (int c = 0; c < C; ++c) {
        const float e = expf(z[c] - m);
        se += e;
        if (c != y) so += e;
      }
      Lsm[b] = m + logf(se) - z[y];
      for (int c = 0; c < C; ++c) z[c] = (c == y ? -(so / se) : expf(z[c] - m) / se) * invB;
    }
    __syncthreads();
    if (tid == 0) {
      float l = 0.f;
      for (int b = 0; b < B; ++b) l += Lsm[b];
      a.loss_part[static_cast<int64_t>(w) * a.max_tau + s] = l;
    }
    // weight gradient and update: item = (class, 4 input features) (or one
    // feature when D % 4 != 0)
    if ((D & 3) == 0) {
      for (int q = tid; q < C * D4; q += kThreads) {
        const int c = q / D4, k4 = q - c * D4;
        float4 g = make_float4(0.f, 0.f, 0.f, 0.f);
        for (int b = 0; b < B; ++b) {
          const float d = Zsm[b * C + c];
          const float4 xv = reinterpret_cast<const float4*>(Xsm + b * D)[k4];
          g.x = fmaf(d, xv.x, g.x);
          g.y = fmaf(d, xv.y, g.y);
          g.z = fmaf(d, xv.z, g.z);
          g.w = fmaf(d, xv.w, g.w);
        }
        float4* wp = reinterpret_cast<float4*>(Wsm + c * D) + k4;
        float4 wv = *wp;
        wv.x = fmaf(-a.lr, g.x, wv.x);
        wv.y = fmaf(-a.lr, g.y, wv.y);
        wv.z = fmaf(-a.lr, g.z, wv.z);
        wv.w = fmaf(-a.lr, g.w, wv.w);
        *wp = wv;
      }
    } else {
      for (int k = tid; k < D; k += kThreads) {
        for (int c = 0; c < C; ++c) {
          float g = 0.f;
          for (int b = 0; b < B; ++b) g = fmaf(Zsm[b * C + c], Xsm[b * D + k], g);
          Wsm[c * D + k] = fmaf(-a.lr, g, Wsm[c * D + k]);
        }
      }
    }
    for (int c = tid; c < C; c += kThreads) {
      float g = 0.f;
      for (int b = 0; b < B; ++b) g += Zsm[b * C + c];
      bsm[c] = fmaf(-a.lr, g, bsm[c]);
    }
  }
  __syncthreads();
  // push: replica <- shared memory
  for (int i = tid; i < C * D; i += kThreads) dst[a.offW + i] = Wsm[i];
  for (int i = tid; i < C; i += kThreads) dst[a.offB + i] = bsm[i];
  if (tid == 0) finish_worker(a, w, tau, cur, n);   // the thread that wrote the loss partials
}

// The same round with each worker on a cluster of kCl CTAs that split the
// input columns: CTA r owns columns [r * Dc, (r + 1) * Dc) (Dc a multiple of
// 4) of W and of every mini-batch row, and the rows b = r (mod kCl) of the
// mini-batch for the softmax.  The bias is column D of W against an input of
// 1, so it needs no code of its own.
//
// A step is a serial chain, so it is built from short parallel phases and
// one-way exchanges (no cluster barrier, no remote read):
//  1. partial logits of the whole mini-batch over the CTA's columns: a warp
//     takes 32 rows x CC classes, a lane 4 rows and every fourth 4-column
//     chunk (4 rows x CC classes in registers); the four lanes of a row
//     reduce-scatter with shuffles, so a lane ends up with one row; with few
//     rows and classes the columns are also split over the warps (KS) and
//     summed in shared memory;
//  2. the partials of a row go to the CTA that owns it with asynchronous
//     16-byte stores (st.async) that complete on the owner's mbarrier; the
//     owner adds the kCl partials in a fixed order and one warp per row (lane =
//     class) computes the softmax cross-entropy;
//  3. the row of dz goes to every CTA the same way;
//  4. weight update of the CTA's columns: a thread sums CC classes x 4
//     columns over a part (1 / BS) of the rows; the parts meet in shared
//     memory.
// Four more warps fetch: the rows of step s + 1 come by cp.async into the
// other of two buffers (and the labels of the CTA's rows beside them) while
// step s runs; they meet the others once a step.
//
// Classes are kept in rows of "slots": groups of CC classes,
// each padded to CCp = a multiple of 4 slots (at most 32 slots in all).
// Every index a thread needs in a step is worked out before the first one or
// by shifts: an integer division by a run-time value costs as much as a
// whole phase of the smaller shapes.  The products are bound by the values
// that shared memory returns (32 a clock, broadcast or not; 128 FMAs a
// clock), hence the register tiles: 4 x CC in phase 1, CC x 4 in phase 4.
//
// Buffer reuse: a CTA sends the partials of step s + 1 only after it has
// received all of dz(s), which an owner sends after it has read its partials
// of step s: so partials(s + 1) never overwrite partials(s) in use.  An owner
// sends dz(s + 1) only after it has received every CTA's partials(s + 1),
// which a CTA sends after its last read of dz(s).
//
// What bounds it: the latency of the chain (784 x 10, 4 workers: issue slots 30%
// busy, 0.3% of DRAM).  Eight steps of one 784 x 10 worker, batch 32: 203 us on one CTA,
// 35 us here (about 3.3 us a step).  A round of 333 x 26, batch 100, 12
// workers, with its merge and pull: 373 us with the earlier cluster kernel
// (cluster barrier, remote reads, one-thread row loops), 128 us now.
// 784 x 10, 4 workers, at most 4 steps: 49 and 35 us.
constexpr int kCl = 8;
// A CTA has NT computing threads and NT / 4 fetching ones, and K CTAs share an
// SM (launch bounds): 512 threads and one (96 registers a thread), 256 and two,
// 128 and four; 128 and two (up to 177 registers) for steps of few products,
// which leave most of 512 threads without work.  More workers than clusters
// that run at once take several waves: see cluster_variant.
constexpr int kClThreads = 512;
constexpr int kClSmallWork = 4096;   // products of a step in a CTA, at most, for 128 threads whatever the workers
constexpr int kClMaxWarps = kClThreads / 32;
// columns per CTA: (D + the bias column) / kCl rounded up to a multiple of 4
__host__ __device__ inline int cluster_cols(int D) { return ((D + 1 + kCl - 1) / kCl + 3) / 4 * 4; }
constexpr int kSlots = 32;   // class slots of a row at most (one lane each)

// The shape-dependent split of a step (host: shared memory; device: offsets).
struct ClPlan {
  int Dc, Xld;     // columns per CTA, row stride of the mini-batch tile
  int ncg, Zp;     // class groups, slots per row
  int KS, BS;      // column splits (logits), row splits (update)
  int R;           // mini-batch rows a CTA owns
  // offsets in floats from the start of shared memory
  int oX, oRed, oPin, oZ, oZst, oEnd;
};
// classes per group: the least padding of C with at most kSlots slots, then
// the larger group (more products per value read)
__host__ __device__ inline int cluster_cc(int C) {
  const int cand[4] = {8, 7, 5, 4};
  int best = 0, waste = 1 << 20;
  for (int i = 0; i < 4; ++i) {
    const int cc = cand[i], g = (C + cc - 1) / cc;
    if (g * ((cc + 3) / 4 * 4) > kSlots) continue;
    if (g * cc - C < waste) {
      waste = g * cc - C;
      best = cc;
    }
  }
  return best;
}
__host__ __device__ inline ClPlan cluster_plan(int D, int C, int B, int CC, int NT) {
  ClPlan p;
  p.Dc = cluster_cols(D);
  p.Xld = (p.Dc / 4) % 2 ? p.Dc : p.Dc + 4;   // an odd number of 16-byte chunks: lanes = rows hit distinct banks
  p.ncg = (C + CC - 1) / CC;
  p.Zp = p.ncg * ((CC + 3) / 4 * 4);
  const int nrb = (B + 31) / 32, nk4 = p.Dc / 4;
  p.KS = NT / 32 / (nrb * p.ncg);
  p.KS = p.KS > 4 ? 4 : p.KS;                          // more splits cost more to sum than they save
  p.KS = p.KS > (nk4 + 3) / 4 ? (nk4 + 3) / 4 : p.KS;  // a warp's lanes take 4 chunks at a time
  p.KS = p.KS < 1 ? 1 : p.KS;
  p.BS = NT / (nk4 * p.ncg);
  p.BS = p.BS > 8 ? 8 : p.BS;
  p.BS = p.BS > B / 8 ? B / 8 : p.BS;                  // at least 8 rows a split: the parts are summed too
  p.BS = p.BS < 1 ? 1 : p.BS;
  p.R = (B + kCl - 1) / kCl;
  const int red1 = p.KS * B * (p.Zp + 4), red2 = p.BS > 1 ? p.BS * p.ncg * CC * p.Dc : 0;
  p.oX = p.ncg * CC * p.Dc;
  p.oRed = p.oX + 2 * B * p.Xld;
  p.oPin = p.oRed + (red1 > red2 ? red1 : red2);
  p.oZ = p.oPin + kCl * p.R * p.Zp;
  p.oZst = p.oZ + B * p.Zp;
  p.oEnd = p.oZst + NT / 32 * kSlots;
  return p;
}
// after the float area (16-byte aligned): loss sums, row offsets, barriers, labels
__host__ __device__ inline size_t cluster_tail_bytes(int B) {
  return sizeof(double) * (kClMaxWarps + kCl) + sizeof(int64_t) * B + 2 * sizeof(uint64_t) +
         sizeof(int) * 2 * ((B + kCl - 1) / kCl);
}

__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async4(void* dst, const void* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

__device__ __forceinline__ float warp_max(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}
__device__ __forceinline__ void fma4(float4& acc, float s, const float4& v) {
  acc.x = fmaf(s, v.x, acc.x);
  acc.y = fmaf(s, v.y, acc.y);
  acc.z = fmaf(s, v.z, acc.z);
  acc.w = fmaf(s, v.w, acc.w);
}
__device__ __forceinline__ void add4(float4& a, const float4& v) {
  a.x += v.x;
  a.y += v.y;
  a.z += v.z;
  a.w += v.w;
}
__device__ __forceinline__ void st_dsmem_f64(double* local, uint32_t rank, double v) {
  asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(cluster_addr(local, rank)), "d"(v) : "memory");
}

template <int CC, int NT, int K>
__global__ void __launch_bounds__(NT + NT / 4, K) softreg_cluster_round_kernel(const __grid_constant__ SoftregArgs a) {
  constexpr int NW = NT / 32, NF = NT / 4;   // computing warps, fetching threads
  extern __shared__ __align__(16) float sm[];
  constexpr int CCp = (CC + 3) / 4 * 4;
  const int D = a.D, C = a.C, B = a.B;
  const ClPlan p = cluster_plan(D, C, B, CC, NT);
  const int Dc = p.Dc, Xld = p.Xld, Zp = p.Zp, zq = p.Zp / 4, R = p.R, ncg = p.ncg;
  const int rank = static_cast<int>(cluster_ctarank());
  const int c0 = rank * Dc;
  const int nc = D - c0 < Dc ? (D - c0 > 0 ? D - c0 : 0) : Dc;   // this CTA's input columns (may be 0)
  const bool has_bias = D >= c0 && D < c0 + Dc;                  // column D: the bias
  const int nk4 = (nc + (has_bias ? 1 : 0) + 3) / 4;             // 4-column chunks in use
  const int R_own = (B - rank + kCl - 1) / kCl;                  // rows rank, rank + kCl, ... (rank <= B + 7)
  float* Wsm = sm;                       // [ncg * CC][Dc], classes past C and columns past the bias zero
  float* Xsm = sm + p.oX;                // [2][B][Xld]
  float* red = sm + p.oRed;              // [KS][B][Zp + 4] partial logits, or [BS][ncg * CC][Dc] gradients
  float* Pin = sm + p.oPin;              // [kCl][R][Zp] partial logits of this CTA's rows
  float* Zsm = sm + p.oZ;                // [B][Zp] dz
  float* zst = sm + p.oZst;              // [warps][kSlots] a row of dz on its way out
  double* lsum = reinterpret_cast<double*>(sm + p.oEnd);    // [warps]
  double* lrank = lsum + kClMaxWarps;                          // [kCl] (rank 0)
  int64_t* Rsm = reinterpret_cast<int64_t*>(lrank + kCl);   // [B] rows of the step being fetched
  uint64_t* pbar = reinterpret_cast<uint64_t*>(Rsm + B);    // the partials of this CTA's rows have landed
  uint64_t* zbar = pbar + 1;                                // dz has landed
  int* Ysm = reinterpret_cast<int*>(zbar + 1);              // [2][R] labels of this CTA's rows, by step parity

  const int w = blockIdx.y;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const bool table = a.tau != nullptr;   // per-worker tables, or one worker's values in the arguments
  const int tau = table ? a.tau[w] : a.tau1;
  const float* gsrc = a.master + static_cast<int64_t>(a.global_slot) * a.slot_stride;
  float* dst = a.master_out + static_cast<int64_t>(w) * a.slot_stride;
  const float* X = table ? a.shard_x[w] : a.x1;
  const int32_t* Y = table ? a.shard_y[w] : a.y1;
  const int64_t n = table ? a.shard_n[w] : a.n1;
  const int64_t cur = table ? a.cursor[w] : a.cursor1;
  const float invB = 1.0f / static_cast<float>(B);

  if (tid == 0) {
    mbar_init(pbar, 1);
    mbar_init(zbar, 1);
    fence_barrier_init();
  }
  // this CTA's columns of each row, in units of 16-byte chunks when every
  // slice is 16-byte aligned, else of single floats: a warp copies 32 / 2^ush
  // rows at a time, 2^ush (the units rounded up, at most 32) lanes a row
  const bool vec = (D & 3) == 0 && (reinterpret_cast<uintptr_t>(X) & 15) == 0;
  const int units = vec ? nc / 4 : nc;
  const int ush = units <= 1 ? 0 : 32 - __clz((units < 32 ? units : 32) - 1);
  // rows of step s: (cursor + s*B + b) mod n, kept in Rsm and advanced by the
  // fetching threads (each the rows b = its index, in steps of NF)
  const int64_t bmod = B % n;
  auto fetch = [&](int s) {   // the fetching warps: rows and labels of step s
    const int ft = tid - NT;
    for (int b = ft; b < B; b += NF) {
      int64_t r = s == 0 ? (cur + b) % n : Rsm[b] + bmod;
      if (s > 0 && r >= n) r -= n;
      Rsm[b] = r;
    }
    bar_named(2, NF);
    float* buf = Xsm + (s & 1) * B * Xld;
    const int fw = warp - NW, u0 = lane & ((1 << ush) - 1), bstep = NF >> ush;
    // four rows at a time: their offsets are read before the first copy goes out
    for (int b = (fw << (5 - ush)) + (lane >> ush); b < B; b += 4 * bstep) {
      const float* from[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) from[i] = X + Rsm[b + i * bstep < B ? b + i * bstep : b] * D + c0;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        if (b + i * bstep >= B) break;
        float* to = buf + (b + i * bstep) * Xld;
        if (vec)
          for (int u = u0; u < units; u += 1 << ush) cp_async16(to + 4 * u, from[i] + 4 * u);
        else
          for (int u = u0; u < units; u += 1 << ush) cp_async4(to + u, from[i] + u);
      }
    }
    for (int l = ft; l < R_own; l += NF) Ysm[(s & 1) * R + l] = Y[Rsm[l * kCl + rank]];
    cp_async_wait_all();
    bar_named(2, NF);   // Rsm is read by all before the next step's rows go in
  };
  const bool fetcher = tid >= NT;
  if (fetcher) {
    if (tau > 0) fetch(0);
  } else {
  // columns past nc of both buffers are never copied: the bias input, then zeros
  for (int i = tid; i < 2 * B; i += NT)
    for (int k = nc; k < 4 * nk4; ++k) Xsm[i * Xld + k] = k == nc && has_bias ? 1.f : 0.f;
  // pull: this CTA's columns of the global model and, in its CTA, the bias
  for (int c = warp; c < ncg * CC; c += NW)
    for (int k = lane; k < Dc; k += 32)
      Wsm[c * Dc + k] = c >= C ? 0.f
                        : k < nc ? gsrc[a.offW + static_cast<int64_t>(c) * D + c0 + k]
                        : k == nc && has_bias ? gsrc[a.offB + c] : 0.f;
  }
  // the class of this lane's slot, or -1
  const int cls0 = lane / CCp * CC + lane % CCp;
  const int cls = lane < Zp && lane % CCp < CC && cls0 < C ? cls0 : -1;
  // phase 1: this warp's column split and class group, its first row block and their step
  const int G = ncg * p.KS, l_ks = warp % p.KS, l_cg = warp / p.KS % ncg;
  const int l_rb = warp / G, l_rbstep = NW / G;   // warps past l_rbstep * G idle
  const int nrb = l_rb < l_rbstep ? (B + 31) / 32 : 0;
  const int l_k0 = l_ks * nk4 / p.KS + (lane >> 3), l_k1 = (l_ks + 1) * nk4 / p.KS;
  // phase 2: thread = (row tid / 8, 16-byte chunk tid % 8 of its slots), rows NT / 8 apart, so with one owner
  const int s_q = tid & 7, s_b = tid >> 3, s_owner = s_b & (kCl - 1);
  static_assert(kCl == 8 && NT / 8 % kCl == 0, "the rows of a thread have one owner");
  const uint32_t s_pin = cluster_addr(Pin + rank * R * Zp + 4 * s_q, s_owner), s_bar = cluster_addr(pbar, s_owner);
  // phase 3: lane = (destination lane % 8, chunk lane / 8)
  const int z_to = lane & 7, z_q = lane >> 3;
  const uint32_t z_dst = cluster_addr(Zsm, z_to), z_bar = cluster_addr(zbar, z_to);
  // phase 4: the first item (kv, cg, bs) of this thread, and its first sum (class, kv)
  const int nkv = Dc / 4, items = nkv * ncg * p.BS;
  const int u_kv = tid % nkv, u_cg = tid / nkv % ncg, u_bs = tid / (nkv * ncg);
  const int u_b0 = u_bs * B / p.BS, u_b1 = (u_bs + 1) * B / p.BS;
  const int r_c = tid / nkv, r_cstep = NT / nkv, r_kvstep = NT % nkv;
  // the warp's row losses over all steps as an unevaluated sum of two floats
  // (2Sum): fp64 adds are two lanes a clock here and sat in the chain
  float loss_hi = 0.f, loss_lo = 0.f;
  bool alive = true;     // no bounded wait has run out
  cluster_sync();        // barriers initialised everywhere; the global model read before anyone can end

  for (int s = 0; s < tau; ++s) {
    __syncthreads();   // X, the labels and W of this step are in place
    if (fetcher) {
      if (s + 1 < tau) fetch(s + 1);
      continue;
    }
    const float* Xs = Xsm + (s & 1) * B * Xld;
    if (tid == 0) {
      if (R_own > 0) mbar_arrive_expect_tx(pbar, static_cast<uint32_t>(kCl * R_own * Zp * 4));
      mbar_arrive_expect_tx(zbar, static_cast<uint32_t>(B * Zp * 4));
    }
    // 1. partial logits over this CTA's columns
    for (int rb = l_rb; rb < nrb; rb += l_rbstep) {
      // lane: rows rb * 32 + lane % 8 + 8 i, chunks l_k0 (= split's first + lane / 8), + 4, ...
      const float* xr[4];
      float acc[4][CC];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int row = rb * 32 + (lane & 7) + 8 * i;
        xr[i] = Xs + (row < B ? row : B - 1) * Xld;
#pragma unroll
        for (int j = 0; j < CC; ++j) acc[i][j] = 0.f;
      }
      const float* wr = Wsm + l_cg * CC * Dc;
#pragma unroll 1
      for (int k4 = l_k0; k4 < l_k1; k4 += 4) {
        float4 xv[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) xv[i] = *reinterpret_cast<const float4*>(xr[i] + 4 * k4);
#pragma unroll
        for (int j = 0; j < CC; ++j) {
          const float4 wv = *reinterpret_cast<const float4*>(wr + j * Dc + 4 * k4);
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            acc[i][j] = fmaf(xv[i].x, wv.x, acc[i][j]);
            acc[i][j] = fmaf(xv[i].y, wv.y, acc[i][j]);
            acc[i][j] = fmaf(xv[i].z, wv.z, acc[i][j]);
            acc[i][j] = fmaf(xv[i].w, wv.w, acc[i][j]);
          }
        }
      }
      // the four lanes of a row set: lane / 8 = i keeps row i
      const bool up = lane & 16, odd = lane & 8;
      float v[CCp];
#pragma unroll
      for (int j = 0; j < CC; ++j) {
        const float k0 = up ? acc[2][j] : acc[0][j], k1 = up ? acc[3][j] : acc[1][j];
        const float g0 = up ? acc[0][j] : acc[2][j], g1 = up ? acc[1][j] : acc[3][j];
        const float h0 = k0 + __shfl_xor_sync(0xffffffffu, g0, 16), h1 = k1 + __shfl_xor_sync(0xffffffffu, g1, 16);
        v[j] = (odd ? h1 : h0) + __shfl_xor_sync(0xffffffffu, odd ? h0 : h1, 8);
      }
#pragma unroll
      for (int j = CC; j < CCp; ++j) v[j] = 0.f;
      const int row = rb * 32 + lane;   // lane % 8 + 8 (lane / 8)
      if (row < B) {
        float* o = red + (l_ks * B + row) * (Zp + 4) + l_cg * CCp;
#pragma unroll
        for (int q = 0; q < CCp / 4; ++q)
          *reinterpret_cast<float4*>(o + 4 * q) = make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
      }
    }
    bar_named(1, NT);
    // 2. each row's partials to its owner
    if (s_q < zq)
      for (int b = s_b; b < B; b += NT / 8) {
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 4
        for (int ks = 0; ks < p.KS; ++ks)
          add4(v, *reinterpret_cast<const float4*>(red + (ks * B + b) * (Zp + 4) + 4 * s_q));
        st_async_v4(s_pin + static_cast<uint32_t>((b >> 3) * Zp * 4),
                    make_uint4(__float_as_uint(v.x), __float_as_uint(v.y), __float_as_uint(v.z), __float_as_uint(v.w)),
                    s_bar);
      }
    // softmax cross-entropy of this CTA's rows, one warp per row, lane = slot
    if (warp < R_own) {
      if (alive) alive = mbar_wait(pbar, s & 1, a.err, kDevTimeoutFull);
      for (int l = warp; l < R_own; l += NW) {
        float part[kCl];
#pragma unroll
        for (int q = 0; q < kCl; ++q) part[q] = lane < Zp ? Pin[(q * R + l) * Zp + lane] : 0.f;
        static_assert(kCl == 8, "the ranks' sum");
        float z = ((part[0] + part[1]) + (part[2] + part[3])) + ((part[4] + part[5]) + (part[6] + part[7]));
        z = cls >= 0 ? z : -INFINITY;
        const int y = Ysm[(s & 1) * R + l], ys = y / CC * CCp + y % CC;
        const float m = warp_max(z);
        // p_c = e_c / s; 1 - p_y = (sum_{c != y} e_c) / s (no cancellation)
        const float e = cls >= 0 ? expf(z - m) : 0.f;
        float se = e, so = lane == ys ? 0.f : e;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
          se += __shfl_xor_sync(0xffffffffu, se, o);
          so += __shfl_xor_sync(0xffffffffu, so, o);
        }
        zst[warp * kSlots + lane] = (lane == ys ? -so : e) / se * invB;
        __syncwarp();
        // 3. the row of dz to every CTA
        for (int q = z_q; q < zq; q += 4)
          st_async_v4(z_dst + static_cast<uint32_t>(((l * kCl + rank) * Zp + 4 * q) * 4),
                      *reinterpret_cast<const uint4*>(zst + warp * kSlots + 4 * q), z_bar);
        const float zy = __shfl_sync(0xffffffffu, z, ys);
        const float row = m + logf(se) - zy, t = loss_hi + row, bb = t - loss_hi;
        loss_lo += (loss_hi - (t - bb)) + (row - bb);
        loss_hi = t;
        __syncwarp();
      }
    }
    // one warp polls for dz, the others wait at a named barrier (with the
    // deeper unrolling below and the fetch's early offsets, 333 x 26, 12
    // workers, a round: 131.5 -> 127.6 us)
    if (warp == NW - 1) {
      if (alive) alive = mbar_wait(zbar, s & 1, a.err, kDevTimeoutFull);
    }
    bar_named(3, NT);
    // 4. weight gradient of this CTA's columns: item = (4 columns, CC classes, 1 / BS of the rows)
    int kv = u_kv, cg = u_cg, bs = u_bs, b0 = u_b0, b1 = u_b1;
    for (int i = tid; i < items;) {
      if (kv < nk4) {
        float4 g[CC];
#pragma unroll
        for (int j = 0; j < CC; ++j) g[j] = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 4
        for (int b = b0; b < b1; ++b) {
          const float4 xv = *reinterpret_cast<const float4*>(Xs + b * Xld + 4 * kv);
          const float* zr = Zsm + b * Zp + cg * CCp;
#pragma unroll
          for (int q = 0; q < CC / 4; ++q) {
            const float4 d = *reinterpret_cast<const float4*>(zr + 4 * q);
            fma4(g[4 * q], d.x, xv);
            fma4(g[4 * q + 1], d.y, xv);
            fma4(g[4 * q + 2], d.z, xv);
            fma4(g[4 * q + 3], d.w, xv);
          }
#pragma unroll
          for (int j = CC / 4 * 4; j < CC; ++j) fma4(g[j], zr[j], xv);
        }
#pragma unroll
        for (int j = 0; j < CC; ++j) {
          const int c = cg * CC + j;
          if (p.BS > 1) {
            *reinterpret_cast<float4*>(red + (bs * ncg * CC + c) * Dc + 4 * kv) = g[j];
          } else {
            float4* wp = reinterpret_cast<float4*>(Wsm + c * Dc + 4 * kv);
            float4 wv = *wp;
            fma4(wv, -a.lr, g[j]);
            *wp = wv;
          }
        }
      }
      i += NT;
      if (i >= items) break;   // nearly always: more items than threads need over 2000 columns
      kv = i % nkv;
      cg = i / nkv % ncg;
      bs = i / (nkv * ncg);
      b0 = bs * B / p.BS;
      b1 = (bs + 1) * B / p.BS;
    }
    if (p.BS > 1) {
      bar_named(1, NT);
      int c = r_c, kv4 = u_kv;
      while (c < C) {
        if (kv4 < nk4) {
          float4 g = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 4
          for (int q = 0; q < p.BS; ++q) add4(g, *reinterpret_cast<const float4*>(red + (q * ncg * CC + c) * Dc + 4 * kv4));
          float4* wp = reinterpret_cast<float4*>(Wsm + c * Dc + 4 * kv4);
          float4 wv = *wp;
          fma4(wv, -a.lr, g);
          *wp = wv;
        }
        c += r_cstep;
        kv4 += r_kvstep;
        if (kv4 >= nkv) {
          kv4 -= nkv;
          ++c;
        }
      }
    }
  }
  // a wait that ran out, in any lane, shows as a NaN loss (the allocation-free entry has no error word)
  alive = __all_sync(0xffffffffu, alive);
  if (!fetcher && lane == 0) {
    double sum = static_cast<double>(loss_hi);
    if (isfinite(loss_hi)) sum += static_cast<double>(loss_lo);   // an infinite row has made it inf - inf
    lsum[warp] = alive ? sum : static_cast<double>(NAN);
  }
  __syncthreads();
  // push: this CTA's columns into the replica
  for (int c = warp; c < C; c += (NT + NF) / 32)
    for (int k = lane; k < nc; k += 32) dst[a.offW + static_cast<int64_t>(c) * D + c0 + k] = Wsm[c * Dc + k];
  if (has_bias && tid < C) dst[a.offB + tid] = Wsm[tid * Dc + nc];
  if (tid == 0) {
    double t = 0.0;
    for (int i = 0; i < NW; ++i) t += lsum[i];
    st_dsmem_f64(lrank + rank, 0, t);
  }
  cluster_sync();   // the loss sums are in; every CTA has read the cursor
  if (rank == 0 && tid == 0) {
    double t = 0.0;
    for (int q = 0; q < kCl; ++q) t += lrank[q];
    a.loss_out[w] = static_cast<float>(t / (static_cast<double>(B) * tau));
    if (a.cursor_next) a.cursor_next[w] = (cur + static_cast<int64_t>(tau) * B) % n;
  }
}

// Mean cross-entropy of the global model, partial sums per block (summed
// afterwards in a fixed order).  The weights sit in shared memory; a warp
// takes 4 samples at a time, lane = every 32nd input, so that a weight read
// from shared memory serves 4 products (with one sample a warp each weight
// read served one: 8192 samples of 784 inputs, 10 classes, took 106 us a
// call, 28 now).  Classes come in G groups of CC; the 4 x CC sums are reduced over the lanes by two
// exchange steps (a lane keeps one sample) and three butterfly steps.
constexpr int kEvalThreads = 512;
template <int CC, int G>
__global__ void __launch_bounds__(kEvalThreads) softreg_eval_kernel(const __grid_constant__ SoftregEvalArgs a) {
  extern __shared__ __align__(16) float Wsm[];   // [C][D]; a group's classes past C read the last row and are ignored
  __shared__ float part[kEvalThreads / 32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int D = a.D, C = a.C;
  for (int i = threadIdx.x; i < C * D; i += kEvalThreads) Wsm[i] = a.master[a.offW + i];
  __syncthreads();
  float mine = 0.f;
  const int64_t step = static_cast<int64_t>(gridDim.x) * (kEvalThreads / 32) * 4;
  for (int64_t i0 = (static_cast<int64_t>(blockIdx.x) * (kEvalThreads / 32) + warp) * 4; i0 < a.n; i0 += step) {
    const float* xr[4];
#pragma unroll
    for (int r = 0; r < 4; ++r) xr[r] = a.x + (i0 + r < a.n ? i0 + r : a.n - 1) * D;
    float z[G][CC];   // of sample i0 + lane / 8
#pragma unroll
    for (int g = 0; g < G; ++g) {
      float acc[4][CC];
#pragma unroll
      for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int c = 0; c < CC; ++c) acc[r][c] = 0.f;
      int woff[CC];
#pragma unroll
      for (int c = 0; c < CC; ++c) woff[c] = (g * CC + c < C ? g * CC + c : C - 1) * D;
#pragma unroll 4
      for (int k = lane; k < D; k += 32) {
        float xv[4];
#pragma unroll
        for (int r = 0; r < 4; ++r) xv[r] = xr[r][k];
#pragma unroll
        for (int c = 0; c < CC; ++c) {
          const float w = Wsm[woff[c] + k];
#pragma unroll
          for (int r = 0; r < 4; ++r) acc[r][c] = fmaf(xv[r], w, acc[r][c]);
        }
      }
      const bool up = lane & 16, odd = lane & 8;
#pragma unroll
      for (int c = 0; c < CC; ++c) {
        const float k0 = up ? acc[2][c] : acc[0][c], k1 = up ? acc[3][c] : acc[1][c];
        const float g0 = up ? acc[0][c] : acc[2][c], g1 = up ? acc[1][c] : acc[3][c];
        const float h0 = k0 + __shfl_xor_sync(0xffffffffu, g0, 16), h1 = k1 + __shfl_xor_sync(0xffffffffu, g1, 16);
        float v = (odd ? h1 : h0) + __shfl_xor_sync(0xffffffffu, odd ? h0 : h1, 8);
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        z[g][c] = v;
      }
    }
    const int64_t i = i0 + (lane >> 3);
    if (i < a.n && (lane & 7) == 0) {
      const int y = a.y[i];
      float m = -INFINITY, zy = 0.f, se = 0.f;
#pragma unroll
      for (int g = 0; g < G; ++g)
#pragma unroll
        for (int c = 0; c < CC; ++c) {
          const int k = g * CC + c;
          if (k >= C) continue;
          z[g][c] += a.master[a.offB + k];
          m = fmaxf(m, z[g][c]);
          if (k == y) zy = z[g][c];
        }
#pragma unroll
      for (int g = 0; g < G; ++g)
#pragma unroll
        for (int c = 0; c < CC; ++c)
          if (g * CC + c < C) se += expf(z[g][c] - m);
      mine += m + logf(se) - zy;
    }
  }
  mine = warp_sum(mine);
  if (lane == 0) part[warp] = mine;
  __syncthreads();
  if (threadIdx.x == 0) {
    float s = 0.f;
    for (int i = 0; i < kEvalThreads / 32; ++i) s += part[i];
    a.loss_sum[blockIdx.x] = s;
  }
}

}  // namespace

size_t softreg_smem_bytes(int D, int C, int B) {
  return sizeof(float) * (static_cast<size_t>(C) * D + 32 + static_cast<size_t>(B) * D +
                          static_cast<size_t>(B) * C + B) +
         sizeof(int) * B + 8 + sizeof(int64_t) * B;
}

cudaError_t launch_softreg_round(const SoftregArgs& a, int W, cudaStream_t s) {
  const size_t smem = softreg_smem_bytes(a.D, a.C, a.B);
  cudaError_t e = allow_smem(softreg_round_kernel, smem);
  if (e != cudaSuccess) return e;
  softreg_round_kernel<<<W, kThreads, smem, s>>>(a);
  return cudaGetLastError();
}

namespace {
size_t cluster_smem_bytes(int D, int C, int B, int NT) {
  const ClPlan p = cluster_plan(D, C, B, cluster_cc(C), NT);
  return sizeof(float) * p.oEnd + cluster_tail_bytes(B);
}

// computing threads where the workers need not share SMs
int cluster_threads_alone(int D, int C, int B) {
  return static_cast<int64_t>(B) * C * cluster_cols(D) <= kClSmallWork ? 128 : kClThreads;
}

template <int CC, int NT, int K>
cudaLaunchConfig_t cluster_config(cudaLaunchAttribute* attr, int W, size_t smem, cudaStream_t s) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(kCl, W, 1);
  cfg.blockDim = dim3(NT + NT / 4, 1, 1);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  attr->id = cudaLaunchAttributeClusterDimension;
  attr->val.clusterDim.x = kCl;
  attr->val.clusterDim.y = 1;
  attr->val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cfg;
}

// Clusters that run at once with k CTAs an SM, k <= 4 (not k SMs / 8: the SMs of
// a cluster share a processor cluster).  Queried once per device.
constexpr int kMaxDevices = 64;
std::atomic<int> g_room[kMaxDevices][4];
template <int NT, int K>
int query_room(size_t smem) {
  int room = 0;
  cudaLaunchAttribute attr;
  const cudaLaunchConfig_t cfg = cluster_config<8, NT, K>(&attr, 1, smem, nullptr);
  if (cudaOccupancyMaxActiveClusters(&room, softreg_cluster_round_kernel<8, NT, K>, &cfg) != cudaSuccess) {
    cudaGetLastError();
    room = 0;
  }
  return room < 1 ? 1 : room;
}
int cluster_room(int k) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) dev = 0;
  std::atomic<int>& r = g_room[dev][k - 1];
  int room = r.load(std::memory_order_relaxed);
  if (room > 0) return room;
  // 3 CTAs an SM: what 2 and 4 leave between them
  room = k == 1   ? query_room<512, 1>(0)
         : k == 2 ? query_room<256, 2>(0)
         : k == 4 ? query_room<128, 4>(0)
                  : (cluster_room(2) + cluster_room(4)) / 2;
  r.store(room, std::memory_order_relaxed);
  return room;
}

// The variant for W workers: the fewest waves, then the most threads.  About 15
// clusters run at once with one CTA an SM: with 512 threads whatever W, more
// workers waited for a second and third wave, and the smaller shapes were slower
// than on the 256-thread cluster kernel before this one, several of whose CTAs
// share an SM.  Rounds of 4 steps with their merge, us, by workers (before /
// 512 threads / this rule):
//   784 x 10, batch 8      1: 27 / 25 / 25    16: 29 / 43 / 27    32: 33 / 60 / 29     64: 56 / 94 / 37
//   64 x 10, batch 64      1: 35 / 25 / 25    16: 38 / 43 / 25    32: 42 / 62 / 29     64: 71 / 98 / 38
//   333 x 26, batch 100    1: 93 / 39 / 39    16: 121 / 74 / 60   32: 126 / 105 / 64   64: 237 / 171 / 118
//   5000 x 4, batch 4      1: 34 / 31 / 31    16: 35 / 53 / 34    32: 38 / 75 / 36     64: 65 / 118 / 46
// The line of 4096 products: a round of 16 x 2, batch 1, 32 workers with its
// merge and pull took 62 us with 512 threads, 40 with 128.
struct ClVariant {
  int NT, K;
};
ClVariant cluster_variant(int D, int C, int B, int W) {
  const ClVariant all[3] = {{512, 1}, {256, 2}, {128, 4}}, few[2] = {{128, 2}, {128, 4}};
  const bool small = cluster_threads_alone(D, C, B) == 128;
  const ClVariant* v = small ? few : all;
  if (W == 1) return v[0];
  ClVariant best = v[0];
  int least = 1 << 30;
  for (int i = 0; i < (small ? 2 : 3) && least > 1; ++i) {
    int k = static_cast<int>(kSmSmem / (cluster_smem_bytes(D, C, B, v[i].NT) + kCtaSmem));
    k = k > v[i].K ? v[i].K : k < 1 ? 1 : k;
    const int room = cluster_room(k), waves = (W + room - 1) / room;
    if (waves < least) {
      least = waves;
      best = v[i];
    }
  }
  return best;
}

template <int CC, int NT, int K>
cudaError_t launch_cluster_nt(const SoftregArgs& a, int W, cudaStream_t s) {
  const size_t smem = cluster_smem_bytes(a.D, a.C, a.B, NT);
  cudaError_t e = allow_smem(softreg_cluster_round_kernel<CC, NT, K>, smem);
  if (e != cudaSuccess) return e;
  cudaLaunchAttribute attr;
  const cudaLaunchConfig_t cfg = cluster_config<CC, NT, K>(&attr, W, smem, s);
  return cudaLaunchKernelEx(&cfg, softreg_cluster_round_kernel<CC, NT, K>, a);
}

template <int CC>
cudaError_t launch_cluster(const SoftregArgs& a, int W, cudaStream_t s) {
  const ClVariant v = cluster_variant(a.D, a.C, a.B, W);
  return v.NT == 512  ? launch_cluster_nt<CC, 512, 1>(a, W, s)
         : v.NT == 256 ? launch_cluster_nt<CC, 256, 2>(a, W, s)
         : v.K == 2    ? launch_cluster_nt<CC, 128, 2>(a, W, s)
                       : launch_cluster_nt<CC, 128, 4>(a, W, s);
}
}  // namespace

bool softreg_cluster_supported(int D, int C, int B) {
  return B <= kSoftregMaxBatch && cluster_smem_bytes(D, C, B, cluster_threads_alone(D, C, B)) <= 220 * 1024;
}

cudaError_t launch_softreg_cluster_round(const SoftregArgs& a, int W, cudaStream_t s) {
  switch (cluster_cc(a.C)) {
    case 4: return launch_cluster<4>(a, W, s);
    case 5: return launch_cluster<5>(a, W, s);
    case 7: return launch_cluster<7>(a, W, s);
    case 8: return launch_cluster<8>(a, W, s);
    default: return cudaErrorInvalidValue;
  }
}

int softreg_eval_blocks(int64_t n, int sms) {
  const int64_t need = (n + kEvalThreads / 8 - 1) / (kEvalThreads / 8);   // 4 samples a warp
  return static_cast<int>(need < sms ? need : sms);
}

namespace {
template <int CC, int G>
cudaError_t launch_eval(const SoftregEvalArgs& a, int blocks, cudaStream_t s) {
  const size_t smem = sizeof(float) * a.C * static_cast<size_t>(a.D);
  cudaError_t e = allow_smem(softreg_eval_kernel<CC, G>, smem);
  if (e != cudaSuccess) return e;
  softreg_eval_kernel<CC, G><<<blocks, kEvalThreads, smem, s>>>(a);
  return cudaGetLastError();
}
}  // namespace

cudaError_t launch_softreg_eval(const SoftregEvalArgs& a, int blocks, cudaStream_t s) {
  if (a.C <= 4) return launch_eval<4, 1>(a, blocks, s);
  if (a.C <= 8) return launch_eval<8, 1>(a, blocks, s);
  if (a.C <= 12) return launch_eval<12, 1>(a, blocks, s);
  if (a.C <= 16) return launch_eval<16, 1>(a, blocks, s);
  if (a.C <= 24) return launch_eval<12, 2>(a, blocks, s);
  return launch_eval<16, 2>(a, blocks, s);
}

}  // namespace oscars
