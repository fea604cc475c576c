// Batched form: thousands of small trajectories in one persistent launch.
//
// The plain loop (runtime.cu) spends one kernel launch per fused gate and a
// host round trip per stage-2 channel; for states of 2^8..2^18 amplitudes
// that is launch- and latency-bound (the paper notes qsim is not tuned for
// small circuits and its translation overhead dominates below 20 qubits,
// Sec. IV.A).  Here every trajectory of the batch, each with its own
// circuit, runs inside one persistent kernel:
//   - CTAs take trajectories from an atomic counter per class of state sizes,
//     largest state first;
//   - a state of up to 2^14 amplitudes lives in its CTA's shared memory, the
//     CTA sized to it, so that an SM holds several small ones; larger states
//     live in a per-CTA slot of global memory (up to 2^20 amplitudes) and come
//     to shared memory tile by tile, several gates to a sweep;
//   - stage 1 of Alg. 2 for every channel is decided on the device with the
//     same Philox4x32-10 draws as the plain loop; stage-2 flush points cut
//     the circuit into segments exactly as in the plain loop, and within a
//     segment a fused gate whose slots all hold their default operator uses
//     its precomputed matrix while any other piece has its members in the
//     segment composed into one matrix in shared memory;
//   - on global-memory states the first segment starts from a product
//     state: every piece that is first on its qubits is folded into the
//     initial state instead of making a pass of its own;
//   - the probability pass, stage 2, and bitstring sampling run in the CTA.
// Host side: circuits are fused on a thread pool (qt_fuse_many) and packed
// once into device tables with every distinct operator set stored once;
// qt_batch_run replays the launch sequence as a CUDA graph.
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstring>
#include <memory>
#include <mutex>
#include <new>
#include <thread>
#include <unordered_map>
#include <vector>

#include "kernels.h"
#include "qt_dfloat.h"
#include "qt_internal.h"
#include "qt_philox.h"

namespace qt {
namespace bt {

constexpr int kMaxW = 6;            // widest fused gate in the batched form
constexpr int kSmemNMax = 14;       // states up to 2^14 amplitudes in shared memory
constexpr int kMaxN = 20;           // widest state of the batched form
// product-state start: sum of 2^w over the folded pieces (disjoint qubits,
// w <= 6, n <= 20 give at most 3 * 64 + 4)
constexpr int kFoldCols = 256;
// classes of trajectories, one launch each (qt_batch::count)
constexpr int kClasses = 5;
inline int class_of(uint32_t n) { return n > 14 ? 0 : (n == 14 ? 1 : (n == 13 ? 2 : (n > 10 ? 3 : 4))); }

struct Traj {
  uint32_t n, gate0, ngates, op0, nops, ch0, nch, chop0;   // ch0: output offset; chop0: ch_op table offset
  uint64_t arena_off;               // amplitude offset of the kept state (keep_states)
  uint32_t gf0, S;                  // offset of this trajectory's per-gate flags (per trajectory, like ch0);
                                    // with per-trajectory parameters: its sample count
  uint64_t seed, tid, soff;         // with per-trajectory parameters: Philox key, trajectory id, first
                                    // sample slot (a merged launch over several requests)
};
struct Op {
  uint8_t kind, q, q0, q1;
  uint32_t set;
  int32_t channel;                  // relative channel ordinal, -1 for gates
  uint32_t gate;                    // fused gate that holds it (relative)
};
struct Set {
  uint32_t nk, q, def, pad;
  uint32_t mat, kraus, mtm, pbar;   // offsets: float2, float2, double, double
  uint64_t thr0;                    // a draw of `bits` / 2^53 is below pbar[0] exactly when bits < thr0
};
struct Gate {
  uint8_t w, t[kMaxW];
  uint8_t pad[1];
  uint32_t mat, mem0, nmem, minpos, maxpos;
};
struct Dev {
  const Traj* traj;
  const Op* ops;
  const Set* sets;
  const Gate* gates;
  const uint32_t* members;
  const uint32_t* ch_op;
  const float2* fmat;
  const double* dmat;
  const uint32_t* order;
  float2* arena;                    // per-CTA slots, or per-trajectory when keeping states
  uint64_t slot_amps;               // amplitudes per CTA slot (0: use traj.arena_off)
  int8_t* kraus;                   // records: bytes (at most 64 operators), -1 undecided
  int8_t* stage;
  uint8_t* gflag;                   // per fused gate of the run: a member channel holds a non-default stage-1 choice
  uint64_t* samples;
  uint32_t* flushes;
  uint32_t* folds;                  // pieces folded into the product-state start, per trajectory (or null)
  unsigned int* counter;
  int* err;
  const uint64_t* run;              // {seed, first_traj} of the current run (device copy)
  uint32_t num, S, keep;
  uint32_t per_traj;                // 1: seed, id and samples from each Traj (merged launches)
  uint32_t lthreads;                // threads that the sums of a trajectory are split over (results depend
                                    // on them, not on the CTA's own size)
  uint32_t wmat;                    // widest fused gate of the launch
};

// ---------------------------------------------------------------------------
// device helpers (all threads of the CTA call them together)
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint32_t insert_zeros32(uint32_t x, int w, const int* sorted) {
  for (int b = 0; b < w; ++b) {
    const int s = sorted[b];
    x = ((x >> s) << (s + 1)) | (x & ((1u << s) - 1u));
  }
  return x;
}

// Clusters of the global class: the CTAs of one trajectory (all their threads
// call cluster_sync together; it orders their global-memory accesses)
__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ uint32_t cluster_size() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// the 32-bit word at p of CTA 0's shared memory
__device__ __forceinline__ uint32_t leader_word(const void* p) {
  uint32_t a = static_cast<uint32_t>(__cvta_generic_to_shared(p)), r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, 0;" : "=r"(a) : "r"(a));
  asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(r) : "r"(a) : "memory");
  return r;
}

// Where amplitude x of a shared-memory state sits: index bits 4..7 are mapped
// linearly into bits 0..3.  The 16 lanes of an 8-byte access differ in the
// four lowest bits that are no target; the map was searched for the fewest
// bank conflicts over the contiguous target runs that chains fuse to (none
// for runs of up to three) and all target sets below bit 10.
__device__ __forceinline__ uint32_t sw(uint32_t x) {
  constexpr uint64_t f = [] {
    const uint32_t img[4] = {15, 10, 12, 8};
    uint64_t t = 0;
    for (int i = 0; i < 16; ++i) {
      uint32_t v = 0;
      for (int b = 0; b < 4; ++b)
        if ((i >> b) & 1) v ^= img[b];
      t |= static_cast<uint64_t>(v) << (4 * i);
    }
    return t;
  }();
  return x ^ (static_cast<uint32_t>(f >> ((x >> 2) & 60u)) & 15u);
}

// amplitude x of a state in global (plain) or shared (swizzled) memory
template <bool SHARED>
__device__ __forceinline__ uint32_t at(uint32_t x) {
  return SHARED ? sw(x) : x;
}

// psi <- A psi for a state in shared memory; A (row-major) in shared memory,
// read two entries at a time (a broadcast); t ascending
template <int W>
__device__ __forceinline__ void smem_apply(float2* psi, int n, const uint8_t* t, const float2* A) {
  constexpr int D = 1 << W;
  int sorted[W];
  uint32_t off[D];
#pragma unroll
  for (int b = 0; b < W; ++b) sorted[b] = t[b];
#pragma unroll
  for (int m = 0; m < D; ++m) {
    uint32_t o = 0;
#pragma unroll
    for (int b = 0; b < W; ++b)
      if ((m >> b) & 1) o |= 1u << sorted[b];
    off[m] = sw(o);                    // sw distributes over disjoint bits
  }
  const uint32_t sets = 1u << (n - W);
  for (uint32_t s = threadIdx.x; s < sets; s += blockDim.x) {
    const uint32_t base = sw(insert_zeros32(s, W, sorted));
    float2 v[D];
#pragma unroll
    for (int m = 0; m < D; ++m) v[m] = psi[base ^ off[m]];
    constexpr int RU = W <= 3 ? D : 4;
#pragma unroll RU
    for (int j = 0; j < D; ++j) {
      float xr = 0.f, xi = 0.f;
#pragma unroll
      for (int m = 0; m < D; m += 2) {
        const float4 a = *reinterpret_cast<const float4*>(A + j * D + m);
        xr = fmaf(a.x, v[m].x, fmaf(-a.y, v[m].y, xr));
        xi = fmaf(a.x, v[m].y, fmaf(a.y, v[m].x, xi));
        xr = fmaf(a.z, v[m + 1].x, fmaf(-a.w, v[m + 1].y, xr));
        xi = fmaf(a.z, v[m + 1].y, fmaf(a.w, v[m + 1].x, xi));
      }
      psi[base ^ off[j]] = make_float2(xr, xi);
    }
  }
}

// widths 5 and 6: one gather set per thread, its 2^w members in a local
// array (registers or, at w = 6, local memory); kept out of line so that its
// register demand does not raise that of the rest of the kernel
template <int W, bool SHARED>
__device__ __noinline__ void cta_apply_wide(float2* psi, int n, const int* order, const float2* A, uint32_t first,
                                            uint32_t stride) {
  constexpr int D = 1 << W;
  int sorted[W];
  for (int b = 0; b < W; ++b) sorted[b] = order[b];
  const uint32_t sets = 1u << (n - W);
  for (uint32_t s = first; s < sets; s += stride) {
    const uint32_t base = insert_zeros32(s, W, sorted);
    float2 v[D];
    for (int m = 0; m < D; ++m) {
      uint32_t o = 0;
      for (int b = 0; b < W; ++b)
        if ((m >> b) & 1) o |= 1u << order[b];
      v[m] = psi[at<SHARED>(base | o)];
    }
    for (int j = 0; j < D; ++j) {
      float xr = 0.f, xi = 0.f;
      for (int m = 0; m < D; ++m) {
        const float2 a = A[j * D + m];
        xr = fmaf(a.x, v[m].x, fmaf(-a.y, v[m].y, xr));
        xi = fmaf(a.x, v[m].y, fmaf(a.y, v[m].x, xi));
      }
      uint32_t o = 0;
      for (int b = 0; b < W; ++b)
        if ((j >> b) & 1) o |= 1u << order[b];
      psi[at<SHARED>(base | o)] = make_float2(xr, xi);
    }
  }
}

// a 5- or 6-qubit gate on a state in global memory; A is in global memory, or
// smat itself when it was composed there
__device__ void cta_apply_wide_glob(float2* psi, int n, const Gate& G, const float2* A, float2* smat) {
  __syncthreads();                     // previous users of smat / psi are done
  if (A != smat) {
    for (int i = threadIdx.x; i < 1 << (2 * G.w); i += blockDim.x) smat[i] = A[i];
    __syncthreads();
  }
  int order[kMaxW];
  for (int b = 0; b < G.w; ++b) order[b] = G.t[b];
  const uint32_t first = cluster_rank() * blockDim.x + threadIdx.x, stride = cluster_size() * blockDim.x;
  if (G.w == 5) cta_apply_wide<5, false>(psi, n, order, smat, first, stride);
  else cta_apply_wide<6, false>(psi, n, order, smat, first, stride);
}

__device__ __forceinline__ float2 cmul_add(float2 a, float2 x, float2 acc) {
  acc.x = fmaf(a.x, x.x, fmaf(-a.y, x.y, acc.x));
  acc.y = fmaf(a.x, x.y, fmaf(a.y, x.x, acc.y));
  return acc;
}

// M <- A M for the 2^q x 2^q operator A (q = 1, 2; index bit b <-> pos[b]
// among the w basis bits of M), scaled by sc: every column of M is a vector
// that A acts on, as in Alg. 1.  M is D x D row-major in shared memory; the
// caller is thread tid of the nt that share the work.
__device__ void left_apply(float2* M, int w, int q, const int* pos, const float2* A, float sc, int tid, int nt) {
  const int D = 1 << w;
  if (q == 1) {
    const float2 a00 = make_float2(A[0].x * sc, A[0].y * sc), a01 = make_float2(A[1].x * sc, A[1].y * sc);
    const float2 a10 = make_float2(A[2].x * sc, A[2].y * sc), a11 = make_float2(A[3].x * sc, A[3].y * sc);
    const int p = pos[0];
    for (int u = tid; u < (D >> 1) * D; u += nt) {
      const int c = u & (D - 1), rr = u >> w;
      const int r0 = ((rr >> p) << (p + 1)) | (rr & ((1 << p) - 1)), r1 = r0 | (1 << p);
      const float2 x0 = M[r0 * D + c], x1 = M[r1 * D + c];
      M[r0 * D + c] = cmul_add(a01, x1, cmul_add(a00, x0, make_float2(0.f, 0.f)));
      M[r1 * D + c] = cmul_add(a11, x1, cmul_add(a10, x0, make_float2(0.f, 0.f)));
    }
    return;
  }
  const int lo = pos[0] < pos[1] ? pos[0] : pos[1], hi = pos[0] < pos[1] ? pos[1] : pos[0];
  for (int u = tid; u < (D >> 2) * D; u += nt) {
    const int c = u & (D - 1);
    int r = u >> w;
    r = ((r >> lo) << (lo + 1)) | (r & ((1 << lo) - 1));
    r = ((r >> hi) << (hi + 1)) | (r & ((1 << hi) - 1));
    int rows[4];
    float2 x[4];
#pragma unroll
    for (int m = 0; m < 4; ++m) {
      rows[m] = r | ((m & 1) << pos[0]) | (((m >> 1) & 1) << pos[1]);
      x[m] = M[rows[m] * D + c];
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      float2 acc = make_float2(0.f, 0.f);
#pragma unroll
      for (int m = 0; m < 4; ++m) {
        const float2 a = A[j * 4 + m];
        acc = cmul_add(make_float2(a.x * sc, a.y * sc), x[m], acc);
      }
      M[rows[j] * D + c] = acc;
    }
  }
}

// Reduced density of the Q qubits order[] -> out[0..4^Q) (layout of
// rdm_unpack), written by thread 0.  The sets are dealt to `lthreads` logical
// threads, FP32 runs of 16 sets each, whatever the CTA's size: logical warp
// after logical warp for the CTA's warps.  Carries in double-floats.
template <int Q, bool SHARED>
__device__ void cta_rdm(const float2* psi, int n, const int* order, int lthreads, double* out, float2 (*red)[16]) {
  constexpr int D = 1 << Q, W = D * D;
  constexpr int U = SHARED ? 1 : 8;                      // sets loaded at once from global memory
  int sorted[Q];
  uint32_t off[D];
  for (int b = 0; b < Q; ++b) sorted[b] = order[b];
  if (Q > 1 && sorted[0] > sorted[Q - 1]) { const int t = sorted[0]; sorted[0] = sorted[Q - 1]; sorted[Q - 1] = t; }
#pragma unroll
  for (int m = 0; m < D; ++m) {
    uint32_t o = 0;
    for (int b = 0; b < Q; ++b)
      if ((m >> b) & 1) o |= 1u << order[b];
    off[m] = o;
  }
  const uint32_t sets = 1u << (n - Q);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5, lw = lthreads >> 5;
  for (int l = warp; l < lw; l += nw) {
    float2 acc[W];
    float f[W];
#pragma unroll
    for (int c = 0; c < W; ++c) { acc[c] = make_float2(0.f, 0.f); f[c] = 0.f; }
    int cnt = 0;
    for (uint32_t s0 = l * 32 + lane; s0 < sets; s0 += U * lthreads) {
      float2 v[U][D];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const uint32_t s = s0 + u * lthreads, base = insert_zeros32(s, Q, sorted);
#pragma unroll
        for (int m = 0; m < D; ++m) v[u][m] = s < sets ? psi[at<SHARED>(base | off[m])] : make_float2(0.f, 0.f);
      }
#pragma unroll
      for (int u = 0; u < U; ++u) {
        int c = 0;
#pragma unroll
        for (int b = 0; b < D; ++b) { f[c] = fmaf(v[u][b].x, v[u][b].x, fmaf(v[u][b].y, v[u][b].y, f[c])); ++c; }
#pragma unroll
        for (int b = 0; b < D; ++b)
#pragma unroll
          for (int a = b + 1; a < D; ++a) {
            f[c] = fmaf(v[u][b].x, v[u][a].x, fmaf(v[u][b].y, v[u][a].y, f[c])); ++c;
            f[c] = fmaf(v[u][b].y, v[u][a].x, fmaf(-v[u][b].x, v[u][a].y, f[c])); ++c;
          }
      }
      if ((cnt += U) == 16) {
#pragma unroll
        for (int k = 0; k < W; ++k) { df_acc(acc[k].x, acc[k].y, f[k]); f[k] = 0.f; }
        cnt = 0;
      }
    }
#pragma unroll
    for (int k = 0; k < W; ++k) df_acc(acc[k].x, acc[k].y, f[k]);
    const float2 r = df_warp_sum<W>(acc, lane);
    constexpr int per = 32 / W;
    if (lane % per == 0) red[l][lane / per] = r;
  }
  __syncthreads();
  if (threadIdx.x < W) {
    float2 v = make_float2(0.f, 0.f);
    for (int w2 = 0; w2 < lw; ++w2) v = df_add(v, red[w2][threadIdx.x]);
    out[threadIdx.x] = df_value(v);
  }
  __syncthreads();
}

__device__ __forceinline__ float warp_scan_f(float v, int lane) {
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const float y = __shfl_up_sync(0xffffffffu, v, o);
    if (lane >= o) v += y;
  }
  return v;
}

// S samples.  The amplitudes are cut into one contiguous range per logical
// warp (lthreads / 32 of them); C(x) inside a range is the running FP32 sum
// of 32-amplitude chunk totals plus the chunk's warp scan; ranges are chained
// by an FP64 scan of their totals.  While the ranges are summed, each group of
// chunks (a chunk of its own up to 2^14 amplitudes) notes the sum before it
// and its largest C, so that a sample finds its group with one vote of the
// warp instead of scanning the range.  32 samples draw at once, a lane each;
// FP64 compares with FP32 sums are made in FP32 against the target rounded
// down (f > t exactly when f > rd(t)).
constexpr int kSampleGroups = 512;
struct SampleScratch {
  double wcum[16];
  float before[kSampleGroups], most[kSampleGroups];
};

template <bool SHARED>
__device__ void cta_sample(const float2* psi, int n, uint64_t seed, uint64_t traj, uint32_t S, uint64_t* out,
                           int lthreads, SampleScratch& sc) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5, lw = lthreads >> 5;
  const uint32_t amps = 1u << n;
  uint32_t per = (amps + lw - 1) / lw;
  per = (per + 31) & ~31u;
  const int chunks = static_cast<int>(per / 32);
  const int gpr = min(chunks, kSampleGroups / lw), gch = chunks / gpr;   // groups per range, chunks per group (2^k)
  const int glog = 31 - __clz(gch);
  // chunks loaded at once from global memory (2^15 amplitudes and more: every
  // chunk is inside the state)
  constexpr int U = SHARED ? 1 : 16;
  auto weight = [&](uint32_t x) {
    float w = 0.f;
    if (!SHARED || x < amps) { const float2 a = psi[at<SHARED>(x)]; w = fmaf(a.x, a.x, a.y * a.y); }
    return w;
  };
  __syncthreads();
  for (int r = warp; r < lw; r += nw) {
    const uint32_t lo = r * per;
    float run = 0.f, most = 0.f;
    for (int c0 = 0; c0 < chunks; c0 += U) {               // chunks is a multiple of U
      float w[U];
#pragma unroll
      for (int u = 0; u < U; ++u) w[u] = weight(lo + (c0 + u) * 32 + lane);
#pragma unroll
      for (int u = 0; u < U; ++u) w[u] = warp_scan_f(w[u], lane);
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int g = (c0 + u) >> glog;
        if (((c0 + u) & (gch - 1)) == 0) {
          if (lane == 0) sc.before[r * gpr + g] = run;
          most = 0.f;
        }
        most = fmaxf(most, run + w[u]);
        run += __shfl_sync(0xffffffffu, w[u], 31);
        if (((c0 + u + 1) & (gch - 1)) == 0) {
          const float all = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(most)));   // not negative
          if (lane == 0) sc.most[r * gpr + g] = all;
        }
      }
    }
    if (lane == 0) sc.wcum[r] = static_cast<double>(run);
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double r = 0.0;
    for (int w = 0; w < lw; ++w) { r += sc.wcum[w]; sc.wcum[w] = r; }
  }
  __syncthreads();
  const double total = sc.wcum[lw - 1];
  const uint32_t batch = min(max((S + nw - 1) / nw, 8u), 32u);   // samples a warp draws at once
  for (uint32_t j0 = warp * batch; j0 < S; j0 += nw * batch) {
    // lane: sample j0 + lane
    int range = 0;
    float below = 0.f;                                     // its target inside the range, rounded down
    double trel = 0.0;
    const bool own = lane < static_cast<int>(batch) && j0 + lane < S;
    if (own) {
      const double t = uniform01(seed, traj, kStreamSample, j0 + lane) * total;
      int last = lw - 1;
      while (range < last) {                               // first range whose end is above t
        const int mid = (range + last) >> 1;
        if (t < sc.wcum[mid]) last = mid; else range = mid + 1;
      }
      trel = t - (range ? sc.wcum[range - 1] : 0.0);
      below = __double2float_rd(trel);
    }
    uint64_t mine = 0;
    for (uint32_t i = 0; i < batch && j0 + i < S; ++i) {
      const int r = __shfl_sync(0xffffffffu, range, i);
      const float b = __shfl_sync(0xffffffffu, below, i);
      const uint32_t lo = r * per;
      int g = gpr;
      for (int g0 = 0; g0 < gpr && g == gpr; g0 += 32) {
        const unsigned hit = __ballot_sync(0xffffffffu, g0 + lane < gpr && sc.most[r * gpr + g0 + lane] > b);
        if (hit) g = g0 + __ffs(hit) - 1;
      }
      uint64_t x = ~0ull;
      if (g < gpr) {
        float run = sc.before[r * gpr + g];
        for (int c = 0; c < gch; ++c) {
          const uint32_t x0 = lo + (g * gch + c) * 32;
          const float inc = warp_scan_f(weight(x0 + lane), lane);
          const unsigned h = __ballot_sync(0xffffffffu, run + inc > b);
          if (h) { x = x0 + __ffs(h) - 1; break; }
          run += __shfl_sync(0xffffffffu, inc, 31);
        }
      }
      if (x >= amps) {
        // rounding put the target past the range (or past the state): its last
        // amplitude of non-zero weight, up to the chunk that would hold the target
        float run = 0.f;
        uint32_t last_nz = lo < amps ? lo : amps - 1;
        for (uint32_t c = lo; c < lo + per; c += 32) {
          const float w = weight(c + lane);
          const float inc = warp_scan_f(w, lane);
          const unsigned nz = __ballot_sync(0xffffffffu, w > 0.f);
          if (nz) last_nz = c + 31 - __clz(nz);
          if (__ballot_sync(0xffffffffu, run + inc > b)) break;
          run += __shfl_sync(0xffffffffu, inc, 31);
        }
        x = last_nz;
      }
      if (lane == static_cast<int>(i)) mine = x;
    }
    if (own) out[j0 + lane] = mine;
  }
}

// The piece of fused gate G over ops [lo, hi): its members there composed in
// FP32 into one matrix over the gate's qubits, left in s_mat (D x D
// row-major; identity on qubits none of them touches).  The channel decided
// in stage 2 at the segment's start (op pend_pos) enters as its Kraus
// operator pend_choice scaled by pend_scale; any other channel as its
// stage-1 choice.
//
// The members' descriptors and operators are first gathered by all threads
// (the table walk is four dependent loads, paid once for 64 members instead
// of by each); up to 3 qubits one warp then multiplies on, without barriers.
constexpr int kListMax = 64;
struct MemberList {
  float2 A[kListMax][16];
  float scale[kListMax];
  int8_t q[kListMax], p0[kListMax], p1[kListMax];    // q = 0: not in the segment
};

__device__ __noinline__ void cta_compose_piece(const Dev& d, const Traj& T, const Gate& G, uint32_t lo, uint32_t hi,
                                               int pend_pos, int pend_choice, float pend_scale, float2* s_mat,
                                               MemberList& list) {
  const int D = 1 << G.w, tid = threadIdx.x, nt = blockDim.x;
  __syncthreads();                 // previous users of s_mat and list are done
  for (int i = tid; i < D * D; i += nt)
    s_mat[i] = make_float2((i >> G.w) == (i & (D - 1)) ? 1.f : 0.f, 0.f);
  for (uint32_t m0 = 0; m0 < G.nmem; m0 += kListMax) {
    const int cnt = static_cast<int>(min(G.nmem - m0, static_cast<uint32_t>(kListMax)));
    if (m0) __syncthreads();
    for (int i = tid; i < cnt * 4; i += nt) {            // four threads a member, four entries each
      const int mi = i >> 2, part = i & 3;
      const uint32_t pos = d.members[G.mem0 + m0 + mi];
      int q = 0;
      if (pos >= lo && pos < hi) {
        const Op op = d.ops[T.op0 + pos];
        const Set st = d.sets[op.set];
        q = op.q;
        const uint32_t dd = 1u << (2 * q);
        const float2* A;
        float sc = 1.f;
        if (op.channel < 0) {
          A = d.fmat + st.mat;
        } else if (static_cast<int>(pos) == pend_pos) {
          A = d.fmat + st.kraus + pend_choice * dd;
          sc = pend_scale;
        } else {
          A = d.fmat + st.mat + d.kraus[T.ch0 + op.channel] * dd;
        }
        for (uint32_t e = part * 4; e < part * 4 + 4 && e < dd; ++e) list.A[mi][e] = A[e];
        if (part == 0) {
          int p0 = 0, p1 = 0;
          for (int b = 0; b < G.w; ++b) {
            if (G.t[b] == op.q0) p0 = b;
            if (q > 1 && G.t[b] == op.q1) p1 = b;
          }
          list.scale[mi] = sc;
          list.p0[mi] = static_cast<int8_t>(p0);
          list.p1[mi] = static_cast<int8_t>(p1);
        }
      }
      if (part == 0) list.q[mi] = static_cast<int8_t>(q);
    }
    __syncthreads();
    const bool one_warp = G.w <= 3;
    if (one_warp && tid >= 32) continue;
    for (int mi = 0; mi < cnt; ++mi) {
      const int q = list.q[mi];
      if (q == 0) continue;
      const int p[2] = {list.p0[mi], list.p1[mi]};
      left_apply(s_mat, G.w, q, p, list.A[mi], list.scale[mi], tid, one_warp ? 32 : nt);
      if (one_warp) __syncwarp();
      else __syncthreads();        // the member's update is complete
    }
  }
}

__device__ __forceinline__ uint32_t gate_mask(const Gate& G) {
  uint32_t m = 0;
  for (int b = 0; b < G.w; ++b) m |= 1u << G.t[b];
  return m;
}

// Product-state start (the first segment, ops [0, hi)).  A piece none of
// whose qubits an earlier piece of the segment touches acts on |0> of its
// own qubits and commutes with every piece before it, so it moves to the
// front: its column U[:, 0] becomes a factor of the initial state
//   psi[x] = prod_f U_f[x restricted to the qubits of f, 0],
// zero where x has a 1 on a qubit that no folded piece holds.  The qubits
// are split at m: the factors of the pieces wholly below m form a table of
// 2^m entries, those wholly from m up one of 2^(n-m) (both in s_mat), so an
// amplitude is one product of two table entries, times the factors of the
// few pieces that straddle m (m is chosen to have the fewest).  Writes the
// whole state, marks the folded gates (gate flag 2: the pass loop of the
// first segment skips them; a later segment treats such a gate, which the
// flush point cut, as a composed piece) and returns their number.
struct FoldPiece {
  uint32_t mask;                   // its qubits
  uint32_t gate;                   // its fused gate
  uint16_t off;                    // its column in s_col
  uint8_t w, q[kMaxW];             // its qubits, basis bit b <-> q[b]
};
constexpr uint32_t kTableAmps = 1u << (2 * kMaxW);   // s_mat holds both tables

__device__ __forceinline__ float2 cmul(float2 a, float2 b) {
  return make_float2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}

// factor U_f[x restricted to the qubits of f, 0]
__device__ __forceinline__ float2 fold_factor(const FoldPiece& F, const float2* s_col, uint32_t x) {
  uint32_t idx = 0;
  for (int b = 0; b < F.w; ++b) idx |= ((x >> F.q[b]) & 1u) << b;
  return s_col[F.off + idx];
}

__device__ __noinline__ int cta_product_start(const Dev& d, const Traj& T, float2* psi, uint32_t hi,
                                              float2* s_mat, float2* s_col, FoldPiece* s_fold, MemberList& list) {
  const uint32_t rank = cluster_rank(), nranks = cluster_size();
  __shared__ int s_split, s_nstr;
  __shared__ uint8_t s_str[kMaxN];
  const int tid = threadIdx.x;
  const int n = static_cast<int>(T.n);
  const uint32_t all = (1u << n) - 1u;
  uint32_t touched = 0, held = 0;
  int nf = 0, off = 0;
  // once every qubit is touched no later piece can fold
  for (uint32_t g = 0; g < T.ngates && touched != all; ++g) {
    const Gate G = d.gates[T.gate0 + g];
    if (G.minpos >= hi) continue;
    const uint32_t gm = gate_mask(G);
    const bool fold = !(gm & touched);
    touched |= gm;
    if (!fold) continue;
    const int D = 1 << G.w;
    const float2* col = d.fmat + G.mat;          // column 0 of the precomputed matrix, stride D
    if (G.maxpos >= hi || d.gflag[T.gf0 + g]) {
      cta_compose_piece(d, T, G, 0, hi, -1, 0, 1.f, s_mat, list);
      __syncthreads();
      col = s_mat;
    }
    for (int i = tid; i < D; i += blockDim.x) s_col[off + i] = col[i * D];
    if (tid == 0) {
      FoldPiece& F = s_fold[nf];
      F.mask = gm;
      F.gate = g;
      F.off = static_cast<uint16_t>(off);
      F.w = G.w;
      for (int b = 0; b < G.w; ++b) F.q[b] = G.t[b];
    }
    held |= gm;
    off += D;
    ++nf;
  }
  cluster_sync();                  // every thread has read the gate flags; s_fold is complete
  if (tid < 32) {
    // lane c scores the split at m = c: fewest straddling pieces, then the
    // most even tables, among the splits whose tables fit s_mat
    const int c = tid;
    uint32_t key = 0xffffffffu;
    if (c <= n && (1u << c) + (1u << (n - c)) <= kTableAmps) {
      int str = 0;
      for (int f = 0; f < nf; ++f) str += (s_fold[f].mask & ((1u << c) - 1u)) && (s_fold[f].mask >> c);
      key = (static_cast<uint32_t>(str) << 16) | (static_cast<uint32_t>(abs(2 * c - n)) << 5) |
            static_cast<uint32_t>(c);
    }
    for (int o = 16; o > 0; o >>= 1) key = min(key, __shfl_xor_sync(0xffffffffu, key, o));
    if (tid == 0) {
      const int m = static_cast<int>(key & 31u);
      s_split = m;
      int ns = 0;
      for (int f = 0; f < nf; ++f)
        if ((s_fold[f].mask & ((1u << m) - 1u)) && (s_fold[f].mask >> m)) s_str[ns++] = static_cast<uint8_t>(f);
      s_nstr = ns;
    }
    // mark the folded gates for the pass loop
    if (rank == 0)
      for (int f = tid; f < nf; f += 32) d.gflag[T.gf0 + s_fold[f].gate] = 2;
  }
  __syncthreads();
  const int m = s_split, ns = s_nstr;
  const uint32_t lmask = (1u << m) - 1u, nlo = 1u << m, nhi = 1u << (n - m);
  const uint32_t zero = all & ~held;                 // qubits no folded piece holds stay |0>
  float2* t_lo = s_mat;
  float2* t_hi = s_mat + nlo;
  for (uint32_t y = tid; y < nlo + nhi; y += blockDim.x) {
    const bool upper = y >= nlo;
    const uint32_t x = upper ? (y - nlo) << m : y;   // the index bits this entry stands for
    const uint32_t half = upper ? ~lmask : lmask;
    float2 v = make_float2(0.f, 0.f);
    if (!(x & zero)) {
      v.x = 1.f;
      for (int f = 0; f < nf; ++f)
        if (!(s_fold[f].mask & ~half)) v = cmul(v, fold_factor(s_fold[f], s_col, x));
    }
    if (upper) t_hi[y - nlo] = v;
    else t_lo[y] = v;
  }
  __syncthreads();
  for (uint32_t x = rank * blockDim.x + tid; x < 1u << n; x += nranks * blockDim.x) {
    float2 v = cmul(t_lo[x & lmask], t_hi[x >> m]);
    for (int j = 0; j < ns; ++j) v = cmul(v, fold_factor(s_fold[s_str[j]], s_col, x));
    psi[x] = v;
  }
  cluster_sync();                  // the marks and the state are visible to the cluster
  return nf;
}

// ---------------------------------------------------------------------------
// the persistent kernels
// ---------------------------------------------------------------------------
// Flush points of the trajectory that a CTA works on: channels that stage 1
// leaves undecided, in no order (past kFlushMax they are found in the stage
// records instead).
constexpr int kFlushMax = 64;
struct TrajShared {
  float2 red[16][16];
  double rho[16];
  SampleScratch sample;
  MemberList list;
  unsigned idx;
  int nflush;                       // entries of flush[] (more than kFlushMax: overflowed)
  uint32_t flush[kFlushMax];
  int next;
  float scale;
  int pend_pos, pend_choice;
};

// Stage 1 of every channel from its draw and the lower bounds; fused gates
// that hold a channel with another operator than its default (or an undecided
// one) get their flag, so that the pass loop reads one flag per gate.  Nearly
// every draw takes the first operator, which an integer compare settles.
// Every CTA of a cluster makes its own list of flush points; the first one
// writes the records and flags.
__device__ __forceinline__ void cta_stage1(const Dev& d, const Traj& T, uint64_t seed, uint64_t traj_id, bool lead,
                                           TrajShared& sh) {
  const int tid = threadIdx.x;
  if (lead)
    for (uint32_t g = tid; g < T.ngates; g += blockDim.x) d.gflag[T.gf0 + g] = 0;
  if (tid == 0) { sh.pend_pos = -1; sh.pend_choice = 0; sh.scale = 1.f; sh.nflush = 0; }
  __syncthreads();
#pragma unroll 2
  for (uint32_t c = tid; c < T.nch; c += blockDim.x) {
    const Op op = d.ops[T.op0 + d.ch_op[T.chop0 + c]];
    const Set& st = d.sets[op.set];
    const uint64_t bits = uniform_bits(seed, traj_id, kStreamChannel, c);
    int ch = -1;
    if (bits < st.thr0) {
      ch = 0;
    } else {
      const double* pbar = d.dmat + st.pbar;
      double rr = static_cast<double>(bits) * 0x1.0p-53 - pbar[0];
      for (uint32_t i = 1; i < st.nk; ++i) {
        if (rr < pbar[i]) { ch = static_cast<int>(i); break; }
        rr -= pbar[i];
      }
    }
    if (lead) {
      d.kraus[T.ch0 + c] = static_cast<int8_t>(ch);
      d.stage[T.ch0 + c] = ch >= 0 ? 1 : 0;
      if (ch != static_cast<int>(st.def)) d.gflag[T.gf0 + op.gate] = 1;
    }
    if (ch < 0) {
      const int k = atomicAdd(&sh.nflush, 1);
      if (k < kFlushMax) sh.flush[k] = c;
    }
  }
  __syncthreads();
}

// first flush point at or after channel cur, -1 if there is none
__device__ __forceinline__ int cta_next_flush(const Dev& d, const Traj& T, uint32_t cur, TrajShared& sh) {
  if (threadIdx.x < 32) {
    uint32_t best = 0xffffffffu;
    if (sh.nflush <= kFlushMax) {
      for (int i = threadIdx.x; i < sh.nflush; i += 32)
        if (sh.flush[i] >= cur) best = min(best, sh.flush[i]);
    } else {
      for (uint32_t c = cur + threadIdx.x; c < T.nch; c += 32)
        if (d.stage[T.ch0 + c] == 0) { best = c; break; }
    }
    best = __reduce_min_sync(0xffffffffu, best);
    if (threadIdx.x == 0) sh.next = static_cast<int>(best);
  }
  __syncthreads();
  return sh.next;
}

// Stage 2 at the flush point: op hi, channel fch (Alg. 2 steps 12-20)
template <bool SHARED>
__device__ __noinline__ void cta_stage2(const Dev& d, const Traj& T, const float2* psi, uint32_t hi, int fch, uint64_t seed,
                                        uint64_t traj_id, TrajShared& sh) {
  const Op op = d.ops[T.op0 + hi];
  const Set st = d.sets[op.set];
  const int order[2] = {op.q0, op.q1};
  __syncthreads();
  if (op.q == 1) cta_rdm<1, SHARED>(psi, static_cast<int>(T.n), order, static_cast<int>(d.lthreads), sh.rho, sh.red);
  else cta_rdm<2, SHARED>(psi, static_cast<int>(T.n), order, static_cast<int>(d.lthreads), sh.rho, sh.red);
  if (threadIdx.x == 0) {
    const int D = 1 << op.q;
    double rho[2 * 16];
    int c = 0;
    for (int b = 0; b < D; ++b) { rho[2 * (b * D + b)] = sh.rho[c++]; rho[2 * (b * D + b) + 1] = 0.0; }
    for (int b = 0; b < D; ++b)
      for (int a = b + 1; a < D; ++a) {
        const double re = sh.rho[c++], im = sh.rho[c++];
        rho[2 * (b * D + a)] = re; rho[2 * (b * D + a) + 1] = im;
        rho[2 * (a * D + b)] = re; rho[2 * (a * D + b) + 1] = -im;
      }
    double N = 0.0;
    for (int b = 0; b < D; ++b) N += rho[2 * (b * D + b)];
    const double* pbar = d.dmat + st.pbar;
    double rr = uniform01(seed, traj_id, kStreamChannel, static_cast<uint32_t>(fch));
    for (uint32_t i = 0; i < st.nk; ++i) rr -= pbar[i];
    int chosen = -1, last = -1, last_pos = -1;
    double Pc = 1.0;
    for (uint32_t i = 0; i < st.nk; ++i) {
      const double* M = d.dmat + st.mtm + static_cast<size_t>(i) * D * D * 2;
      double P = 0.0;                                  // tr(M rho)
      for (int a = 0; a < D; ++a)
        for (int b = 0; b < D; ++b) {
          const double mr = M[2 * (a * D + b)], mi2 = M[2 * (a * D + b) + 1];
          const double rr2 = rho[2 * (b * D + a)], ri = rho[2 * (b * D + a) + 1];
          P += mr * rr2 - mi2 * ri;
        }
      double dlt = P / N - pbar[i];
      if (dlt < 0.0) dlt = 0.0;
      if (dlt > 0.0) last = static_cast<int>(i);
      if (P > 0.0) last_pos = static_cast<int>(i);
      if (chosen < 0 && rr < dlt) { chosen = static_cast<int>(i); Pc = P; }
      if (chosen < 0) rr -= dlt;
    }
    if (chosen < 0) {
      chosen = last >= 0 ? last : (last_pos >= 0 ? last_pos : static_cast<int>(st.def));
      const double* M = d.dmat + st.mtm + static_cast<size_t>(chosen) * D * D * 2;
      Pc = 0.0;
      for (int a = 0; a < D; ++a)
        for (int b = 0; b < D; ++b)
          Pc += M[2 * (a * D + b)] * rho[2 * (b * D + a)] - M[2 * (a * D + b) + 1] * rho[2 * (b * D + a) + 1];
    }
    d.kraus[T.ch0 + fch] = static_cast<int8_t>(chosen);
    d.stage[T.ch0 + fch] = 2;
    sh.pend_pos = static_cast<int>(hi);
    sh.pend_choice = chosen;
    sh.scale = static_cast<float>(1.0 / sqrt(Pc > 0.0 ? Pc : 1.0));
  }
  __syncthreads();
}

// the next trajectory of the launch; false when there is none left
__device__ __forceinline__ bool next_trajectory(const Dev& d, TrajShared& sh, uint32_t& ti) {
  __syncthreads();
  if (threadIdx.x == 0) sh.idx = atomicAdd(d.counter, 1u);
  __syncthreads();
  if (sh.idx >= d.num) return false;
  ti = d.order[sh.idx];
  return true;
}

__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"(static_cast<uint32_t>(__cvta_generic_to_shared(dst))), "l"(src)
               : "memory");
}
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// States of at most 2^14 amplitudes, held in the CTA's shared memory.  Passes
// are short (2^n / 2^w sets over a few hundred threads), so what bounds them
// is latency: the CTA is sized to the state (128 threads up to 10 qubits, 256
// up to 13, 512 at 14) so that several trajectories share an SM; a window of
// gate descriptors with what to do about each is brought to shared memory at
// once; and the matrix of the next gate is copied (cp.async, two buffers)
// while this one is applied, which leaves one barrier per gate.
// 1600 trajectories of 8 to 12 qubits, k = 3: 4.14 -> 0.90 ms of device time
// (every state had one CTA of 512 threads per SM before, and each gate fetched
// its descriptor, flag and matrix in turn between two barriers).  Now 40 % of
// the issue slots; 4 CTAs of 256 threads at 64 registers, or CTAs of 128
// threads from 11 qubits on, measured 2-3 % slower.
constexpr int kWindow = 128;        // gates of a descriptor window
enum : uint8_t { kSkip = 0, kDefault = 1, kCompose = 2 };

template <int TB, int MINB>
__global__ void __launch_bounds__(TB, MINB) k_batch_smem(const __grid_constant__ Dev d, uint32_t max_amps) {
  extern __shared__ __align__(16) float2 s_dyn[];
  __shared__ TrajShared sh;
  __shared__ Gate s_gate[kWindow];
  __shared__ uint8_t s_kind[kWindow];
  float2* const psi = s_dyn;
  const uint32_t wbuf = min(d.wmat, 4u);
  float2* const buf = s_dyn + max_amps;                  // two matrices of up to 2^wbuf
  float2* const big = buf + (2u << (2 * wbuf));          // one wider matrix (wmat > 4)
  const int tid = threadIdx.x;
  uint32_t ti;
  while (next_trajectory(d, sh, ti)) {
    const Traj T = d.traj[ti];
    const int n = static_cast<int>(T.n);
    const uint32_t amps = 1u << n;
    const uint64_t seed = d.per_traj ? T.seed : d.run[0];
    const uint64_t traj_id = d.per_traj ? T.tid : d.run[1] + ti;
    const uint32_t S = d.per_traj ? T.S : d.S;
    uint64_t* samples = d.samples + (d.per_traj ? T.soff : static_cast<uint64_t>(ti) * d.S);
    for (uint32_t x = tid; x < amps; x += blockDim.x) psi[x] = make_float2(x == 0 ? 1.f : 0.f, 0.f);   // sw(0) = 0
    cta_stage1(d, T, seed, traj_id, true, sh);
    uint32_t lo = 0, cur_ch = 0, nflush = 0;
    for (;;) {
      const int fch = cta_next_flush(d, T, cur_ch, sh);
      const uint32_t hi = fch >= 0 ? d.ch_op[T.chop0 + fch] : T.nops;
      const int pend_pos = sh.pend_pos, pend_choice = sh.pend_choice;
      const float pend_scale = sh.scale;
      // the channel decided in stage 2 at this segment's start is applied as
      // its normalized Kraus operator, so the gate holding it is never default
      const uint32_t pend_gate = pend_pos >= 0 ? d.ops[T.op0 + pend_pos].gate : 0xffffffffu;
      // apply ops [lo, hi): fused gates restricted to the segment
      for (uint32_t g0 = 0; g0 < T.ngates; g0 += kWindow) {
        const int cnt = static_cast<int>(min(T.ngates - g0, static_cast<uint32_t>(kWindow)));
        __syncthreads();                                 // the previous window and its buffers are done with
        for (int i = tid; i < cnt; i += TB) {
          const Gate G = d.gates[T.gate0 + g0 + i];
          uint8_t kind = kSkip;
          if (G.maxpos >= lo && G.minpos < hi)
            kind = G.minpos >= lo && G.maxpos < hi && !d.gflag[T.gf0 + g0 + i] && g0 + i != pend_gate ? kDefault : kCompose;
          s_gate[i] = G;
          s_kind[i] = kind;
        }
        __syncthreads();
        auto next_active = [&](int g) {
          while (g < cnt && s_kind[g] == kSkip) ++g;
          return g;
        };
        auto prefetch = [&](int g, int b) {              // a default gate's matrix into buffer b
          if (g < cnt && s_kind[g] == kDefault && s_gate[g].w <= 4) {
            const float2* src = d.fmat + s_gate[g].mat;
            float2* dst = buf + (static_cast<uint32_t>(b) << (2 * wbuf));
            const int words = 1 << (2 * s_gate[g].w - 1);
            for (int i = tid; i < words; i += TB) cp_async16(dst + 2 * i, src + 2 * i);
          }
        };
        int g = next_active(0), b = 0;
        prefetch(g, 0);
        while (g < cnt) {
          const int w = s_gate[g].w;
          float2* A = w <= 4 ? buf + (static_cast<uint32_t>(b) << (2 * wbuf)) : big;
          if (s_kind[g] == kCompose) {
            // a piece that is cut by the segment or holds a non-default operator:
            // its members in [lo, hi) as one matrix over the gate's qubits
            const Gate G = s_gate[g];
            cta_compose_piece(d, T, G, lo, hi, pend_pos, pend_choice, pend_scale, A, sh.list);
          } else if (w > 4) {
            __syncthreads();
            const float2* src = d.fmat + s_gate[g].mat;
            for (int i = tid; i < 1 << (2 * w); i += TB) A[i] = src[i];
          } else {
            cp_async_wait();
          }
          __syncthreads();                               // the matrix is there; the previous pass is complete
          const int nx = next_active(g + 1);
          prefetch(nx, b ^ 1);
          const uint8_t* t = s_gate[g].t;
          switch (w) {
            case 1: smem_apply<1>(psi, n, t, A); break;
            case 2: smem_apply<2>(psi, n, t, A); break;
            case 3: smem_apply<3>(psi, n, t, A); break;
            case 4: smem_apply<4>(psi, n, t, A); break;
            default: {
              int order[kMaxW];
              for (int k = 0; k < w; ++k) order[k] = t[k];
              if (w == 5) cta_apply_wide<5, true>(psi, n, order, A, tid, blockDim.x);
              else cta_apply_wide<6, true>(psi, n, order, A, tid, blockDim.x);
            }
          }
          g = nx;
          b ^= 1;
        }
      }
      if (fch < 0) break;
      cta_stage2<true>(d, T, psi, hi, fch, seed, traj_id, sh);
      ++nflush;
      lo = hi;
      cur_ch = static_cast<uint32_t>(fch) + 1;
    }
    __syncthreads();
    if (S) cta_sample<true>(psi, n, seed, traj_id, S, samples, static_cast<int>(d.lthreads), sh.sample);
    if (d.keep)
      for (uint32_t x = tid; x < amps; x += blockDim.x) d.arena[T.arena_off + x] = psi[sw(x)];
    if (tid == 0) {
      d.flushes[ti] = nflush;
      if (d.folds) d.folds[ti] = 0;
    }
  }
}

// Larger states (2^15..2^20 amplitudes), each in its cluster's slot of global
// memory (a cluster is one CTA in a batch with trajectories enough, see
// glob_cluster).  One pass per gate was bound by the latency and traffic of
// the slot (156 us a pass at 18 qubits, 13 bytes a clock and SM), so
// consecutive gates share a sweep: in circuit order, gates are taken as long
// as their qubits and the lowest kTileLow ones number at most kTileBits.  A
// sweep brings the state tile by tile (2^13 amplitudes over the group's
// qubits, rows of at least 128 bytes, cp.async) to shared memory, applies
// every gate of the group and writes the tile back.  At 18 qubits and k = 3
// that is about 43 sweeps for 164 gates; what bounds it now is the tile's
// arithmetic and the shared-memory reads that feed it (4700 clocks a gate and
// tile, of which the FMAs take 2050).  Gates keep their order and an amplitude
// its operations: states and samples are those of one pass per gate, bit for
// bit.  660 trajectories of 8 to 18 qubits: 21.2 -> 11.3 ms (18.8 with one
// CTA per trajectory and both halves of it on one tile).
constexpr int kTileBits = 13, kTileLow = 4;
constexpr int kTileSets = 32;                              // members a thread holds
constexpr int kGroupGates = 16, kGroupEntries = 1024;      // matrices of a sweep: at most 1024 entry pairs
constexpr int kTileChunks = 1 << (kTileBits - 1);          // 16-byte chunks of a tile

// place of amplitude x of a staged tile: as sw, but whole 16-byte chunks move
__device__ __forceinline__ uint32_t sw16(uint32_t x) { return x ^ ((sw(x) ^ x) & 14u); }

// the set bits of `mask`, ascending, receive the low bits of x
__device__ __forceinline__ uint32_t deposit(uint32_t x, uint32_t mask) {
  uint32_t r = 0;
  for (uint32_t m = mask; m; m &= m - 1, x >>= 1)
    if (x & 1u) r |= m & (0u - m);
  return r;
}

struct Sweep {
  uint8_t gate[kGroupGates], w[kGroupGates], pos[kGroupGates][4];   // window index, width, tile positions
  uint16_t mat[kGroupGates];                                        // first entry of its matrix
  uint16_t member[kGroupGates][16], step[kGroupGates][8];           // places of member m and of a thread's set b
  int ng;
  uint32_t tile, rest;                                              // qubit masks
  uint32_t off[64], place[64];                                      // per chunk step: memory and tile offset
};

// sets of a w-qubit gate that a thread takes at once
__host__ __device__ constexpr int tile_sets(int w) { return kTileSets >> w > 8 ? 8 : kTileSets >> w; }

// psi <- A psi on a staged tile.  A shared-memory read returns 128 bytes a
// clock however many lanes ask for the same word, so a matrix entry read for
// one set costs as much as its FMAs: a thread takes B sets (32 / 2^W of them,
// 128 registers of members) and two rows at a time.  M4 entry (row pair, m) is
// (Re, Re, Im, Im) of the two rows, the members are held doubled, and packed
// FMAs sum P = sum Re v and Q = sum Im v for both rows; the outputs are
// (P.x - Q.y, P.y + Q.x).
template <int W>
__device__ __forceinline__ void tile_apply(float2* tile, const Sweep& g, int k, const float4* M4, int tid, int nt) {
  constexpr int D = 1 << W, B = tile_sets(W);
  int p[W];
  uint32_t off[D], step[B];
#pragma unroll
  for (int b = 0; b < W; ++b) p[b] = g.pos[k][b];
#pragma unroll
  for (int m = 0; m < D; ++m) off[m] = g.member[k][m];
#pragma unroll
  for (int b = 0; b < B; ++b) step[b] = g.step[k][b];
  constexpr uint32_t sets = 1u << (kTileBits - W);
  for (uint32_t s0 = tid; s0 < sets; s0 += B * nt) {       // sets is a multiple of B nt
    const uint32_t first = sw16(insert_zeros32(s0, W, p));
    uint32_t base[B];
    float2 vx[B][D], vy[B][D];
#pragma unroll
    for (int b = 0; b < B; ++b) {
      base[b] = first ^ step[b];
#pragma unroll
      for (int m = 0; m < D; ++m) {
        const float2 v = tile[base[b] ^ off[m]];
        vx[b][m] = make_float2(v.x, v.x);
        vy[b][m] = make_float2(v.y, v.y);
      }
    }
#pragma unroll 1
    for (int j = 0; j < D; j += 2) {
      float2 px[B], py[B], qx[B], qy[B];
#pragma unroll
      for (int b = 0; b < B; ++b) px[b] = py[b] = qx[b] = qy[b] = make_float2(0.f, 0.f);
#pragma unroll
      for (int m = 0; m < D; ++m) {
        const float4 a = M4[(j >> 1) * D + m];
        const float2 re = make_float2(a.x, a.y), im = make_float2(a.z, a.w);
#pragma unroll
        for (int b = 0; b < B; ++b) {
          px[b] = __ffma2_rn(re, vx[b][m], px[b]);
          py[b] = __ffma2_rn(re, vy[b][m], py[b]);
          qx[b] = __ffma2_rn(im, vx[b][m], qx[b]);
          qy[b] = __ffma2_rn(im, vy[b][m], qy[b]);
        }
      }
      const uint32_t o0 = g.member[k][j], o1 = g.member[k][j + 1];
#pragma unroll
      for (int b = 0; b < B; ++b) {
        tile[base[b] ^ o0] = make_float2(px[b].x - qy[b].x, py[b].x + qx[b].x);
        tile[base[b] ^ o1] = make_float2(px[b].y - qy[b].y, py[b].y + qx[b].y);
      }
    }
  }
}

__device__ __forceinline__ void cp_async16_l2(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(static_cast<uint32_t>(__cvta_generic_to_shared(dst))), "l"(src)
               : "memory");
}

// One sweep over the state: the group's matrices are in place.  Each half of
// the CTA stages and works on tiles of its own (named barriers), so that one
// half's copies, gathers and barriers pass under the other's arithmetic; the
// tiles are dealt to the halves of all the cluster's CTAs.
__device__ __noinline__ void cta_sweep(float2* __restrict__ psi, int n, float2* tiles, const float4* mats, const Sweep& g) {
  const int half = threadIdx.x >= blockDim.x / 2, gs = blockDim.x / 2, tid = threadIdx.x - half * gs;
  const int steps = kTileChunks / gs;
  const uint32_t my_off = deposit(2u * tid, g.tile), my_place = sw16(2u * tid), rest = g.rest;
  const int ntiles = 1 << (n - kTileBits);
  float2* const tile = tiles + (half << kTileBits);
  auto sync = [&] { asm volatile("bar.sync %0, %1;" ::"r"(1 + half), "r"(gs) : "memory"); };
  for (int t = cluster_rank() * 2 + half; t < ntiles; t += cluster_size() * 2) {
    float2* const mem = psi + (deposit(t, rest) | my_off);
#pragma unroll 4
    for (int i = 0; i < steps; ++i) cp_async16_l2(tile + (my_place ^ g.place[i]), mem + g.off[i]);
    cp_async_wait();
    sync();
    for (int i = 0; i < g.ng; ++i) {
      const float4* const M4 = mats + g.mat[i];
      switch (g.w[i]) {
        case 1: tile_apply<1>(tile, g, i, M4, tid, gs); break;
        case 2: tile_apply<2>(tile, g, i, M4, tid, gs); break;
        case 3: tile_apply<3>(tile, g, i, M4, tid, gs); break;
        default: tile_apply<4>(tile, g, i, M4, tid, gs); break;
      }
      sync();
    }
#pragma unroll 4
    for (int i = 0; i < steps; ++i)
      *reinterpret_cast<float4*>(mem + g.off[i]) = *reinterpret_cast<const float4*>(tile + (my_place ^ g.place[i]));
    // this thread's own chunks are in its registers: the next copies may overwrite
    // them, and no one else reads this tile before the next barrier
  }
}

constexpr int kGlobThreads = 256;

__global__ void __launch_bounds__(kGlobThreads) k_batch_glob(const __grid_constant__ Dev d) {
  extern __shared__ __align__(16) float2 s_dyn[];
  float2* const tiles = s_dyn;                      // two staged tiles; between sweeps, one matrix of up to
  float2* const s_mat = s_dyn;                      // 64 x 64 or the product-state tables
  float4* const mats = reinterpret_cast<float4*>(s_dyn + (2u << kTileBits));   // the sweep's matrices
  __shared__ TrajShared sh;
  __shared__ Gate s_gate[kWindow];
  __shared__ uint8_t s_kind[kWindow];
  __shared__ Sweep s_sweep;
  __shared__ float2 s_col[kFoldCols];               // columns U[:, 0] of the folded pieces
  __shared__ FoldPiece s_fold[kMaxN];
  const int tid = threadIdx.x, nt = blockDim.x;
  const bool lead = cluster_rank() == 0;
  for (;;) {
    cluster_sync();                                 // the previous trajectory is done with
    if (lead && tid == 0) sh.idx = atomicAdd(d.counter, 1u);
    cluster_sync();
    const uint32_t idx = leader_word(&sh.idx);
    if (idx >= d.num) break;
    const uint32_t ti = d.order[idx];
    const Traj T = d.traj[ti];
    const int n = static_cast<int>(T.n);
    const uint64_t seed = d.per_traj ? T.seed : d.run[0];
    const uint64_t traj_id = d.per_traj ? T.tid : d.run[1] + ti;
    const uint32_t S = d.per_traj ? T.S : d.S;
    uint64_t* samples = d.samples + (d.per_traj ? T.soff : static_cast<uint64_t>(ti) * d.S);
    float2* psi = d.keep ? d.arena + T.arena_off : d.arena + blockIdx.x / cluster_size() * d.slot_amps;
    cta_stage1(d, T, seed, traj_id, lead, sh);
    cluster_sync();                                 // the records and flags are there
    uint32_t lo = 0, cur_ch = 0, nflush = 0;
    for (;;) {
      const int fch = cta_next_flush(d, T, cur_ch, sh);
      const uint32_t hi = fch >= 0 ? d.ch_op[T.chop0 + fch] : T.nops;
      const int pend_pos = sh.pend_pos, pend_choice = sh.pend_choice;
      const float pend_scale = sh.scale;
      const uint32_t pend_gate = pend_pos >= 0 ? d.ops[T.op0 + pend_pos].gate : 0xffffffffu;
      const bool first = lo == 0 && nflush == 0;
      if (first) {
        const int nf = cta_product_start(d, T, psi, hi, s_mat, s_col, s_fold, sh.list);
        if (lead && tid == 0 && d.folds) d.folds[ti] = static_cast<uint32_t>(nf);
      }
      // apply ops [lo, hi): fused gates restricted to the segment (in the
      // first segment, those not folded into the initial state)
      for (uint32_t g0 = 0; g0 < T.ngates; g0 += kWindow) {
        const int cnt = static_cast<int>(min(T.ngates - g0, static_cast<uint32_t>(kWindow)));
        __syncthreads();                                 // the previous window is done with
        for (int i = tid; i < cnt; i += nt) {
          const Gate G = d.gates[T.gate0 + g0 + i];
          const uint8_t flag = d.gflag[T.gf0 + g0 + i];
          uint8_t kind = kSkip;
          if (G.maxpos >= lo && G.minpos < hi && !(first && flag == 2))
            kind = G.minpos >= lo && G.maxpos < hi && !flag && g0 + i != pend_gate ? kDefault : kCompose;
          s_gate[i] = G;
          s_kind[i] = kind;
        }
        __syncthreads();
        for (int g = 0; g < cnt;) {
          if (s_kind[g] == kSkip) { ++g; continue; }
          if (s_gate[g].w > 4) {                         // a pass of its own
            const Gate G = s_gate[g];
            const float2* A = d.fmat + G.mat;
            if (s_kind[g] == kCompose) {
              cta_compose_piece(d, T, G, lo, hi, pend_pos, pend_choice, pend_scale, s_mat, sh.list);
              A = s_mat;
            }
            cta_apply_wide_glob(psi, n, G, A, s_mat);
            cluster_sync();
            ++g;
            continue;
          }
          // the group: every thread walks the same descriptors
          uint32_t mask = (1u << kTileLow) - 1u;
          int ng = 0, entries = 0, end = g;
          for (; end < cnt; ++end) {
            if (s_kind[end] == kSkip) continue;
            const int w = s_gate[end].w;
            if (w > 4 || ng == kGroupGates || entries + (1 << (2 * w - 1)) > kGroupEntries) break;
            const uint32_t m = mask | gate_mask(s_gate[end]);
            if (__popc(m) > kTileBits) break;
            mask = m;
            entries += 1 << (2 * w - 1);
            ++ng;
          }
          for (uint32_t q = 0; __popc(mask) < kTileBits; ++q) mask |= 1u << q;   // n >= 15: enough qubits
          __syncthreads();
          if (tid == 0) {
            int k = 0, e = 0;
            for (int i = g; i < end; ++i) {
              if (s_kind[i] == kSkip) continue;
              const int w = s_gate[i].w;
              s_sweep.gate[k] = static_cast<uint8_t>(i);
              s_sweep.w[k] = static_cast<uint8_t>(w);
              for (int b = 0; b < w; ++b)
                s_sweep.pos[k][b] = static_cast<uint8_t>(__popc(mask & ((1u << s_gate[i].t[b]) - 1u)));
              s_sweep.mat[k] = static_cast<uint16_t>(e);
              e += 1 << (2 * w - 1);
              ++k;
            }
            s_sweep.ng = ng;
            s_sweep.tile = mask;
            s_sweep.rest = ((1u << n) - 1u) & ~mask;
          }
          if (tid >= 64 && tid < 128) {
            const uint32_t l = static_cast<uint32_t>(nt) * (tid - 64);   // 2 x (nt / 2) threads of a half
            s_sweep.off[tid - 64] = deposit(l, mask);
            s_sweep.place[tid - 64] = sw16(l);
          }
          __syncthreads();
          for (int x = tid; x < ng * 24; x += nt) {      // 16 members, 8 sets a gate
            const int k = x / 24, e = x % 24, w = s_sweep.w[k];
            int p[4];
            for (int b = 0; b < w; ++b) p[b] = s_sweep.pos[k][b];
            if (e < 16) {
              uint32_t o = 0;
              for (int b = 0; b < w; ++b)
                if ((e >> b) & 1) o |= 1u << p[b];
              s_sweep.member[k][e] = static_cast<uint16_t>(sw16(o));
            } else {
              s_sweep.step[k][e - 16] =
                  static_cast<uint16_t>(sw16(insert_zeros32(static_cast<uint32_t>((e - 16) * (nt / 2)), w, p)));
            }
          }
          for (int k = 0; k < ng; ++k) {
            const int i = s_sweep.gate[k], w = s_sweep.w[k];
            float4* const M4 = mats + s_sweep.mat[k];
            const float2* A = d.fmat + s_gate[i].mat;
            if (s_kind[i] == kCompose) {
              const Gate G = s_gate[i];
              cta_compose_piece(d, T, G, lo, hi, pend_pos, pend_choice, pend_scale, s_mat, sh.list);
              __syncthreads();
              A = s_mat;
            }
            for (int x = tid; x < 1 << (2 * w - 1); x += nt) {
              const int r = (x >> w) << (w + 1) | (x & ((1 << w) - 1));   // row 2 (x >> w), column x mod 2^w
              const float2 a0 = A[r], a1 = A[r + (1 << w)];
              M4[x] = make_float4(a0.x, a1.x, a0.y, a1.y);
            }
          }
          __syncthreads();                               // matrices complete, s_mat free for the tiles
          cta_sweep(psi, n, tiles, mats, s_sweep);
          cluster_sync();                                // the sweep is complete, and done with its shared memory
          g = end;
        }
      }
      if (fch < 0) break;
      if (lead) cta_stage2<false>(d, T, psi, hi, fch, seed, traj_id, sh);
      cluster_sync();
      if (!lead && tid == 0) {
        sh.pend_pos = static_cast<int>(leader_word(&sh.pend_pos));
        sh.pend_choice = static_cast<int>(leader_word(&sh.pend_choice));
        sh.scale = __uint_as_float(leader_word(&sh.scale));
      }
      ++nflush;
      lo = hi;
      cur_ch = static_cast<uint32_t>(fch) + 1;
    }
    if (lead && S) cta_sample<false>(psi, n, seed, traj_id, S, samples, static_cast<int>(d.lthreads), sh.sample);
    if (lead && tid == 0) d.flushes[ti] = nflush;
  }
  cluster_sync();                                   // no CTA leaves while its shared memory may be read
}

}  // namespace bt

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
namespace {

uint64_t fnv1a(const void* p, size_t n, uint64_t h = 1469598103934665603ull) {
  const uint8_t* b = static_cast<const uint8_t*>(p);
  for (size_t i = 0; i < n; ++i) { h ^= b[i]; h *= 1099511628211ull; }
  return h;
}

// a distinct operator set (gate or channel)
struct SetKey {
  uint64_t h;
  const Op* op;
};

bool same_set(const Op& a, const Op& b) {
  if (a.kind != b.kind || a.q != b.q || a.num_ops != b.num_ops) return false;
  if (a.mats.size() != b.mats.size() || std::memcmp(a.mats.data(), b.mats.data(), sizeof(cd) * a.mats.size()) != 0)
    return false;
  if (a.probs.size() != b.probs.size()) return false;
  return a.probs.empty() || std::memcmp(a.probs.data(), b.probs.data(), sizeof(double) * a.probs.size()) == 0;
}

uint64_t set_hash(const Op& op) {
  uint64_t h = fnv1a(&op.kind, sizeof(op.kind));
  h = fnv1a(&op.q, sizeof(op.q), h);
  h = fnv1a(op.mats.data(), sizeof(cd) * op.mats.size(), h);
  if (!op.probs.empty()) h = fnv1a(op.probs.data(), sizeof(double) * op.probs.size(), h);
  return h;
}

}  // namespace

struct DevMem {
  void* p = nullptr;
  size_t bytes = 0;
  ~DevMem() { if (p) cudaFree(p); }
  bool alloc(size_t b) {
    if (p) cudaFree(p);
    p = nullptr;
    bytes = 0;                               // until there is memory: callers keep a buffer that is large enough
    if (b == 0) return true;
    if (cudaMalloc(&p, b) != cudaSuccess) { cudaGetLastError(); p = nullptr; return false; }
    bytes = b;
    return true;
  }
};

}  // namespace qt

using namespace qt;

struct qt_batch {
  uint32_t num = 0;
  uint32_t total_ch = 0;
  uint64_t total_amps = 0;
  uint32_t max_n = 0;
  std::vector<bt::Traj> traj;
  std::vector<uint32_t> order;
  DevMem tables, arena, outs, counter;
  uint64_t* hrun = nullptr;         // pinned {seed, first_traj}; the graph copies it to counter+32
  bt::Dev dev{};
  size_t off_kraus = 0, off_stage = 0, off_samples = 0, off_flushes = 0, off_folds = 0, off_err = 0, off_gflag = 0;
  uint64_t total_gates = 0;         // sum of the trajectories' fused-gate counts (one flag each per run)
  uint32_t S = 0, keep = 0;
  std::vector<uint8_t> host;        // host image of the device tables
  uint64_t lane_samples = 0;        // merged launches: total sample slots
  qt_batch_params last{};
  // results on the host
  std::vector<int8_t> kraus, stage;
  std::vector<uint64_t> samples;
  std::vector<uint32_t> flushes, folds;
  double device_ms = 0.0;
  uint64_t gate_ops = 0, fused_gates = 0;
  // Classes of trajectories by state size, largest first as in `order`: states
  // in global memory (n > 14), then shared-memory states of 14, 13, 11..12 and
  // up to 10 qubits.  Each is one persistent launch, on streams of their own so
  // that their CTAs share the SMs.
  uint32_t count[bt::kClasses] = {}, wmat[bt::kClasses] = {}, top_n[bt::kClasses] = {};
  cudaStream_t side[bt::kClasses - 1] = {};
  cudaEvent_t ev_fork = nullptr, ev_join[bt::kClasses - 1] = {};
  // CUDA graph of the launch sequence
  cudaGraphExec_t gexec = nullptr;
  cudaGraph_t graph = nullptr;
  uint32_t g_threads = 0, g_threads_glob = 0, g_S = 0, g_keep = 0;
  ~qt_batch() {
    if (gexec) cudaGraphExecDestroy(gexec);
    if (graph) cudaGraphDestroy(graph);
    if (hrun) cudaFreeHost(hrun);
    if (ev_fork) cudaEventDestroy(ev_fork);
    for (auto e : ev_join)
      if (e) cudaEventDestroy(e);
    for (auto st : side)
      if (st) cudaStreamDestroy(st);
  }
};

// Pack num fused circuits (trajectory i runs fused[i]) into B's host fields
// and device tables: B->tables grows when the image does not fit, and the
// image is copied with cudaMemcpyAsync on st (the call returns once the
// pageable source has been staged).  per (optional): per-trajectory seed,
// trajectory id and sample count of a merged launch.
static qt_status pack_batch(qt_batch* B, uint32_t num, const qt_fused* const* fused, const LaneTraj* per,
                            const char* who, cudaStream_t st) {
  B->num = num;
  B->total_ch = 0;
  B->total_amps = 0;
  B->max_n = 0;
  for (int c = 0; c < bt::kClasses; ++c) B->count[c] = B->wmat[c] = B->top_n[c] = 0;
  B->total_gates = 0;
  B->gate_ops = 0;
  B->fused_gates = 0;
  B->traj.assign(num, bt::Traj{});
  // ---- per-circuit checks and distinct operator sets ----
  std::unordered_map<uint64_t, std::vector<uint32_t>> set_index;
  std::vector<const Op*> sets;
  std::vector<bt::Op> ops;
  std::vector<bt::Gate> gates;
  std::vector<uint32_t> members, ch_op;
  std::vector<float2> fmat;
  std::vector<double> dmat;
  std::vector<uint32_t> set_fmat, set_kraus, set_mtm, set_pbar;
  // a fused circuit that appears several times (e.g. many trajectories of one
  // request) is packed once; its trajectories share the tables
  std::unordered_map<const qt_fused*, uint32_t> first_use;
  std::vector<uint32_t> widest(num, 1);               // widest fused gate of each trajectory's circuit
  for (uint32_t i = 0; i < num; ++i) {
    const qt_fused* f = fused[i];
    if (!f) return set_error(QT_ERR_INVALID_ARG, "%s: fused %u is NULL", who, i);
    auto seen = first_use.find(f);
    if (seen != first_use.end()) {
      const bt::Traj& P = B->traj[seen->second];
      bt::Traj& T = B->traj[i];
      T = P;
      T.ch0 = B->total_ch;                 // outputs and per-run flags are per trajectory
      B->total_ch += T.nch;
      T.gf0 = static_cast<uint32_t>(B->total_gates);
      B->total_gates += T.ngates;
      B->gate_ops += f->gate_ops;
      widest[i] = widest[seen->second];
      continue;
    }
    first_use.emplace(f, i);
    const Circuit& c = *f->c;
    if (c.n > static_cast<uint32_t>(bt::kMaxN) || c.n < 1)
      return set_error(QT_ERR_UNSUPPORTED, "%s: circuit %u has %u qubits (batched form: 1..%d)", who, i, c.n,
                       bt::kMaxN);
    bt::Traj& T = B->traj[i];
    T.n = c.n;
    T.op0 = static_cast<uint32_t>(ops.size());
    T.nops = static_cast<uint32_t>(c.ops.size());
    T.ch0 = B->total_ch;
    T.chop0 = static_cast<uint32_t>(ch_op.size());
    T.nch = static_cast<uint32_t>(c.channel_op.size());
    T.gate0 = static_cast<uint32_t>(gates.size());
    T.ngates = static_cast<uint32_t>(f->gates.size());
    T.gf0 = static_cast<uint32_t>(B->total_gates);
    B->total_gates += T.ngates;
    B->total_ch += T.nch;
    B->max_n = std::max(B->max_n, c.n);
    std::vector<uint32_t> local_sets;   // set ids by op
    // within-circuit cache: consecutive ops mostly repeat a handful of sets
    std::vector<std::pair<const Op*, uint32_t>> recent;
    for (uint32_t oi = 0; oi < c.ops.size(); ++oi) {
      const Op& op = c.ops[oi];
      if (op.q > 2) return set_error(QT_ERR_UNSUPPORTED, "%s: circuit %u op %u has %u qubits (batched form: <= 2)", who, i, oi, op.q);
      uint32_t sid = UINT32_MAX;
      for (auto& r : recent)
        if (same_set(*r.first, op)) { sid = r.second; break; }
      if (sid == UINT32_MAX) {
        const uint64_t h = set_hash(op);
        auto& bucket = set_index[h];
        for (uint32_t cand : bucket)
          if (same_set(*sets[cand], op)) { sid = cand; break; }
        if (sid == UINT32_MAX) {
          sid = static_cast<uint32_t>(sets.size());
          sets.push_back(&op);
          bucket.push_back(sid);
        }
        recent.emplace_back(&op, sid);
        if (recent.size() > 16) recent.erase(recent.begin());
      }
      bt::Op o{};
      o.kind = static_cast<uint8_t>(op.kind);
      o.q = static_cast<uint8_t>(op.q);
      o.q0 = static_cast<uint8_t>(op.qubits[0]);
      o.q1 = static_cast<uint8_t>(op.q > 1 ? op.qubits[1] : 0);
      o.set = sid;
      o.channel = op.channel;
      ops.push_back(o);
      if (op.channel >= 0) ch_op.push_back(oi);
      if (op.kind == QT_OP_GATE) B->gate_ops++;
    }
    for (uint32_t oi = 0; oi < c.ops.size(); ++oi) ops[T.op0 + oi].gate = f->gate_of_op[oi];
    for (const FusedGate& fg : f->gates) {
      if (fg.targets.size() > static_cast<size_t>(bt::kMaxW))
        return set_error(QT_ERR_UNSUPPORTED, "%s: fused width %zu > %d in circuit %u", who, fg.targets.size(),
                         bt::kMaxW, i);
      bt::Gate g{};
      g.w = static_cast<uint8_t>(fg.targets.size());
      widest[i] = std::max<uint32_t>(widest[i], g.w);
      for (size_t b = 0; b < fg.targets.size(); ++b) g.t[b] = static_cast<uint8_t>(fg.targets[b]);
      g.mat = static_cast<uint32_t>(fmat.size());
      for (const cd& x : fg.def) fmat.push_back(make_float2(static_cast<float>(x.real()), static_cast<float>(x.imag())));
      g.mem0 = static_cast<uint32_t>(members.size());
      g.nmem = static_cast<uint32_t>(fg.members.size());
      g.minpos = UINT32_MAX;
      g.maxpos = 0;
      for (uint32_t m : fg.members) {
        members.push_back(m);
        g.minpos = std::min(g.minpos, m);
        g.maxpos = std::max(g.maxpos, m);
      }
      gates.push_back(g);
      B->fused_gates++;
    }
    if (fmat.size() > 0x7fffffffu) return set_error(QT_ERR_UNSUPPORTED, "%s: matrix table too large", who);
  }
  // operator-set tables
  std::vector<bt::Set> dsets(sets.size());
  for (size_t s = 0; s < sets.size(); ++s) {
    const Op& op = *sets[s];
    bt::Set& S = dsets[s];
    S.nk = op.num_ops;
    S.q = op.q;
    S.def = static_cast<uint32_t>(op.def);
    S.mat = static_cast<uint32_t>(fmat.size());
    for (const cd& x : op.mats) fmat.push_back(make_float2(static_cast<float>(x.real()), static_cast<float>(x.imag())));
    S.kraus = static_cast<uint32_t>(fmat.size());
    const std::vector<cd>& kr = op.kind == QT_OP_GATE ? op.mats : op.kraus;
    for (const cd& x : kr) fmat.push_back(make_float2(static_cast<float>(x.real()), static_cast<float>(x.imag())));
    S.mtm = static_cast<uint32_t>(dmat.size());
    for (const cd& x : op.mtm) { dmat.push_back(x.real()); dmat.push_back(x.imag()); }
    S.pbar = static_cast<uint32_t>(dmat.size());
    for (double p : op.pbar) dmat.push_back(p);
    if (op.pbar.empty()) dmat.push_back(0.0);
    // u01 = bits * 2^-53 exactly, so bits * 2^-53 < p is bits < ceil(p 2^53)
    const double p0 = op.pbar.empty() ? 0.0 : op.pbar[0];
    S.thr0 = p0 > 0.0 ? static_cast<uint64_t>(std::ceil(std::min(p0, 1.0) * 0x1.0p53)) : 0;
  }
  // processing order: largest states first
  B->order.resize(num);
  for (uint32_t i = 0; i < num; ++i) B->order[i] = i;
  std::stable_sort(B->order.begin(), B->order.end(),
                   [&](uint32_t a, uint32_t b) { return B->traj[a].n > B->traj[b].n; });
  uint64_t soff = 0;
  for (uint32_t i = 0; i < num; ++i) {
    bt::Traj& T = B->traj[i];
    T.arena_off = B->total_amps;
    B->total_amps += 1ull << T.n;
    const int cls = bt::class_of(T.n);
    B->count[cls]++;
    B->top_n[cls] = std::max(B->top_n[cls], T.n);
    B->wmat[cls] = std::max(B->wmat[cls], widest[i]);
    T.seed = per ? per[i].seed : 0;
    T.tid = per ? per[i].traj : 0;
    T.S = per ? per[i].S : 0;
    T.soff = soff;
    soff += T.S;
  }
  B->lane_samples = soff;
  // ---- one device buffer for all tables ----
  auto align = [](size_t x) { return (x + 255) & ~size_t(255); };
  size_t off = 0;
  const size_t o_traj = off; off = align(off + sizeof(bt::Traj) * num);
  const size_t o_ops = off; off = align(off + sizeof(bt::Op) * ops.size());
  const size_t o_sets = off; off = align(off + sizeof(bt::Set) * dsets.size());
  const size_t o_gates = off; off = align(off + sizeof(bt::Gate) * std::max<size_t>(gates.size(), 1));
  const size_t o_mem = off; off = align(off + sizeof(uint32_t) * std::max<size_t>(members.size(), 1));
  const size_t o_chop = off; off = align(off + sizeof(uint32_t) * std::max<size_t>(ch_op.size(), 1));
  const size_t o_fmat = off; off = align(off + sizeof(float2) * fmat.size());
  const size_t o_dmat = off; off = align(off + sizeof(double) * std::max<size_t>(dmat.size(), 1));
  const size_t o_order = off; off = align(off + sizeof(uint32_t) * num);
  if (B->tables.bytes < off && !B->tables.alloc(off))
    return set_error(QT_ERR_OUT_OF_MEMORY, "%s: device tables (%zu bytes)", who, off);
  std::vector<uint8_t>& host = B->host;
  host.assign(off, 0);
  auto put = [&](size_t o, const void* src, size_t n) { if (n) std::memcpy(host.data() + o, src, n); };
  put(o_traj, B->traj.data(), sizeof(bt::Traj) * num);
  put(o_ops, ops.data(), sizeof(bt::Op) * ops.size());
  put(o_sets, dsets.data(), sizeof(bt::Set) * dsets.size());
  put(o_gates, gates.data(), sizeof(bt::Gate) * gates.size());
  put(o_mem, members.data(), sizeof(uint32_t) * members.size());
  put(o_chop, ch_op.data(), sizeof(uint32_t) * ch_op.size());
  put(o_fmat, fmat.data(), sizeof(float2) * fmat.size());
  put(o_dmat, dmat.data(), sizeof(double) * dmat.size());
  put(o_order, B->order.data(), sizeof(uint32_t) * num);
  cudaError_t e = cudaMemcpyAsync(B->tables.p, host.data(), off, cudaMemcpyHostToDevice, st);
  if (e != cudaSuccess) return set_error(QT_ERR_CUDA, "%s: cudaMemcpyAsync: %s", who, cudaGetErrorString(e));
  uint8_t* base = static_cast<uint8_t*>(B->tables.p);
  bt::Dev& d = B->dev;
  d.traj = reinterpret_cast<const bt::Traj*>(base + o_traj);
  d.ops = reinterpret_cast<const bt::Op*>(base + o_ops);
  d.sets = reinterpret_cast<const bt::Set*>(base + o_sets);
  d.gates = reinterpret_cast<const bt::Gate*>(base + o_gates);
  d.members = reinterpret_cast<const uint32_t*>(base + o_mem);
  d.ch_op = reinterpret_cast<const uint32_t*>(base + o_chop);
  d.fmat = reinterpret_cast<const float2*>(base + o_fmat);
  d.dmat = reinterpret_cast<const double*>(base + o_dmat);
  d.order = reinterpret_cast<const uint32_t*>(base + o_order);
  d.num = num;
  return QT_OK;
}

// counters, pinned run parameters, and the side streams of the classes
static qt_status init_batch_runtime(qt_batch* B, const char* who) {
  bt::Dev& d = B->dev;
  // work counters of the launches (4 B each, 28 B), error flag (4 B), run parameters at +32 (2 x 8 B)
  if (!B->counter.alloc(48)) return set_error(QT_ERR_OUT_OF_MEMORY, "%s: counter", who);
  d.counter = static_cast<unsigned int*>(B->counter.p);
  d.err = reinterpret_cast<int*>(static_cast<unsigned int*>(B->counter.p) + 7);
  d.run = reinterpret_cast<const uint64_t*>(static_cast<uint8_t*>(B->counter.p) + 32);
  if (cudaMallocHost(&B->hrun, 2 * sizeof(uint64_t)) != cudaSuccess)
    return set_error(QT_ERR_OUT_OF_MEMORY, "%s: pinned parameters", who);
  bool ok = cudaEventCreateWithFlags(&B->ev_fork, cudaEventDisableTiming) == cudaSuccess;
  for (int c = 0; ok && c < bt::kClasses - 1; ++c)
    ok = cudaStreamCreateWithFlags(&B->side[c], cudaStreamNonBlocking) == cudaSuccess &&
         cudaEventCreateWithFlags(&B->ev_join[c], cudaEventDisableTiming) == cudaSuccess;
  if (!ok) return set_error(QT_ERR_CUDA, "%s: side streams", who);
  return QT_OK;
}

// dynamic shared memory of the global class: two tiles (one of them holds the
// 64 x 64 matrix area between sweeps) and the matrices of a sweep
constexpr size_t kSmemGlob = sizeof(float2) * (2u << bt::kTileBits) + sizeof(float4) * bt::kGroupEntries;
// of a shared-memory class: the state, two matrices of up to 4 qubits and,
// where there are wider gates, one of their width
static size_t smem_class_bytes(uint32_t n, uint32_t wmat) {
  const uint32_t wbuf = std::min(wmat, 4u);
  return sizeof(float2) * ((size_t{1} << n) + (size_t{2} << (2 * wbuf)) + (wmat > 4 ? size_t{1} << (2 * wmat) : 0));
}

// The shared-memory classes ask for the largest carveout, so that their CTAs
// fit an SM together; the global class keeps its L1.
template <typename K>
static cudaError_t smem_kernel_attr(K kern) {
  const size_t most = smem_class_bytes(bt::kSmemNMax, bt::kMaxW);
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(most));
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
  return e;
}

static cudaError_t batch_kernel_attrs() {
  static PerDevice attr_set;
  return static_cast<cudaError_t>(attr_set.get([] {
    cudaError_t e = cudaFuncSetAttribute(bt::k_batch_glob, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         static_cast<int>(kSmemGlob));
    if (e == cudaSuccess) e = smem_kernel_attr(bt::k_batch_smem<512, 1>);
    if (e == cudaSuccess) e = smem_kernel_attr(bt::k_batch_smem<256, 3>);
    if (e == cudaSuccess) e = smem_kernel_attr(bt::k_batch_smem<128, 7>);
    return static_cast<int>(e);
  }));
}

template <typename K>
static cudaError_t launch_smem_class(K kern, uint32_t threads, size_t smem, const bt::Dev& d, uint32_t amps, cudaStream_t s) {
  int occ = 0;
  cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, static_cast<int>(threads), smem);
  if (e != cudaSuccess) return e;
  const unsigned grid = static_cast<unsigned>(std::min<uint64_t>(static_cast<uint64_t>(sm_count()) * std::max(occ, 1), d.num));
  kern<<<grid, threads, smem, s>>>(d, amps);
  return cudaGetLastError();
}

// CTAs per trajectory of the global class: one where the batch has
// trajectories enough to even out over the SMs, two below two per SM (240 of
// 15 to 18 qubits: 17.6 ms with one, 12.1 with two, 14.4 with four, whose
// smaller states have fewer tiles than the cluster has halves and whose
// clusters leave SMs over), more where SMs would stay idle: up to four and
// eight, in ms of at most two / four / eight CTAs (depth 24, k = 3),
//   4 of 16 to 18 qubits  1.28 2.68 5.03 / 0.84 1.64 2.87 / 0.84 1.11 1.79
//   4 of 20               20.9 / 11.2 / 6.3
//   30 of 18              5.52 / 3.17 / 3.58 (19 clusters of eight fit)
//   30 of 15 to 18        5.48 / 3.17 / 1.99
static unsigned glob_cluster(uint32_t num, uint32_t top_n) {
  const uint32_t sms = static_cast<uint32_t>(sm_count());
  const unsigned most = std::min(8u, 1u << (top_n - bt::kTileBits - 1));   // at least a tile per half
  unsigned c = num < 2 * sms ? 2 : 1;
  while (c < most && num * c < sms) c *= 2;
  return c;
}

static cudaError_t launch_glob_class(uint32_t threads, const bt::Dev& d, uint32_t top_n, cudaStream_t s) {
  const unsigned c = glob_cluster(d.num, top_n);
  const unsigned clusters = static_cast<unsigned>(std::min<uint64_t>(static_cast<uint64_t>(sm_count()) / c, d.num));
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = c;
  at.val.clusterDim.y = at.val.clusterDim.z = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(std::max(clusters, 1u) * c);
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = kSmemGlob;
  cfg.stream = s;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, bt::k_batch_glob, d);
  if (e != cudaSuccess) cudaGetLastError();          // not for the calls that come after
  return e;
}

// CTA size of class c where the caller asks for `threads`: the largest that
// its kernel is built for (k_batch_smem, k_batch_glob)
static uint32_t class_threads(int c, uint32_t threads) {
  static constexpr uint32_t most[bt::kClasses] = {bt::kGlobThreads, 512, 256, 256, 128};
  return std::min(threads, most[c]);
}

// One run's persistent launches, with tables, outputs and arena as d holds
// them: the work counters are zeroed on s, then every class launches, the
// first one present on s and the others on side streams forked from and
// joined back into s.  `threads` bounds a shared-memory class's CTA and fixes
// the logical threads its sums are split over.
static cudaError_t launch_classes(qt_batch* b, const bt::Dev& d, uint32_t threads, uint32_t threads_glob,
                                  cudaStream_t s) {
  cudaError_t r = cudaMemsetAsync(b->counter.p, 0, 32, s);
  int present = 0;
  for (uint32_t c : b->count) present += c != 0;
  if (r == cudaSuccess && present > 1) r = cudaEventRecord(b->ev_fork, s);
  uint32_t off = 0;
  int used = 0;
  for (int c = 0; c < bt::kClasses && r == cudaSuccess; ++c) {
    if (!b->count[c]) continue;
    cudaStream_t st = s;
    if (used > 0) {
      st = b->side[used - 1];
      r = cudaStreamWaitEvent(st, b->ev_fork, 0);
      if (r != cudaSuccess) return r;
    }
    bt::Dev dc = d;
    dc.order = d.order + off;
    dc.num = b->count[c];
    dc.counter = d.counter + c;
    dc.wmat = b->wmat[c];
    if (c == 0) {
      dc.lthreads = threads_glob;
      r = launch_glob_class(class_threads(c, threads_glob), dc, b->top_n[c], st);
    } else {
      dc.lthreads = threads;
      const uint32_t tb = class_threads(c, threads);
      const size_t smem = smem_class_bytes(b->top_n[c], dc.wmat);
      const uint32_t amps = 1u << b->top_n[c];
      r = tb == 512   ? launch_smem_class(bt::k_batch_smem<512, 1>, tb, smem, dc, amps, st)
          : tb == 256 ? launch_smem_class(bt::k_batch_smem<256, 3>, tb, smem, dc, amps, st)
                      : launch_smem_class(bt::k_batch_smem<128, 7>, tb, smem, dc, amps, st);
    }
    if (r == cudaSuccess && used > 0) r = cudaEventRecord(b->ev_join[used - 1], st);
    off += b->count[c];
    ++used;
  }
  for (int k = 0; k + 1 < used && r == cudaSuccess; ++k) r = cudaStreamWaitEvent(s, b->ev_join[k], 0);
  return r;
}

extern "C" {

qt_status qt_fuse_many(uint32_t num, const qt_circuit* const* circuits, uint32_t max_fused_qubits,
                       uint32_t threads, qt_fused** out) {
  clear_error();
  if (!circuits || !out) return set_error(QT_ERR_INVALID_ARG, "qt_fuse_many: NULL argument");
  for (uint32_t i = 0; i < num; ++i) {
    out[i] = nullptr;
    if (!circuits[i]) return set_error(QT_ERR_INVALID_ARG, "qt_fuse_many: circuit %u is NULL", i);
  }
  if (max_fused_qubits > QT_MAX_FUSED_QUBITS)
    return set_error(QT_ERR_INVALID_ARG, "qt_fuse_many: max_fused_qubits %u > 6", max_fused_qubits);
  unsigned nt = threads ? threads : std::max(1u, std::thread::hardware_concurrency());
  nt = std::min<unsigned>(nt, std::max<uint32_t>(num, 1));
  std::atomic<uint32_t> next{0};
  std::atomic<int> failed{0};
  auto work = [&] {
    for (;;) {
      const uint32_t i = next.fetch_add(1);
      if (i >= num) return;
      const qt_circuit* c = circuits[i];
      uint32_t k = max_fused_qubits ? max_fused_qubits : (c->n >= 20 ? 4 : (c->n >= 12 ? 3 : 2));
      k = std::min<uint32_t>(k, c->n);
      qt_fused* f = new (std::nothrow) qt_fused();
      if (!f || fuse_circuit(*c, k, *f) != QT_OK) {
        delete f;
        failed = 1;
        continue;
      }
      out[i] = f;
    }
  };
  std::vector<std::thread> pool;
  for (unsigned t = 1; t < nt; ++t) pool.emplace_back(work);
  work();
  for (auto& t : pool) t.join();
  if (failed) {
    for (uint32_t i = 0; i < num; ++i) { delete out[i]; out[i] = nullptr; }
    return set_error(QT_ERR_INTERNAL, "qt_fuse_many: fusion failed");
  }
  return QT_OK;
}

qt_status qt_batch_create(uint32_t num, const qt_fused* const* fused, qt_batch** out) {
  clear_error();
  if (!fused || !out || num == 0) return set_error(QT_ERR_INVALID_ARG, "qt_batch_create: NULL argument or empty batch");
  *out = nullptr;
  std::unique_ptr<qt_batch> B(new (std::nothrow) qt_batch());
  if (!B) return set_error(QT_ERR_OUT_OF_MEMORY, "qt_batch_create: host allocation");
  qt_status s = pack_batch(B.get(), num, fused, nullptr, "qt_batch_create", nullptr);
  if (s == QT_OK) s = init_batch_runtime(B.get(), "qt_batch_create");
  if (s != QT_OK) return s;
  const cudaError_t e = cudaStreamSynchronize(nullptr);   // the tables are on the device
  if (e != cudaSuccess) return set_error(QT_ERR_CUDA, "qt_batch_create: %s", cudaGetErrorString(e));
  *out = B.release();
  return QT_OK;
}

qt_status qt_batch_run(qt_batch* b, const qt_batch_params* p) {
  clear_error();
  TraceRange tr("qt batched run");
  if (!b || !p) return set_error(QT_ERR_INVALID_ARG, "qt_batch_run: NULL argument");
  if (p->samples_per_traj > 1u << 20) return set_error(QT_ERR_INVALID_ARG, "qt_batch_run: samples_per_traj too large");
  const uint32_t threads = p->threads ? p->threads : 512;
  const uint32_t threads_glob = p->threads_global ? p->threads_global : threads;
  for (uint32_t t : {threads, threads_glob})
    if (t != 128 && t != 256 && t != 512)
      return set_error(QT_ERR_INVALID_ARG, "qt_batch_run: threads %u (128, 256 or 512)", t);
  cudaStream_t st = static_cast<cudaStream_t>(p->stream);
  bt::Dev& d = b->dev;
  const bool relayout = !b->outs.p || p->samples_per_traj != b->S || (p->keep_states != 0) != (b->keep != 0);
  if (relayout) {
    if (b->gexec) { cudaGraphExecDestroy(b->gexec); b->gexec = nullptr; }
    if (b->graph) { cudaGraphDestroy(b->graph); b->graph = nullptr; }
    b->S = p->samples_per_traj;
    b->keep = p->keep_states ? 1u : 0u;
    auto align = [](size_t x) { return (x + 255) & ~size_t(255); };
    size_t off = 0;
    b->off_kraus = off; off = align(off + std::max<size_t>(b->total_ch, 1));
    b->off_stage = off; off = align(off + std::max<size_t>(b->total_ch, 1));
    b->off_samples = off; off = align(off + sizeof(uint64_t) * std::max<uint64_t>(uint64_t(b->num) * b->S, 1));
    b->off_flushes = off; off = align(off + sizeof(uint32_t) * b->num);
    b->off_folds = off; off = align(off + sizeof(uint32_t) * b->num);
    b->off_gflag = off; off = align(off + std::max<uint64_t>(b->total_gates, 1));
    if (!b->outs.alloc(off)) return set_error(QT_ERR_OUT_OF_MEMORY, "qt_batch_run: outputs");
    uint8_t* o = static_cast<uint8_t*>(b->outs.p);
    d.kraus = reinterpret_cast<int8_t*>(o + b->off_kraus);
    d.stage = reinterpret_cast<int8_t*>(o + b->off_stage);
    d.samples = reinterpret_cast<uint64_t*>(o + b->off_samples);
    d.flushes = reinterpret_cast<uint32_t*>(o + b->off_flushes);
    d.folds = reinterpret_cast<uint32_t*>(o + b->off_folds);
    d.gflag = o + b->off_gflag;
    int sms = sm_count();
    const uint64_t slot = b->max_n > static_cast<uint32_t>(bt::kSmemNMax) ? (1ull << b->max_n) : 0;
    const uint64_t arena_amps = b->keep ? b->total_amps : slot * sms;
    if (!b->arena.alloc(sizeof(float2) * arena_amps)) {
      b->outs.alloc(0);                      // no layout: the next run lays out again
      b->keep = 0;
      return set_error(QT_ERR_OUT_OF_MEMORY, "qt_batch_run: state arena (%llu amplitudes)",
                       static_cast<unsigned long long>(arena_amps));
    }
    d.arena = static_cast<float2*>(b->arena.p);
    d.slot_amps = slot;
    d.keep = b->keep;
    d.S = b->S;
    b->kraus.assign(b->total_ch, 0);
    b->stage.assign(b->total_ch, 0);
    b->samples.assign(static_cast<size_t>(b->num) * b->S, 0);
    b->flushes.assign(b->num, 0);
    b->folds.assign(b->num, 0);
  }
  b->hrun[0] = p->seed;
  b->hrun[1] = p->first_traj;
  const cudaError_t attr = batch_kernel_attrs();
  if (attr != cudaSuccess) return set_error(QT_ERR_CUDA, "qt_batch_run: smem attribute: %s", cudaGetErrorString(attr));
  struct Events {                   // the run's timing events, destroyed on every return
    cudaEvent_t a = nullptr, b = nullptr;
    ~Events() {
      if (a) cudaEventDestroy(a);
      if (b) cudaEventDestroy(b);
    }
  } ev;
  cudaError_t e = cudaEventCreate(&ev.a);
  if (e == cudaSuccess) e = cudaEventCreate(&ev.b);
  if (e != cudaSuccess) return set_error(QT_ERR_CUDA, "qt_batch_run: cudaEventCreate: %s", cudaGetErrorString(e));
  cudaEvent_t e0 = ev.a, e1 = ev.b;
  auto enqueue = [&](cudaStream_t s) -> cudaError_t {
    cudaError_t r = cudaMemcpyAsync(static_cast<uint8_t*>(b->counter.p) + 32, b->hrun, 2 * sizeof(uint64_t),
                                    cudaMemcpyHostToDevice, s);
    if (r != cudaSuccess) return r;
    return launch_classes(b, d, threads, threads_glob, s);
  };
  e = cudaEventRecord(e0, st);
  if (e == cudaSuccess && p->use_graph && st) {
    // the graph copies the run parameters from pinned memory when it runs, so
    // it is rebuilt only when the launch shape changes
    if (b->gexec && (b->g_threads != threads || b->g_threads_glob != threads_glob)) {
      cudaGraphExecDestroy(b->gexec); b->gexec = nullptr;
      cudaGraphDestroy(b->graph); b->graph = nullptr;
    }
    if (!b->gexec) {
      e = cudaStreamBeginCapture(st, cudaStreamCaptureModeThreadLocal);
      if (e == cudaSuccess) {
        cudaError_t r = enqueue(st);
        e = cudaStreamEndCapture(st, &b->graph);
        if (r != cudaSuccess) e = r;
      }
      if (e == cudaSuccess) e = cudaGraphInstantiate(&b->gexec, b->graph, 0);
      b->g_threads = threads;
      b->g_threads_glob = threads_glob;
    }
    if (e == cudaSuccess) e = cudaGraphLaunch(b->gexec, st);
  } else if (e == cudaSuccess) {
    e = enqueue(st);
  }
  if (e == cudaSuccess) e = cudaEventRecord(e1, st);
  b->last = *p;
  if (e == cudaSuccess) e = cudaMemcpyAsync(b->kraus.data(), d.kraus, b->total_ch, cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaMemcpyAsync(b->stage.data(), d.stage, b->total_ch, cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess && b->S)
    e = cudaMemcpyAsync(b->samples.data(), d.samples, sizeof(uint64_t) * b->samples.size(), cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaMemcpyAsync(b->flushes.data(), d.flushes, sizeof(uint32_t) * b->num, cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaMemcpyAsync(b->folds.data(), d.folds, sizeof(uint32_t) * b->num, cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  float ms = 0.f;
  if (e == cudaSuccess) e = cudaEventElapsedTime(&ms, e0, e1);
  if (e != cudaSuccess) return set_error(QT_ERR_CUDA, "qt_batch_run: %s", cudaGetErrorString(e));
  b->device_ms = ms;
  return QT_OK;
}

qt_status qt_batch_samples(const qt_batch* b, uint64_t* out, size_t cap) {
  clear_error();
  if (!b || (!out && !b->samples.empty())) return set_error(QT_ERR_INVALID_ARG, "qt_batch_samples: NULL argument");
  if (cap < b->samples.size()) return set_error(QT_ERR_INVALID_ARG, "qt_batch_samples: cap %zu < %zu", cap, b->samples.size());
  if (!b->samples.empty()) std::memcpy(out, b->samples.data(), sizeof(uint64_t) * b->samples.size());
  return QT_OK;
}

qt_status qt_batch_kraus_indices(const qt_batch* b, uint32_t i, int32_t* kraus, int32_t* stage, size_t cap,
                                 uint32_t* num_channels) {
  clear_error();
  if (!b) return set_error(QT_ERR_INVALID_ARG, "qt_batch_kraus_indices: NULL batch");
  if (i >= b->num) return set_error(QT_ERR_INVALID_ARG, "qt_batch_kraus_indices: index %u out of range", i);
  const bt::Traj& T = b->traj[i];
  if (num_channels) *num_channels = T.nch;
  if ((kraus || stage) && cap < T.nch) return set_error(QT_ERR_INVALID_ARG, "qt_batch_kraus_indices: cap %zu < %u", cap, T.nch);
  if (kraus) std::copy_n(b->kraus.data() + T.ch0, T.nch, kraus);
  if (stage) std::copy_n(b->stage.data() + T.ch0, T.nch, stage);
  return QT_OK;
}

qt_status qt_batch_state(const qt_batch* b, uint32_t i, void* dst, size_t bytes) {
  clear_error();
  if (!b || !dst) return set_error(QT_ERR_INVALID_ARG, "qt_batch_state: NULL argument");
  if (!b->keep) return set_error(QT_ERR_INVALID_ARG, "qt_batch_state: the last run did not keep its states");
  if (i >= b->num) return set_error(QT_ERR_INVALID_ARG, "qt_batch_state: index %u out of range", i);
  const bt::Traj& T = b->traj[i];
  const size_t sb = sizeof(float2) << T.n;
  if (bytes < sb) return set_error(QT_ERR_INVALID_ARG, "qt_batch_state: %zu bytes < %zu", bytes, sb);
  // the kept state is un-normalized (deferred operators): normalize a device copy
  DevMem tmp, part;
  if (!tmp.alloc(sb) || !part.alloc(sizeof(double) * (kPartialDoubles + kResultDoubles)))
    return set_error(QT_ERR_OUT_OF_MEMORY, "qt_batch_state: buffers");
  Scratch scr;
  scr.partial = static_cast<double*>(part.p);
  scr.result = scr.partial + kPartialDoubles;
  double N = 0.0;
  cudaError_t e = cudaMemcpy(tmp.p, static_cast<float2*>(b->arena.p) + T.arena_off, sb, cudaMemcpyDeviceToDevice);
  if (e == cudaSuccess) e = launch_expect(static_cast<const float2*>(tmp.p), static_cast<int>(T.n), 0, nullptr, scr, 0);
  if (e == cudaSuccess) e = cudaMemcpy(&N, scr.result, sizeof(double), cudaMemcpyDeviceToHost);
  if (e == cudaSuccess)
    e = launch_scale(static_cast<float2*>(tmp.p), static_cast<int>(T.n), static_cast<float>(1.0 / std::sqrt(N)), 0);
  if (e == cudaSuccess) e = cudaMemcpy(dst, tmp.p, sb, cudaMemcpyDeviceToHost);
  if (e != cudaSuccess) return set_error(QT_ERR_CUDA, "qt_batch_state: %s", cudaGetErrorString(e));
  return QT_OK;
}

qt_status qt_batch_stats(const qt_batch* b, qt_batch_stats_t* out) {
  clear_error();
  if (!b || !out) return set_error(QT_ERR_INVALID_ARG, "qt_batch_stats: NULL argument");
  out->num_traj = b->num;
  out->num_channels = b->total_ch;
  out->total_amps = b->total_amps;
  out->fused_gates = b->fused_gates;
  out->gate_ops = b->gate_ops;
  uint64_t f = 0;
  for (uint32_t x : b->flushes) f += x;
  out->flushes = f;
  out->device_ms = b->device_ms;
  uint64_t fo = 0;
  for (uint32_t x : b->folds) fo += x;
  out->folded_pieces = fo;
  return QT_OK;
}

void qt_batch_destroy(qt_batch* b) { delete b; }

qt_status qt_batch_autotune(uint32_t num, const qt_circuit* const* circuits, uint32_t sample, uint32_t kmin,
                            uint32_t kmax, void* stream, qt_batch_tuning* best, double* table) {
  clear_error();
  if (!circuits || !best || num == 0)
    return set_error(QT_ERR_INVALID_ARG, "qt_batch_autotune: NULL argument or empty batch");
  kmin = std::max<uint32_t>(kmin, 1);
  kmax = std::min<uint32_t>(kmax, bt::kMaxW);
  if (kmin > kmax) return set_error(QT_ERR_INVALID_ARG, "qt_batch_autotune: empty k range");
  static const uint32_t kThreadOpts[3] = {128, 256, 512};
  const uint32_t nk = kmax - kmin + 1;
  best->k_shared = best->k_global = kmin;
  best->threads_shared = best->threads_global = 512;
  if (table)
    for (uint32_t i = 0; i < 2 * nk * 3; ++i) table[i] = 0.0;
  // the two classes of the batched kernel: states in shared memory (n <= 14)
  // and states in global memory, each tuned on a spread sample of its own
  for (int cls = 0; cls < 2; ++cls) {
    std::vector<const qt_circuit*> members;
    for (uint32_t i = 0; i < num; ++i) {
      if (!circuits[i]) return set_error(QT_ERR_INVALID_ARG, "qt_batch_autotune: circuit %u is NULL", i);
      if ((circuits[i]->n > static_cast<uint32_t>(bt::kSmemNMax)) == (cls == 1)) members.push_back(circuits[i]);
    }
    if (members.empty()) continue;
    const uint32_t nm = static_cast<uint32_t>(members.size());
    const uint32_t ns = std::max<uint32_t>(1, std::min(sample ? sample : 256u, nm));
    std::vector<const qt_circuit*> sub(ns);
    for (uint32_t i = 0; i < ns; ++i) sub[i] = members[static_cast<uint64_t>(i) * nm / ns];
    double best_ms = 1e300;
    for (uint32_t k = kmin; k <= kmax; ++k) {
      std::vector<qt_fused*> f(ns, nullptr);
      qt_status s = qt_fuse_many(ns, sub.data(), k, 0, f.data());
      if (s != QT_OK) return s;
      qt_batch* b = nullptr;
      s = qt_batch_create(ns, const_cast<const qt_fused* const*>(f.data()), &b);
      for (auto* x : f) qt_fused_destroy(x);
      if (s != QT_OK) return s;
      // sizes that launch the same CTAs are timed once and stand for the largest
      // of them: the value also fixes how sums are split, which noise is not to pick
      double timed[3];
      for (int ti = 2; ti >= 0; --ti) {
        int same = -1;
        for (int tj = ti + 1; tj < 3 && same < 0; ++tj) {
          same = tj;
          for (int c = 0; c < bt::kClasses; ++c)
            if (b->count[c] && class_threads(c, kThreadOpts[ti]) != class_threads(c, kThreadOpts[tj])) same = -1;
        }
        double ms = 0.0;
        if (same < 0) {
          qt_batch_params p{};
          p.seed = 0x5eed;
          p.samples_per_traj = 16;
          p.threads = kThreadOpts[ti];
          p.threads_global = kThreadOpts[ti];
          p.stream = stream;
          for (int rep = 0; rep < 3 && s == QT_OK; ++rep) {
            p.first_traj = rep;
            s = qt_batch_run(b, &p);
            if (rep > 0) ms += b->device_ms;     // the first run is warm-up
          }
          if (s != QT_OK) { qt_batch_destroy(b); return s; }
        }
        timed[ti] = same < 0 ? ms / 2.0 : timed[same];
        if (table) table[(cls * nk + (k - kmin)) * 3 + ti] = timed[ti];
        if (same < 0 && ms < best_ms) {
          best_ms = ms;
          if (cls == 0) { best->k_shared = k; best->threads_shared = kThreadOpts[ti]; }
          else { best->k_global = k; best->threads_global = kThreadOpts[ti]; }
        }
      }
      qt_batch_destroy(b);
    }
  }
  return QT_OK;
}

}  // extern "C"

// ---------------------------------------------------------------------------
// merged launches of the serving form (the batch lane)
// ---------------------------------------------------------------------------
namespace qt {

struct BatchLane {
  qt_batch B;
  cudaStream_t st = nullptr;
  uint32_t max_n = 0;
  uint64_t slot = 0;                // amplitudes per global-memory state slot
  std::vector<const qt_fused*> fused;
};

qt_status lane_create(uint32_t max_n, void* stream, BatchLane** out) {
  if (!out) return set_error(QT_ERR_INVALID_ARG, "lane_create: NULL argument");
  *out = nullptr;
  if (max_n < 1 || max_n > static_cast<uint32_t>(bt::kMaxN))
    return set_error(QT_ERR_INVALID_ARG, "lane_create: max_n %u outside 1..%d", max_n, bt::kMaxN);
  std::unique_ptr<BatchLane> L(new (std::nothrow) BatchLane());
  if (!L) return set_error(QT_ERR_OUT_OF_MEMORY, "lane_create: host allocation");
  L->st = static_cast<cudaStream_t>(stream);
  L->max_n = max_n;
  qt_status s = init_batch_runtime(&L->B, "lane_create");
  if (s != QT_OK) return s;
  if (max_n > static_cast<uint32_t>(bt::kSmemNMax)) {
    L->slot = 1ull << max_n;
    if (!L->B.arena.alloc(sizeof(float2) * L->slot * sm_count()))
      return set_error(QT_ERR_OUT_OF_MEMORY, "lane_create: state slots (%u qubits)", max_n);
  }
  *out = L.release();
  return QT_OK;
}

void lane_destroy(BatchLane* l) { delete l; }

qt_status lane_run(BatchLane* L, uint32_t num, const LaneTraj* tr, uint64_t* samples, uint32_t* flushes) {
  TraceRange range("qt merged batched launch");
  if (!L || !tr || num == 0) return set_error(QT_ERR_INVALID_ARG, "lane_run: NULL argument or no trajectories");
  qt_batch* b = &L->B;
  L->fused.resize(num);
  for (uint32_t i = 0; i < num; ++i) {
    if (!tr[i].f) return set_error(QT_ERR_INVALID_ARG, "lane_run: trajectory %u has no circuit", i);
    if (tr[i].f->c->n > L->max_n)
      return set_error(QT_ERR_UNSUPPORTED, "lane_run: %u qubits > the lane's %u", tr[i].f->c->n, L->max_n);
    L->fused[i] = tr[i].f;
  }
  qt_status s = pack_batch(b, num, L->fused.data(), tr, "lane_run", L->st);
  if (s != QT_OK) return s;
  auto align = [](size_t x) { return (x + 255) & ~size_t(255); };
  size_t off = 0;
  const size_t o_kraus = off; off = align(off + std::max<size_t>(b->total_ch, 1));
  const size_t o_stage = off; off = align(off + std::max<size_t>(b->total_ch, 1));
  const size_t o_samp = off; off = align(off + sizeof(uint64_t) * std::max<uint64_t>(b->lane_samples, 1));
  const size_t o_flush = off; off = align(off + sizeof(uint32_t) * num);
  const size_t o_gflag = off; off = align(off + std::max<uint64_t>(b->total_gates, 1));
  if (b->outs.bytes < off && !b->outs.alloc(off)) return set_error(QT_ERR_OUT_OF_MEMORY, "lane_run: outputs");
  uint8_t* o = static_cast<uint8_t*>(b->outs.p);
  bt::Dev d = b->dev;
  d.kraus = reinterpret_cast<int8_t*>(o + o_kraus);
  d.stage = reinterpret_cast<int8_t*>(o + o_stage);
  d.samples = reinterpret_cast<uint64_t*>(o + o_samp);
  d.flushes = reinterpret_cast<uint32_t*>(o + o_flush);
  d.folds = nullptr;
  d.gflag = o + o_gflag;
  d.arena = static_cast<float2*>(b->arena.p);
  d.slot_amps = L->slot;
  d.keep = 0;
  d.S = 0;
  d.per_traj = 1;
  cudaError_t e = batch_kernel_attrs();
  if (e == cudaSuccess) e = launch_classes(b, d, 512, 512, L->st);
  if (e == cudaSuccess && b->lane_samples)
    e = cudaMemcpyAsync(samples, d.samples, sizeof(uint64_t) * b->lane_samples, cudaMemcpyDeviceToHost, L->st);
  if (e == cudaSuccess && flushes)
    e = cudaMemcpyAsync(flushes, d.flushes, sizeof(uint32_t) * num, cudaMemcpyDeviceToHost, L->st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(L->st);
  if (e != cudaSuccess) return set_error(QT_ERR_CUDA, "lane_run: %s", cudaGetErrorString(e));
  return QT_OK;
}

}  // namespace qt
