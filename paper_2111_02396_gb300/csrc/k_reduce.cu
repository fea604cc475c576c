// Read-only passes over the state: branch probabilities (Alg. 2 step 14),
// Z-string expectations and bitstring sampling, plus state init / scale.
//
// Precision: products are formed in FP32 from the complex64 state; partial
// sums over a short run of terms stay in FP32 and are then carried in
// double-floats (qt_dfloat.h: FP64 throughput on this part is low) and leave
// as FP64.  Every reduction has a fixed grid and a fixed combination order,
// so results are bitwise reproducible run to run.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <mutex>

#include "kernels.h"
#include "qt_dfloat.h"
#include "qt_philox.h"

namespace qt {

// A dependent launch: its blocks may become resident while the kernel before
// it on the stream still runs, and wait there (cudaGridDependencySynchronize)
// for that kernel's results.  The short kernels that follow a reduction start
// without a launch gap this way.  An error of that kernel's launch is returned
// instead; no error stays behind for the calls that come after.
template <typename... P, typename... A>
static cudaError_t launch_dependent(void (*kern)(P...), dim3 grid, unsigned block, cudaStream_t st, A... args) {
  const cudaError_t before = cudaGetLastError();
  if (before != cudaSuccess) return before;
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(block);
  cfg.stream = st;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, kern, static_cast<P>(args)...);
  if (e != cudaSuccess) cudaGetLastError();
  return e;
}

// ---------------------------------------------------------------------------
// block-wide sums of W per-thread double-floats into partial[block][W]
// ---------------------------------------------------------------------------
template <int W>
__device__ __forceinline__ void block_reduce_store(const float (&h)[W], const float (&l)[W],
                                                   float2* __restrict__ partial) {
  constexpr int P = W >= 16 ? 16 : (W >= 4 ? 4 : 2), REST = W - P;   // one transposed group and the rest
  __shared__ float2 sm[kRedThreads / 32][W];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  float2 v[P];
#pragma unroll
  for (int c = 0; c < P; ++c) v[c] = make_float2(h[c], l[c]);
  const float2 s = df_warp_sum<P>(v, lane);
  constexpr int per = 32 / P;                          // lanes that hold the same sum
  if (lane % per == 0) sm[warp][lane / per] = s;
#pragma unroll
  for (int c = W - REST; c < W; ++c) {
    float2 r = make_float2(h[c], l[c]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) r = df_add(r, df_shfl_xor(r, o));
    if (lane == 0) sm[warp][c] = r;
  }
  __syncthreads();
  const int nw = static_cast<int>(blockDim.x >> 5);    // blocks of at most kRedThreads threads
  for (int c = threadIdx.x; c < W; c += blockDim.x) {
    float2 r = make_float2(0.f, 0.f);
    for (int w = 0; w < nw; ++w) r = df_add(r, sm[w][c]);
    partial[static_cast<size_t>(blockIdx.x) * W + c] = r;
  }
}

// out[c] = sum over blocks of partial[block][c].  CB columns per block of 1024
// threads, 1024 / CB of them per column: a handful of independent loads each
// at the largest grid.  (One thread per column chained up to 1216 FP64 adds:
// 55 us after a 29-qubit pass, 14 after a 17-qubit one, now 4 and 3.)
constexpr int kSumThreads = 1024;

template <int CB>
__device__ __forceinline__ float2 column_sum(const float2* partial, int nblocks, int W, int col) {
  constexpr int SL = kSumThreads / CB;
  __shared__ float2 sm[SL][CB];
  const int cl = threadIdx.x % CB, sl = threadIdx.x / CB;
  float2 r = make_float2(0.f, 0.f);
  if (col < W) {
#pragma unroll 4
    for (int b = sl; b < nblocks; b += SL) r = df_add(r, partial[static_cast<size_t>(b) * W + col]);
  }
  // lanes of a warp that hold the same column, then the warps
  if constexpr (CB < 32) {
#pragma unroll
    for (int o = CB; o < 32; o <<= 1) r = df_add(r, df_shfl_xor(r, o));
  }
  constexpr int PER = CB < 32 ? 32 / CB : 1;             // slices of a warp
  if (sl % PER == 0) sm[sl / PER][cl] = r;
  __syncthreads();
#pragma unroll
  for (int o = SL / PER / 2; o > 0; o >>= 1) {
    if (sl < o) sm[sl][cl] = df_add(sm[sl][cl], sm[sl + o][cl]);
    __syncthreads();
  }
  return sm[0][cl];
}

template <int CB>
__global__ void __launch_bounds__(kSumThreads) k_finalize(const float2* partial, int nblocks, int W, double* out) {
  cudaGridDependencySynchronize();
  const int col = blockIdx.x * CB + threadIdx.x % CB;
  const float2 r = column_sum<CB>(partial, nblocks, W, col);
  if (threadIdx.x < CB && col < W) out[col] = df_value(r);
}

static cudaError_t finalize(const float2* partial, int nblocks, int W, double* out, cudaStream_t st) {
  return launch_dependent(k_finalize<4>, dim3((W + 3) / 4), kSumThreads, st, partial, nblocks, W, out);
}

template <typename Kern>
static int red_grid(Kern kern, uint64_t work_items) {
  // one full wave of resident blocks, capped by the work and by the scratch
  int occ = 0;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, kRedThreads, 0);
  if (occ <= 0) occ = 1;
  uint64_t g = static_cast<uint64_t>(sm_count()) * occ;
  const uint64_t need = (work_items + kRedThreads - 1) / kRedThreads;
  if (g > need) g = need;
  if (g > static_cast<uint64_t>(kMaxRedBlocks)) g = kMaxRedBlocks;
  if (g < 1) g = 1;
  return static_cast<int>(g);
}

// ---------------------------------------------------------------------------
// Reduced density block of qubits Q: rho[b][a] = sum_rest psi[rest,b] conj(psi[rest,a]),
// with basis bit j = the j-th lowest qubit (the callers reorder).
//
// q = 1, 2 (k_rdm): every entry in registers, W = 4^q reals: the 2^q diagonal
// entries, then (re, im) of each b < a.  Bound by HBM: a thread keeps 4 to 16
// 128-bit loads in flight (LOW0: qubit 0 is in Q, so members 2j and 2j + 1 of a
// set share a load; otherwise two neighbouring sets do).  A call at n =
// 29: q = 1 754 -> 670 us, q = 2 901 -> 660 (one set of 8-byte loads at a time
// and FP64 carries before); 4 GiB read at the copy rate take 634.
//
// The FP32 runs are fixed, whatever the launch: with T streams (rdm_blocks),
// stream t takes the sets t, t + T, t + 2 T, ... and carries after every
// kRdmChunk of them.  A run's rounding (1e-10 of an entry at 20 qubits) goes
// into the branch that a channel picks, normalized by 1 / sqrt(P) and rounded
// to FP32: other runs would give other last bits of the state.  A thread has
// two streams, 2p and 2p + 1, or with LOW0 one.
// ---------------------------------------------------------------------------
// f + Im(b conj a), added as (-b.x a.y), (b.y a.x), or the other way round (rev)
__device__ __forceinline__ float cross(float2 b, float2 a, float f, bool rev) {
  const float u = rev ? b.y : -b.x, v = rev ? a.x : a.y, w = rev ? -b.x : b.y, z = rev ? a.y : a.x;
  return fmaf(w, z, fmaf(u, v, f));
}

// whether sorted member b comes after member a in the caller's order of the
// qubits (his basis bit j is the rank[j]-th lowest of them): the two products
// of an imaginary part are added in that order, which shows in the last bits
// of small states
static bool member_after(int q, const int* rank, int b, int a) {
  int ub = 0, ua = 0;
  for (int j = 0; j < q; ++j) {
    ub |= ((b >> rank[j]) & 1) << j;
    ua |= ((a >> rank[j]) & 1) << j;
  }
  return ub > ua;
}

template <int Q>
struct RdmArgs {
  uint64_t offs[1 << Q];      // 128-bit word offset of load m within a group
  uint32_t ins[Q + 1];        // ascending bit positions to insert zeros at
  uint64_t num_groups;
  bool rev;                   // q = 2: the caller's members 1 and 2 are swapped
  float down;                 // Scratch::down
};

constexpr int kRdmChunk = 16;     // sets summed in FP32 before the carry
constexpr int kRdmThreads = kRedThreads / 2;

// T: 8 (q = 2: 3) times kRedThreads an SM, not more than the sets need
template <int Q>
static int rdm_blocks(uint64_t sets) {
  const uint64_t need = (sets + kRedThreads - 1) / kRedThreads;
  return static_cast<int>(std::min<uint64_t>({need, static_cast<uint64_t>(sm_count()) * (Q == 1 ? 8 : 3),
                                              static_cast<uint64_t>(kMaxRedBlocks)}));
}

// streams of a thread
__host__ __device__ constexpr int rdm_streams(bool low0) { return low0 ? 1 : 2; }

template <int Q, bool LOW0>
__global__ void __launch_bounds__(kRdmThreads, Q == 1 && LOW0 ? 16 : 1) k_rdm(const float4* __restrict__ psi,
                                                     const __grid_constant__ RdmArgs<Q> a,
                                                     float2* __restrict__ partial) {
  constexpr int D = 1 << Q, W = D * D;
  constexpr int NV = LOW0 ? D / 2 : D;        // loads per group
  constexpr int SPG = LOW0 ? 1 : 2;           // sets per group
  constexpr int NI = LOW0 ? Q : Q + 1;        // zeros inserted into the group index
  constexpr int ST = rdm_streams(LOW0);
  constexpr int U = (LOW0 ? 4 * Q : 8 * Q) / NV;   // groups in flight
  cudaTriggerProgrammaticLaunchCompletion();
  float h[W], l[W], f[ST][W];
#pragma unroll
  for (int c = 0; c < W; ++c) { h[c] = l[c] = f[0][c] = f[ST - 1][c] = 0.f; }
  auto carry = [&] {
#pragma unroll
    for (int t = 0; t < ST; ++t)
#pragma unroll
      for (int k = 0; k < W; ++k) { df_acc(h[k], l[k], f[t][k] * a.down); f[t][k] = 0.f; }
  };
  const uint64_t stride = static_cast<uint64_t>(gridDim.x) * blockDim.x;
  auto load = [&](uint64_t g, float4 (&v)[NV]) {
    uint64_t base = g;
#pragma unroll
    for (int b = 0; b < NI; ++b) {
      const uint32_t s = a.ins[b];
      base = ((base >> s) << (s + 1)) | (base & ((1ull << s) - 1ull));
    }
#pragma unroll
    for (int m = 0; m < NV; ++m) v[m] = __ldg(psi + (base >> 1) + a.offs[m]);
  };
  auto add = [&](const float4 (&v)[NV]) {
#pragma unroll
    for (int s = 0; s < SPG; ++s) {
      float2 x[D];
#pragma unroll
      for (int m = 0; m < D; ++m) {
        const float4 w = v[LOW0 ? m / 2 : m];
        const bool second = LOW0 ? (m & 1) : s == 1;
        x[m] = second ? make_float2(w.z, w.w) : make_float2(w.x, w.y);
      }
      float* const r = f[LOW0 ? 0 : s];
      int c = 0;
#pragma unroll
      for (int b = 0; b < D; ++b) { r[c] = fmaf(x[b].x, x[b].x, fmaf(x[b].y, x[b].y, r[c])); ++c; }
#pragma unroll
      for (int b = 0; b < D; ++b)
#pragma unroll
        for (int aa = b + 1; aa < D; ++aa) {
          // x_b conj(x_a)
          r[c] = fmaf(x[b].x, x[aa].x, fmaf(x[b].y, x[aa].y, r[c])); ++c;
          r[c] = cross(x[b], x[aa], r[c], Q == 2 && b == 1 && aa == 2 && a.rev); ++c;
        }
    }
  };
  int cnt = 0;
  uint64_t i = static_cast<uint64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  // whole batches: no condition between the loads, or they would wait for one another
  for (; i + (U - 1) * stride < a.num_groups; i += U * stride) {
    float4 v[U][NV];
#pragma unroll
    for (int u = 0; u < U; ++u) load(i + u * stride, v[u]);
#pragma unroll
    for (int u = 0; u < U; ++u) add(v[u]);
    cnt += U * SPG;                           // sets of the ST streams
    if (cnt == ST * kRdmChunk) {
      carry();
      cnt = 0;
    }
  }
#pragma unroll
  for (int u = 0; u < U; ++u)
    if (i + u * stride < a.num_groups) {
      float4 v[NV];
      load(i + u * stride, v);
      add(v);
    }
  carry();
  block_reduce_store<W>(h, l, partial);
}

// sorted copy of q qubits
template <int Q>
static void sort_qubits(const uint32_t* qubits, uint32_t* s) {
  for (int b = 0; b < Q; ++b) s[b] = qubits[b];
  for (int i = 1; i < Q; ++i)
    for (int j = i; j > 0 && s[j - 1] > s[j]; --j) { const uint32_t t = s[j]; s[j] = s[j - 1]; s[j - 1] = t; }
}

template <int Q, bool LOW0>
static cudaError_t rdm_low(const float2* psi, int n, const uint32_t* qubits, const uint32_t* s, const Scratch& scr,
                           cudaStream_t st) {
  RdmArgs<Q> a{};
  a.rev = Q == 2 && qubits[0] != s[0];
  a.down = scr.down;
  int ni = 0;
  if (!LOW0) a.ins[ni++] = 0;
  for (int b = 0; b < Q; ++b) a.ins[ni++] = s[b];
  for (int m = 0; m < (1 << Q); ++m) {
    uint64_t o = 0;
    const int mem = LOW0 ? 2 * m : m;            // the even member of load m
    for (int b = 0; b < Q; ++b)
      if ((mem >> b) & 1) o |= 1ull << s[b];
    a.offs[m] = o >> 1;
  }
  a.num_groups = 1ull << (n - Q - (LOW0 ? 0 : 1));
  const int g = rdm_blocks<Q>(1ull << (n - Q)) * (2 / rdm_streams(LOW0));
  k_rdm<Q, LOW0><<<g, kRdmThreads, 0, st>>>(reinterpret_cast<const float4*>(psi), a, scr.partials());
  return finalize(scr.partials(), g, 1 << (2 * Q), scr.result, st);
}

// ---------------------------------------------------------------------------
// q = 3 (k_rdm3): 64 reals do not fit one thread with their carries, so a pair
// of lanes (l, l ^ 16) shares a group: each loads the four members with its
// value of the highest qubit, gets the other four by shuffles, and sums half
// of the block: the triangle over its own members (16 reals) and two columns
// of the 4 x 4 corner between the halves (16 reals).  The carries sit in
// shared memory, which leaves the registers to loads in flight.
// n = 29: 1856 -> 936 us (64 FP64 accumulators a thread, 8 warps an SM).
// ---------------------------------------------------------------------------
struct Rdm3Args {
  uint64_t offs[4];           // 128-bit word offset of load m of the half-group
  uint64_t half;              // 128-bit word offset of the upper half
  uint32_t ins[4];            // ascending bit positions to insert zeros at
  uint64_t num_groups;
  int run;                    // sets summed in FP32 before the carry
  uint32_t rev;               // pairs in the other order: bits 0..5 within a half, 8 + 4 y + x of the corner
  float down;                 // Scratch::down
};

constexpr int kRdm3Threads = 128;
constexpr int kRdm3OrderLog = 18;   // fewer sets than this: imaginary parts in the caller's order (3e-11 of an entry beyond)

template <bool LOW0, bool PERM>
__global__ void __launch_bounds__(kRdm3Threads, 4) k_rdm3(const float4* __restrict__ psi, const __grid_constant__ Rdm3Args a,
                                                          float2* __restrict__ partial) {
  constexpr int NV = LOW0 ? 2 : 4;            // loads per half-group
  constexpr int SPG = LOW0 ? 1 : 2;           // sets per group
  constexpr int NI = LOW0 ? 3 : 4;
  constexpr int U = LOW0 ? 4 : 2;             // groups in flight
  __shared__ float2 carry[32][kRdm3Threads];
  cudaTriggerProgrammaticLaunchCompletion();
  const int tid = threadIdx.x;
  const bool upper = tid & 16;
  float f[32];
#pragma unroll
  for (int k = 0; k < 32; ++k) { f[k] = 0.f; carry[k][tid] = make_float2(0.f, 0.f); }
  int run = 0;
  auto flush = [&] {
#pragma unroll
    for (int k = 0; k < 32; ++k) {
      float2 c = carry[k][tid];
      df_acc(c.x, c.y, f[k] * a.down);
      carry[k][tid] = c;
      f[k] = 0.f;
    }
  };
  // pairs of lanes: pair index within the grid
  const uint64_t pair = (static_cast<uint64_t>(blockIdx.x) * kRdm3Threads + tid) >> 5 << 4 | (tid & 15);
  const uint64_t stride = static_cast<uint64_t>(gridDim.x) * (kRdm3Threads / 2);
  const uint64_t first = pair - (tid & 15);   // of the warp: the loop is uniform over it
  for (uint64_t w0 = first; w0 < a.num_groups; w0 += U * stride) {
    float4 v[U][NV];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const uint64_t g = w0 + (tid & 15) + u * stride;
      uint64_t base = g;
#pragma unroll
      for (int b = 0; b < NI; ++b) {
        const uint32_t s = a.ins[b];
        base = ((base >> s) << (s + 1)) | (base & ((1ull << s) - 1ull));
      }
      base >>= 1;
      if (upper) base += a.half;
#pragma unroll
      for (int m = 0; m < NV; ++m)
        v[u][m] = g < a.num_groups ? __ldg(psi + base + a.offs[m]) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
#pragma unroll
    for (int u = 0; u < U; ++u)
#pragma unroll
      for (int s = 0; s < SPG; ++s) {
        float2 own[4], x[4], y[2];
#pragma unroll
        for (int m = 0; m < 4; ++m) {
          const float4 w = v[u][LOW0 ? m / 2 : m];
          const bool second = LOW0 ? (m & 1) : s == 1;
          own[m] = second ? make_float2(w.z, w.w) : make_float2(w.x, w.y);
        }
        // corner: rows = the upper half's members, columns 0, 1 (lower lanes)
        // or 2, 3 (upper lanes) of the lower half's
#pragma unroll
        for (int m = 0; m < 4; ++m) {
          const float2 o = make_float2(__shfl_xor_sync(0xffffffffu, own[m].x, 16), __shfl_xor_sync(0xffffffffu, own[m].y, 16));
          x[m] = upper ? own[m] : o;
          if (m < 2 && !upper) y[m] = own[m];
          if (m >= 2 && upper) y[m - 2] = o;
        }
        int c = 0;
#pragma unroll
        for (int b = 0; b < 4; ++b) { f[c] = fmaf(own[b].x, own[b].x, fmaf(own[b].y, own[b].y, f[c])); ++c; }
        int pair = 0;
#pragma unroll
        for (int b = 0; b < 4; ++b)
#pragma unroll
          for (int aa = b + 1; aa < 4; ++aa) {
            f[c] = fmaf(own[b].x, own[aa].x, fmaf(own[b].y, own[aa].y, f[c])); ++c;
            f[c] = cross(own[b], own[aa], f[c], PERM && ((a.rev >> pair) & 1u)); ++c; ++pair;
          }
#pragma unroll
        for (int p = 0; p < 4; ++p)
#pragma unroll
          for (int q = 0; q < 2; ++q) {
            // y_q conj(x_p)
            f[c] = fmaf(y[q].x, x[p].x, fmaf(y[q].y, x[p].y, f[c])); ++c;
            f[c] = cross(y[q], x[p], f[c], PERM && ((a.rev >> (8 + 4 * (upper ? q + 2 : q) + p)) & 1u)); ++c;
          }
        if (++run == a.run) { flush(); run = 0; }
      }
  }
  flush();
  __syncthreads();
  // value (half, k): sum over the half's 64 threads, by two threads of 32
  __shared__ float2 part[kRdm3Threads];
  const int o = tid & 63, k = o & 31, hf = o >> 5, which = tid >> 6;
  float2 sum = make_float2(0.f, 0.f);
  for (int i = 0; i < 32; ++i) {
    const int j = which * 32 + ((i + tid) & 31);           // rotated: neighbouring threads read other banks
    sum = df_add(sum, carry[k][(j >> 4 << 5) | (hf << 4) | (j & 15)]);
  }
  part[tid] = sum;
  __syncthreads();
  if (tid < 64) partial[static_cast<size_t>(blockIdx.x) * 64 + tid] = df_add(part[tid], part[tid + 64]);
}

// Sets summed in FP32 before the carry.  The rounding of a run of R sets leaves
// about R / sqrt(3 sets) * 3e-8 of an entry (3e-10 at 2^20 sets with R = 16),
// but it does not average out in small states.
static int carry_run(double scale, int log_sets, int cap) {
  const double r = scale * exp2(0.5 * log_sets);
  return r < 1.0 ? 1 : (r > cap ? cap : static_cast<int>(r));
}

template <bool LOW0, bool PERM>
static cudaError_t rdm3_low(const float2* psi, int n, const uint32_t* s, uint32_t rev, const Scratch& scr,
                            cudaStream_t st) {
  Rdm3Args a{};
  int ni = 0;
  if (!LOW0) a.ins[ni++] = 0;
  for (int b = 0; b < 3; ++b) a.ins[ni++] = s[b];
  for (int m = 0; m < 4; ++m) {
    const int mem = LOW0 ? (2 * m) & 3 : m;                // the even member of load m
    a.offs[m] = ((mem & 1 ? 1ull << s[0] : 0) | (mem & 2 ? 1ull << s[1] : 0)) >> 1;
  }
  a.half = (1ull << s[2]) >> 1;
  a.num_groups = 1ull << (n - 3 - (LOW0 ? 0 : 1));
  a.run = carry_run(0.01, n - 3, kRdmChunk);
  a.rev = rev;
  a.down = scr.down;
  static PerDevice grid_dev;
  const int grid = grid_dev.get([] {
    int occ = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_rdm3<LOW0, PERM>, kRdm3Threads, 0);
    return sm_count() * (occ > 0 ? occ : 1);
  });
  const uint64_t per = static_cast<uint64_t>(kRdm3Threads / 2) * (LOW0 ? 4 : 2);
  uint64_t g = (a.num_groups + per - 1) / per;
  if (g > static_cast<uint64_t>(grid)) g = grid;
  if (g > static_cast<uint64_t>(kPartialDoubles / 64)) g = kPartialDoubles / 64;
  k_rdm3<LOW0, PERM><<<static_cast<unsigned>(g), kRdm3Threads, 0, st>>>(reinterpret_cast<const float4*>(psi), a, scr.partials());
  return finalize(scr.partials(), static_cast<int>(g), 64, scr.result, st);
}

// ---------------------------------------------------------------------------
// q = 4, 5 (k_gram): the block is a Hermitian rank-k update, 4 * 2^q FMA per
// amplitude counting both triangles, so the lower triangle is cut into 4 x 4
// complex tiles and a thread owns one (its "role": tile rows bi, columns bj)
// for the gather sets of its group: 8 members from shared memory feed 64
// FMAs.  Bound by FP32 FMA and the shared-memory reads that feed them.  A CTA
// stages 4096 amplitudes at a time, one set after the other; the next tile's
// loads are in flight while this one is multiplied.  Member m of a set sits
// at m + m / 16 of a row of odd pitch: the blocks a warp reads together then
// fall into different banks.  FP32 runs are carried in double-floats held in
// shared memory, which leaves 128 registers a thread, two CTAs an SM.  A run
// is 12 sets, the longest for which probabilities from the block are no
// further off than sums of |K_i v|^2 (rule at k_kraus_trace).
// n = 25, q = 4 / 5: 151 / 184 us (138 / 158 with runs of 30); the products K_i v that gave these
// channels' probabilities before took 2719 / 1584 us for each 16 / 4 operators.
// ---------------------------------------------------------------------------
template <int Q>
struct Gram {
  static constexpr int D = 1 << Q;
  static constexpr int NB = D / 4;                       // 4-member blocks
  static constexpr int ROLES = NB * (NB + 1) / 2;        // tiles of the lower triangle
  static constexpr int THREADS = 256;
  static constexpr int GROUPS = THREADS / ROLES;         // 25, 7 sets at a time
  static constexpr int TILE = 4096;                      // amplitudes staged at a time
  static constexpr int SETS = TILE / D;
  static constexpr int PITCH = D + 1;
  static constexpr int OUT = ROLES * 32;
  static constexpr size_t SMEM = sizeof(float2) * (SETS * PITCH + 32 * THREADS);
  static constexpr int NCH = TILE / 2 / THREADS;         // 8 128-bit loads a thread and tile
};

template <int Q>
struct GramArgs {
  uint64_t offs[1 << Q];      // amplitude offset of member m within a set
  uint64_t coff[8];           // what chunk c adds to a thread's address (amplitudes)
  uint32_t cset[8], cmem[8];  // what chunk c adds to the thread's set and member
  uint32_t ins[Q + 1];        // ascending bit positions to insert zeros at
  uint64_t num_tiles;
};

constexpr int kGramRun = 12;  // sets summed in FP32 before the carry

// bi, bj (bj <= bi) of tile r of the lower triangle
__device__ __forceinline__ void gram_tile(int r, int& bi, int& bj) {
  bi = 0;
  while ((bi + 1) * (bi + 2) / 2 <= r) ++bi;
  bj = r - bi * (bi + 1) / 2;
}

template <int Q, bool LOW0>
__global__ void __launch_bounds__(Gram<Q>::THREADS, 2) k_gram(const float2* __restrict__ psi,
                                                              const __grid_constant__ GramArgs<Q> a,
                                                              float2* __restrict__ partial) {
  using G = Gram<Q>;
  constexpr int NI = LOW0 ? Q : Q + 1;
  constexpr int LOGJ = (LOW0 ? 12 : 11) - Q;             // log2 of the sets (set pairs) of a tile
  extern __shared__ __align__(16) float2 s_gram[];
  float2* const tile_s = s_gram;                         // [SETS][PITCH]
  float2* const carry = s_gram + G::SETS * G::PITCH;     // [32][THREADS]
  cudaTriggerProgrammaticLaunchCompletion();
  const int tid = threadIdx.x;
  // chunk c of this thread is 128-bit word e = tid + 256 c of the tile: set
  // (pair) e mod 2^LOGJ, member (pair) e >> LOGJ; both split into a thread
  // part and a part that only depends on c
  const uint32_t j0 = tid & ((1u << (LOGJ < 8 ? LOGJ : 8)) - 1u);
  const uint32_t m0 = LOGJ < 8 ? static_cast<uint32_t>(tid) >> LOGJ : 0u;
  const uint32_t set0 = LOW0 ? j0 : 2u * j0, mem0 = LOW0 ? 2u * m0 : m0;
  auto spread = [&](uint64_t x) {
#pragma unroll
    for (int b = 0; b < NI; ++b) {
      const uint32_t s = a.ins[b];
      x = ((x >> s) << (s + 1)) | (x & ((1ull << s) - 1ull));
    }
    return x;
  };
  const uint64_t toff = spread(j0) | a.offs[mem0];
  const int role = tid % G::ROLES, group = tid / G::ROLES;
  const bool active = group < G::GROUPS;
  int bi, bj;
  gram_tile(role, bi, bj);
  const int xo = 4 * bi + (bi >> 2), yo = 4 * bj + (bj >> 2);
  float f[32];
#pragma unroll
  for (int k = 0; k < 32; ++k) {
    f[k] = 0.f;
    carry[k * G::THREADS + tid] = make_float2(0.f, 0.f);
  }
  float4 buf[G::NCH];
  auto load = [&](uint64_t tile) {
    const uint64_t base = spread(tile << LOGJ) | toff;
#pragma unroll
    for (int c = 0; c < G::NCH; ++c) buf[c] = __ldg(reinterpret_cast<const float4*>(psi + (base | a.coff[c])));
  };
  auto flush = [&] {
#pragma unroll
    for (int k = 0; k < 32; ++k) {
      float2 c = carry[k * G::THREADS + tid];
      df_acc(c.x, c.y, f[k]);
      carry[k * G::THREADS + tid] = c;
      f[k] = 0.f;
    }
  };
  uint64_t tile = blockIdx.x;
  load(tile);                                            // the grid has at most num_tiles blocks
  int run = 0;
  for (; tile < a.num_tiles; tile += gridDim.x) {
#pragma unroll
    for (int c = 0; c < G::NCH; ++c) {
      const uint32_t m = mem0 + a.cmem[c];
      float2* const d = tile_s + (set0 + a.cset[c]) * G::PITCH + m + (m >> 4);
      d[0] = make_float2(buf[c].x, buf[c].y);
      d[LOW0 ? 1 : G::PITCH] = make_float2(buf[c].z, buf[c].w);
    }
    __syncthreads();
    if (tile + gridDim.x < a.num_tiles) load(tile + gridDim.x);
    if (active) {
      for (int s = group; s < G::SETS; s += G::GROUPS) {
        const float2* const v = tile_s + s * G::PITCH;
        float2 x[4], y[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) { x[k] = v[xo + k]; y[k] = v[yo + k]; }
#pragma unroll
        for (int p = 0; p < 4; ++p)
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            // x_p conj(y_q)
            f[4 * p + q] = fmaf(x[p].x, y[q].x, fmaf(x[p].y, y[q].y, f[4 * p + q]));
            f[16 + 4 * p + q] = fmaf(x[p].y, y[q].x, fmaf(-x[p].x, y[q].y, f[16 + 4 * p + q]));
          }
        if (++run == kGramRun) { flush(); run = 0; }
      }
    }
    __syncthreads();                                     // the tile is read: its buffer is free
  }
  if (active) flush();
  __syncthreads();
  for (int o = tid; o < G::OUT; o += G::THREADS) {
    const int r = o >> 5, k = o & 31;
    float2 sum = make_float2(0.f, 0.f);
    for (int g = 0; g < G::GROUPS; ++g) sum = df_add(sum, carry[k * G::THREADS + g * G::ROLES + r]);
    partial[static_cast<size_t>(blockIdx.x) * G::OUT + o] = sum;
  }
}

// rho (2^Q x 2^Q, entry [b][a] at b * 2^Q + a) as double-floats
// (re.h, re.l, im.h, im.l) from the blocks' partial tiles
template <int Q>
__global__ void __launch_bounds__(kSumThreads) k_gram_matrix(const float2* partial, int nblocks, float4* rho) {
  using G = Gram<Q>;
  cudaGridDependencySynchronize();
  cudaTriggerProgrammaticLaunchCompletion();
  const int col = blockIdx.x * 32 + threadIdx.x % 32;    // OUT is a multiple of 32: block = one role
  float2 v = column_sum<32>(partial, nblocks, G::OUT, col);
  if (threadIdx.x >= 32) return;
  // lanes 0..15 hold the real parts of the tile's entries, 16..31 the imaginary ones
  const float2 w = df_shfl_xor(v, 16);
  int bi, bj;
  gram_tile(static_cast<int>(blockIdx.x), bi, bj);
  const int b = 4 * bi + ((threadIdx.x & 15) >> 2), c = 4 * bj + (threadIdx.x & 3);
  if (b < c) return;                                     // upper half of a diagonal tile
  if (threadIdx.x < 16) rho[b * G::D + c] = b == c ? make_float4(v.x, v.y, 0.f, 0.f) : make_float4(v.x, v.y, w.x, w.y);
  else if (b > c) rho[c * G::D + b] = make_float4(w.x, w.y, -v.x, -v.y);
}

template <int Q, bool LOW0>
static cudaError_t gram_low(const float2* psi, int n, const uint32_t* s, float2* partial, int max_blocks, int* blocks,
                            cudaStream_t st) {
  using G = Gram<Q>;
  constexpr int LOGJ = (LOW0 ? 12 : 11) - Q;
  GramArgs<Q> a{};
  int ni = 0;
  if (!LOW0) a.ins[ni++] = 0;
  for (int b = 0; b < Q; ++b) a.ins[ni++] = s[b];
  for (int m = 0; m < G::D; ++m) {
    uint64_t o = 0;
    for (int b = 0; b < Q; ++b)
      if ((m >> b) & 1) o |= 1ull << s[b];
    a.offs[m] = o;
  }
  for (int c = 0; c < 8; ++c) {
    const uint32_t e = 256u * c;
    const uint32_t j = e & ((1u << LOGJ) - 1u), m = e >> LOGJ;
    a.cset[c] = LOW0 ? j : 2 * j;
    a.cmem[c] = LOW0 ? 2 * m : m;
    uint64_t x = j;
    for (int b = 0; b < ni; ++b) x = ((x >> a.ins[b]) << (a.ins[b] + 1)) | (x & ((1ull << a.ins[b]) - 1ull));
    a.coff[c] = x | a.offs[a.cmem[c]];
  }
  a.num_tiles = 1ull << (n - 12);                        // n - Q >= kGramMinLog: whole tiles
  static PerDevice setup;
  const int grid = setup.get([] {
    if (cudaFuncSetAttribute(k_gram<Q, LOW0>, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(G::SMEM)) !=
        cudaSuccess)
      return 0;
    int occ = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_gram<Q, LOW0>, G::THREADS, G::SMEM);
    return sm_count() * (occ > 0 ? occ : 1);
  });
  if (grid <= 0) return cudaErrorInvalidConfiguration;
  uint64_t g = a.num_tiles;
  if (g > static_cast<uint64_t>(grid)) g = grid;
  if (g > static_cast<uint64_t>(max_blocks)) g = max_blocks;
  *blocks = static_cast<int>(g);
  k_gram<Q, LOW0><<<static_cast<unsigned>(g), G::THREADS, G::SMEM, st>>>(psi, a, partial);
  return cudaGetLastError();
}

template <int Q>
static cudaError_t gram_q(const float2* psi, int n, const uint32_t* qubits, float2* partial, int max_blocks, int* blocks,
                          cudaStream_t st) {
  uint32_t s[Q];
  sort_qubits<Q>(qubits, s);
  return s[0] == 0 ? gram_low<Q, true>(psi, n, s, partial, max_blocks, blocks, st)
                   : gram_low<Q, false>(psi, n, s, partial, max_blocks, blocks, st);
}

template <int Q>
static cudaError_t rdm_q(const float2* psi, int n, const uint32_t* qubits, const Scratch& scr, cudaStream_t st) {
  uint32_t s[Q];
  sort_qubits<Q>(qubits, s);
  return s[0] == 0 ? rdm_low<Q, true>(psi, n, qubits, s, scr, st) : rdm_low<Q, false>(psi, n, qubits, s, scr, st);
}

cudaError_t launch_rdm(const float2* psi, int n, int q, const uint32_t* qubits, const Scratch& scr,
                       cudaStream_t st) {
  if (q > n) return cudaErrorInvalidValue;
  switch (q) {
    case 1: return rdm_q<1>(psi, n, qubits, scr, st);
    case 2: return rdm_q<2>(psi, n, qubits, scr, st);
    case 3: {
      uint32_t s[3];
      sort_qubits<3>(qubits, s);
      uint32_t rev = 0;
      if (n - 3 < kRdm3OrderLog) {
        int rank[3], pair = 0;
        for (int j = 0; j < 3; ++j) rank[j] = (qubits[j] > s[0]) + (qubits[j] > s[1]);
        for (int b = 0; b < 4; ++b)
          for (int a = b + 1; a < 4; ++a) rev |= static_cast<uint32_t>(member_after(3, rank, b, a)) << pair++;
        for (int y = 0; y < 4; ++y)
          for (int x = 0; x < 4; ++x) rev |= static_cast<uint32_t>(member_after(3, rank, y, 4 + x)) << (8 + 4 * y + x);
      }
      if (rev) return s[0] == 0 ? rdm3_low<true, true>(psi, n, s, rev, scr, st) : rdm3_low<false, true>(psi, n, s, rev, scr, st);
      return s[0] == 0 ? rdm3_low<true, false>(psi, n, s, 0, scr, st) : rdm3_low<false, false>(psi, n, s, 0, scr, st);
    }
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t read_rdm(const float2* psi, int n, int q, const uint32_t* qubits, Scratch scr, cudaStream_t st, double* r) {
  const int W = 1 << (2 * q);
  for (;;) {
    cudaError_t e = launch_rdm(psi, n, q, qubits, scr, st);
    if (e == cudaSuccess) e = cudaMemcpyAsync(r, scr.result, sizeof(double) * W, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) return e;
    if (scr.down != 1.f) {
      for (int k = 0; k < W; ++k) r[k] /= scr.down;
      return cudaSuccess;
    }
    if (std::all_of(r, r + W, [](double x) { return std::isfinite(x); })) return cudaSuccess;
    scr.down = kRangeDown;
  }
}

void rdm_unpack(int q, const uint32_t* qubits, const double* r, double* rho) {
  const int D = 1 << q;
  // basis index over `qubits` of basis index x over the sorted qubits
  auto user = [&](int x) {
    int u = 0;
    for (int b = 0; b < q; ++b) {
      int pos = 0;
      for (int k = 0; k < q; ++k) pos += qubits[k] < qubits[b];
      u |= ((x >> pos) & 1) << b;
    }
    return u;
  };
  auto put = [&](int sb, int sa, double re, double im) {   // rho[b][a] = sum psi_b conj(psi_a), Hermitian
    const int b = user(sb), a = user(sa);
    rho[2 * (b * D + a)] = re;
    rho[2 * (b * D + a) + 1] = im;
    rho[2 * (a * D + b)] = re;
    rho[2 * (a * D + b) + 1] = a == b ? im : -im;
  };
  if (q == 3) {                                            // per half: its triangle, two columns of the corner
    for (int h = 0; h < 2; ++h, r += 32) {
      for (int b = 0; b < 4; ++b) put(4 * h + b, 4 * h + b, r[b], 0.0);
      int c = 4;
      for (int b = 0; b < 4; ++b)
        for (int a = b + 1; a < 4; ++a, c += 2) put(4 * h + b, 4 * h + a, r[c], r[c + 1]);
      for (int p = 0; p < 4; ++p)
        for (int k = 0; k < 2; ++k, c += 2) put(2 * h + k, 4 + p, r[c], r[c + 1]);
    }
    return;
  }
  int c = 0;
  for (int b = 0; b < D; ++b) put(b, b, r[c++], 0.0);
  for (int b = 0; b < D; ++b)
    for (int a = b + 1; a < D; ++a) {
      const double re = r[c++], im = r[c++];
      put(b, a, re, im);
    }
}

// ---------------------------------------------------------------------------
// Branch probabilities of a channel on 4 or 5 qubits (Alg. 2 step 14).  With
// rho the reduced density block, P_i = <psi|K_i^dag K_i|psi> is
//   sum_j k_j rho k_j^dag   over the rows k_j of K_i,
// so one pass over the state serves every operator of the channel, where
// forming |K_i v|^2 per operator costs twice the arithmetic of rho each.  The
// contraction (2^(3q) products per operator) is far below the pass but wants
// more than FP32; FP64 is slow here, so rho enters as double-floats and the
// products keep their FMA error term.  The operators are complex64.
//
// The rounding of rho's entries, independent of one another, moves P_i by about
// 1.5e-7 E_i, E_i^2 = sum_ab |(K_i^dag K_i)_ab|^2 rho_aa rho_bb, and where the
// terms of P_i cancel (a state near the kernel of K_i) that is all there is: a
// true 1e-6 N comes out 10 % off, a true 0 negative.  |K_i v|^2 keeps its
// relative accuracy, 1.5e-7 of P_i.  So an operator with E_i > P_i is left to
// k_kraus_norms by the caller.  Relative errors with E_i <= P_i, runs of 12
// sets, all sets alike (nothing averages out), 4-qubit operators, rms here /
// of |K_i v|^2: E_i in (0.8, 1] P_i dense 1.2e-7 / 1.6e-7, a single entry 1.2e-7 /
// 1.3e-7; in (1, 2] P_i, left out, 1.6e-7..1.9e-7 / 1.7e-7; runs of 16 sets, a
// single entry 1.7e-7.  A maximally mixed rho has E_i <= P_i for every K_i.
//
// From 2^18 gather sets on (kGramMinLog), where on states whose sets differ
// the FP32 rounding of both forms averages out below 1e-9.  For q = 6 the
// rows of 128 FP32 terms of k_norms64 leave a mean of -6e-10 at any size, which
// the two forms would then differ by; it has no such pass.
// ---------------------------------------------------------------------------
// acc += x y, x a double-float
__device__ __forceinline__ void df_mul_acc(float2& acc, float xh, float xl, float y) {
  const float p = xh * y;
  const float e = fmaf(xl, y, fmaf(xh, y, -p));
  df_acc(acc.x, acc.y, p);
  acc.y += e;
}

// block (x, i): 256 of the terms (eight b, entry a, row j) of operator i,
// Re(k_ja sum_b rho[a][b] conj(k_jb)), summed into out[i * gridDim.x + x]; the
// last D^2 / 256 blocks of an operator put 256 terms each of E_i^2 there
template <int Q>
__global__ void __launch_bounds__(256) k_kraus_trace(const float4* rho, const float2* __restrict__ ops, double* out) {
  constexpr int D = 1 << Q;
  __shared__ float2 s_sum[8];
  cudaGridDependencySynchronize();
  constexpr int TERMS = D * D * D / 8 / 256;             // blocks of P_i
  if (blockIdx.x >= TERMS) {
    __shared__ double s_part[8];
    const float2* const K = ops + static_cast<size_t>(blockIdx.y) * D * D;
    const int e = (blockIdx.x - TERMS) * 256 + threadIdx.x, x = e % D, y = e / D;
    float gr = 0.f, gi = 0.f;
#pragma unroll 8
    for (int r = 0; r < D; ++r) {
      const float2 u = __ldg(K + r * D + x), v = __ldg(K + r * D + y);
      gr = fmaf(u.x, v.x, fmaf(u.y, v.y, gr));
      gi = fmaf(u.x, v.y, fmaf(-u.y, v.x, gi));
    }
    const double g = gr, h = gi;                         // products of four factors would leave FP32's range
    double s = (g * g + h * h) * (static_cast<double>(rho[x * (D + 1)].x) * static_cast<double>(rho[y * (D + 1)].x));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if ((threadIdx.x & 31) == 0) s_part[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
      for (int w = 1; w < 8; ++w) s += s_part[w];
      out[blockIdx.y * gridDim.x + blockIdx.x] = s;
    }
    return;
  }
  const int idx = blockIdx.x * 256 + threadIdx.x, a = idx % D, j = (idx / D) % D, b0 = idx / (D * D) * 8;
  const float2* const k = ops + (static_cast<size_t>(blockIdx.y) * D + j) * D;
  float2 tr = make_float2(0.f, 0.f), ti = make_float2(0.f, 0.f);
#pragma unroll 4
  for (int b = b0; b < b0 + 8; ++b) {
    // rho[a][b] = conj(rho[b][a]); lanes read neighbouring a
    const float4 r = rho[b * D + a];
    const float2 c = __ldg(k + b);
    // conj(r) conj(c)
    df_mul_acc(tr, r.x, r.y, c.x);
    df_mul_acc(tr, -r.z, -r.w, c.y);
    df_mul_acc(ti, -r.x, -r.y, c.y);
    df_mul_acc(ti, -r.z, -r.w, c.x);
  }
  const float2 c = __ldg(k + a);
  float2 v[1] = {make_float2(0.f, 0.f)};
  df_mul_acc(v[0], tr.x, tr.y, c.x);
  df_mul_acc(v[0], ti.x, ti.y, -c.y);
  const float2 s = df_warp_sum<1>(v, threadIdx.x & 31);
  if ((threadIdx.x & 31) == 0) s_sum[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    float2 r = s_sum[0];
    for (int w = 1; w < 8; ++w) r = df_add(r, s_sum[w]);
    out[blockIdx.y * gridDim.x + blockIdx.x] = df_value(r);
  }
}

int kraus_error_slices(int q) { return (1 << (2 * q)) / 256; }
int kraus_slices(int q) { return (1 << (3 * q - 3)) / 256 + kraus_error_slices(q); }

// the result rows, padded so that the operators after them are 16-byte aligned
size_t kraus_results(int q, int nops) { return (static_cast<size_t>(nops) * kraus_slices(q) + 1) & ~size_t(1); }

static int kraus_grid() { return sm_count() * 2; }

size_t kraus_scratch_bytes(int q, int nops) {
  const size_t D = 1ull << q, nb = D / 4, out = nb * (nb + 1) / 2 * 32;
  return sizeof(double) * kraus_results(q, nops) + sizeof(float2) * nops * D * D + sizeof(float4) * D * D +
         sizeof(float2) * kraus_grid() * out;
}

void kraus_sort_columns(int q, const uint32_t* qubits, const double* K, float2* out) {
  const int D = 1 << q;
  for (int a = 0; a < D; ++a) {                          // column of sorted-basis index a
    int u = 0;
    for (int b = 0; b < q; ++b) {
      int pos = 0;
      for (int k = 0; k < q; ++k) pos += qubits[k] < qubits[b];
      u |= ((a >> pos) & 1) << b;
    }
    for (int j = 0; j < D; ++j)
      out[j * D + a] = make_float2(static_cast<float>(K[2 * (j * D + u)]), static_cast<float>(K[2 * (j * D + u) + 1]));
  }
}

template <int Q>
static cudaError_t kraus_q(const float2* psi, int n, const uint32_t* qubits, int nops, void* scratch, cudaStream_t st) {
  using G = Gram<Q>;
  double* const out = static_cast<double*>(scratch);
  float2* const ops = reinterpret_cast<float2*>(out + kraus_results(Q, nops));
  float4* const rho = reinterpret_cast<float4*>(ops + static_cast<size_t>(nops) * G::D * G::D);
  float2* const partial = reinterpret_cast<float2*>(rho + G::D * G::D);
  int g = 0;
  cudaError_t e = gram_q<Q>(psi, n, qubits, partial, kraus_grid(), &g, st);
  if (e == cudaSuccess) e = launch_dependent(k_gram_matrix<Q>, dim3(G::ROLES), kSumThreads, st, partial, g, rho);
  if (e == cudaSuccess)
    e = launch_dependent(k_kraus_trace<Q>, dim3(kraus_slices(Q), nops), 256, st, rho, ops, out);
  return e;
}

cudaError_t launch_kraus_probs(const float2* psi, int n, int q, const uint32_t* qubits, int nops, void* scratch,
                               cudaStream_t st) {
  if (q > n || nops < 1) return cudaErrorInvalidValue;
  switch (q) {
    case 4: return kraus_q<4>(psi, n, qubits, nops, scratch, st);
    case 5: return kraus_q<5>(psi, n, qubits, nops, scratch, st);
    default: return cudaErrorInvalidValue;
  }
}

// Channels on 4 and 5 qubits of smaller states: for G operators at a time, P_i = sum over gather sets of
// |K_i v|^2, plus N = <psi|psi>.  Each thread takes whole gather sets, staged
// column-wise in shared memory (member m of thread t at v[m * blockDim + t],
// conflict-free), with the G operators in shared memory.  Products and row
// sums in FP32; runs of kKrausChunk sets in FP32, carried in double-floats.
// result[0] = N, result[1 + i] = P_i.
constexpr int kKrausThreads = 128;
constexpr int kKrausChunk = 16;

template <int Q>
struct KrausArgs {
  uint64_t offs[1 << Q];
  uint32_t ins[Q];
  uint64_t num_sets;
  const float2* ops;            // G matrices 2^Q x 2^Q, row-major (basis bit b <-> qubits[b])
  float down;                   // Scratch::down
};

template <int Q, int G>
__global__ void __launch_bounds__(kKrausThreads) k_kraus_norms(const float2* __restrict__ psi,
                                                               const __grid_constant__ KrausArgs<Q> a,
                                                               float2* __restrict__ partial) {
  constexpr int D = 1 << Q, W = G + 1;
  extern __shared__ __align__(16) float2 s_dyn[];
  float2* sK = s_dyn;                          // G * D * D
  float2* sv = s_dyn + G * D * D;              // D * blockDim
  cudaTriggerProgrammaticLaunchCompletion();
  for (int i = threadIdx.x; i < G * D * D; i += blockDim.x) sK[i] = a.ops[i];
  __syncthreads();
  float ah[W], al[W], f[W];
#pragma unroll
  for (int c = 0; c < W; ++c) { ah[c] = 0.f; al[c] = 0.f; f[c] = 0.f; }
  int cnt = 0;
  const int t = threadIdx.x, bd = blockDim.x;
  const uint64_t stride = static_cast<uint64_t>(gridDim.x) * blockDim.x;
  for (uint64_t i = static_cast<uint64_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < a.num_sets;
       i += stride) {
    uint64_t base = i;
#pragma unroll
    for (int b = 0; b < Q; ++b) {
      const uint32_t s = a.ins[b];
      base = ((base >> s) << (s + 1)) | (base & ((1ull << s) - 1ull));
    }
    for (int m = 0; m < D; ++m) {
      const float2 v = __ldg(psi + base + a.offs[m]);
      sv[m * bd + t] = v;
      f[0] = fmaf(v.x, v.x, fmaf(v.y, v.y, f[0]));
    }
#pragma unroll
    for (int g = 0; g < G; ++g) {
      const float2* K = sK + g * D * D;
      float row = 0.f;
      for (int j = 0; j < D; ++j) {
        float wr = 0.f, wi = 0.f;
#pragma unroll 8
        for (int m = 0; m < D; ++m) {
          const float2 k = K[j * D + m];
          const float2 v = sv[m * bd + t];
          wr = fmaf(k.x, v.x, fmaf(-k.y, v.y, wr));
          wi = fmaf(k.x, v.y, fmaf(k.y, v.x, wi));
        }
        row = fmaf(wr, wr, fmaf(wi, wi, row));
      }
      f[1 + g] += row;
    }
    if (++cnt == kKrausChunk) {
#pragma unroll
      for (int k = 0; k < W; ++k) { df_acc(ah[k], al[k], f[k] * a.down); f[k] = 0.f; }
      cnt = 0;
    }
  }
#pragma unroll
  for (int k = 0; k < W; ++k) df_acc(ah[k], al[k], f[k] * a.down);
  block_reduce_store<W>(ah, al, partial);
}

template <int Q, int G>
static cudaError_t kraus_norms_q(const float2* psi, int n, const uint32_t* qubits, const float2* ops_dev,
                                 const Scratch& scr, cudaStream_t st) {
  constexpr int D = 1 << Q;
  KrausArgs<Q> a;
  uint32_t s[Q];
  for (int b = 0; b < Q; ++b) s[b] = qubits[b];
  for (int i = 1; i < Q; ++i)
    for (int j = i; j > 0 && s[j - 1] > s[j]; --j) { const uint32_t t = s[j]; s[j] = s[j - 1]; s[j - 1] = t; }
  for (int b = 0; b < Q; ++b) a.ins[b] = s[b];
  for (int m = 0; m < D; ++m) {
    uint64_t o = 0;
    for (int b = 0; b < Q; ++b)
      if ((m >> b) & 1) o |= 1ull << qubits[b];
    a.offs[m] = o;
  }
  a.num_sets = 1ull << (n - Q);
  a.ops = ops_dev;
  a.down = scr.down;
  const size_t smem = sizeof(float2) * (static_cast<size_t>(G) * D * D + static_cast<size_t>(D) * kKrausThreads);
  static PerDevice setup;
  const int grid = setup.get([smem] {
    if (cudaFuncSetAttribute(k_kraus_norms<Q, G>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             static_cast<int>(smem)) != cudaSuccess)
      return 0;
    int occ = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_kraus_norms<Q, G>, kKrausThreads, smem);
    const int g = sm_count() * (occ > 0 ? occ : 1);
    return g < kMaxRedBlocks ? g : kMaxRedBlocks;
  });
  if (grid <= 0) return cudaErrorInvalidConfiguration;
  const uint64_t need = (a.num_sets + kKrausThreads - 1) / kKrausThreads;
  const int g = static_cast<int>(need < static_cast<uint64_t>(grid) ? need : grid);
  k_kraus_norms<Q, G><<<g, kKrausThreads, smem, st>>>(psi, a, scr.partials());
  return finalize(scr.partials(), g, G + 1, scr.result, st);
}

int kraus_group(int q) { return q <= 4 ? 16 : (q == 5 ? 4 : 1); }

cudaError_t launch_kraus_norms(const float2* psi, int n, int q, const uint32_t* qubits, int nops,
                               const float2* ops_dev, const Scratch& scr, cudaStream_t st) {
  if (q > n || nops != kraus_group(q)) return cudaErrorInvalidValue;
  switch (q) {
    case 4: return kraus_norms_q<4, 16>(psi, n, qubits, ops_dev, scr, st);
    case 5: return kraus_norms_q<5, 4>(psi, n, qubits, ops_dev, scr, st);
    case 6: {                             // k_mat64.cu
      int g = 0;
      const cudaError_t e = launch_norms64(psi, n, qubits, ops_dev, scr.down, scr.partials(), &g, st);
      return e != cudaSuccess ? e : finalize(scr.partials(), g, 2, scr.result, st);
    }
    default: return cudaErrorInvalidValue;
  }
}

// ---------------------------------------------------------------------------
// Z-string expectations: result[0] = N, result[1+m] = sum_x |psi_x|^2 (-1)^popc(x & mask_m)
// ---------------------------------------------------------------------------
struct ExpArgs {
  uint64_t masks[kExpGroup];
  int nm;
  uint64_t num_pairs;
  float down;                   // Scratch::down
};

constexpr int kExpChunk = 64;

__global__ void __launch_bounds__(kRedThreads) k_expect(const float2* __restrict__ psi,
                                                        const __grid_constant__ ExpArgs a,
                                                        float2* __restrict__ partial) {
  constexpr int W = kExpGroup + 1;
  cudaTriggerProgrammaticLaunchCompletion();
  float ah[W], al[W], f[W];
#pragma unroll
  for (int c = 0; c < W; ++c) { ah[c] = 0.f; al[c] = 0.f; f[c] = 0.f; }
  int cnt = 0;
  const uint64_t stride = static_cast<uint64_t>(gridDim.x) * blockDim.x;
  for (uint64_t i = static_cast<uint64_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < a.num_pairs;
       i += stride) {
    const float4 v = __ldg(reinterpret_cast<const float4*>(psi) + i);
    const float w0 = fmaf(v.x, v.x, v.y * v.y), w1 = fmaf(v.z, v.z, v.w * v.w);
    const uint64_t x0 = 2 * i;
    f[0] += w0 + w1;
#pragma unroll
    for (int m = 0; m < kExpGroup; ++m) {
      if (m < a.nm) {
        const uint64_t mk = a.masks[m];
        const int s0 = __popcll(x0 & mk) & 1;
        const int s1 = s0 ^ static_cast<int>(mk & 1ull);
        f[1 + m] += (s0 ? -w0 : w0) + (s1 ? -w1 : w1);
      }
    }
    if (++cnt == kExpChunk) {
#pragma unroll
      for (int k = 0; k < W; ++k) { df_acc(ah[k], al[k], f[k] * a.down); f[k] = 0.f; }
      cnt = 0;
    }
  }
#pragma unroll
  for (int k = 0; k < W; ++k) df_acc(ah[k], al[k], f[k] * a.down);
  block_reduce_store<W>(ah, al, partial);
}

// n >= 9: a warp takes blocks of 512 amplitudes and lane l holds the 16
// amplitudes x = (blk << 9) | (j << 6) | (l << 1) | e, j = 0..7, e = 0..1,
// read with eight coalesced 128-bit loads.  Over the bits that vary inside
// the thread (0, 6, 7, 8) its 16 weights are Walsh-Hadamard transformed,
//   W[u] = sum_v (-1)^popc(u & v) w[v],   v = e | (j << 1),
// so that the block's share of sum_x |psi_x|^2 (-1)^popc(x & m) is
// (-1)^(parity of m on the fixed bits) * W[u_m], u_m being m's bits 0, 6, 7,
// 8.  The parity over the lane bits (1..5) is fixed per thread and the one
// over the block bits (>= 9) is one popc, so a mask costs a few instructions
// per 16 amplitudes.  FP32 runs cover 8 blocks (128 amplitudes per thread),
// then a carry.
struct ExpWArgs {
  uint32_t mblk[kExpGroup];     // mask bits >= 9, shifted down by 9
  uint32_t mlane[kExpGroup];    // mask bits 1..5, shifted down by 1
  uint32_t u[kExpGroup];        // mask bits (0, 6, 7, 8) as a 4-bit index
  int nm;
  uint64_t num_blocks;          // 2^(n - 9)
  float down;                   // Scratch::down
};

constexpr int kExpWChunk = 8;

__global__ void __launch_bounds__(kRedThreads) k_expect_wht(const float2* __restrict__ psi,
                                                            const __grid_constant__ ExpWArgs a,
                                                            float2* __restrict__ partial) {
  constexpr int W = kExpGroup + 1;
  __shared__ float s_w[kRedThreads][17];        // each thread's transformed weights (padded row)
  cudaTriggerProgrammaticLaunchCompletion();
  float ah[W], al[W], f[W];
#pragma unroll
  for (int c = 0; c < W; ++c) { ah[c] = 0.f; al[c] = 0.f; f[c] = 0.f; }
  const uint32_t lane = threadIdx.x & 31u;
  const uint64_t warp = (static_cast<uint64_t>(blockIdx.x) * blockDim.x + threadIdx.x) >> 5;
  const uint64_t nwarps = (static_cast<uint64_t>(gridDim.x) * blockDim.x) >> 5;
  uint32_t slane = 0;                           // bit m: parity of mask m on the lane bits
  for (int m = 0; m < a.nm; ++m) slane |= (static_cast<uint32_t>(__popc(lane & a.mlane[m])) & 1u) << m;
  const float4* p4 = reinterpret_cast<const float4*>(psi);
  float* row = s_w[threadIdx.x];
  int cnt = 0;
  for (uint64_t blk = warp; blk < a.num_blocks; blk += nwarps) {
    float w[16];
    float4 q[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) q[j] = __ldg(p4 + (blk << 8) + j * 32 + lane);
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      w[2 * j] = fmaf(q[j].x, q[j].x, q[j].y * q[j].y);
      w[2 * j + 1] = fmaf(q[j].z, q[j].z, q[j].w * q[j].w);
    }
    if (a.nm > 0) {
#pragma unroll
      for (int h = 1; h < 16; h <<= 1)
#pragma unroll
        for (int i = 0; i < 16; ++i)
          if ((i & h) == 0) {
            const float x = w[i], y = w[i | h];
            w[i] = x + y;
            w[i | h] = x - y;
          }
      f[0] += w[0];
#pragma unroll
      for (int u = 0; u < 16; ++u) row[u] = w[u];
      const uint32_t b32 = static_cast<uint32_t>(blk);
#pragma unroll
      for (int m = 0; m < kExpGroup; ++m) {
        if (m < a.nm) {
          const float val = row[a.u[m]];
          const uint32_t sgn = (static_cast<uint32_t>(__popc(b32 & a.mblk[m])) ^ (slane >> m)) & 1u;
          f[1 + m] += sgn ? -val : val;
        }
      }
    } else {
      float t = 0.f;
#pragma unroll
      for (int v = 0; v < 16; ++v) t += w[v];
      f[0] += t;
    }
    if (++cnt == kExpWChunk) {
#pragma unroll
      for (int k = 0; k < W; ++k) { df_acc(ah[k], al[k], f[k] * a.down); f[k] = 0.f; }
      cnt = 0;
    }
  }
#pragma unroll
  for (int k = 0; k < W; ++k) df_acc(ah[k], al[k], f[k] * a.down);
  block_reduce_store<W>(ah, al, partial);
}

cudaError_t launch_expect(const float2* psi, int n, int nm, const uint64_t* masks,
                          const Scratch& scr, cudaStream_t st) {
  if (nm > kExpGroup || n < 1) return cudaErrorInvalidValue;
  if (n >= 9) {
    ExpWArgs a;
    for (int m = 0; m < kExpGroup; ++m) {
      const uint64_t mk = m < nm ? masks[m] : 0;
      a.mblk[m] = static_cast<uint32_t>(mk >> 9);
      a.mlane[m] = static_cast<uint32_t>((mk >> 1) & 31u);
      a.u[m] = static_cast<uint32_t>((mk & 1u) | (((mk >> 6) & 7u) << 1));
    }
    a.nm = nm;
    a.num_blocks = 1ull << (n - 9);
    a.down = scr.down;
    static PerDevice gridw_dev;
    const int gridw = gridw_dev.get([] { return red_grid(k_expect_wht, ~0ull >> 1); });
    const uint64_t need = (a.num_blocks * 32 + kRedThreads - 1) / kRedThreads;
    const int g = static_cast<int>(need < static_cast<uint64_t>(gridw) ? need : gridw);
    k_expect_wht<<<g, kRedThreads, 0, st>>>(psi, a, scr.partials());
    return finalize(scr.partials(), g, kExpGroup + 1, scr.result, st);
  }
  ExpArgs a;
  for (int m = 0; m < kExpGroup; ++m) a.masks[m] = m < nm ? masks[m] : 0;
  a.nm = nm;
  a.num_pairs = 1ull << (n - 1);
  a.down = scr.down;
  static PerDevice grid_dev;
  const int grid = grid_dev.get([] { return red_grid(k_expect, ~0ull >> 1); });
  const uint64_t need = (a.num_pairs + kRedThreads - 1) / kRedThreads;
  const int g = static_cast<int>(need < static_cast<uint64_t>(grid) ? need : grid);
  k_expect<<<g, kRedThreads, 0, st>>>(psi, a, scr.partials());
  return finalize(scr.partials(), g, kExpGroup + 1, scr.result, st);
}

// ---------------------------------------------------------------------------
// Sampling.  C(x) is built in three levels with one fixed arithmetic, used
// both to build the block table and to search inside a block, so that the
// search sees the same cumulative values the table was built from:
//   chunk      64 amplitudes, warp inclusive scan in FP32 of (|a0|^2+|a1|^2)
//   sub-block  16 chunks, running FP32 sum of chunk totals  -> cdf_sub
//   block      64 sub-blocks, warp inclusive scan in FP64   -> block totals
//   table      inclusive FP64 scan of the block totals      -> cdf_cum
// A sample with uniform u targets t = u * C(2^n - 1) and returns the
// smallest x with t < C(x).
// ---------------------------------------------------------------------------
__device__ __forceinline__ float warp_incl_scan_f(float v, int lane) {
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const float y = __shfl_up_sync(0xffffffffu, v, o);
    if (lane >= o) v += y;
  }
  return v;
}

__device__ __forceinline__ double warp_incl_scan_d(double v, int lane) {
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const double y = __shfl_up_sync(0xffffffffu, v, o);
    if (lane >= o) v += y;
  }
  return v;
}

// weights of the two amplitudes a lane owns in a chunk (0 past the end)
__device__ __forceinline__ void chunk_weights(const float2* __restrict__ psi, uint64_t namps,
                                              uint64_t x0, float& w0, float& w1) {
  w0 = 0.f;
  w1 = 0.f;
  if (x0 < namps) {
    const float4 v = __ldg(reinterpret_cast<const float4*>(psi + x0));
    w0 = fmaf(v.x, v.x, v.y * v.y);
    w1 = fmaf(v.z, v.z, v.w * v.w);
  }
}

// Sums of a sub-block's 16 chunks, each in the order in which lane 31 of an
// inclusive warp scan forms it (a binary tree over neighbouring lanes): lane
// l (any l with the same low four bits) returns the sum of chunk l & 15.
// Transposed: step o combines lanes o apart and halves the chunks a lane
// holds, 16 exchanges for 16 chunks where one scan per chunk makes 80.
__device__ __forceinline__ float chunk_sums(float (&p)[16], int lane) {
  int c = 16;
#pragma unroll
  for (int o = 1; o < 16; o <<= 1) {
    c >>= 1;
    const bool up = lane & o;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      if (k >= c) break;
      // chunks with bit o set go to the lanes with bit o set
      const float keep = up ? p[2 * k + 1] : p[2 * k], send = up ? p[2 * k] : p[2 * k + 1];
      p[k] = keep + __shfl_xor_sync(0xffffffffu, send, o);
    }
  }
  return p[0] + __shfl_xor_sync(0xffffffffu, p[0], 16);
}

// One warp per sub-block, its 1024 amplitudes (8 KB) loaded before any
// arithmetic.  Bound by HBM; n = 29: 782 -> 612 us (one chunk at a time, a
// scan for each, before).
__global__ void __launch_bounds__(256) k_cdf_sub(const float2* __restrict__ psi, uint64_t namps, uint64_t nsub,
                                                 float* __restrict__ sub) {
  constexpr int CH = 1 << (kCdfSubLog - kCdfChunkLog);
  static_assert(CH == 16);
  cudaTriggerProgrammaticLaunchCompletion();
  const int lane = threadIdx.x & 31;
  const uint64_t warp = (static_cast<uint64_t>(blockIdx.x) * blockDim.x + threadIdx.x) >> 5;
  const uint64_t nwarps = (static_cast<uint64_t>(gridDim.x) * blockDim.x) >> 5;
  for (uint64_t s = warp; s < nsub; s += nwarps) {
    float4 v[CH];
#pragma unroll
    for (int c = 0; c < CH; ++c) {
      const uint64_t x0 = (s << kCdfSubLog) + (static_cast<uint64_t>(c) << kCdfChunkLog) + 2 * lane;
      v[c] = x0 < namps ? __ldg(reinterpret_cast<const float4*>(psi + x0)) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
    float p[CH];
#pragma unroll
    for (int c = 0; c < CH; ++c)
      p[c] = fmaf(v[c].x, v[c].x, v[c].y * v[c].y) + fmaf(v[c].z, v[c].z, v[c].w * v[c].w);
    const float sum = chunk_sums(p, lane);
    float run = 0.f;
#pragma unroll
    for (int c = 0; c < CH; ++c) run += __shfl_sync(0xffffffffu, sum, c);
    if (lane == 0) sub[s] = run;
  }
}

// lane values of block b: (double)sub[2L] + (double)sub[2L+1]
__device__ __forceinline__ void block_lane_values(const float* sub, uint64_t nsub,
                                                  uint64_t b, int lane, double& s0, double& s1) {
  const uint64_t i0 = (b << 6) + 2 * lane;
  s0 = i0 < nsub ? static_cast<double>(sub[i0]) : 0.0;
  s1 = i0 + 1 < nsub ? static_cast<double>(sub[i0 + 1]) : 0.0;
}

__global__ void k_cdf_blk(const float* sub, uint64_t nsub, uint64_t nblk, double* cum) {
  cudaGridDependencySynchronize();
  cudaTriggerProgrammaticLaunchCompletion();
  const int lane = threadIdx.x & 31;
  const uint64_t warp = (static_cast<uint64_t>(blockIdx.x) * blockDim.x + threadIdx.x) >> 5;
  const uint64_t nwarps = (static_cast<uint64_t>(gridDim.x) * blockDim.x) >> 5;
  for (uint64_t b = warp; b < nblk; b += nwarps) {
    double s0, s1;
    block_lane_values(sub, nsub, b, lane, s0, s1);
    const double incl = warp_incl_scan_d(s0 + s1, lane);
    if (lane == 31) cum[b] = incl;
  }
}

// In-place inclusive scan of nblk doubles by one block of 1024 threads, a
// contiguous run per thread: warp scans of the run sums, then a scan of the
// 32 warp totals (one thread chained the 1024 run sums before: 56-65 us at
// 17 to 29 qubits, now 3 to 14).
__global__ void __launch_bounds__(1024) k_cdf_scan(double* cum, uint64_t nblk) {
  __shared__ double tot[32];
  cudaGridDependencySynchronize();
  cudaTriggerProgrammaticLaunchCompletion();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint64_t per = (nblk + 1023) / 1024;
  const uint64_t lo = threadIdx.x * per;
  const uint64_t hi = lo + per < nblk ? lo + per : nblk;
  const bool idle = (static_cast<uint64_t>(warp) << 5) * per >= nblk;   // the whole warp is past the end
  double s = 0.0, incl = 0.0;
  if (!idle) {
    for (uint64_t i = lo; i < hi; ++i) s += cum[i];
    incl = warp_incl_scan_d(s, lane);
  }
  if (lane == 31) tot[warp] = incl;
  __syncthreads();
  if (warp == 0) tot[lane] = warp_incl_scan_d(tot[lane], lane);
  __syncthreads();
  if (idle) return;
  double before = __shfl_up_sync(0xffffffffu, incl, 1);
  if (lane == 0) before = 0.0;
  double r = (warp ? tot[warp - 1] : 0.0) + before;
  for (uint64_t i = lo; i < hi; ++i) { r += cum[i]; cum[i] = r; }
}

// first b in [0, n) with t < cum[b], n - 1 if there is none: 32 probes a step.
// cum[b - 1], when b > 0, was probed and is not above t.
__device__ __forceinline__ uint64_t warp_search(const double* cum, uint64_t n, double t, int lane) {
  uint64_t lo = 0, hi = n - 1;                           // the answer is in [lo, hi]
  while (lo < hi) {
    const uint64_t step = (hi - lo + 31) / 32;           // probes lo + step - 1, lo + 2 step - 1, ... below hi
    const uint64_t p = lo + step * (lane + 1) - 1;
    const unsigned hit = __ballot_sync(0xffffffffu, p < hi && t < cum[p]);
    const unsigned in = __ballot_sync(0xffffffffu, p < hi);
    const int first = hit ? __ffs(hit) - 1 : __popc(in); // probes before it are not above t
    if (hit) hi = lo + step * (first + 1) - 1;
    lo += step * first;
  }
  return lo;
}

// ro (optional): readout errors (Sec. V.A), 2 per qubit: qubit q of value b
// is reported as 1 - b when u01(seed, traj, 2, (j << 6) | q) < ro[2q + b];
// lane l decides qubits l and l + 32, and the flips are OR-combined.
__global__ void __launch_bounds__(256) k_sample(const float2* __restrict__ psi, uint64_t namps, const float* sub,
                                                uint64_t nsub, const double* cum, uint64_t nblk, uint64_t seed,
                                                uint64_t traj, uint32_t S, uint64_t* __restrict__ out, int n,
                                                const double* __restrict__ ro) {
  constexpr int CH = 1 << (kCdfSubLog - kCdfChunkLog);
  cudaGridDependencySynchronize();
  const int lane = threadIdx.x & 31;
  const uint64_t warp = (static_cast<uint64_t>(blockIdx.x) * blockDim.x + threadIdx.x) >> 5;
  const uint64_t nwarps = (static_cast<uint64_t>(gridDim.x) * blockDim.x) >> 5;
  for (uint64_t j = warp; j < S; j += nwarps) {
    const double total = cum[nblk - 1];
    const double t = uniform01(seed, traj, kStreamSample, static_cast<uint32_t>(j)) * total;
    const uint64_t b = warp_search(cum, nblk, t, lane);
    double trel = t - (b ? cum[b - 1] : 0.0);
    // sub-block inside the block (same lane values and scan as k_cdf_blk)
    double s0, s1;
    block_lane_values(sub, nsub, b, lane, s0, s1);
    const double incl = warp_incl_scan_d(s0 + s1, lane);
    double excl = __shfl_up_sync(0xffffffffu, incl, 1);
    if (lane == 0) excl = 0.0;
    unsigned hit = __ballot_sync(0xffffffffu, trel < incl);
    int L = hit ? __ffs(hit) - 1 : 31;
    const double eL = __shfl_sync(0xffffffffu, excl, L);
    const double s0L = __shfl_sync(0xffffffffu, s0, L);
    uint64_t sidx = (b << 6) + 2 * L;
    double base = eL;
    if (!(trel < eL + s0L)) { base = eL + s0L; sidx += 1; }
    if (sidx >= nsub) sidx = nsub - 1;
    trel -= base;
    // chunks inside the sub-block (same chunk arithmetic as k_cdf_sub), all
    // of it loaded before the search
    float4 v[CH];
#pragma unroll
    for (int c = 0; c < CH; ++c) {
      const uint64_t x0 = (sidx << kCdfSubLog) + (static_cast<uint64_t>(c) << kCdfChunkLog) + 2 * lane;
      v[c] = x0 < namps ? __ldg(reinterpret_cast<const float4*>(psi + x0)) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
    float run = 0.f;
    uint64_t x = ~0ull, last_nz = sidx << kCdfSubLog;
#pragma unroll
    for (int c = 0; c < CH; ++c) {
      const float w0 = fmaf(v[c].x, v[c].x, v[c].y * v[c].y), w1 = fmaf(v[c].z, v[c].z, v[c].w * v[c].w);
      const float inc = warp_incl_scan_f(w0 + w1, lane);
      const float tot = __shfl_sync(0xffffffffu, inc, 31);
      const float cend = run + inc;
      const float cstart = cend - (w0 + w1);
      const unsigned h = __ballot_sync(0xffffffffu, trel < static_cast<double>(cend));
      const unsigned nz = __ballot_sync(0xffffffffu, (w0 + w1) > 0.f);
      if (nz) {
        const int ln = 31 - __clz(nz);
        const float w1n = __shfl_sync(0xffffffffu, w1, ln);
        last_nz = (sidx << kCdfSubLog) + (static_cast<uint64_t>(c) << kCdfChunkLog) + 2 * ln + (w1n > 0.f ? 1 : 0);
      }
      if (h) {
        const int l2 = __ffs(h) - 1;
        const float cs = __shfl_sync(0xffffffffu, cstart, l2);
        const float a0 = __shfl_sync(0xffffffffu, w0, l2);
        x = (sidx << kCdfSubLog) + (static_cast<uint64_t>(c) << kCdfChunkLog) + 2 * l2 +
            (trel < static_cast<double>(cs + a0) ? 0 : 1);
        break;
      }
      run += tot;
    }
    if (x == ~0ull) x = last_nz;     // rounding put t past the sub-block end
    if (ro) {
      unsigned long long flips = 0ull;
      for (int q = lane; q < n; q += 32) {
        const uint32_t b = static_cast<uint32_t>((x >> q) & 1ull);
        const double u = uniform01(seed, traj, kStreamReadout, (static_cast<uint32_t>(j) << 6) | static_cast<uint32_t>(q));
        if (u < ro[2 * q + b]) flips |= 1ull << q;
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) flips |= __shfl_xor_sync(0xffffffffu, flips, o);
      x ^= flips;
    }
    if (lane == 0) out[j] = x;
  }
}

// C(x) for every x, exactly as k_sample compares against it: the FP64 table
// up to the block, the FP64 lane scan up to the sub-block, and the FP32 run
// inside the sub-block up to x (one warp per sub-block, same chunk arithmetic)
__global__ void k_cdf_values(const float2* __restrict__ psi, uint64_t namps, const float* __restrict__ sub,
                             uint64_t nsub, const double* __restrict__ cum, double* __restrict__ out) {
  const int lane = threadIdx.x & 31;
  const uint64_t warp = (static_cast<uint64_t>(blockIdx.x) * blockDim.x + threadIdx.x) >> 5;
  const uint64_t nwarps = (static_cast<uint64_t>(gridDim.x) * blockDim.x) >> 5;
  for (uint64_t s = warp; s < nsub; s += nwarps) {
    const uint64_t b = s >> 6;
    double s0, s1;
    block_lane_values(sub, nsub, b, lane, s0, s1);
    const double incl = warp_incl_scan_d(s0 + s1, lane);
    double excl = __shfl_up_sync(0xffffffffu, incl, 1);
    if (lane == 0) excl = 0.0;
    const int L = static_cast<int>((s & 63) >> 1);
    const double eL = __shfl_sync(0xffffffffu, excl, L);
    const double s0L = __shfl_sync(0xffffffffu, s0, L);
    const double base = (b ? cum[b - 1] : 0.0) + ((s & 1) ? eL + s0L : eL);
    float run = 0.f;
    for (int c = 0; c < (1 << (kCdfSubLog - kCdfChunkLog)); ++c) {
      const uint64_t x0 = (s << kCdfSubLog) + (static_cast<uint64_t>(c) << kCdfChunkLog) + 2 * lane;
      float w0, w1;
      chunk_weights(psi, namps, x0, w0, w1);
      const float inc = warp_incl_scan_f(w0 + w1, lane);
      const float tot = __shfl_sync(0xffffffffu, inc, 31);
      const float cend = run + inc;
      const float cstart = cend - (w0 + w1);
      if (x0 < namps) {
        out[x0] = base + static_cast<double>(cstart + w0);
        out[x0 + 1] = base + static_cast<double>(cend);
      }
      run += tot;
    }
  }
}

// the three table levels of the sampling CDF (sub-block runs, block scans,
// FP64 table) into scr.cdf_sub / scr.cdf_cum
static cudaError_t build_cdf_tables(const float2* psi, int n, const Scratch& scr, cudaStream_t st) {
  const uint64_t namps = 1ull << n;
  const uint64_t nsub = cdf_num_sub(n), nblk = cdf_num_blk(n);
  const int threads = 256, wpb = threads / 32;
  uint64_t g = (nsub + wpb - 1) / wpb;
  const uint64_t cap = static_cast<uint64_t>(sm_count()) * 8;
  if (g > cap) g = cap;
  k_cdf_sub<<<static_cast<unsigned>(g), threads, 0, st>>>(psi, namps, nsub, scr.cdf_sub);
  uint64_t gb = (nblk + wpb - 1) / wpb;
  if (gb > cap) gb = cap;
  cudaError_t e = launch_dependent(k_cdf_blk, dim3(static_cast<unsigned>(gb)), threads, st, scr.cdf_sub, nsub, nblk,
                                   scr.cdf_cum);
  if (e == cudaSuccess) e = launch_dependent(k_cdf_scan, dim3(1), 1024, st, scr.cdf_cum, nblk);
  return e == cudaSuccess ? cudaGetLastError() : e;
}

cudaError_t launch_cdf_values(const float2* psi, int n, const Scratch& scr, double* out, cudaStream_t st) {
  if (n < 1) return cudaErrorInvalidValue;
  const cudaError_t e = build_cdf_tables(psi, n, scr, st);
  if (e != cudaSuccess) return e;
  const uint64_t nsub = cdf_num_sub(n);
  const int threads = 256, wpb = threads / 32;
  uint64_t g = (nsub + wpb - 1) / wpb;
  const uint64_t cap = static_cast<uint64_t>(sm_count()) * 8;
  if (g > cap) g = cap;
  k_cdf_values<<<static_cast<unsigned>(g), threads, 0, st>>>(psi, 1ull << n, scr.cdf_sub, nsub, scr.cdf_cum, out);
  return cudaGetLastError();
}

cudaError_t launch_sample(const float2* psi, int n, uint64_t seed, uint64_t traj, uint32_t S,
                          uint64_t* out, const Scratch& scr, cudaStream_t st, const double* readout) {
  if (n < 1) return cudaErrorInvalidValue;
  const uint64_t namps = 1ull << n;
  const uint64_t nsub = cdf_num_sub(n), nblk = cdf_num_blk(n);
  const int threads = 256, wpb = threads / 32;
  const uint64_t cap = static_cast<uint64_t>(sm_count()) * 8;
  const cudaError_t e = build_cdf_tables(psi, n, scr, st);
  if (e != cudaSuccess || S == 0) return e;
  uint64_t gs = (S + wpb - 1) / wpb;
  if (gs > cap) gs = cap;
  return launch_dependent(k_sample, dim3(static_cast<unsigned>(gs)), threads, st, psi, namps, scr.cdf_sub, nsub,
                          scr.cdf_cum, nblk, seed, traj, S, out, n, readout);
}

// ---------------------------------------------------------------------------
__global__ void k_init(float4* __restrict__ psi, uint64_t npairs) {
  const uint64_t stride = static_cast<uint64_t>(gridDim.x) * blockDim.x;
  for (uint64_t i = static_cast<uint64_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < npairs; i += stride)
    psi[i] = make_float4(i == 0 ? 1.f : 0.f, 0.f, 0.f, 0.f);
}

cudaError_t kernel_arch(int* binary_version, int* ptx_version) {
  cudaFuncAttributes a{};
  const cudaError_t e = cudaFuncGetAttributes(&a, k_init);
  if (e != cudaSuccess) return e;
  *binary_version = a.binaryVersion;
  *ptx_version = a.ptxVersion;
  return cudaSuccess;
}

__global__ void k_scale(float4* __restrict__ psi, uint64_t npairs, float f) {
  const uint64_t stride = static_cast<uint64_t>(gridDim.x) * blockDim.x;
  for (uint64_t i = static_cast<uint64_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < npairs; i += stride) {
    float4 v = psi[i];
    v.x *= f; v.y *= f; v.z *= f; v.w *= f;
    psi[i] = v;
  }
}

static unsigned stream_grid(uint64_t items) {
  uint64_t g = (items + 255) / 256;
  const uint64_t cap = static_cast<uint64_t>(sm_count()) * 8;
  return static_cast<unsigned>(g < cap ? (g ? g : 1) : cap);
}

// ---------------------------------------------------------------------------
// Product-state preparation.  Fused gates that are the first to act on each
// of their qubits, on disjoint qubits, take |0...0> to the tensor product of
// their first columns (U |0> = U[:, 0]) with |0> on every other qubit.  With
// the qubits split at m, each factor on the low or on the high side, the
// amplitude is psi[x] = H[x >> m] * L[x mod 2^m]: the two tables are built
// first (FP64 products of the factors, rounded once), then one write pass
// fills the state, in place of the |0...0> pass and one pass per factor.
// ---------------------------------------------------------------------------
__global__ void k_fold_table(float2* __restrict__ out, uint32_t size, const __grid_constant__ FoldSpec s) {
  const uint32_t stride = gridDim.x * blockDim.x;
  for (uint32_t e = blockIdx.x * blockDim.x + threadIdx.x; e < size; e += stride) {
    double re = 0.0, im = 0.0;
    if (!(e & s.zmask)) {
      re = 1.0;
      for (int f = 0; f < s.nf; ++f) {
        uint32_t j = 0;
        for (int b = 0; b < s.w[f]; ++b) j |= ((e >> s.q[f][b]) & 1u) << b;
        const float2 v = s.v[s.off[f] + j];
        const double a = re * v.x - im * v.y;
        im = re * v.y + im * v.x;
        re = a;
      }
    }
    out[e] = make_float2(static_cast<float>(re), static_cast<float>(im));
  }
}

__global__ void __launch_bounds__(256) k_init_outer(float4* __restrict__ psi, const float2* __restrict__ tl,
                                                    const float2* __restrict__ th, int m, uint64_t npairs) {
  const uint64_t lmask = (1ull << m) - 1ull;
  const uint64_t stride = static_cast<uint64_t>(gridDim.x) * blockDim.x;
  for (uint64_t i = static_cast<uint64_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < npairs; i += stride) {
    const uint64_t x = 2ull * i;                  // even: both amplitudes share H[x >> m] (m >= 1)
    const float4 l = *reinterpret_cast<const float4*>(tl + (x & lmask));
    const float2 h = th[x >> m];
    __stcs(psi + i, make_float4(h.x * l.x - h.y * l.y, h.x * l.y + h.y * l.x,
                                h.x * l.z - h.y * l.w, h.x * l.w + h.y * l.z));
  }
}

cudaError_t launch_init_product(float2* psi, int n, int m, const FoldSpec& lo, const FoldSpec& hi,
                                float2* tables, cudaStream_t st) {
  if (n < 2 || m < 1 || m >= n || m > kFoldTableBits || n - m > kFoldTableBits) return cudaErrorInvalidValue;
  const uint32_t nl = 1u << m, nhi = 1u << (n - m);
  float2* tl = tables;
  float2* th = tables + nl;                      // nl even: th stays 16-byte aligned
  k_fold_table<<<stream_grid(nl), 256, 0, st>>>(tl, nl, lo);
  k_fold_table<<<stream_grid(nhi), 256, 0, st>>>(th, nhi, hi);
  const uint64_t np = 1ull << (n - 1);
  k_init_outer<<<stream_grid(np), 256, 0, st>>>(reinterpret_cast<float4*>(psi), tl, th, m, np);
  return cudaGetLastError();
}

cudaError_t launch_init_state(float2* psi, int n, cudaStream_t st) {
  if (n < 1) return cudaErrorInvalidValue;
  const uint64_t np = 1ull << (n - 1);
  k_init<<<stream_grid(np), 256, 0, st>>>(reinterpret_cast<float4*>(psi), np);
  return cudaGetLastError();
}

cudaError_t launch_scale(float2* psi, int n, float f, cudaStream_t st) {
  if (n < 1) return cudaErrorInvalidValue;
  const uint64_t np = 1ull << (n - 1);
  k_scale<<<stream_grid(np), 256, 0, st>>>(reinterpret_cast<float4*>(psi), np, f);
  return cudaGetLastError();
}

}  // namespace qt
