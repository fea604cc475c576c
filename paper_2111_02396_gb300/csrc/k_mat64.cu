// 64 x 64 complex matrices on CUDA cores (FP32): 6-qubit fused gates (Alg. 1)
// and the branch norms |K psi|^2 of 6-qubit channels (Alg. 2 step 14).
//
// Both are the product of one matrix with 2^(n-6) gather sets, 256 FMAs an
// amplitude, so FP32 FMA is the bound (0.93 ms at n = 27, where the bytes take
// 0.32).  A CTA of 256 threads stages the matrix once and 128 sets at a time,
// and a thread owns 8 rows x 4 sets: per member 6 shared-memory reads of 16
// bytes feed 64 packed FMAs.  A read returns 128 bytes a clock and SM however
// many lanes share its words, so smaller tiles are bound by reads.  The packed
// FMAs pair two rows, whose matrix entries lie together; the members are
// doubled in registers.  Two CTAs an SM cover each other's copies and
// barriers.  n = 27: 2.77 -> 1.40 ms (1.54 with qubit 0 among the targets);
// |K psi|^2 at n = 25: 879 -> 335 us.  Before, a thread took one set, 16 rows
// at a time (the channel's: one row), with a read per multiply-add.
//
// Each output sums its 64 members in ascending order, the product with the
// imaginary part first.
#include <cuda_runtime.h>

#include "kernels.h"
#include "qt_dfloat.h"

namespace qt {

namespace m64 {

constexpr int kThreads = 256;
constexpr int kSets = 128;                  // gather sets of a tile
constexpr int kChunks = kSets * 64 / 2 / kThreads;   // 16-byte chunks per thread and tile
constexpr size_t kSmem = sizeof(float4) * (64 * 32 + 64 * kSets / 2);

struct Args {
  uint64_t offs[64];          // amplitude offset of member m within a set
  uint64_t coff[kChunks];     // what chunk c adds to a thread's address
  int cmem[kChunks];          // and to its member
  int z;                      // member bit of qubit 0 (if it is a target)
  uint32_t ins[7];            // ascending bit positions to insert zeros at
  uint64_t num_sets, num_tiles;
  const float2* u;            // row-major matrix (device)
  float down;                 // factor of the FP32 runs at their carry (norms)
};

// 16-byte word of (row m, sets 2 c, 2 c + 1) of a staged tile: the threads of
// a quarter-warp that write together differ in m / 2 mod 8
__device__ __forceinline__ int word(int m, int c) { return m * (kSets / 2) + (c ^ ((m >> 1) & 7)); }

// x with a zero inserted at bit z
__host__ __device__ __forceinline__ int skip(int x, int z) { return ((x >> z) << (z + 1)) | (x & ((1 << z) - 1)); }

// LOW0: qubit 0 is a target, so a 16-byte word of the state holds the two
// members of a set that differ in it; otherwise one member of two neighbouring
// sets
template <bool LOW0>
struct Tile {
  static constexpr int NI = LOW0 ? 6 : 7, LOGJ = LOW0 ? 7 : 6;
  const Args& a;
  int j, m;                   // this thread's set (pair) and member, chunk 0
  uint64_t off;
  __device__ __forceinline__ uint64_t spread(uint64_t x) const {
#pragma unroll
    for (int b = 0; b < NI; ++b) {
      const uint32_t s = a.ins[b];
      x = ((x >> s) << (s + 1)) | (x & ((1ull << s) - 1ull));
    }
    return x;
  }
  __device__ __forceinline__ explicit Tile(const Args& args) : a(args) {
    j = threadIdx.x & ((1 << LOGJ) - 1);
    m = LOW0 ? skip(threadIdx.x >> LOGJ, a.z) : threadIdx.x >> LOGJ;
    off = spread(j) | a.offs[m];
  }
  // fewer than a tile of sets (one partial tile): the rest is zero, not stored
  __device__ __forceinline__ bool inside() const { return static_cast<uint64_t>(LOW0 ? j : 2 * j) < a.num_sets; }
  __device__ __forceinline__ void load(const float2* psi, uint64_t tile, float4* v) const {
    const float2* const p = psi + (spread(tile << LOGJ) | off);
    const bool in = inside();
    float4 buf[kChunks];
#pragma unroll
    for (int c = 0; c < kChunks; ++c)
      buf[c] = in ? __ldcs(reinterpret_cast<const float4*>(p + a.coff[c])) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int c = 0; c < kChunks; ++c) {
      const int r = m | a.cmem[c];
      if (LOW0) {
        reinterpret_cast<float2*>(v + word(r, j >> 1))[j & 1] = make_float2(buf[c].x, buf[c].y);
        reinterpret_cast<float2*>(v + word(r | 1 << a.z, j >> 1))[j & 1] = make_float2(buf[c].z, buf[c].w);
      } else {
        v[word(r, j)] = buf[c];
      }
    }
  }
  __device__ __forceinline__ void store(float2* psi, uint64_t tile, const float4* v) const {
    if (!inside()) return;
    float2* const p = psi + (spread(tile << LOGJ) | off);
#pragma unroll
    for (int c = 0; c < kChunks; ++c) {
      const int r = m | a.cmem[c];
      float4 x;
      if (LOW0) {
        const float2 lo = reinterpret_cast<const float2*>(v + word(r, j >> 1))[j & 1];
        const float2 hi = reinterpret_cast<const float2*>(v + word(r | 1 << a.z, j >> 1))[j & 1];
        x = make_float4(lo.x, lo.y, hi.x, hi.y);
      } else {
        x = v[word(r, j)];
      }
      __stcs(reinterpret_cast<float4*>(p + a.coff[c]), x);
    }
  }
};

// entry (m, p): rows 2p and 2p + 1 of column m as (re, re, im, im)
__device__ __forceinline__ void stage_matrix(const float2* __restrict__ u, float4* s) {
  for (int i = threadIdx.x; i < 64 * 32; i += kThreads) {
    const int p = i >> 6, m = i & 63;
    const float2 x = u[(2 * p) * 64 + m], y = u[(2 * p + 1) * 64 + m];
    s[m * 32 + p] = make_float4(x.x, y.x, x.y, y.y);
  }
}

// v <- U v for the staged tile, both in shared memory; all threads
__device__ __forceinline__ void multiply(const float4* s, float4* v) {
  const int rg = threadIdx.x & 7, c0 = (threadIdx.x >> 3) * 2;   // row pairs rg + 8 i, words c0 and c0 + 1
  float2 xr[4][4], xi[4][4];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int q = 0; q < 4; ++q) xr[i][q] = xi[i][q] = make_float2(0.f, 0.f);
#pragma unroll 2
  for (int m = 0; m < 64; ++m) {
    const float4 a = v[word(m, c0)], b = v[word(m, c0 + 1)];
    const float x[4] = {a.x, a.z, b.x, b.z}, y[4] = {a.y, a.w, b.y, b.w};
    float4 u[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) u[i] = s[m * 32 + rg + 8 * i];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const float2 vx = make_float2(x[q], x[q]), vy = make_float2(y[q], y[q]), ny = make_float2(-y[q], -y[q]);
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const float2 re = make_float2(u[i].x, u[i].y), im = make_float2(u[i].z, u[i].w);
        xr[i][q] = __ffma2_rn(re, vx, __ffma2_rn(im, ny, xr[i][q]));
        xi[i][q] = __ffma2_rn(re, vy, __ffma2_rn(im, vx, xi[i][q]));
      }
    }
  }
  __syncthreads();                                       // every member is read
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int r = 2 * (rg + 8 * i);
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      v[word(r, c0 + h)] = make_float4(xr[i][2 * h].x, xi[i][2 * h].x, xr[i][2 * h + 1].x, xi[i][2 * h + 1].x);
      v[word(r + 1, c0 + h)] = make_float4(xr[i][2 * h].y, xi[i][2 * h].y, xr[i][2 * h + 1].y, xi[i][2 * h + 1].y);
    }
  }
  __syncthreads();
}

}  // namespace m64

template <bool LOW0>
__global__ void __launch_bounds__(m64::kThreads, 2) k_apply64(float2* __restrict__ psi,
                                                              const __grid_constant__ m64::Args a) {
  extern __shared__ __align__(16) float4 s_m64[];
  float4* const v = s_m64 + 64 * 32;
  m64::stage_matrix(a.u, s_m64);
  const m64::Tile<LOW0> t(a);
  for (uint64_t tile = blockIdx.x; tile < a.num_tiles; tile += gridDim.x) {
    t.load(psi, tile, v);
    __syncthreads();
    m64::multiply(s_m64, v);
    t.store(psi, tile, v);
    __syncthreads();                                     // the tile is read
  }
}

// N = <psi|psi> and P = |K psi|^2: thread t < 128 sums set t of every tile of
// its CTA, in runs of 16 sets, as k_kraus_norms does for narrower channels
constexpr int kNormRun = 16;

template <bool LOW0>
__global__ void __launch_bounds__(m64::kThreads, 2) k_norms64(const float2* __restrict__ psi,
                                                              const __grid_constant__ m64::Args a,
                                                              float2* __restrict__ partial) {
  extern __shared__ __align__(16) float4 s_m64[];
  __shared__ float2 s_sum[m64::kSets / 32][2];
  float4* const v = s_m64 + 64 * 32;
  cudaTriggerProgrammaticLaunchCompletion();
  m64::stage_matrix(a.u, s_m64);
  const m64::Tile<LOW0> t(a);
  const int set = threadIdx.x;                           // of the first 128 threads
  float f[2] = {0.f, 0.f}, h[2] = {0.f, 0.f}, l[2] = {0.f, 0.f};
  auto at = [&](int m) { return reinterpret_cast<const float2*>(v + m64::word(m, set >> 1))[set & 1]; };
  int run = 0;
  for (uint64_t tile = blockIdx.x; tile < a.num_tiles; tile += gridDim.x) {
    t.load(psi, tile, v);
    __syncthreads();
    if (set < m64::kSets) {
#pragma unroll 8
      for (int m = 0; m < 64; ++m) {
        const float2 x = at(m);
        f[0] = fmaf(x.x, x.x, fmaf(x.y, x.y, f[0]));
      }
    }
    m64::multiply(s_m64, v);
    if (set < m64::kSets) {
      float row = 0.f;
#pragma unroll 8
      for (int m = 0; m < 64; ++m) {
        const float2 w = at(m);
        row = fmaf(w.x, w.x, fmaf(w.y, w.y, row));
      }
      f[1] += row;
      if (++run == kNormRun) {
        for (int k = 0; k < 2; ++k) { df_acc(h[k], l[k], f[k] * a.down); f[k] = 0.f; }
        run = 0;
      }
    }
    __syncthreads();
  }
  if (set < m64::kSets) {
    for (int k = 0; k < 2; ++k) {
      df_acc(h[k], l[k], f[k] * a.down);
      float2 x = make_float2(h[k], l[k]);
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) x = df_add(x, df_shfl_xor(x, o));
      if ((set & 31) == 0) s_sum[set >> 5][k] = x;
    }
  }
  __syncthreads();
  if (set < 2) {
    float2 x = s_sum[0][set];
    for (int w = 1; w < m64::kSets / 32; ++w) x = df_add(x, s_sum[w][set]);
    partial[static_cast<size_t>(blockIdx.x) * 2 + set] = x;
  }
}

// member bit b of u's columns <-> qubits[b]
static m64::Args m64_args(int n, const uint32_t* qubits, const float2* udev) {
  m64::Args a{};
  uint32_t t[6];
  for (int b = 0; b < 6; ++b) t[b] = qubits[b];
  for (int i = 1; i < 6; ++i)
    for (int j = i; j > 0 && t[j - 1] > t[j]; --j) { const uint32_t x = t[j]; t[j] = t[j - 1]; t[j - 1] = x; }
  const bool low0 = t[0] == 0;
  int ni = 0;
  if (!low0) a.ins[ni++] = 0;
  for (int b = 0; b < 6; ++b) {
    a.ins[ni++] = t[b];
    if (qubits[b] == 0) a.z = b;
  }
  for (int m = 0; m < 64; ++m)
    for (int b = 0; b < 6; ++b)
      if ((m >> b) & 1) a.offs[m] |= 1ull << qubits[b];
  for (int c = 0; c < m64::kChunks; ++c) {
    a.cmem[c] = low0 ? m64::skip(2 * c, a.z) : 4 * c;
    a.coff[c] = a.offs[a.cmem[c]];
  }
  a.num_sets = 1ull << (n - 6);
  a.num_tiles = (a.num_sets + m64::kSets - 1) / m64::kSets;
  a.u = udev;
  return a;
}

static bool has_qubit0(const uint32_t* qubits) {
  for (int b = 0; b < 6; ++b)
    if (qubits[b] == 0) return true;
  return false;
}

template <typename K>
static int m64_grid(K kern) {
  if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(m64::kSmem)) != cudaSuccess)
    return 0;
  int occ = 0;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, m64::kThreads, m64::kSmem);
  return sm_count() * (occ > 0 ? occ : 1);
}

template <bool LOW0>
static cudaError_t apply64(float2* psi, const m64::Args& a, cudaStream_t st) {
  static PerDevice setup;
  const int grid = setup.get([] { return m64_grid(k_apply64<LOW0>); });
  if (grid <= 0) return cudaErrorInvalidConfiguration;
  const unsigned g = static_cast<unsigned>(a.num_tiles < static_cast<uint64_t>(grid) ? a.num_tiles : grid);
  k_apply64<LOW0><<<g, m64::kThreads, m64::kSmem, st>>>(psi, a);
  return cudaGetLastError();
}

cudaError_t launch_apply6_fp32(float2* psi, int n, const uint32_t* targets, const float2* udev, cudaStream_t st) {
  if (n < 13) return cudaErrorInvalidValue;
  const m64::Args a = m64_args(n, targets, udev);
  return targets[0] == 0 ? apply64<true>(psi, a, st) : apply64<false>(psi, a, st);
}

template <bool LOW0>
static cudaError_t norms64(const float2* psi, const m64::Args& a, float2* partial, int* blocks, cudaStream_t st) {
  static PerDevice setup;
  const int grid = setup.get([] { return m64_grid(k_norms64<LOW0>); });
  if (grid <= 0) return cudaErrorInvalidConfiguration;
  *blocks = static_cast<int>(a.num_tiles < static_cast<uint64_t>(grid) ? a.num_tiles : grid);
  k_norms64<LOW0><<<static_cast<unsigned>(*blocks), m64::kThreads, m64::kSmem, st>>>(psi, a, partial);
  return cudaGetLastError();
}

cudaError_t launch_norms64(const float2* psi, int n, const uint32_t* qubits, const float2* kdev, float down,
                           float2* partial, int* blocks, cudaStream_t st) {
  if (n < 6) return cudaErrorInvalidValue;
  m64::Args a = m64_args(n, qubits, kdev);
  a.down = down;
  return has_qubit0(qubits) ? norms64<true>(psi, a, partial, blocks, st) : norms64<false>(psi, a, partial, blocks, st);
}

}  // namespace qt
