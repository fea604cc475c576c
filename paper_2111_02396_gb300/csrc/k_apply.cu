// Fused-gate application (Alg. 1, Sec. III.A) on a complex64 state.
//
// The state is 2^n interleaved (re, im) float pairs.  A k-qubit fused gate
// splits it into 2^(n-k) gather sets of 2^k amplitudes (the set's base
// index with every combination of the target bits); each set is one
// 2^k x 2^k matrix-vector product.
//
// k_apply_tile (the main kernel): a CTA of 128 threads owns one tile of
// 128 gather sets = 2^(7+k) amplitudes.  The tile is 2^h rows (h = number
// of "high" targets) of 2^C contiguous amplitudes, where C is the smallest
// width such that the row holds every "low" target plus 7 free bits; so a
// row is at least 1 KB and every warp-wide 128-bit load or store of the
// tile is fully coalesced whatever the target pattern.  The tile is staged
// in shared memory with an XOR swizzle (8-byte slot ^= a per-launch linear
// image of index bits 4..7) chosen so that the strided gathers of every
// target pattern are free of bank conflicts.  Each thread then gathers one
// set, multiplies, and scatters it back; the tile is stored with the same
// coalesced pattern.
//
// The matrix is a __grid_constant__ kernel parameter: its entries reach the
// FMAs through uniform registers loaded from the constant bank.  The complex
// products use the three-multiply form: with U = c + i d and v = a + i b,
// precomputing e = c + d and f = d - c per entry and s = a + b per amplitude,
//   Re(U v) = sum c s - sum b e,   Im(U v) = sum c s + sum a f,
// i.e. 3 FMA per complex multiply-add instead of 4.  The two sums that
// share an entry pair, (sum c s, sum e b), run as one packed FP32x2 FMA on
// the (c, e) pair, so a complex multiply-add issues 2 instructions.
//
// k_apply (direct, for states smaller than one tile): one thread per
// gather set (or per pair of sets that differ in bit 0), members loaded
// straight into registers.
//
// Bytes per launch: 16 * 2^n (every amplitude read once and written once).
// FLOPs per launch: 2^(k+2) * 2^(n+1) (the paper's count).
#include <cuda_runtime.h>

#include <mutex>

#include "kernels.h"

namespace qt {

template <int K>
struct ApplyArgs {
  float2 u[1 << K][1 << K];     // row-major gate matrix
  uint64_t offs[1 << K];        // amplitude offset of member m within a set
  uint32_t ins[K + 1];          // ascending bit positions to insert zeros at
  uint64_t num_sets;            // sets (or set pairs) to process
};

template <int K, bool PAIR>
__global__ void __launch_bounds__(256) k_apply(float2* __restrict__ psi,
                                               const __grid_constant__ ApplyArgs<K> a) {
  constexpr int M = 1 << K;
  constexpr int NI = PAIR ? K + 1 : K;
  const uint64_t stride = static_cast<uint64_t>(gridDim.x) * blockDim.x;
  for (uint64_t i = static_cast<uint64_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < a.num_sets;
       i += stride) {
    uint64_t base = i;
#pragma unroll
    for (int b = 0; b < NI; ++b) {
      const uint32_t s = a.ins[b];
      base = ((base >> s) << (s + 1)) | (base & ((1ull << s) - 1ull));
    }
    if constexpr (PAIR) {
      float4 v[M];
#pragma unroll
      for (int m = 0; m < M; ++m) v[m] = __ldcs(reinterpret_cast<const float4*>(psi + base + a.offs[m]));
#pragma unroll 2
      for (int j = 0; j < M; ++j) {
        float xr = 0.f, xi = 0.f, yr = 0.f, yi = 0.f;
#pragma unroll
        for (int m = 0; m < M; ++m) {
          const float ur = a.u[j][m].x, ui = a.u[j][m].y;
          xr = fmaf(ur, v[m].x, xr);
          xr = fmaf(-ui, v[m].y, xr);
          xi = fmaf(ur, v[m].y, xi);
          xi = fmaf(ui, v[m].x, xi);
          yr = fmaf(ur, v[m].z, yr);
          yr = fmaf(-ui, v[m].w, yr);
          yi = fmaf(ur, v[m].w, yi);
          yi = fmaf(ui, v[m].z, yi);
        }
        __stcs(reinterpret_cast<float4*>(psi + base + a.offs[j]), make_float4(xr, xi, yr, yi));
      }
    } else {
      float2 v[M];
#pragma unroll
      for (int m = 0; m < M; ++m) v[m] = __ldcs(psi + base + a.offs[m]);
#pragma unroll 2
      for (int j = 0; j < M; ++j) {
        float xr = 0.f, xi = 0.f;
#pragma unroll
        for (int m = 0; m < M; ++m) {
          const float ur = a.u[j][m].x, ui = a.u[j][m].y;
          xr = fmaf(ur, v[m].x, xr);
          xr = fmaf(-ui, v[m].y, xr);
          xi = fmaf(ur, v[m].y, xi);
          xi = fmaf(ui, v[m].x, xi);
        }
        __stcs(psi + base + a.offs[j], make_float2(xr, xi));
      }
    }
  }
}

int sm_count() {
  static PerDevice sms;
  return sms.get([] {
    int dev = 0, v = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev);
    return v > 0 ? v : 1;
  });
}


// ---------------------------------------------------------------------------
// tiled kernel
// ---------------------------------------------------------------------------
constexpr int kTileThreads = 128;       // = gather sets per tile

// 16-byte aligned so that the matrix pairs sit on aligned constant-bank words
template <int K>
struct alignas(16) TileArgs {
  float2 ce[1 << K][1 << K];  // (Re U, Re U + Im U)
  float f[1 << K][1 << K];    // Im U - Re U
  uint64_t roff[1 << K];      // memory offset of tile row r
  uint64_t poff[1 << K];      // memory offset of tile index 256 c (chunk c of every thread)
  uint32_t smoff[1 << K];     // swizzled tile-local offset of member m
  uint32_t tins[K];           // tile-local target positions, ascending
  uint32_t hins[K];           // memory positions of the high targets, ascending
  uint8_t swzt[16];           // swizzle table: slot = l ^ swzt[(l >> 4) & 15]
  int nh;                     // number of high targets
  int C;                      // contiguous low bits per row
  uint64_t num_tiles;
};

// The swizzle of the tile kernel is chosen per launch.  It XORs a linear
// (GF(2)) image of index bits 4..7 into bits 0..3, slot = l ^ G(l >> 4 & 15).
// A half-warp's 16 lanes differ in the 4 lowest non-target tile positions;
// those below 4 stay put, and G maps those in 4..7 onto the target positions
// below 4, so every 8-byte gather and scatter of a half-warp hits 16
// distinct bank pairs, whatever the targets.  (No fixed map does this for
// every pattern: the single-target cases force every entry of G to 1.)  The
// image of bit 4 also sets bit 0, which keeps the coalesced staging stores
// (lane t writes index 2t) conflict-free.
__device__ __forceinline__ uint32_t swz_t(uint32_t l, const uint8_t* t) { return l ^ t[(l >> 4) & 15u]; }

static void swizzle_table(const uint32_t* tpos, int K, uint8_t* tab) {
  uint32_t tmask = 0;
  for (int b = 0; b < K; ++b) tmask |= 1u << tpos[b];
  int lane[4], nl = 0;
  for (uint32_t p = 0; nl < 4; ++p)
    if (!((tmask >> p) & 1u)) lane[nl++] = static_cast<int>(p);
  uint32_t g[4] = {1u, 2u, 4u, 8u};    // image of bit 4 + i (the fixed map)
  if (lane[3] < 8) {
    int low = 0;                       // target positions below 4, ascending
    for (int i = 0; i < 4; ++i)
      if (lane[i] >= 4) {
        while (!((tmask >> low) & 1u)) ++low;
        g[lane[i] - 4] = 1u << low++;
      }
  }
  g[0] |= 1u;
  for (int x = 0; x < 16; ++x) {
    uint32_t v = 0;
    for (int i = 0; i < 4; ++i)
      if ((x >> i) & 1) v ^= g[i];
    tab[x] = static_cast<uint8_t>(v);
  }
}

// RU: unroll factor of the row loop; MINB: CTAs per SM that the register
// allocation must allow.  At K = 4 the kernel is issue-bound: rows go four
// at a time under an 8-CTA bound (64 registers), which gives the scheduler
// the most warps to choose from; a full row unroll keeps more values live
// than even 255 registers hold.
//
// Index arithmetic is hoisted out of the per-amplitude work with two
// identities.  The swizzle distributes over an OR of disjoint bit sets,
// swz(x | y) = swz(x) ^ swz(y), so member m of the thread's set sits at
// swz(sbase) ^ smoff[m] with smoff[m] = swz(moff[m]) precomputed.  The map
// from a tile index to its memory offset deposits bits (the row bits go to
// the high-target positions), so it too distributes over disjoint bits:
// thread t's chunk c (tile index 2t + 256c) is at offset(2t) | poff[c].
template <int K, int RU = 2, int MINB = 1>
__global__ void __launch_bounds__(kTileThreads, MINB) k_apply_tile(float2* __restrict__ psi,
                                                             const __grid_constant__ TileArgs<K> a) {
  constexpr int M = 1 << K;
  constexpr int TILE = kTileThreads * M;       // amplitudes per tile
  constexpr int NCH = TILE / 2 / kTileThreads; // float4 chunks per thread
  __shared__ __align__(16) float2 sm[TILE];
  const uint32_t tid = threadIdx.x;
  // this thread's gather set inside the tile (same for every tile)
  uint32_t sbase = tid;
#pragma unroll
  for (int b = 0; b < K; ++b) {
    const uint32_t t = a.tins[b];
    sbase = ((sbase >> t) << (t + 1)) | (sbase & ((1u << t) - 1u));
  }
  const uint32_t ss = swz_t(sbase, a.swzt);
  // one tile per CTA: a loop over tiles would make the matrix entries
  // loop-invariant, and the compiler would then hold them in registers
  {
    const uint64_t tile = blockIdx.x;
    uint64_t base = tile << a.C;
    for (int j = 0; j < a.nh; ++j) {
      const uint32_t h = a.hins[j];
      base = ((base >> h) << (h + 1)) | (base & ((1ull << h) - 1ull));
    }
    const uint32_t l0 = 2u * tid;
    float2* const pt = psi + (base | a.roff[l0 >> a.C] | (l0 & ((1u << a.C) - 1u)));
    // bits 4..7 of the tile index 2t + 256c are bits 3..6 of t, so the
    // swizzle of both amplitudes of a chunk is the same for every c
    const uint32_t fl = a.swzt[(tid >> 3) & 15u];
    const uint32_t s0 = l0 ^ fl, s1 = (l0 + 1u) ^ fl;
    // load rows -> shared (coalesced 128-bit)
    float4 buf[NCH];
#pragma unroll
    for (int c = 0; c < NCH; ++c) buf[c] = __ldcs(reinterpret_cast<const float4*>(pt + a.poff[c]));
#pragma unroll
    for (int c = 0; c < NCH; ++c) {
      sm[s0 + 256u * c] = make_float2(buf[c].x, buf[c].y);
      sm[s1 + 256u * c] = make_float2(buf[c].z, buf[c].w);
    }
    __syncthreads();
    // one gather set per thread
    float va[M];
    float2 sb[M];    // (a + b, b) of member m
#pragma unroll
    for (int m = 0; m < M; ++m) {
      const float2 v = sm[ss ^ a.smoff[m]];
      va[m] = v.x;
      sb[m] = make_float2(v.x + v.y, v.y);
    }
    // rows RU at a time: the matrix entries come in through uniform
    // constant loads (warp-uniform row index)
#pragma unroll RU
    for (int j = 0; j < M; ++j) {
      float2 tr = make_float2(0.f, 0.f);    // (sum c s, sum e b)
      float im = 0.f;
#pragma unroll
      for (int m = 0; m < M; ++m) {
        tr = __ffma2_rn(a.ce[j][m], sb[m], tr);
        im = fmaf(a.f[j][m], va[m], im);
      }
      sm[ss ^ a.smoff[j]] = make_float2(tr.x - tr.y, tr.x + im);
    }
    __syncthreads();
    // shared -> rows (coalesced 128-bit)
#pragma unroll
    for (int c = 0; c < NCH; ++c) {
      const float2 x = sm[s0 + 256u * c], y = sm[s1 + 256u * c];
      __stcs(reinterpret_cast<float4*>(pt + a.poff[c]), make_float4(x.x, x.y, y.x, y.y));
    }
    __syncthreads();
  }
}

template <int K>
static cudaError_t launch_tile(float2* psi, int n, const uint32_t* targets, const float2* U,
                               cudaStream_t st) {
  constexpr int M = 1 << K;
  TileArgs<K> a;
  for (int j = 0; j < M; ++j)
    for (int m = 0; m < M; ++m) {
      const float re = U[j * M + m].x, im = U[j * M + m].y;
      a.ce[j][m] = make_float2(re, re + im);
      a.f[j][m] = im - re;
    }
  // C = 7 + number of targets below C
  int C = 7;
  for (;;) {
    int low = 0;
    for (int b = 0; b < K; ++b) low += targets[b] < static_cast<uint32_t>(C);
    if (C - low >= 7) break;
    ++C;
  }
  a.C = C;
  int nh = 0;
  uint32_t tpos[K];
  for (int b = 0; b < K; ++b) {
    if (targets[b] < static_cast<uint32_t>(C)) {
      tpos[b] = targets[b];
    } else {
      tpos[b] = static_cast<uint32_t>(C + nh);
      a.hins[nh++] = targets[b];
    }
  }
  a.nh = nh;
  for (int b = 0; b < K; ++b) a.tins[b] = tpos[b];   // ascending: low targets, then C, C+1, ...
  swizzle_table(tpos, K, a.swzt);
  for (int m = 0; m < M; ++m) {
    uint32_t o = 0;
    for (int b = 0; b < K; ++b)
      if ((m >> b) & 1) o |= 1u << tpos[b];
    a.smoff[m] = o ^ a.swzt[(o >> 4) & 15u];
  }
  for (int r = 0; r < M; ++r) {
    uint64_t o = 0;
    for (int j = 0; j < nh; ++j)
      if ((r >> j) & 1) o |= 1ull << a.hins[j];
    a.roff[r] = r < (1 << nh) ? o : 0;
  }
  // chunk c of every thread starts at tile index 256 c (< 2^(7+K))
  for (int c = 0; c < M; ++c) {
    const uint32_t l = 256u * static_cast<uint32_t>(c);
    a.poff[c] = c < M / 2 ? (a.roff[l >> C] | (l & ((1u << C) - 1u))) : 0;
  }
  a.num_tiles = 1ull << (n - C - nh);
  if constexpr (K == 4)
    k_apply_tile<4, 4, 8><<<static_cast<unsigned>(a.num_tiles), kTileThreads, 0, st>>>(psi, a);
  else if constexpr (K == 5)
    k_apply_tile<5, 2, 3><<<static_cast<unsigned>(a.num_tiles), kTileThreads, 0, st>>>(psi, a);
  else
    k_apply_tile<K><<<static_cast<unsigned>(a.num_tiles), kTileThreads, 0, st>>>(psi, a);
  return cudaGetLastError();
}

// smallest n for which one tile fits: 7 free bits + k targets
static inline bool tile_fits(int n, int k) { return n >= 7 + k; }

template <int K, bool PAIR>
static cudaError_t launch_k(float2* psi, int n, const uint32_t* targets, const float2* U,
                            cudaStream_t st) {
  static PerDevice occ_dev;
  const int occ = occ_dev.get([] {
    int v = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&v, k_apply<K, PAIR>, 256, 0);
    return v > 0 ? v : 1;
  });
  ApplyArgs<K> a;
  constexpr int M = 1 << K;
  for (int j = 0; j < M; ++j)
    for (int m = 0; m < M; ++m) a.u[j][m] = U[j * M + m];
  for (int m = 0; m < M; ++m) {
    uint64_t o = 0;
    for (int b = 0; b < K; ++b)
      if ((m >> b) & 1) o |= 1ull << targets[b];
    a.offs[m] = o;
  }
  int ni = 0;
  if (PAIR) a.ins[ni++] = 0;
  for (int b = 0; b < K; ++b) a.ins[ni++] = targets[b];
  a.num_sets = 1ull << (n - K - (PAIR ? 1 : 0));
  const uint64_t want = (a.num_sets + 255) / 256;
  const uint64_t cap = static_cast<uint64_t>(sm_count()) * occ;
  const unsigned grid = static_cast<unsigned>(want < cap ? want : cap);
  k_apply<K, PAIR><<<grid, 256, 0, st>>>(psi, a);
  return cudaGetLastError();
}

cudaError_t launch_apply(float2* psi, int n, int k, const uint32_t* targets, const float2* U,
                         cudaStream_t st) {
  // targets ascending; pair mode needs qubit 0 free and at least one spare bit
  if (tile_fits(n, k)) {
    switch (k) {
      case 1: return launch_tile<1>(psi, n, targets, U, st);
      case 2: return launch_tile<2>(psi, n, targets, U, st);
      case 3: return launch_tile<3>(psi, n, targets, U, st);
      case 4: return launch_tile<4>(psi, n, targets, U, st);
      case 5: return launch_tile<5>(psi, n, targets, U, st);
      default: return cudaErrorInvalidValue;
    }
  }
  const bool pair = (targets[0] != 0) && (n >= k + 1);
  switch (k) {
    case 1: return pair ? launch_k<1, true>(psi, n, targets, U, st) : launch_k<1, false>(psi, n, targets, U, st);
    case 2: return pair ? launch_k<2, true>(psi, n, targets, U, st) : launch_k<2, false>(psi, n, targets, U, st);
    case 3: return pair ? launch_k<3, true>(psi, n, targets, U, st) : launch_k<3, false>(psi, n, targets, U, st);
    case 4: return pair ? launch_k<4, true>(psi, n, targets, U, st) : launch_k<4, false>(psi, n, targets, U, st);
    case 5: return launch_k<5, false>(psi, n, targets, U, st);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace qt
