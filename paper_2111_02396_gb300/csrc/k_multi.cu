// Several fused gates in one pass over the state (Alg. 1 on a staged tile).
//
// A pass over a large state costs its bytes (16 an amplitude, 0.71 clocks of
// an SM's share of HBM); the arithmetic of a 4-qubit gate is 0.38 clocks of
// FP32 FMA.  So consecutive pieces whose qubits, with the lowest kMultiLow
// ones, fit a tile of 2^kMultiBits amplitudes go in one pass: a CTA brings its
// tile to shared memory, applies every gate in order and writes it back once.
// States of at most 2^kMultiBits amplitudes are one tile, and a launch takes
// as many gates as its parameters hold.
//
// The gates keep their order and the sums theirs: with c, e, f of an entry
// U = (c, d) and member a + i b as in k_apply.cu (e = c + d, f = d - c, s = a +
// b), an output is (sum c s - sum e b, sum c s + sum f a).  The outputs are the
// same bits as one pass per gate (k_apply_tile).
//
// What feeds the FMAs decides the form.  The matrix sits in the kernel
// parameters and comes through uniform loads (8 bytes at most) from the
// constant bank.
//   - One tile (n <= kMultiFewLog): 512 threads, a set each; what counts is the
//     chain of dependent loads of a gate.  Whole warps drop out together where
//     there are fewer sets, which keeps the matrix loads uniform (per-thread
//     ones: n = 12, 26 -> 46 us a pass of 8 gates on 4 qubits; n = 10, 25 -> 33
//     of 32 on 2).
//   - Many tiles: 128 threads, 4 CTAs an SM; a thread takes 8 sets of 1 or 2
//     qubits, 4 of 3, 2 of 4 (96 registers of members), so that an entry is
//     loaded once for all of them.  The FMAs are scalar: they take an entry
//     from its uniform register however often it is used, where a packed FMA
//     takes a pair of them only once and otherwise wants it moved to registers
//     (n = 28, packed and scalar: 2 qubits 58.8 and 51.0 ms, 3 qubits 60.4 and
//     45.7).  64 threads with 4 sets of 4 qubits need 15% fewer instructions
//     but leave 8 warps an SM: 51.8 ms for 44.6.
// Bound by issue (85-89% of the slots with 4-qubit gates, 59% of them FMAs) rather
// than HBM from two gates a pass on.  Grouping pays at every size, so whatever
// fits is grouped.  Device time of a grid circuit, one pass a gate -> grouped,
// fused to at most 2, 3 and 4 qubits (in ms; n = 28: 211, 121 and 70 gates in
// 47, 46 and 33 passes):
//   n = 28   129 -> 51.0   79.6 -> 45.7   51.4 -> 44.6
//   n = 20  1.57 -> 0.55   0.97 -> 0.46   0.69 -> 0.45
// and of 200 gates on random qubits, n = 26: 15.4 -> 5.8, 9.3 -> 4.9, 7.1 -> 6.0;
// n = 13: 0.92 -> 0.22, 0.52 -> 0.19, 0.39 -> 0.21.
#include <cuda_runtime.h>

#include <cstddef>

#include "kernels.h"

namespace qt {

namespace multi {

constexpr int kThreads = 128, kFewThreads = 512;

struct alignas(16) Gate {       // the parameters stay 16-byte aligned from gate to gate
  uint32_t smoff[16];         // swizzled tile offset of member m, in bytes
  uint32_t step[8];           // and of a thread's set b from its first
  uint32_t mat;               // first entry of its matrix
  uint8_t k, tins[4], pad[7];
};

// CAP: matrix entries of a launch.  Parameters are copied with every launch
// (12 us of the host for 32 KB, 4 for 12), so there are smaller forms: 512 for
// the one or two gates common in large states, 1024 for 48 gates on 2 qubits.
template <int CAP>
struct alignas(16) Args {
  float4 ce[CAP / 2];         // (c, e) of two entries, row-major per gate
  float4 f[CAP / 4];          // f of four
  uint64_t poff[16];          // memory offset of tile index 256 c (chunk c of every thread)
  Gate g[kMultiGates];
  uint32_t q[kMultiBits];     // qubit of tile bit i, ascending
  uint64_t swz;               // slot = l ^ nibble (l >> 4) & 15 (lanes differ: no table in the constant bank)
  int ng, bits, C;            // gates; tile bits; contiguous low bits of a row
};
// matrix entries come through 8- and 16-byte loads of the constant bank
template <int CAP>
constexpr bool kAligned = offsetof(Args<CAP>, ce) % 16 == 0 && offsetof(Args<CAP>, f) % 16 == 0 &&
                          offsetof(Args<CAP>, poff) % 16 == 0 && offsetof(Args<CAP>, g) % 16 == 0 &&
                          offsetof(Args<CAP>, swz) % 8 == 0 && sizeof(Args<CAP>) % 16 == 0;
static_assert(sizeof(Gate) % 16 == 0 && kAligned<512> && kAligned<1024> && kAligned<kMultiEntries>);
static_assert(sizeof(Args<kMultiEntries>) <= 32764);   // what a launch's parameters may hold

__device__ __forceinline__ float2* slot(float2* sm, uint32_t bytes) {
  return reinterpret_cast<float2*>(reinterpret_cast<char*>(sm) + bytes);
}

__device__ __forceinline__ uint32_t swizzle(uint32_t l, uint64_t t) {
  return l ^ (static_cast<uint32_t>(t >> ((l >> 2) & 60u)) & 15u);
}

template <int K, int B, int T, int CAP>
__device__ __forceinline__ void gate(float2* sm, const Args<CAP>& a, const Gate& g, uint32_t warp) {
  constexpr int M = 1 << K;
  const uint32_t sets = 1u << (a.bits - K);        // 128 or more; with B > 1 a multiple of B T
  // whole warps loop together: a condition on the thread would make every
  // matrix entry a per-thread load instead of a uniform one
  for (uint32_t w = warp; w < sets; w += B * T) {
    const uint32_t s0 = w + (threadIdx.x & 31u);
    uint32_t base[B];
    float va[B][M], vb[B][M], vs[B][M];            // a, b and s = a + b of member m
    uint32_t s = s0;
#pragma unroll
    for (int i = 0; i < K; ++i) {
      const uint32_t t = g.tins[i];
      s = ((s >> t) << (t + 1)) | (s & ((1u << t) - 1u));
    }
    s = swizzle(s, a.swz);
#pragma unroll
    for (int b = 0; b < B; ++b) {
      base[b] = (8 * s) ^ g.step[b];               // the swizzle distributes over disjoint bits
#pragma unroll
      for (int m = 0; m < M; ++m) {
        const float2 v = *slot(sm, base[b] ^ g.smoff[m]);
        va[b][m] = v.x;
        vb[b][m] = v.y;
        vs[b][m] = v.x + v.y;
      }
    }
    const float4* const ce = a.ce + g.mat / 2;
    const float4* const ff = a.f + g.mat / 4;
#pragma unroll 8
    for (int j = 0; j < M; ++j) {
      float cs[B], eb[B], fa[B];
#pragma unroll
      for (int b = 0; b < B; ++b) cs[b] = eb[b] = fa[b] = 0.f;
#pragma unroll
      for (int m = 0; m < M; ++m) {
        const int x = j * M + m;
        const float4 u = ce[x >> 1], w = ff[x >> 2];
        const float c = x & 1 ? u.z : u.x, e = x & 1 ? u.w : u.y;
        const float f = x & 2 ? (x & 1 ? w.w : w.z) : (x & 1 ? w.y : w.x);
#pragma unroll
        for (int b = 0; b < B; ++b) {
          cs[b] = fmaf(c, vs[b][m], cs[b]);
          eb[b] = fmaf(e, vb[b][m], eb[b]);
          fa[b] = fmaf(f, va[b][m], fa[b]);
        }
      }
#pragma unroll
      for (int b = 0; b < B; ++b) *slot(sm, base[b] ^ g.smoff[j]) = make_float2(cs[b] - eb[b], cs[b] + fa[b]);
    }
  }
}

template <int T, int CAP>
__global__ void __launch_bounds__(T, T == kThreads ? 4 : 1) k_multi(float2* __restrict__ psi,
                                                                    const __grid_constant__ Args<CAP> a) {
  constexpr bool FEW = T == kFewThreads;
  __shared__ __align__(16) float2 sm[1 << kMultiBits];
  const uint32_t tid = threadIdx.x, l0 = 2u * tid;
  uint64_t base = static_cast<uint64_t>(blockIdx.x) << a.C;
  for (int i = a.C; i < a.bits; ++i) {
    const uint32_t h = a.q[i];
    base = ((base >> h) << (h + 1)) | (base & ((1ull << h) - 1ull));
  }
  uint64_t off = l0 & ((1u << a.C) - 1u);
  constexpr int TB = FEW ? 10 : 8;                           // bits of l0
  for (int i = a.C; i < TB && i < a.bits; ++i)
    if ((l0 >> i) & 1u) off |= 1ull << a.q[i];
  float2* const pt = psi + (base | off);
  // bits 4..7 of 2t + 2 T c are those of 2t
  const uint32_t s0 = swizzle(l0, a.swz), s1 = s0 ^ 1u;
  constexpr int NC = (1 << kMultiBits) / 2 / T;              // 16-byte chunks per thread of a full tile
  constexpr int STEP = 2 * T / 256;                          // chunk c is at tile index 256 STEP c
  // a state below 2^kMultiBits (FEW only): idle threads, fewer chunks
  const bool in = !FEW || l0 < (1u << a.bits);
  const int chunks = FEW ? max((1 << a.bits) / 2 / T, 1) : NC;
  {
    float4 buf[NC];
#pragma unroll
    for (int c = 0; c < NC; ++c)
      if (c < chunks && in) buf[c] = __ldcs(reinterpret_cast<const float4*>(pt + a.poff[STEP * c]));
#pragma unroll
    for (int c = 0; c < NC; ++c)
      if (c < chunks && in) {
        sm[s0 + 2u * T * c] = make_float2(buf[c].x, buf[c].y);
        sm[s1 + 2u * T * c] = make_float2(buf[c].z, buf[c].w);
      }
  }
  const uint32_t warp = __shfl_sync(0xffffffffu, tid & ~31u, 0);   // first thread of the warp
  for (int i = 0; i < a.ng; ++i) {
    __syncthreads();
    const Gate& g = a.g[i];
    switch (g.k) {
      case 1: gate<1, FEW ? 1 : 8, T, CAP>(sm, a, g, warp); break;
      case 2: gate<2, FEW ? 1 : 8, T, CAP>(sm, a, g, warp); break;
      case 3: gate<3, FEW ? 1 : 4, T, CAP>(sm, a, g, warp); break;
      default: gate<4, FEW ? 1 : 2, T, CAP>(sm, a, g, warp); break;
    }
  }
  __syncthreads();
#pragma unroll
  for (int c = 0; c < NC; ++c)
    if (c < chunks && in) {
      const float2 x = sm[s0 + 2u * T * c], y = sm[s1 + 2u * T * c];
      __stcs(reinterpret_cast<float4*>(pt + a.poff[STEP * c]), make_float4(x.x, x.y, y.x, y.y));
    }
}

}  // namespace multi

bool multi_fits(int n, int ng, const MultiPiece* p) {
  if (ng < 1 || ng > kMultiGates) return false;
  uint64_t mask = (1ull << kMultiLow) - 1ull;
  int entries = 0;
  for (int i = 0; i < ng; ++i) {
    if (p[i].k < 1 || p[i].k > 4 || n < 7 + p[i].k) return false;
    for (int b = 0; b < p[i].k; ++b) mask |= 1ull << p[i].targets[b];
    entries += 1 << (2 * p[i].k);
  }
  return __builtin_popcountll(mask) <= (n < kMultiBits ? n : kMultiBits) && entries <= kMultiEntries;
}

// 16-lane accesses of a gate that fall on the same bank pair: lanes differ in
// the four lowest positions that are no target; positions 4..7 map to the bits
// img[0..3], lower ones stay
static int conflict_log(const uint32_t* tpos, int k, const uint32_t* img, int bits) {
  uint32_t rows[4], nr = 0, tm = 0;
  for (int b = 0; b < k; ++b) tm |= 1u << tpos[b];
  for (int p = 0; nr < 4 && p < bits; ++p)
    if (!((tm >> p) & 1u)) rows[nr++] = p < 4 ? 1u << p : (p < 8 ? img[p - 4] : 0u);
  int rank = 0;
  for (int b = 0; b < 4; ++b) {
    uint32_t pivot = nr;
    for (uint32_t i = rank; i < nr; ++i)
      if ((rows[i] >> b) & 1u) { pivot = i; break; }
    if (pivot == nr) continue;
    const uint32_t t = rows[pivot]; rows[pivot] = rows[rank]; rows[rank] = t;
    for (uint32_t i = 0; i < nr; ++i)
      if (static_cast<int>(i) != rank && ((rows[i] >> b) & 1u)) rows[i] ^= rows[rank];
    ++rank;
  }
  return static_cast<int>(nr) - rank;
}

template <int CAP>
static cudaError_t launch_cap(float2* psi, int n, int ng, const MultiPiece* p, cudaStream_t st) {
  multi::Args<CAP> a;
  a.bits = n < kMultiBits ? n : kMultiBits;
  a.ng = ng;
  uint64_t mask = (1ull << kMultiLow) - 1ull;
  for (int i = 0; i < ng; ++i)
    for (int b = 0; b < p[i].k; ++b) mask |= 1ull << p[i].targets[b];
  for (int q = 0; __builtin_popcountll(mask) < a.bits; ++q) mask |= 1ull << q;
  a.C = 0;
  while (a.C < a.bits && ((mask >> a.C) & 1ull)) ++a.C;
  int nb = 0;
  for (int q = 0; q < 64; ++q)
    if ((mask >> q) & 1ull) a.q[nb++] = static_cast<uint32_t>(q);
  auto pos = [&](uint32_t q) { return static_cast<uint32_t>(__builtin_popcountll(mask & ((1ull << q) - 1ull))); };
  uint32_t tpos[kMultiGates][4], off = 0;
  for (int i = 0; i < ng; ++i) {
    multi::Gate& g = a.g[i];
    const int k = p[i].k, M = 1 << k;
    g.k = static_cast<uint8_t>(k);
    g.mat = off;
    for (int b = 0; b < k; ++b) {
      tpos[i][b] = pos(p[i].targets[b]);
      g.tins[b] = static_cast<uint8_t>(tpos[i][b]);
    }
    for (int e = 0; e < M * M; ++e) {
      const float re = p[i].u[e].x, im = p[i].u[e].y;
      float4& ce = a.ce[(off + e) / 2];
      (e & 1 ? ce.z : ce.x) = re;
      (e & 1 ? ce.w : ce.y) = re + im;
      float4& f = a.f[(off + e) / 4];
      (e & 2 ? (e & 1 ? f.w : f.z) : (e & 1 ? f.y : f.x)) = im - re;
    }
    off += static_cast<uint32_t>(M * M);
  }
  // the swizzle: of a few linear maps, the one with the fewest conflicts over
  // the gates (the image of bit 4 sets bit 0, for the staging accesses).  The
  // first is free of them for runs of up to three neighbouring qubits, the
  // others for single gates with targets below position 4.
  static const uint32_t maps[][4] = {{15, 10, 12, 8}, {1, 2, 4, 8}, {3, 6, 12, 9}, {9, 5, 14, 2}, {5, 11, 6, 12},
                                     {7, 9, 4, 10},   {13, 6, 3, 8}, {11, 14, 8, 5}, {1, 4, 8, 2}, {1, 8, 2, 4},
                                     {3, 12, 5, 10},  {9, 2, 12, 7}};
  int best = 1 << 30;
  const uint32_t* img = maps[0];
  for (const auto& m : maps) {
    int cost = 0;
    for (int i = 0; i < ng; ++i) cost += (1 << conflict_log(tpos[i], p[i].k, m, a.bits)) << p[i].k;
    if (cost < best) { best = cost; img = m; }
  }
  uint32_t tab[16];
  a.swz = 0;
  for (int x = 0; x < 16; ++x) {
    tab[x] = 0;
    for (int b = 0; b < 4; ++b)
      if ((x >> b) & 1) tab[x] ^= img[b];
    a.swz |= static_cast<uint64_t>(tab[x]) << (4 * x);
  }
  for (int i = 0; i < ng; ++i) {
    for (int m = 0; m < (1 << p[i].k); ++m) {
      uint32_t o = 0;
      for (int b = 0; b < p[i].k; ++b)
        if ((m >> b) & 1) o |= 1u << tpos[i][b];
      a.g[i].smoff[m] = 8 * (o ^ tab[(o >> 4) & 15u]);
    }
    for (uint32_t e = 0; e < 8; ++e) {             // set b is multi::kThreads sets on (FEW: one set a thread)
      uint32_t o = e * multi::kThreads;
      for (int b = 0; b < p[i].k; ++b) o = ((o >> tpos[i][b]) << (tpos[i][b] + 1)) | (o & ((1u << tpos[i][b]) - 1u));
      a.g[i].step[e] = 8 * (o ^ tab[(o >> 4) & 15u]);
    }
  }
  for (int c = 0; c < 16; ++c) {
    const uint32_t l = 256u * static_cast<uint32_t>(c);
    uint64_t o = 0;
    for (int i = 0; i < a.bits; ++i)
      if ((l >> i) & 1u) o |= 1ull << a.q[i];
    a.poff[c] = o;
  }
  const unsigned grid = static_cast<unsigned>(1ull << (n - a.bits));
  if (n <= kMultiFewLog) multi::k_multi<multi::kFewThreads, CAP><<<grid, multi::kFewThreads, 0, st>>>(psi, a);
  else multi::k_multi<multi::kThreads, CAP><<<grid, multi::kThreads, 0, st>>>(psi, a);
  return cudaGetLastError();
}

cudaError_t launch_multi(float2* psi, int n, int ng, const MultiPiece* p, cudaStream_t st) {
  if (!multi_fits(n, ng, p)) return cudaErrorInvalidValue;
  int entries = 0;
  for (int i = 0; i < ng; ++i) entries += 1 << (2 * p[i].k);
  if (entries <= 512) return launch_cap<512>(psi, n, ng, p, st);
  if (entries <= 1024) return launch_cap<1024>(psi, n, ng, p, st);
  return launch_cap<kMultiEntries>(psi, n, ng, p, st);
}

}  // namespace qt
