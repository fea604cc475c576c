// Double-float sums: a value held as the unevaluated sum of two floats.
//
// FP64 runs at about 2 operations per clock and SM on sm_103a (1/64 of the
// FP32 rate; one warp-wide FP64 add holds its scheduler's FP64 pipe for 64
// clocks), so the reductions carry their FP32 runs in double-floats, with
// Knuth's error-free addition (The Art of Computer Programming, vol. 2,
// 4.2.2, theorem B): ~48 bits, well below the rounding of the FP32 runs
// themselves.  One carry is 7 FADDs instead of a conversion and an FP64 add.
// Results leave as FP64.
#pragma once
#include <cuda_runtime.h>

namespace qt {

// (h, l) += f
__device__ __forceinline__ void df_acc(float& h, float& l, float f) {
  const float s = h + f;
  const float b = s - h;
  l += (h - (s - b)) + (f - b);
  h = s;
}

__device__ __forceinline__ float2 df_add(float2 x, float2 y) {
  const float s = x.x + y.x;
  const float b = s - x.x;
  const float e = (x.x - (s - b)) + (y.x - b);
  return make_float2(s, (x.y + y.y) + e);
}

// a non-finite sum leaves its error term undefined (inf - inf): the sum alone counts
__device__ __forceinline__ double df_value(float2 x) {
  return isfinite(x.x) ? static_cast<double>(x.x) + static_cast<double>(x.y) : static_cast<double>(x.x);
}

__device__ __forceinline__ float2 df_shfl_xor(float2 v, int o) {
  return make_float2(__shfl_xor_sync(0xffffffffu, v.x, o), __shfl_xor_sync(0xffffffffu, v.y, o));
}

// Sums of P values over the warp (P a power of two, at most 32), transposed:
// each step halves the values a lane holds, so the warp does ~P exchanges
// instead of 5 P.  Lane l ends with the sum of value l >> (5 - log2 P).
template <int P>
__device__ __forceinline__ float2 df_warp_sum(float2 (&v)[P], int lane) {
  int c = P;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    if (c > 1) {
      c >>= 1;
      const bool up = lane & o;
#pragma unroll
      for (int k = 0; k < P / 2; ++k) {
        if (k >= c) break;
        const float2 keep = up ? v[k + c] : v[k], send = up ? v[k] : v[k + c];
        v[k] = df_add(keep, df_shfl_xor(send, o));
      }
    } else {
      v[0] = df_add(v[0], df_shfl_xor(v[0], o));
    }
  }
  return v[0];
}

}  // namespace qt
