// Values and running sums of three FP32 words, for sums that need the accuracy of FP64
// on a part that executes 2 FP64 operations per clock and SM against 128 in FP32.
#pragma once

#include <cuda_runtime.h>

namespace lbm {

// A value h + l + m of three FP32 words, |l| <= 2^-24 |h| and m of the order of
// 2^-48 |h| (a rounded remainder, so the value is good to about 2^-70).
struct Words {
  float h, l, m;
};
// s + e = a + b exactly (Knuth)
__device__ __forceinline__ float two_sum(float a, float b, float& e) {
  const float s = __fadd_rn(a, b), t = __fsub_rn(s, a);
  e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, t)), __fsub_rn(b, t));
  return s;
}
// s += v, every remainder kept.
__device__ __forceinline__ void add_full(Words& s, const Words& v) {
  float e, e1, e2;
  s.h = two_sum(s.h, v.h, e);
  const float w = two_sum(e, v.l, e1);
  s.l = two_sum(s.l, w, e2);
  s.m = __fadd_rn(s.m, __fadd_rn(v.m, __fadd_rn(e1, e2)));
}
__device__ __forceinline__ Words shfl_xor(const Words& v, int mask) {
  return Words{__shfl_xor_sync(0xffffffffu, v.h, mask), __shfl_xor_sync(0xffffffffu, v.l, mask),
               __shfl_xor_sync(0xffffffffu, v.m, mask)};
}
__device__ __forceinline__ double to_double(const Words& v) { return (double)v.h + ((double)v.l + (double)v.m); }

// Sum 16 values over the warp's 32 lanes, value i ending in lanes 2 i and 2 i + 1: each
// of the first four steps halves the values a lane holds (16 additions instead of 80).
__device__ __forceinline__ Words warp_sum16(Words (&a)[16], int lane) {
#pragma unroll
  for (int s = 16; s > 1; s >>= 1) {
    const bool up = (lane & s) != 0;
#pragma unroll
    for (int i = 0; i < s / 2; ++i) {
      const Words lo = a[i], hi = a[i + s / 2];
      Words keep = up ? hi : lo;
      add_full(keep, shfl_xor(up ? lo : hi, s));
      a[i] = keep;
    }
  }
  add_full(a[0], shfl_xor(a[0], 1));
  return a[0];
}
__device__ __forceinline__ double warp_sum16(double (&a)[16], int lane) {
#pragma unroll
  for (int s = 16; s > 1; s >>= 1) {
    const bool up = (lane & s) != 0;
#pragma unroll
    for (int i = 0; i < s / 2; ++i) {
      const double lo = a[i], hi = a[i + s / 2];
      a[i] = (up ? hi : lo) + __shfl_xor_sync(0xffffffffu, up ? lo : hi, s);
    }
  }
  return a[0] + __shfl_xor_sync(0xffffffffu, a[0], 1);
}

}  // namespace lbm
