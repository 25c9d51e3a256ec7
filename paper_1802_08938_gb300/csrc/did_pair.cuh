#pragma once
// Pairs of float32 (hi + lo, about 45 to 48 bits) for the sums and scalars that
// need more than float32: float64 runs at 2 FMA per cycle and SM.  The
// sums are Knuth's two-sum, the products exact by FMA.  The range is float32's:
// a product of entries below about 1e-19 loses bits, below 1e-23 it is zero.
#include <cuda_runtime.h>

namespace did {

struct df {
  float h, l;
};
__device__ __forceinline__ df df_zero() { return df{0.f, 0.f}; }
// a + b, two-sum of the high parts (Knuth), renormalised.
__device__ __forceinline__ df df_add(df a, df b) {
  const float s = __fadd_rn(a.h, b.h);
  const float t = __fsub_rn(s, a.h);
  float e = __fadd_rn(__fsub_rn(a.h, __fsub_rn(s, t)), __fsub_rn(b.h, t));
  e = __fadd_rn(e, __fadd_rn(a.l, b.l));
  df r;
  r.h = __fadd_rn(s, e);
  r.l = __fsub_rn(e, __fsub_rn(r.h, s));
  return r;
}
// acc + x y (the product exact as p + fma(x, y, -p)).
__device__ __forceinline__ df df_fma(float x, float y, df acc) {
  const float p = __fmul_rn(x, y);
  return df_add(acc, df{p, __fmaf_rn(x, y, -p)});
}
// acc + x y for a pair y.
__device__ __forceinline__ df df_fma(float x, df y, df acc) {
  const float p = __fmul_rn(x, y.h);
  return df_add(acc, df{p, __fmaf_rn(x, y.l, __fmaf_rn(x, y.h, -p))});
}
// acc + v, the compensation collected without renormalising (running sums).
__device__ __forceinline__ void df_acc(df& a, float v) {
  const float s = __fadd_rn(a.h, v);
  const float t = __fsub_rn(s, a.h);
  a.l = __fadd_rn(a.l, __fadd_rn(__fsub_rn(a.h, __fsub_rn(s, t)), __fsub_rn(v, t)));
  a.h = s;
}
// a / b: a float32 quotient and its correction (a float64 division by all 16
// warps costs about 2 us).
__device__ __forceinline__ df df_div(df a, df b) {
  const float q = __fdiv_rn(a.h, b.h);
  const float p = __fmul_rn(q, b.h);
  const float e = __fmaf_rn(q, b.h, -p);
  const float r = __fadd_rn(__fsub_rn(a.h, p), __fsub_rn(a.l, __fmaf_rn(q, b.l, e)));
  return df_add(df{q, 0.f}, df{__fdiv_rn(r, b.h), 0.f});
}
// The product of two pairs, rounded to float32.
__device__ __forceinline__ float df_mul_f32(df a, df b) {
  const float p = __fmul_rn(a.h, b.h);
  return p + (__fmaf_rn(a.h, b.h, -p) + __fmaf_rn(a.h, b.l, __fmul_rn(a.l, b.h)));
}
__device__ __forceinline__ df df_shfl_xor(df a, int m) {
  return df{__shfl_xor_sync(0xffffffffu, a.h, m), __shfl_xor_sync(0xffffffffu, a.l, m)};
}
// Sums over the 32 lanes of eight values at once: lane i (and i + 8, ...)
// returns the total of v[i % 8].  Nine pair additions instead of forty.
__device__ __forceinline__ df df_warp_sum8(df v[8]) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int w = 4; w >= 1; w >>= 1) {
    const bool up = (lane & w) != 0;
#pragma unroll
    for (int i = 0; i < w; ++i) {
      const df send = up ? v[i] : v[i + w];
      const df keep = up ? v[i + w] : v[i];
      v[i] = df_add(keep, df_shfl_xor(send, w));
    }
  }
  df s = df_add(v[0], df_shfl_xor(v[0], 8));
  return df_add(s, df_shfl_xor(s, 16));
}
__device__ __forceinline__ df df_warp_sum(df a) {
#pragma unroll
  for (int m = 16; m >= 1; m >>= 1) a = df_add(a, df_shfl_xor(a, m));
  return a;
}

}  // namespace did
