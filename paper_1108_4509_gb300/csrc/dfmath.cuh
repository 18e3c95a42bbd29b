// Double-float arithmetic: a value is a pair of FP32 numbers hi + lo
// (|lo| <= ulp(hi)/2, about 48 significant bits). Sums use Knuth's TwoSum,
// products Dekker's TwoProduct through a fused multiply-add; both are exact
// transformations, so the only errors are the final roundings of the lo
// parts (a few units of 2^-48 relative to the magnitudes involved). The code
// must be compiled without fast-math reassociation (the build does not use
// it).
#pragma once

#include <cstdint>

namespace trm {

struct F2 {
  float h, l;
};

// s + e = a + b exactly (any magnitudes).
__device__ __forceinline__ F2 two_sum(float a, float b) {
  const float s = a + b;
  const float bb = s - a;
  return {s, (a - (s - bb)) + (b - bb)};
}
// s + e = a + b exactly when |a| >= |b| or a == 0.
__device__ __forceinline__ F2 quick_two_sum(float a, float b) {
  const float s = a + b;
  return {s, b - (s - a)};
}
__device__ __forceinline__ F2 df_add(F2 a, F2 b) {
  F2 s = two_sum(a.h, b.h);
  s.l += a.l + b.l;
  return quick_two_sum(s.h, s.l);
}
__device__ __forceinline__ F2 df_mul(F2 a, F2 b) {
  const float p = a.h * b.h;
  float e = fmaf(a.h, b.h, -p);
  e = fmaf(a.h, b.l, e);
  e = fmaf(a.l, b.h, e);
  return quick_two_sum(p, e);
}
__device__ __forceinline__ F2 df_of(double v) {
  const float h = __double2float_rn(v);
  return {h, __double2float_rn(v - (double)h)};
}
// FP64 -> (hi, lo) on the integer pipe: hi = fl32(v) rounded to nearest even
// from the bits, and v - hi is the signed integer made of the dropped bits,
// whose conversion to FP32 is lo's only rounding (the scaling by a power of
// two is exact, in two factors so that neither is subnormal). The same bits as
// df_of, without its three FP64-pipe instructions; magnitudes outside
// [2^-97, 2^127) other than zero take df_of.
__device__ __forceinline__ F2 df_of_bits(double v) {
  const long long u = __double_as_longlong(v);
  const int ef = (int)((u >> 52) & 0x7FF);
  const uint32_t sign = (uint32_t)(u >> 32) & 0x80000000u;
  if (ef < 926 || ef >= 1150) {  // 926 = 1023 - 97, 1150 = 1023 + 127
    if (ef == 0) return {__uint_as_float(sign), __uint_as_float(sign)};
    return df_of(v);
  }
  const uint32_t low = (uint32_t)u & 0x1FFFFFFFu;  // the 29 dropped bits
  const uint32_t top = (uint32_t)(((unsigned long long)u >> 29) & 0x7FFFFFu) |
                       ((uint32_t)(ef - 896) << 23);
  const uint32_t up =
      (low > 0x10000000u || (low == 0x10000000u && (top & 1u))) ? 1u : 0u;
  const int d = (int)low - (int)(up << 29);
  const float r = (float)(sign ? -d : d) * 9.094947017729282379e-13f;  // 2^-40
  return {__uint_as_float((top + up) | sign),
          r * __uint_as_float((uint32_t)(ef - 908) << 23)};  // 2^(e - 12)
}
__device__ __forceinline__ double to_double(F2 a) {
  return (double)a.h + (double)a.l;
}

// Accumulator of products of pairs: a.b by a fused multiply-add TwoProduct
// of the high parts plus the cross terms, added by TwoSum into the high part
// and plainly into the low part; norm() renormalises (call it every few
// dozen products). About 2^-46 relative to the sum of |a||b|.
struct DfAcc {
  float h = 0.f, l = 0.f;
  __device__ __forceinline__ void fma(float ah, float al, float bh, float bl) {
    const float p = ah * bh;
    float e = fmaf(ah, bh, -p);
    e = fmaf(ah, bl, e);
    e = fmaf(al, bh, e);
    const F2 t = two_sum(h, p);
    h = t.h;
    l += t.l + e;
  }
  __device__ __forceinline__ void norm() {
    const F2 t = quick_two_sum(h, l);
    h = t.h;
    l = t.l;
  }
};

}  // namespace trm
