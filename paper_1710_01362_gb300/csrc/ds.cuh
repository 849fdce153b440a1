// Double-single arithmetic (unevaluated sums h + l of two floats, 48-bit significand) and
// FP64 <-> FP32 conversions on the integer pipes.
//
// Error-free transformations: TwoSum (Knuth: s + e = a + b exactly) and TwoProduct through
// the fused multiply-add (p + e = a b exactly); the _rn intrinsics keep the compiler from
// contracting or reassociating them.  Products accumulate as a running float sum plus a
// float sum of all rounding errors, renormalised once at the end (the compensated dot
// product of Ogita, Rump and Oishi, SIAM J. Sci. Comput. 26 (2005), with double-single
// inputs).
#pragma once

namespace ttns {

// Conversions by integer arithmetic on the bit patterns (the FP64 <-> FP32 conversion
// instructions run on the narrow FP64 pipe).  ds_from: the head is the double rounded to
// nearest-even float (from the 29 dropped significand bits), the tail the exact remainder
// rounded to a float, scaled by a power of two; values below 2^-126 give zero, values beyond
// FP32's range take the conversion instruction.  Identical to h = (float) x,
// l = (float) (x - h) for |x| >= 2^-74.
__device__ __forceinline__ float magic_i2f(int n) {  // exact for |n| < 2^22
  return __uint_as_float(0x4B400000u + (unsigned)n) - 12582912.0f;
}
__device__ __forceinline__ float2 ds_from(double x) {
  const unsigned hi32 = (unsigned)__double2hiint(x), lo32 = (unsigned)__double2loint(x);
  const int e = (int)((hi32 >> 20) & 0x7FFu);
  if (e < 897) return make_float2(0.f, 0.f);
  if (e > 1149) return make_float2(__double2float_rn(x), 0.f);
  unsigned fb = (hi32 & 0x80000000u) | ((unsigned)(e - 896) << 23) | ((hi32 & 0xFFFFFu) << 3) | (lo32 >> 29);
  const unsigned rest = lo32 & 0x1FFFFFFFu;
  const unsigned up = (rest > 0x10000000u) || (rest == 0x10000000u && (fb & 1u));
  fb += up;  // a carry into the exponent field is the correct rounding
  const int lrem = (int)rest - (int)(up << 29);  // x - h in units of 2^(e - 1075)
  float l = __fmaf_rn(magic_i2f(lrem >> 14), 16384.0f, magic_i2f(lrem & 0x3FFF));
  const int se = e - 948;
  l = se >= 1 ? __fmul_rn(l, __uint_as_float((unsigned)se << 23))
              : __fmul_rn(__fmul_rn(l, 5.421010862427522e-20f), __uint_as_float((unsigned)(se + 64) << 23));
  if (hi32 & 0x80000000u) l = -l;
  return make_float2(__uint_as_float(fb), l);
}
// float -> double by the bit pattern (zero and normal floats; others by the instruction)
__device__ __forceinline__ double f2d_bits(float f) {
  const unsigned u = __float_as_uint(f);
  const unsigned ef = (u >> 23) & 0xFFu;
  if ((u << 1) == 0u) return __hiloint2double((int)(u & 0x80000000u), 0);
  if (ef == 0u || ef == 255u) return (double)f;
  return __hiloint2double((int)((u & 0x80000000u) | ((ef + 896u) << 20) | ((u & 0x7FFFFFu) >> 3)), (int)((u & 7u) << 29));
}
__device__ __forceinline__ double ds_to(float2 a) { return f2d_bits(a.x) + f2d_bits(a.y); }
// double -> float, rounded to nearest even, by the bit pattern: the head of ds_from
__device__ __forceinline__ float d2f_bits(double x) {
  const unsigned hi32 = (unsigned)__double2hiint(x), lo32 = (unsigned)__double2loint(x);
  const int e = (int)((hi32 >> 20) & 0x7FFu);
  if (e == 0) return __uint_as_float(hi32 & 0x80000000u);  // zero, or far below FP32's range
  if (e < 897 || e > 1149) return __double2float_rn(x);
  unsigned fb = (hi32 & 0x80000000u) | ((unsigned)(e - 896) << 23) | ((hi32 & 0xFFFFFu) << 3) | (lo32 >> 29);
  const unsigned rest = lo32 & 0x1FFFFFFFu;
  fb += (rest > 0x10000000u) || (rest == 0x10000000u && (fb & 1u));
  return __uint_as_float(fb);
}
__device__ __forceinline__ double to_f64(double x) { return x; }
__device__ __forceinline__ double to_f64(float x) { return f2d_bits(x); }
// s + t renormalised to a head and a tail (exact when |s| >= |t|)
__device__ __forceinline__ float2 ds_quick(float s, float t) {
  const float h = __fadd_rn(s, t);
  return make_float2(h, __fsub_rn(t, __fsub_rn(h, s)));
}
__device__ __forceinline__ float2 ds_add(float2 a, float2 b) {
  const float s = __fadd_rn(a.x, b.x);
  const float v = __fsub_rn(s, a.x);
  const float e = __fadd_rn(__fsub_rn(a.x, __fsub_rn(s, v)), __fsub_rn(b.x, v));
  return ds_quick(s, __fadd_rn(e, __fadd_rn(a.y, b.y)));
}
__device__ __forceinline__ float2 ds_neg(float2 a) { return make_float2(-a.x, -a.y); }
__device__ __forceinline__ float2 ds_re(float4 z) { return make_float2(z.x, z.y); }
__device__ __forceinline__ float2 ds_im(float4 z) { return make_float2(z.z, z.w); }
__device__ __forceinline__ float4 ds_c(float2 re, float2 im) { return make_float4(re.x, re.y, im.x, im.y); }
__device__ __forceinline__ float4 ds_cfrom(double2 z) { return ds_c(ds_from(z.x), ds_from(z.y)); }
__device__ __forceinline__ double2 ds_cto(float4 z) { return make_double2(ds_to(ds_re(z)), ds_to(ds_im(z))); }

struct DsAcc {
  float s, c;  // running sum and the sum of its rounding errors
  __device__ __forceinline__ void init(float2 a) {
    s = a.x;
    c = a.y;
  }
  __device__ __forceinline__ void mac(float2 x, float2 y) {  // += x y (the lo*lo term is below the format)
    const float p = __fmul_rn(x.x, y.x);
    float e = __fmaf_rn(x.x, y.x, -p);
    e = __fmaf_rn(x.x, y.y, e);
    e = __fmaf_rn(x.y, y.x, e);
    const float t = __fadd_rn(s, p);
    const float v = __fsub_rn(t, s);
    c = __fadd_rn(c, __fadd_rn(__fadd_rn(__fsub_rn(s, __fsub_rn(t, v)), __fsub_rn(p, v)), e));
    s = t;
  }
  __device__ __forceinline__ float2 val() const { return ds_quick(s, c); }
};

__device__ __forceinline__ float2 shfl_xor_ds(float2 v, int o) {
  return make_float2(__shfl_xor_sync(0xffffffffu, v.x, o), __shfl_xor_sync(0xffffffffu, v.y, o));
}

}  // namespace ttns
