// Pairs of floats, the unevaluated sum of a high and a low part of 48 bits together: what
// stands in for FP64 where its rate, one warp-wide instruction in 76 clocks on GB300
// (measured), would bound a kernel. The operations are the classical ones: Knuth's two-sum,
// an FMA for a product's rounding (Dekker 1971; Hida, Li & Bailey 2001).
#pragma once

#include "letkf_device.cuh"

namespace {

struct Df {
  float h, l;
};

__device__ __forceinline__ Df df(float a) { return Df{a, 0.f}; }
__device__ __forceinline__ Df df_of(double a) {
  const float h = (float)a;
  return Df{h, (float)(a - (double)h)};
}
__device__ __forceinline__ float pow2f(int e) {               // -126 <= e <= 127
  return __int_as_float((127 + e) << 23);
}
// v 2^sh by its bits (a conversion instruction from FP64 takes as long as an FP64 FMA, 76
// clocks): the upper 24 bits of its significand and the lower 29 rounded to 24. Zero below
// 2^-70, NaN above 2^100.
__device__ __forceinline__ Df df_split(double v, int sh) {
  const int H = __double2hiint(v), L = __double2loint(v), eb = (H >> 20) & 0x7ff;
  const int e = eb - 1023 + sh, sg = H & 0x80000000;
  const float hi = __int_as_float(sg | (e + 127) << 23 | (H & 0xfffff) << 3 | (unsigned)L >> 29);
  const float lo = (float)(L & 0x1fffffff) * __int_as_float(sg | (e - 52 + 127) << 23);
  const float s = __fadd_rn(hi, lo);
  Df r = Df{s, __fsub_rn(lo, __fsub_rn(s, hi))};
  if (eb == 0x7ff || e > 100) r = Df{__int_as_float(0x7fffffff), 0.f};
  if (eb == 0 || e < -70) r = Df{0.f, 0.f};
  return r;
}
// the exponent e with |v| < 2^e (-1022 for zero)
__device__ __forceinline__ int exponent64(double v) {
  return ((__double2hiint(v) >> 20) & 0x7ff) - 1022;
}
// The double (v.h + v.l) 2^sh, the parts normalised, again by bits; zero below the normal
// range.
__device__ __forceinline__ double df_to_double(Df v, int sh) {
  const int u = __float_as_int(v.h), eb = (u >> 23) & 0xff, E = eb - 127 + 1023 + sh;
  // the low part in units of the result's last place (2^-52 of the leading bit)
  int li = __float2int_rn(v.l * __int_as_float((254 - eb) << 23) * 4503599627370496.f);
  if (u < 0) li = -li;
  if ((u & 0x7fffff) == 0 && li < 0) li += li;       // into the binade below, its unit half
  const long long b = ((long long)E << 52 | (long long)(u & 0x7fffff) << 29) + li;
  double r = __longlong_as_double(b | (long long)(u & 0x80000000) << 32);
  if (eb == 0 || E < 2) r = 0.0;
  if (eb == 0xff || E > 2046) r = __hiloint2double(0x7ff80000, 0);
  return r;
}
__device__ __forceinline__ Df df_quick(float h, float l) {   // |h| >= |l|
  const float s = __fadd_rn(h, l);
  return Df{s, __fsub_rn(l, __fsub_rn(s, h))};
}
__device__ __forceinline__ Df df_add(Df a, Df b) {
  const float s = __fadd_rn(a.h, b.h), bb = __fsub_rn(s, a.h);
  const float e = __fadd_rn(__fsub_rn(a.h, __fsub_rn(s, bb)), __fsub_rn(b.h, bb));
  return df_quick(s, __fadd_rn(e, __fadd_rn(a.l, b.l)));
}
__device__ __forceinline__ Df df_neg(Df a) { return Df{-a.h, -a.l}; }
__device__ __forceinline__ Df df_mul(Df a, Df b) {
  const float p = __fmul_rn(a.h, b.h);
  return df_quick(p, fmaf(a.l, b.h, fmaf(a.h, b.l, fmaf(a.h, b.h, -p))));
}
__device__ __forceinline__ Df df_rcp(Df a) {                 // one Newton step from 1 / a.h
  const float r = __fdividef(1.f, a.h);
  const float e = fmaf(-a.l, r, fmaf(-a.h, r, 1.f));
  return df_quick(r, __fmul_rn(r, e));
}
__device__ __forceinline__ Df df_sqrt(Df a) {                // a > 0
  const float s = sqrtf(a.h), p = __fmul_rn(s, s);
  const float e = __fadd_rn(__fadd_rn(__fsub_rn(a.h, p), -fmaf(s, s, -p)), a.l);
  return df_quick(s, __fdividef(0.5f * e, s));
}
__device__ __forceinline__ Df df_shfl(Df a, int src) {
  return Df{__shfl_sync(FULL, a.h, src), __shfl_sync(FULL, a.l, src)};
}
__device__ __forceinline__ Df df_shfl_xor(Df a, int o) {
  return Df{__shfl_xor_sync(FULL, a.h, o), __shfl_xor_sync(FULL, a.l, o)};
}
__device__ __forceinline__ Df df_warp_sum(Df v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = df_add(v, df_shfl_xor(v, o));
  return v;
}
// Sum over the warp of values below 2^E, to 2^(E-51) each: two 26-bit integer parts through
// the warp's integer reduction (a third of the instructions and of the latency of five
// exchanges with pair additions).
__device__ __forceinline__ Df df_redux(Df v, int E) {
  const float S = pow2f(25 - E), R = pow2f(E - 25);
  const int i0 = __float2int_rn(__fmul_rn(v.h, S));
  const float rem = __fadd_rn(fmaf(-(float)i0, R, v.h), v.l);
  const int i1 = __float2int_rn(__fmul_rn(__fmul_rn(rem, S), 67108864.f));
  const int s0 = __reduce_add_sync(FULL, i0), s1 = __reduce_add_sync(FULL, i1);
  const float h = (float)s0, l = fmaf((float)s1, 1.f / 67108864.f, (float)(s0 - (int)h));
  return df_quick(__fmul_rn(h, R), __fmul_rn(l, R));
}
// the exponent E with every lane's |x| below 2^E (bounded; NaN and infinity count as largest)
__device__ __forceinline__ int warp_exponent(float x) {
  const int e = (int)(__reduce_max_sync(FULL, __float_as_uint(x) & 0x7fffffffu) >> 23) - 126;
  return e < -100 ? -100 : e > 100 ? 100 : e;
}
__device__ __forceinline__ void df_warp_sum2(Df &v0, Df &v1) {
  const bool u = threadIdx.x & 16;
  Df a = df_add(u ? v1 : v0, df_shfl_xor(u ? v0 : v1, 16));
#pragma unroll
  for (int o = 8; o > 0; o >>= 1) a = df_add(a, df_shfl_xor(a, o));
  v0 = df_shfl(a, 0);
  v1 = df_shfl(a, 16);
}

// Packed pairs (two columns of the lane's row).
__device__ __forceinline__ float2 dup2(float a) { return make_float2(a, a); }
// a b rounded by itself: a product that an addition follows must not become one
// FMA with it (the packed multiply may), or the two-sums below lose its rounding
__device__ __forceinline__ float2 prod2(float2 a, float2 b) {
  return __ffma2_rn(a, b, make_float2(-0.f, -0.f));
}
// a - b (no separate negation of a pair)
__device__ __forceinline__ float2 sub2(float2 a, float2 b) {
  return __ffma2_rn(b, make_float2(-1.f, -1.f), a);
}
__device__ __forceinline__ float2 neg2(float2 a) {
  return __ffma2_rn(a, make_float2(-1.f, -1.f), make_float2(-0.f, -0.f));
}
// (s, e): s = a + b rounded, e the rounding error (Knuth)
__device__ __forceinline__ void two_sum2(float2 a, float2 b, float2 &s, float2 &e) {
  s = __fadd2_rn(a, b);
  const float2 bb = sub2(s, a);
  e = __fadd2_rn(sub2(a, sub2(s, bb)), sub2(b, bb));
}

// the same of a - b
__device__ __forceinline__ void two_diff2(float2 a, float2 b, float2 &s, float2 &e) {
  s = sub2(a, b);
  const float2 bb = sub2(s, a);
  e = sub2(sub2(a, sub2(s, bb)), __fadd2_rn(b, bb));
}
// (S, F) += a b, pairs of products (ah + al) (bh + bl), na = -ah: S by two-sums, what is
// lost of it in F
__device__ __forceinline__ void df_fma2(float2 &S, float2 &F, float2 ah, float2 na, float2 al,
                                        float2 bh, float2 bl) {
  const float2 p = prod2(ah, bh), d = __ffma2_rn(na, bh, p);
  float2 e;
  two_sum2(S, p, S, e);
  F = __ffma2_rn(ah, bl, __ffma2_rn(al, bh, F));
  F = __fadd2_rn(F, sub2(e, d));
}

}  // namespace
