// Double-float arithmetic: a value is the unevaluated sum h + l of two FP32 numbers, about 48
// significant bits.  GB300 completes one FP64 warp instruction per 64 cycles per warp, an FP32
// one per 4, and the FP32 pipe issues every cycle: a double-float product is four dependent FP32
// instructions (16 cycles), a sum eleven, so a serial chain that can do with 46 bits per
// operation runs several times faster here than on the FP64 pipe.
//
// Building blocks: the error-free sum (Knuth, TAOCP vol. 2, Sec. 4.2.2, Theorem B) and its short
// form for ordered operands (Dekker 1971, Numer. Math. 18, 224), and the error-free product by a
// fused multiply-add.  Every operation is an explicitly rounded intrinsic, so the compiler can
// neither contract nor reassociate them.  Negating all operands negates every result exactly.
#pragma once

struct df {
  float h, l;
};

__device__ __forceinline__ df mk(float h, float l) { df r; r.h = h; r.l = l; return r; }
__device__ __forceinline__ df neg(df a) { return mk(-a.h, -a.l); }

// a + b exactly, as sum and error
__device__ __forceinline__ df two_sum(float a, float b) {
  const float s = __fadd_rn(a, b), bb = __fsub_rn(s, a);
  return mk(s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb)));
}
// the same for |a| >= |b| or a = 0
__device__ __forceinline__ df fast_two_sum(float a, float b) {
  const float s = __fadd_rn(a, b);
  return mk(s, __fsub_rn(b, __fsub_rn(s, a)));
}
__device__ __forceinline__ df add(df a, df b) {
  const df s = two_sum(a.h, b.h);
  return fast_two_sum(s.h, __fadd_rn(s.l, __fadd_rn(a.l, b.l)));
}
// sum, not renormalised (an addend of another sum)
__device__ __forceinline__ df add_u(df a, df b) {
  const df s = two_sum(a.h, b.h);
  return mk(s.h, __fadd_rn(s.l, __fadd_rn(a.l, b.l)));
}
// c - a for |c| >= |a|, not renormalised
__device__ __forceinline__ df from(float c, df a) {
  const df s = fast_two_sum(c, -a.h);
  return mk(s.h, __fsub_rn(s.l, a.l));
}
// product, not renormalised: |l| may reach a few units in the last place of h
__device__ __forceinline__ df mul(df a, df b) {
  const float p = __fmul_rn(a.h, b.h);
  float e = __fmaf_rn(a.h, b.h, -p);
  e = __fmaf_rn(a.h, b.l, e);
  return mk(p, __fmaf_rn(a.l, b.h, e));
}
__device__ __forceinline__ df mul(df a, float b) {
  const float p = __fmul_rn(a.h, b);
  return mk(p, __fmaf_rn(a.l, b, __fmaf_rn(a.h, b, -p)));
}
__device__ __forceinline__ df sqr(df a) {
  const float p = __fmul_rn(a.h, a.h);
  return mk(p, __fmaf_rn(__fadd_rn(a.h, a.h), a.l, __fmaf_rn(a.h, a.h, -p)));
}
__device__ __forceinline__ df renorm(df a) { return fast_two_sum(a.h, a.l); }
// a < b for renormalised operands
__device__ __forceinline__ bool less(df a, df b) { return a.h < b.h || (a.h == b.h && a.l < b.l); }

// a . b and a . a over three components
__device__ __forceinline__ df dot3(const df (&a)[3], const df (&b)[3]) {
  const df p = mul(a[0], b[0]), q = mul(a[1], b[1]), r = mul(a[2], b[2]);
  const df s = two_sum(p.h, q.h), t = two_sum(s.h, r.h);
  return fast_two_sum(t.h, __fadd_rn(__fadd_rn(s.l, t.l), __fadd_rn(__fadd_rn(p.l, q.l), r.l)));
}
__device__ __forceinline__ df norm2(const df (&a)[3]) {
  float p[3], c = 0.0f, e = 0.0f;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    p[k] = __fmul_rn(a[k].h, a[k].h);
    e = __fadd_rn(e, __fmaf_rn(a[k].h, a[k].h, -p[k]));
    c = __fmaf_rn(a[k].h, a[k].l, c);
  }
  const df s = two_sum(p[0], p[1]), t = two_sum(s.h, p[2]);
  return fast_two_sum(t.h, __fadd_rn(__fadd_rn(s.l, t.l), __fmaf_rn(2.0f, c, e)));
}

__device__ __forceinline__ float rsqrt_seed(float x) {
  float y;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// The powers of s^(-1/2) share one seed y (22 bits), its exact square t and the residual
// e = 1 - s y^2 (|e| < 2^-21, formed to 2^-46): s^(-1/2) = y (1 + e/2 + 3e^2/8 + ...).
struct df_root {
  float y, e;
  df t;
};
__device__ __forceinline__ df_root root_from(df s, float y) {
  df_root r;
  r.y = y;
  r.t.h = __fmul_rn(r.y, r.y);
  r.t.l = __fmaf_rn(r.y, r.y, -r.t.h);
  const float e = __fmaf_rn(-s.h, r.t.l, __fmaf_rn(-s.h, r.t.h, 1.0f));
  r.e = __fmaf_rn(-s.l, r.t.h, e);
  return r;
}
__device__ __forceinline__ df_root root(df s) { return root_from(s, rsqrt_seed(s.h)); }
// the same from a seed corrected once (24 bits): e and with it the error of every power is four times
// smaller, for factors that stay the same over many sub-steps
__device__ __forceinline__ df_root root_fine(df s) {
  const float y = rsqrt_seed(s.h);
  return root_from(s, __fmaf_rn(y, 0.5f * __fmaf_rn(-s.h, __fmul_rn(y, y), 1.0f), y));
}
// s^(1/2) = s y (1 + e/2 + 3e^2/8)
__device__ __forceinline__ df root_of(df s, const df_root &r) {
  const float p = __fmul_rn(s.h, r.y);
  const float q = __fmaf_rn(s.l, r.y, __fmaf_rn(s.h, r.y, -p));
  return fast_two_sum(p, __fmaf_rn(p, __fmul_rn(r.e, __fmaf_rn(r.e, 0.375f, 0.5f)), q));
}
// s^(-1) = y^2 (1 + e + e^2)
__device__ __forceinline__ df inverse(const df_root &r) {
  return fast_two_sum(r.t.h, __fmaf_rn(r.t.h, __fmaf_rn(r.e, r.e, r.e), r.t.l));
}
// s^(-3/2) = y^3 (1 + 3e/2 + 15e^2/8)
__device__ __forceinline__ df inverse_cube(const df_root &r) {
  const float p = __fmul_rn(r.y, r.t.h);
  const float q = __fmaf_rn(r.y, r.t.l, __fmaf_rn(r.y, r.t.h, -p));
  return fast_two_sum(p, __fmaf_rn(p, __fmul_rn(r.e, __fmaf_rn(r.e, 1.875f, 1.5f)), q));
}

// The double equal to a normal FP32 value, on the integer pipe; zeros and subnormals give zero.
__device__ __forceinline__ double f32_to_f64(float f) {
  const unsigned b = __float_as_uint(f);
  const unsigned e = (b >> 23) & 0xFFu;
  const unsigned hi = (b & 0x80000000u) | ((e + 896u) << 20) | ((b & 0x7FFFFFu) >> 3);
  return e == 0u ? 0.0 : __hiloint2double((int)hi, (int)(b << 29));
}
// A double as its leading 24 bits and the next 24 (truncated at 2^-47 of itself), on the integer
// pipe, for magnitudes in the normal FP32 range; the low part of values below 2^-103 is left out.
__device__ __forceinline__ df split(double a) {
  const unsigned hi = (unsigned)__double2hiint(a), lo = (unsigned)__double2loint(a);
  const unsigned mag = hi & 0x7FFFFFFFu, sgn = hi & 0x80000000u;
  if (mag < 0x38100000u || mag >= 0x47F00000u) return mk(mag < 0x38100000u ? 0.0f : __int_as_float(sgn | 0x7F800000u), 0.0f);
  df r;
  r.h = __uint_as_float((__funnelshift_l(lo, mag, 3) + 0x40000000u) | sgn);
  const int e = (int)(mag >> 20) - 896 - 23;           // biased FP32 exponent of 2^(E - 23)
  const float s = e > 0 ? __uint_as_float(((unsigned)e << 23) | sgn) : 0.0f;
  r.l = __fmul_rn(__fmul_rn(__uint2float_rn(lo & 0x1FFFFFFFu), 1.8626451e-9f), s);   // 2^-29
  return fast_two_sum(r.h, r.l);
}
// a 2^k on the exponent field; zero, and zero for results below the normal range
__device__ __forceinline__ double scale2(double a, int k) {
  const int hi = __double2hiint(a);
  const int e = ((hi >> 20) & 0x7FF);
  const int n = e + k;
  return e == 0 || n <= 0 ? 0.0 : __hiloint2double(hi + (k << 20), __double2loint(a));
}
// A sum of scaled accelerations as a double, scaled back by 2^k.
__device__ __forceinline__ double kick_value(df a, int k) {
  return scale2(__dadd_rn(f32_to_f64(a.h), f32_to_f64(a.l)), k);
}
