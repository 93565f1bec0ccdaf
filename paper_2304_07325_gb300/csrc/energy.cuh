// Exact sums of doubles held in registers, and the pair terms of the energy on the integer pipe.
//
// The energy is the correctly rounded sum of its terms, and every term is fixed to the last bit
// (correctly rounded operations in a stated order).  For the O(N^2) pair terms two things cost time:
// the shared-memory atomics of the exact accumulator, whose 32 lanes mostly hit the same digits, and
// the FP64 instructions of a root and a quotient (about 20 of 29 per term, at 16 cycles of an SM per
// warp instruction).  So each thread sums into a 128-bit integer (the window), joined over the warp
// once at the end; and root and quotient are formed on integers: a double-float estimate good to 46
// bits, one correction from the exact residual, and the comparison with the rounding boundary that
// makes the result the nearest double.  Nine FP64 instructions a term are left, 0.78 ms of issue for
// 10,000 bodies; the energy of those took 10.17 ms with the atomics, roots and quotients and takes
// 1.15 ms (1.04 to 1.10 of it the pair kernel).
#pragma once
#include "df32.cuh"
#include "internal.cuh"

// A signed 128-bit sum per lane in units of 2^base.  The base is one for the warp and set by its first
// terms, 2^-25 below the largest of them; terms from there to 2^25 above that largest fit.  Room for
// WIN_TERMS terms a lane: 2^(54 + WIN_SPAN) WIN_TERMS 32 < 2^127.
#define WIN_SPAN 50
#define WIN_TERMS (1 << 16)
#define WIN_NONE (-100000)
struct Window {
  unsigned long long lo;
  long long hi;
  int base;
};
__device__ __forceinline__ void win_clear(Window &w) { w.lo = 0ull; w.hi = 0ll; w.base = WIN_NONE; }
// every lane of the warp calls it; e: exponent of this lane's lowest bit, use: the lane has a term
__device__ __forceinline__ void win_base(Window &w, bool use, int e) {
  if (w.base != WIN_NONE) return;
  const int top = __reduce_max_sync(0xffffffffu, use ? e : WIN_NONE);
  if (top != WIN_NONE) w.base = max(top - WIN_SPAN / 2, -1074);
}
// += q 2^e (q < 2^54), or minus; false when it does not fit the window
__device__ __forceinline__ bool win_put(Window &w, unsigned long long q, int e, bool minus) {
  const int sh = e - w.base;
  if ((unsigned)sh > (unsigned)WIN_SPAN) return false;
  const unsigned long long lo = q << sh, hi = (q >> 1) >> (63 - sh);
  if (minus) {
    const unsigned long long t = w.lo - lo;
    w.hi -= (long long)hi + (t > w.lo ? 1ll : 0ll);
    w.lo = t;
  } else {
    const unsigned long long t = w.lo + lo;
    w.hi += (long long)hi + (t < lo ? 1ll : 0ll);
    w.lo = t;
  }
  return true;
}
// += x (0.0 from a lane without a term; every lane calls it): into the window, or straight into the
// digits where it does not fit
__device__ __forceinline__ void win_add(Window &w, unsigned long long *dig, double x) {
  const long long bits = __double_as_longlong(x);
  const int ex = (int)((bits >> 52) & 0x7FF);
  const bool use = ex != 0 && ex != 0x7FF;
  win_base(w, use, ex - 1075);
  const unsigned long long q = ((unsigned long long)bits & 0xFFFFFFFFFFFFFull) | (1ull << 52);
  if (!use || !win_put(w, q, ex - 1075, bits < 0)) sa_add(dig, x);
}
// the warp's sum into the digits, and an empty window (every lane calls it)
__device__ __forceinline__ void win_flush(Window &w, unsigned long long *dig) {
  if (w.base == WIN_NONE) return;
  unsigned long long lo = w.lo, hi = (unsigned long long)w.hi;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long l = __shfl_down_sync(0xffffffffu, lo, o), t = lo + l;
    hi += __shfl_down_sync(0xffffffffu, hi, o) + (t < l ? 1ull : 0ull);
    lo = t;
  }
  if ((threadIdx.x & 31) == 0) {
    const bool minus = (long long)hi < 0;
    if (minus) { lo = 0ull - lo; hi = ~hi + (lo == 0ull ? 1ull : 0ull); }
    const int p = w.base + 1088, k = p >> 5, s = p & 31;
    const unsigned long long a = lo << s, b = (hi << s) | (s ? lo >> (64 - s) : 0ull), c = s ? hi >> (64 - s) : 0ull;
    const unsigned long long part[5] = {a & 0xFFFFFFFFull, a >> 32, b & 0xFFFFFFFFull, b >> 32, c};
#pragma unroll
    for (int i = 0; i < 5; ++i)
      if (part[i]) atomicAdd(&dig[k + i], minus ? 0ull - part[i] : part[i]);
  }
  win_clear(w);
}

// The double nearest c / r with r the double nearest sqrt(s) (both roundings as IEEE 754 has them), as
// q 2^e; false (nothing done) where an operand or a result is not a normal number.
__device__ __forceinline__ bool quotient_by_root(double c, double s, unsigned long long &q, int &e) {
  const long long sb = __double_as_longlong(s), cb = __double_as_longlong(c);
  const int se = (int)(sb >> 52), ce = (int)(cb >> 52);            // sign bit included: positive only
  e = 0;
  if (se < 1 || se > 2046 || ce < 1 || ce > 2046) return false;
  const unsigned long long S = ((unsigned long long)sb & 0xFFFFFFFFFFFFFull) | (1ull << 52);
  const unsigned long long Cm = ((unsigned long long)cb & 0xFFFFFFFFFFFFFull) | (1ull << 52);
  // s = M 2^es, es even, M in [2^52, 2^54); R = sqrt(M 2^52) to the nearest, in [2^52, 2^53]
  const int odd = (se - 1075) & 1, es = se - 1075 - odd;
  const unsigned long long M = S << odd;
  df m;                                                            // M 2^-52 in [1, 4)
  m.h = __uint2float_rn((unsigned)(M >> 30)) * 2.3841858e-7f;      // 2^-22
  m.l = __uint2float_rn((unsigned)M & 0x3FFFFFFFu) * 2.2204460e-16f;   // 2^-52
  const df_root rt = root_fine(m);                                 // seed to half a last place
  const df r = root_of(m, rt);
  const float y = rt.y;
  const unsigned long long Rh = (unsigned long long)((__float_as_uint(r.h) & 0x7FFFFFu) | 0x800000u) << 29;
  // (r.h may round to 2 when s is close below 4: its exponent then stands for one more bit)
  long long R = (long long)(Rh << ((__float_as_uint(r.h) >> 23) - 127)) + __float2int_rn(r.l * 4.5035996e15f);   // 2^52
  long long D = (long long)((M << 52) - (unsigned long long)R * (unsigned long long)R);
  long long t = __float2int_rn((float)(int)(D >> 32) * (y * 4.7683716e-7f));      // 2^32 2^-53
  D -= t * (2 * R + t);
  R += t;
  if (D > R) R += 1;
  else if (D <= -R) R -= 1;
  // c / r: Q = Cm 2^k / R to the nearest, k = 52 or 53 so that Q >= 2^52
  const int k = Cm >= (unsigned long long)R ? 52 : 53;
  const float sc = k == 52 ? 1.0f : 2.0f;
  df a;                                                            // Cm 2^(k - 104) in [1, 2]
  a.h = __uint2float_rn((unsigned)(Cm >> 29)) * (1.1920929e-7f * sc);              // 2^-23
  a.l = __uint2float_rn((unsigned)Cm & 0x1FFFFFFFu) * (2.2204460e-16f * sc);
  const float qh = a.h * y;
  const float el = __fmaf_rn(-qh, r.h, a.h) + __fmaf_rn(-qh, r.l, a.l);
  const unsigned qb = __float_as_uint(qh);
  const int qe = (int)(qb >> 23) - 127;                            // -1, 0 or 1
  const unsigned long long Qm = (unsigned long long)((qb & 0x7FFFFFu) | 0x800000u) << 30;
  long long Q = (long long)(Qm >> (1 - qe)) + __float2int_rn(el * y * 4.5035996e15f);
  long long E = (long long)((Cm << k) - (unsigned long long)Q * (unsigned long long)R);
  t = __float2int_rn((float)(int)(E >> 32) * (y * 9.5367432e-7f));                 // 2^32 2^-52
  E -= t * R;
  Q += t;
  if (2 * E > R) Q += 1;
  else if (2 * E < -R) Q -= 1;
  q = (unsigned long long)Q;
  // value of the last place: 2^(ce - 1075) 2^-k 2^-(es / 2 - 26)
  e = (ce - 1075) - k - (es / 2 - 26);
  return e > -1074 && e < 970;
}

// -c / |d|, c = (G m_i) m_j, of a lane with a pair (every lane calls it)
static __device__ __noinline__ void pair_term_general(unsigned long long *dig, double c, double s) {
  sa_add(dig, -__ddiv_rn(c, __dsqrt_rn(s)));
}
__device__ __forceinline__ void energy_pair(Window &w, unsigned long long *dig, bool use, double c,
                                            double dx, double dy, double dz) {
  const double s = __dadd_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)), __dmul_rn(dz, dz));
  unsigned long long q;
  int e;
  const bool ok = quotient_by_root(c, s, q, e) && use;
  win_base(w, ok, e);
  // (a massless body's term is zero unless the two coincide)
  if (use && (!ok || !win_put(w, q, e, true)) && !(c == 0.0 && s > 0.0)) pair_term_general(dig, c, s);
}

// columns of a strip: whole tiles once every warp has at least two, quarters below that (a warp's terms
// are one after the other: 1,500 bodies on 4,864 warps have 1,100 tiles)
__device__ __forceinline__ int energy_cols(long long tiles, long long nwarps) { return tiles < 2 * nwarps ? 8 : 32; }

// terms of one body: (0.5 m) v^2, -(G m0) m / r, and m (x_c1 v_c2 - x_c2 v_c1)
__device__ __forceinline__ void body_terms(double m, double x, double y, double z, double vx, double vy,
                                           double vz, double Gm0, double t[5]) {
  const double v2 = __dadd_rn(__dadd_rn(__dmul_rn(vx, vx), __dmul_rn(vy, vy)), __dmul_rn(vz, vz));
  t[0] = __dmul_rn(__dmul_rn(0.5, m), v2);
  const double r = __dsqrt_rn(__dadd_rn(__dadd_rn(__dmul_rn(x, x), __dmul_rn(y, y)), __dmul_rn(z, z)));
  t[1] = -__ddiv_rn(__dmul_rn(Gm0, m), r);
  t[2] = __dmul_rn(m, __dsub_rn(__dmul_rn(y, vz), __dmul_rn(z, vy)));
  t[3] = __dmul_rn(m, __dsub_rn(__dmul_rn(z, vx), __dmul_rn(x, vz)));
  t[4] = __dmul_rn(m, __dsub_rn(__dmul_rn(x, vy), __dmul_rn(y, vx)));
}
