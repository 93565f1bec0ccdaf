// Kepler drift over any interval: the elliptic solution with one FP64 evaluation of the orbit equation.
//
// What costs time is FP64 instructions, 64 cycles of a warp each, however few of its lanes drift.  So
// the anomaly is found in FP32 first, and FP64 evaluates sin, 1 - cos and X - sin X once, takes the
// one correction left (below 1e-6) and turns the three by it through their Taylor series.  Roots and
// reciprocals start from FP32 seeds, and each of the final coefficients is written without a division
// of its own.  Against three or four evaluations (sincos and three divisions each): a sub-step of a
// pair on this solver 13.2 -> 6.1 us, the drift of 100 to 10,000 lone bodies 21 -> 12 us.  Error against
// quadruple precision over e < 0.99, n dt from 0.002 to 1,000: 0.85 to 1.0 of theirs.
#pragma once
#include "df32.cuh"
#include "internal.cuh"

// 1/a to about one last place: FP32 seed and y (1 + e + e^2), e = 1 - a y; outside FP32's range the
// plain division
__device__ __forceinline__ double recip_fp64(double a) {
  const float f = f32_trunc(a), m = fabsf(f);
  if (!(m > 1e-37f && m < 1e37f)) return 1.0 / a;
  float yf;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(yf) : "f"(f));
  const double y = f32_to_f64(yf);
  const double e = fma(-a, y, 1.0);
  return fma(y, fma(e, e, e), y);
}

// E with X = th + E, X - ec sin X + es (1 - cos X) = th, to about 2e-7 (1 + e)/(1 - e)
__device__ __forceinline__ float kepler_guess(float th, float ec, float es) {
  float E = 0.0f;
  for (int it = 0; it < 6; ++it) {
    const float X = th + E;
    const float s = __sinf(X), c = __cosf(X);
    const float F = fmaf(es, 1.0f - c, fmaf(-ec, s, E));
    const float Fp = fmaf(es, s, fmaf(-ec, c, 1.0f)), hpp = 0.5f * fmaf(ec, s, es * c);
    const float d1 = __fdividef(-F, Fp);
    const float d = __fdividef(-F, fmaf(d1, hpp, Fp));
    E += d;
    if (fabsf(d) <= 1e-3f) break;          // the next one would be below 1e-8
  }
  return E;
}

// S = sin X, O = 1 - cos X, D = X - sin X, no digits lost at small X.  To |X| = 1/2 the Taylor series,
// whose terms from X^11 (X^12) on are below 6e-10 (1e-11) of the sum and come in FP32; to |X| = 1 the
// same at X/2, doubled; beyond that sincos(X/2).
__device__ __forceinline__ void kepler_trig(double X, double &S, double &O, double &D) {
  const float Xf = f32_trunc(X);
  if (fabsf(Xf) < 1.0f) {
    const bool dbl = fabsf(Xf) >= 0.5f;
    const double Y = dbl ? 0.5 * X : X;
    const float Yf = dbl ? 0.5f * Xf : Xf;
    const double z = Y * Y;
    const float zf = Yf * Yf;
    // D/X^3 = 1/6 - z/120 + z^2/5040 - z^3/362880 + z^4 (1/11! - z/13! + z^2/15!)
    const float dt = fmaf(zf, fmaf(zf, 7.6471637e-13f, -1.6059044e-10f), 2.5052108e-8f);
    double p = fma(z, f32_to_f64(dt), -1.0 / 362880.0);
    p = fma(p, z, 1.0 / 5040.0);
    p = fma(p, z, -1.0 / 120.0);
    p = fma(p, z, 1.0 / 6.0);
    // O/X^2 = 1/2 - z/24 + z^2/720 - z^3/40320 + z^4/3628800 - z^5 (1/12! - z/14! + z^2/16!)
    const float ot = -fmaf(zf, fmaf(zf, 4.7794773e-14f, -1.1470746e-11f), 2.0876757e-9f);
    double q = fma(z, f32_to_f64(ot), 1.0 / 3628800.0);
    q = fma(q, z, -1.0 / 40320.0);
    q = fma(q, z, 1.0 / 720.0);
    q = fma(q, z, -1.0 / 24.0);
    q = fma(q, z, 0.5);
    D = (Y * z) * p;
    O = z * q;
    S = Y - D;
    if (dbl) {
      const double so = S * O;
      D = 2.0 * (D + so);
      O = 2.0 * (S * S);
      S = 2.0 * (S - so);
    }
    return;
  }
  double s, c;
  sincos(0.5 * X, &s, &c);
  O = 2.0 * (s * s);
  S = 2.0 * (s * c);
  D = X - S;
}

// f - 1, g, f', g' - 1 of an ellipse (alpha = 2 mu / r0 - v^2 > 0) over dt; ir0 = 1/r0, u = x.v.
// X is the eccentric-anomaly difference: X - ec sin X + es (1 - cos X) = n dt with
// ec = 1 - r0/a, es = u / sqrt(mu a).
__device__ __forceinline__ int kepler_ellipse(double mu, double dt, double r0, double ir0, double u, double alpha,
                                              double &fm1, double &g, double &fdot, double &gdm1) {
  const double imu = recip_fp64(mu), isa = rsqrt_fp64(alpha);
  double sa = alpha * isa;                                   // sqrt(alpha), and 1/a = alpha/mu: the mean
  sa = fma(fma(-sa, sa, alpha), 0.5 * isa, sa);              // motion hangs on both, so each gets its
  double ia = alpha * imu;                                   // last digit back
  ia = fma(fma(-ia, mu, alpha), imu, ia);
  const double nn = ia * sa, ndt = nn * dt;
  const double ec = fma(-r0, ia, 1.0), es = u * (sa * imu);
  double th = ndt;
  if (fabsf(f32_trunc(th)) > 3.0f) th -= 6.283185307179586 * rint(th * 0.15915494309189535);
  double X = ndt + f32_to_f64(kepler_guess(f32_trunc(th), f32_trunc(ec), f32_trunc(es)));
  double S, O, D, d = 0.0;
  bool ok = false;
  for (int it = 0; it < 12; ++it) {
    kepler_trig(X, S, O, D);
    const double C = 1.0 - O;
    const double F = fma(es, O, fma(-ec, S, X - ndt));
    const double Fp = fma(es, S, fma(-ec, C, 1.0)), iFp = recip_fp64(Fp);
    // Newton and the second-order term; the third, d^3 (1 + |F''|)^2 / Fp^2, is below 1e-18 at the bound
    d = -F * iFp;
    const float df_ = f32_trunc(d), hpp = 0.5f * fmaf(f32_trunc(ec), f32_trunc(S), f32_trunc(es) * f32_trunc(C));
    d = fma(d, f32_to_f64(-df_ * hpp * f32_trunc(iFp)), d);
    if (fabsf(df_) <= 1e-6f * fminf(1.0f, f32_trunc(Fp))) { ok = true; break; }
    X += d;
  }
  if (!ok) {
    double lo = ndt - 2.5, hi = ndt + 2.5;                   // |X - ndt| <= ec + 2 es
    X = ndt;
    d = 0.0;
    for (int it = 0; it < 200; ++it) {
      kepler_trig(X, S, O, D);
      const double F = fma(es, O, fma(-ec, S, X - ndt)), Fp = fma(es, S, fma(-ec, 1.0 - O, 1.0));
      if (F > 0.0) hi = X; else lo = X;
      const double dX = -F / Fp;
      double Xn = X + dX;
      if (fabs(dX) <= 1e-15 * fmax(1.0, fabs(X))) { X = Xn; ok = true; break; }
      if (!(Xn > lo && Xn < hi)) Xn = 0.5 * (lo + hi);
      X = Xn;
    }
    if (!ok) return SYMBA_E_KEPLER;
    kepler_trig(X, S, O, D);
  }
  // X -> X + d
  const double C = 1.0 - O, h = 0.5 * d, d3 = d * (1.0 / 3.0);
  const double a1 = fma(d3, C, S), b1 = fma(-d3, S, C);
  const double o1 = fma(h, a1, O), s1 = fma(h, b1, S);       // d o1 = D(X + d) - D(X), d s1 = O(X + d) - O(X)
  D = fma(d, o1, D);
  S = fma(d, 1.0 - o1, S);
  O = fma(d, s1, O);
  const double q = fma(es, S, fma(-ec, 1.0 - O, 1.0));       // r / a
  const double iq = recip_fp64(q);
  fm1 = -O * (mu * (isa * isa)) * ir0;
  g = dt - D * (mu * (isa * isa) * isa);
  fdot = -(sa * ir0) * (iq * S);
  gdm1 = -O * iq;
  return SYMBA_OK;
}

// the same for every other orbit: universal variable s with Stumpff functions, bracketed Newton
__device__ inline void stumpff4(double z, double c[4]) {
  if (fabs(z) < 0.1) {
    for (int k = 0; k < 4; ++k) {
      double term = 1.0, s = 0.0;
      for (int i = 2; i <= k; ++i) term /= (double)i;
      for (int j = 0; j < 24; ++j) {
        s += term;
        term *= -z / ((double)(2 * j + k + 1) * (double)(2 * j + k + 2));
      }
      c[k] = s;
    }
    return;
  }
  if (z > 0.0) {
    const double sz = sqrt(z);
    double sn, cs;
    sincos(sz, &sn, &cs);
    c[0] = cs;
    c[1] = sn / sz;
  } else {
    const double sz = sqrt(-z);
    c[0] = cosh(sz);
    c[1] = sinh(sz) / sz;
  }
  c[2] = (1.0 - c[0]) / z;
  c[3] = (1.0 - c[1]) / z;
}
__device__ __noinline__ static int kepler_universal(double mu, double dt, double r0, double u, double alpha, double &fm1,
                                                    double &g, double &fdot, double &gdm1) {
  const double sgn = dt >= 0.0 ? 1.0 : -1.0;
  double c[4];
  double lo = 0.0, hi = fabs(dt) / r0;
  if (hi == 0.0) { fm1 = g = fdot = gdm1 = 0.0; return SYMBA_OK; }
  bool found = false;
  for (int it = 0; it < 200; ++it) {
    const double s = sgn * hi;
    stumpff4(alpha * s * s, c);
    const double F = r0 * s * c[1] + u * s * s * c[2] + mu * s * s * s * c[3] - dt;
    if (sgn * F >= 0.0) { found = true; break; }
    lo = hi;
    hi *= 2.0;
  }
  if (!found) return SYMBA_E_KEPLER;
  double sa = 0.5 * (lo + hi);
  bool ok = false;
  for (int it = 0; it < 400; ++it) {
    const double s = sgn * sa;
    stumpff4(alpha * s * s, c);
    const double G1 = s * c[1], G2 = s * s * c[2], G3 = s * s * s * c[3];
    const double F = r0 * G1 + u * G2 + mu * G3 - dt;
    const double Fp = r0 * c[0] + u * G1 + mu * G2;
    if (sgn * F > 0.0) hi = sa; else lo = sa;
    const double ds = -F / Fp;
    double sn = sa + sgn * ds;
    if (fabs(ds) <= 1e-15 * fmax(1e-300, fabs(sa))) { sa = sn; ok = true; break; }
    if (!(sn > lo && sn < hi)) sn = 0.5 * (lo + hi);
    sa = sn;
  }
  if (!ok) return SYMBA_E_KEPLER;
  const double s = sgn * sa;
  stumpff4(alpha * s * s, c);
  const double G1 = s * c[1], G2 = s * s * c[2], G3 = s * s * s * c[3];
  const double r = r0 * c[0] + u * G1 + mu * G2;
  fm1 = -mu * G2 / r0;
  g = dt - mu * G3;
  fdot = -mu * G1 / (r * r0);
  gdm1 = -mu * G2 / r;
  return SYMBA_OK;
}

// Kepler drift (f and g functions): advance (x, v) by dt on the orbit of parameter mu.
// Returns SYMBA_OK or SYMBA_E_KEPLER / SYMBA_E_NONFINITE (state untouched).
// The new state is x0 + ((f - 1) x0 + g v0), v0 + (f' x0 + (g' - 1) v0): f - 1 and g' - 1 are
// formed apart from the 1, which they would be rounded into when small.
__device__ inline int kepler_drift(double mu, double dt, double &x, double &y, double &z,
                                   double &vx, double &vy, double &vz) {
  const double r2 = fma(z, z, fma(y, y, x * x));
  const double v2 = fma(vz, vz, fma(vy, vy, vx * vx));
  const double u = fma(z, vz, fma(y, vy, x * vx));
  const unsigned ex = (unsigned)__double2hiint(r2) >> 20;
  double r0, ir0;
  if (ex - 897u <= 253u) {
    ir0 = rsqrt_fp64(r2);
    r0 = r2 * ir0;
    r0 = fma(fma(-r0, r0, r2), 0.5 * ir0, r0);
  } else {                                 // outside the range of the FP32 seeds
    r0 = sqrt(r2);
    ir0 = 1.0 / r0;
  }
  const double alpha = fma(2.0 * mu, ir0, -v2);
  if (!(r0 > 0.0) || !isfinite(alpha) || !isfinite(u)) return SYMBA_E_NONFINITE;
  double fm1, g, fdot, gdm1;
  const int st = alpha > 0.0 ? kepler_ellipse(mu, dt, r0, ir0, u, alpha, fm1, g, fdot, gdm1)
                             : kepler_universal(mu, dt, r0, u, alpha, fm1, g, fdot, gdm1);
  if (st != SYMBA_OK) return st;
  const double x0 = x, y0 = y, z0 = z, vx0 = vx, vy0 = vy, vz0 = vz;
  x = x0 + fma(fm1, x0, g * vx0);
  y = y0 + fma(fm1, y0, g * vy0);
  z = z0 + fma(fm1, z0, g * vz0);
  vx = vx0 + fma(gdm1, vx0, fdot * x0);
  vy = vy0 + fma(gdm1, vy0, fdot * y0);
  vz = vz0 + fma(gdm1, vz0, fdot * z0);
  return SYMBA_OK;
}
