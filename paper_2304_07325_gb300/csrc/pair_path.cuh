// The single-pair path of the group recursion (included by k_recur.cu): once F_{k-1} = {q} holds
// one pair, every sub-step of levels >= k touches only the pair's two bodies.  Close and bound
// pairs take 10^4 to 10^6 such sub-steps one after another, and the longest of these chains sets
// the step time, so what counts is the latency of one sub-step in one warp.
//
// Arithmetic.  FP64 costs 64 cycles per warp instruction here, and a result that passes through
// any other unit 46 more; FP32 costs 4.  So a body's position and velocity are kept as an FP64
// anchor that stands still plus a double-float offset (df32.cuh),
//     x = X0 + dl,   v = V0 + nu,
// and the sub-steps only ever form increments, in double-float: each increment is a small
// fraction of what it is added to (in the order-2 regime below 2^-20 of x and, for the sun's
// pull, of v; a pair's kick is below 2^-11 of v), and the offset is a small fraction of its anchor,
// so 2^-46 of an increment and 2^-48 of an offset lie below the FP64 rounding of x and v, which the
// FP64 form committed at every update.  The anchors absorb the offsets (exactly but for one FP64
// rounding) every ANCHOR_N sub-steps, and earlier when the elapsed time makes |dl| grow past a
// set fraction of |x|.  The separation is d = (X0_b - X0_a) + (dl_b - dl_a): the difference of the
// anchors is exact, so unlike a difference of rounded positions d keeps its digits as the pair
// closes in.
//
// Layout.  Even lanes hold body a, odd lanes body b, all three components in the lane (the other
// lanes repeat them): sums over components and the scalar chains need no exchange, three
// components give the FP32 pipe three independent chains, and one shuffle round per sub-step hands
// the displacement over.  d points from this lane's body to the other,
// so both lanes run the same instructions, and every quantity of the pair is the same in both bit
// for bit (negating operands negates results).  Units are scaled by powers of two so that
// |x|, |v| ~ 1.
//
// Sub-steps.  pair_run() walks the level stack: one pass of its loop evaluates the force once (at new
// positions d, r, r^-3 and the shell function g; on a change of level at unchanged positions only
// what the level changes), and decides the sub-step.  A closing kick and the opening kick of the next
// sub-step of the same level are the same, so the opening applies both ("pend") and a closing kick
// stands alone only where a level ends.  Most sub-steps belong to a pair that stays between R_j and
// R_{j-1}: one FP32 test clears M of them at once, and run_order2() / run_series() take them with no
// decision inside, ending and starting the levels below by a weight of the kick.  Drifts:
//   order 2 (s < 5e-13, s = h^2 max(u, p^2, |q|), with u = mu/r^3, p = (x.v)/r^2, q = v^2/r^2 - u):
//     x' = x + h v - (u h^2/2) x,  v' = v - u h (1 - 3/2 p h) (x + h/2 v); 1/r^3 of the sun distance
//     is carried along by the factor (1 + w)^(-3/2), w = 2 p h + q h^2 the relative change of r^2
//     (|w| < 2e-6, formed in FP32 to 2^-43), and formed in full at every anchor;
//   s <= 1.3e-4: the Lagrange f and g series, to order 6 as in drift_series() and above s = 2e-6 to
//     order 10, 1/r^3, u, p and the leading coefficients in double-float;
//   longer intervals: the FP64 Kepler solver on the anchors.
//
// Cost and bound (one GB300 at 2.07 GHz).  A cleared order-2 sub-step is ~410 warp instructions, 95 %
// of them FP32, on a dependent path of ~500 cycles, and takes ~720; the component-packed FP64 form it
// replaces issued 22 FP64 and ~480 other instructions in 2,360.  Recursion time over the sub-steps of
// the longest chain, before and now: 10,000-body disk 1.12 -> 0.28 us (first step 113 -> 28 ms),
// 5,000 1.16 -> 0.30, 1,000 + 100,000 field 1.15 -> 0.30; chains of shallow levels, where a sub-step
// takes 0.6 us (order 6), 1.3 (order 10) or 6 to 12 (the Kepler solver), 4.4 -> 0.7 (1,000-body disk).
// Error against an 80-bit integration of 430 two- and many-body systems, one step: 0.054 of the FP64
// form's on the geometric mean (the separation is exact here, see above).
// The routine is inlined into its caller: as a function of its own the calling convention left
// the compiler too few registers to interleave the chains (0.40 against 0.26 us per sub-step).
#include "df32.cuh"

#define ANCHOR_N 128         // sub-steps between anchors

// per-level constants of a group in its scaled units (shared memory, one per warp)
struct GroupTab {
  float2 h[SYM_MAX_LEVELS + 2];    // sub-step h_j
  float2 rh[SYM_MAX_LEVELS + 2];   // 1 / h_j
  float2 mh[SYM_MAX_LEVELS + 2];   // mu h_j^2
  float2 A[SYM_MAX_LEVELS + 2];    // argument of g_j about the middle of its zone: y = A r/R_0 + B =
  float2 B[SYM_MAX_LEVELS + 2];    // 2 (r - R_{j+1}) / (R_j - R_{j+1}) - 1
  float2 c2[SYM_MAX_LEVELS + 2];   // (R_j / R_0)^2
};
// and those of one pair
struct PairTab {
  float2 ga[SYM_MAX_LEVELS + 2];   // G m_b h_j / 2, the kick's factor on body a
  float2 gb[SYM_MAX_LEVELS + 2];   // G m_a h_j / 2, on body b
  float2 ha[SYM_MAX_LEVELS + 2];   // h_j times the same
  float2 hb[SYM_MAX_LEVELS + 2];
  float2 R2[SYM_MAX_LEVELS + 2];   // R_j^2
  float2 A[SYM_MAX_LEVELS + 2];    // A of the group's table over R_0
  double X0[3][2], V0[3][2];       // the anchors of bodies a, b
};
__device__ __forceinline__ df ld(const float2 &v) { return mk(v.x, v.y); }

// f_3((1 + y)/2) - 1/2 = y (35/32 - z (35/32 - z (21/32 - 5/32 z))), z = y^2: the partition function
// of order 3 about the middle of its zone, where it is odd (its derivative is (35/32)(1 - y^2)^3), so
// that g and 1 - g are 1/2 plus and minus one value.  Coefficients are exact FP32 numbers and on
// [-1, 1] every difference takes the smaller from the larger.
__device__ __forceinline__ df partition3_odd(df y) {
  const df z = sqr(y);
  const df q = from(0.65625f, mul(z, 0.15625f));
  const df p = from(1.09375f, mul(z, q));
  return mul(y, from(1.09375f, mul(z, p)));
}

// What a run of sub-steps works on; x0, d0 and hv0 (h V0) stand still.  Velocities and kicks are times h.
struct Run {
  df x0[3], d0[3], hv0[3], Ap, Bp;
  df hn[3], dl[3], d[3], hk;       // h nu, dl, separation, the kick due at it is hk d
  df r3s;                          // 1/r^3 from the sun, and FP32 1/r^2
  df r2, r, r3, yp;                // of the separation; yp = g - 1/2 of zone j - 1
  float ri2s, ph, qh, uh;          // p h, q h^2, u h^2 of the last drift
};

// yp at r in the zone of A, B (fast_two_sum(B, r A): |B| >= r A, or r A <= 2 |B| and the sum is exact)
__device__ __forceinline__ df zone_odd(df r, df A, df B) {
  const df p = mul(r, A), y = fast_two_sum(B.h, p.h);
  return partition3_odd(mk(y.h, __fadd_rn(y.l, __fadd_rn(p.l, B.l))));
}
// The force at d and the kick due there: that of a whole sub-step, 2 (1 - g), or of one that also
// ends and starts level j - 1, 2 (1 - g) + 2 M g (cM = M, else 0).  gh: G m h^2 / 2.
#define RUN_KICK(cM)                                                                             \
  do {                                                                                           \
    r2 = norm2(d);                                                                               \
    const df_root q_ = root(r2);                                                                 \
    r = root_of(r2, q_);                                                                         \
    r3 = inverse_cube(q_);                                                                       \
    yp = zone_odd(r, Ap, Bp);                                                                    \
    hk = mul(from(1.0f + (cM), mul(yp, 2.0f - 2.0f * (cM))), mul(r3, gh));                       \
  } while (0)

// sub-steps cj .. end - 1 of a level by the order-2 drift
__device__ __forceinline__ void run_order2(Run &S, df gh, df mhh, int cj, int end, int M) {
  const float fM = (float)M;
  df x0[3], hv0[3], hn[3], dl[3], d[3];
#pragma unroll
  for (int c = 0; c < 3; ++c) { x0[c] = S.x0[c]; hv0[c] = S.hv0[c]; hn[c] = S.hn[c]; dl[c] = S.dl[c]; d[c] = S.d[c]; }
  const df Ap = S.Ap, Bp = S.Bp;
  df hk = S.hk, r3s = S.r3s, r2, r, r3, yp;
  float ri2s = S.ri2s, ph, qh, uh;
#pragma unroll 1
  for (int i = cj; i < end; ++i) {
    // x' = x + h v - (u h^2/2) x, h v' = h v - f'' h (x + h/2 v), f'' h = u h^2 (1 - 3/2 p h), both
    // from the v after the opening kick
    const df u = mul(mhh, r3s);
    float xf[3], vf[3], rv = 0.0f, vv = 0.0f;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      xf[c] = x0[c].h + dl[c].h;
      vf[c] = hv0[c].h + fmaf(hk.h, d[c].h, hn[c].h);
      rv = fmaf(xf[c], vf[c], rv);
      vv = fmaf(vf[c], vf[c], vv);
    }
    ph = rv * ri2s;
    qh = fmaf(vv, ri2s, -u.h);
    uh = u.h;
    const df fp = mk(-u.h, -__fmaf_rn(u.h, -1.5f * ph, u.l));
    const float uq = -0.5f * u.h;
    df hv[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const df m = add_u(hn[c], mul(hk, d[c]));
      hv[c] = add_u(hv0[c], m);
      hv[c].l = __fmaf_rn(uq, xf[c], hv[c].l);
      df a = mul(fp, x0[c]);
      a.l = __fmaf_rn(fp.h, dl[c].h, __fmaf_rn(uq, vf[c], a.l));
      hn[c] = add(m, a);
    }
    // 1/r^3 and 1/r^2 from the sun: the drift changes r^2 by the factor 1 + w
    const float w = fmaf(2.0f, ph, qh);
    r3s = fast_two_sum(r3s.h, __fmaf_rn(r3s.h, w * fmaf(1.875f, w, -1.5f), r3s.l));
    ri2s = fmaf(-ri2s, w, ri2s);
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const float oh = __shfl_xor_sync(FULL, hv[c].h, 1), ol = __shfl_xor_sync(FULL, hv[c].l, 1);
      dl[c] = add(dl[c], hv[c]);
      const df t = two_sum(oh, -hv[c].h), e = two_sum(d[c].h, t.h);
      d[c] = fast_two_sum(e.h, __fadd_rn(e.l, __fadd_rn(t.l, __fadd_rn(__fsub_rn(ol, hv[c].l), d[c].l))));
    }
    RUN_KICK(i + 1 == M ? fM : 0.0f);
  }

#pragma unroll
  for (int c = 0; c < 3; ++c) { S.hn[c] = hn[c]; S.dl[c] = dl[c]; S.d[c] = d[c]; }
  S.hk = hk; S.r3s = r3s; S.ri2s = ri2s; S.r2 = r2; S.r = r; S.r3 = r3; S.yp = yp;
  S.ph = ph; S.qh = qh; S.uh = uh;
}

// The Lagrange f and g series at position xx with velocity hv / h: increments dx of the position and
// dv / h of the velocity.  mhh: mu h^2.  Orders to 6 as in drift_series(), and to 10 for intervals with
// s > 2e-6 (far).
struct Series {
  df r3s;                          // 1/r^3 from the sun
  float ri2s, P, Q, U;             // 1/r^2, p h, q h^2, u h^2
};
// Without the orders above 6 such an interval was 4 to 16 equal drifts: a level of them 2.24 -> 1.32 us
// per sub-step, with the levels around it; 260 disks of 500 to 4,000 bodies 3 % faster (geometric mean).
// Orders 7 to 10 of both series over U = u h^2, from the recurrences of u' = -3 u p, p' = q - 2 p^2,
// w' = -2 p (u + w), w = v^2/r^2 = q + u, f'' = -u f: sums of c_k, k c_k, g_k and k g_k.
// (Called, not inlined: its 40 temporaries would be taken from the sub-steps that do not need it.)
static __device__ __noinline__ float4 series_tail(float U, float P, float W) {
  float e[9], p[8], w[8], c[11], g[11];
  e[0] = 1.0f;
  p[0] = P;
  w[0] = W;
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    float a = 0.0f, b = 0.0f, m = 0.0f;
#pragma unroll
    for (int j = 0; j <= k; ++j) {
      a = fmaf(e[j], p[k - j], a);
      b = fmaf(p[j], p[k - j], b);
      m = fmaf(p[j], fmaf(U, e[k - j], w[k - j]), m);
    }
    const float i = 1.0f / (float)(k + 1);
    e[k + 1] = -3.0f * i * a;
    if (k < 7) {
      p[k + 1] = i * (fmaf(-U, e[k], w[k]) - 2.0f * b);
      w[k + 1] = -2.0f * i * m;
    }
  }
#pragma unroll
  for (int k = 0; k <= 8; ++k) {                               // c_2 .. c_10, g_3 .. g_10
    float a = 0.0f, b = 0.0f;
#pragma unroll
    for (int j = 0; j + 2 <= k; ++j) {
      a = fmaf(e[j], c[k - j], a);
      if (j + 3 <= k) b = fmaf(e[j], g[k - j], b);
    }
    const float i = -1.0f / (float)((k + 1) * (k + 2));
    c[k + 2] = i * fmaf(U, a, e[k]);
    if (k > 0) g[k + 2] = i * fmaf(U, b, e[k - 1]);
  }
  return make_float4((c[7] + c[8]) + (c[9] + c[10]),
                     fmaf(7.0f, c[7], 8.0f * c[8]) + fmaf(9.0f, c[9], 10.0f * c[10]),
                     (g[7] + g[8]) + (g[9] + g[10]),
                     fmaf(7.0f, g[7], 8.0f * g[8]) + fmaf(9.0f, g[9], 10.0f * g[10]));
}
__device__ __forceinline__ Series series_increments(const df (&xx)[3], const df (&hv)[3], df mhh, bool wide, bool far,
                                                    df (&dx)[3], df (&dv)[3]) {
  // Coefficients over u h^2: FP32 where what they multiply is below 1e-17 of x and 1e-16 of v: their error,
  // unlike a rounding of x or v, is the same from one sub-step to the next and adds up.  With
  // s > 1e-8 (wide) that leaves out c4 in f' and g - h, with s > 2e-6 c4 everywhere, c5 in f' and the
  // fifth order of g' too.
  Series o;
  const df sixth = mk(0.16666667f, -4.967054e-09f);
  const df_root q = root_fine(norm2(xx));
  const df ri2 = inverse(q);
  o.r3s = inverse_cube(q);
  o.ri2s = ri2.h;
  const df u = renorm(mul(mhh, o.r3s));                      // u h^2
  const df pd = renorm(mul(dot3(xx, hv), ri2));              // p h
  const float U = u.h, P = pd.h, P2 = P * P;
  float Q;                                                   // q h^2
  df qd, c4d;                                                // 4 c4
  if (wide) {
    qd = add(mul(norm2(hv), ri2), neg(u));
    Q = qd.h;
    c4d = mul(add(add(mul(qd, 3.0f), u), mul(sqr(pd), -15.0f)), sixth);
  } else {
    Q = fmaf(fmaf(hv[2].h, hv[2].h, fmaf(hv[1].h, hv[1].h, hv[0].h * hv[0].h)), ri2.h, -U);
    qd = mk(Q, 0.0f);
    c4d = mk((3.0f * Q - 15.0f * P2 + U) * (1.0f / 6.0f), 0.0f);
  }
  const float c5 = P * (7.0f * P2 - 3.0f * Q - U) * 0.125f;
  const float c6 = (P2 * (-945.0f * P2 + 630.0f * Q + 210.0f * U) - 45.0f * Q * Q - 24.0f * U * Q - U * U) *
                   (1.0f / 720.0f);
  const float d5 = (9.0f * Q - 45.0f * P2 + U) * (1.0f / 120.0f);
  const float d6 = P * (14.0f * P2 - 6.0f * Q - U) * (1.0f / 24.0f);
  // the brackets' terms from order 4 (5 in g) on
  df fr = mk(0.5f * c4d.h + 2.0f * (c5 + c6), 0.0f), fdr = mk(c4d.h, c4d.l + (5.0f * c5 + 6.0f * c6));
  df gr = mk(10.0f * d5 + 12.0f * d6, 0.0f);
  float gmr = 6.0f * (d5 + d6);
  if (far) {
    const float4 t = series_tail(U, P, Q + U);
    // 5 c5 = 5/8 P (7 P^2 - 3 Q - U), 10 d5 = 3/2 (4 c4) - U / 6
    const df c5d = mul(mul(pd, 0.625f), add(add(mul(sqr(pd), 7.0f), mul(qd, -3.0f)), neg(u)));
    fr = mk(0.5f * c4d.h, 0.5f * c4d.l + 2.0f * (c5 + c6 + t.x));
    fdr = add(c4d, c5d);
    fdr.l += 6.0f * c6 + t.y;
    gr = add(mk(1.5f * c4d.h, 1.5f * c4d.l), neg(mul(u, sixth)));
    gr.l += 12.0f * d6 + 2.0f * t.w;
    gmr += 6.0f * t.z;
  }
  // f - 1 = (u h^2/2) (-1 + p h + ...), h f' = u h^2 (-1 + 3/2 p h + ...), g' - 1 = (u h^2/2)
  // (-1 + 2 p h + ...), g - h = h (u h^2/6) (-1 + 3/2 p h + ...)
  auto bracket = [&](float k, df rest) {
    const df p = mul(pd, k), t = fast_two_sum(-1.0f, p.h), b = fast_two_sum(t.h, rest.h);
    return mk(b.h, __fadd_rn(__fadd_rn(b.l, t.l), __fadd_rn(p.l, rest.l)));
  };
  const df u2 = mk(0.5f * u.h, 0.5f * u.l);
  const df fm1 = mul(u2, bracket(1.0f, fr));
  const df fd = mul(u, bracket(1.5f, fdr));
  const df gdm = mul(u2, bracket(2.0f, gr));
  const float gf = U * fmaf(0.25f, P, -1.0f / 6.0f);
  df gm = mk(0.0f, 0.0f);
  if (wide) gm = mul(mul(u, sixth), bracket(1.5f, mk(gmr, 0.0f)));
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    dv[c] = add_u(mul(fd, xx[c]), mul(gdm, hv[c]));
    df hp = hv[c];
    if (wide) hp = add_u(hp, mul(gm, hv[c]));
    else hp.l = __fmaf_rn(gf, hv[c].h, hp.l);
    dx[c] = add_u(hp, mul(fm1, xx[c]));
  }
  o.P = P;
  o.Q = Q;
  o.U = U;
  return o;
}

// the same by the series
__device__ __forceinline__ void run_series(Run &S, df gh, df mhh, int cj, int end, int M, bool wide, bool far) {
  const float fM = (float)M;
  df x0[3], d0[3], hv0[3], hn[3], dl[3], d[3];
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    x0[c] = S.x0[c]; d0[c] = S.d0[c]; hv0[c] = S.hv0[c];
    hn[c] = S.hn[c]; dl[c] = S.dl[c]; d[c] = S.d[c];
  }
  const df Ap = S.Ap, Bp = S.Bp;
  df hk = S.hk, r3s, r2, r, r3, yp;
  float ri2s, ph, qh, uh;
#pragma unroll 1
  for (int i = cj; i < end; ++i) {
    df xx[3], m[3], hv[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      xx[c] = add(x0[c], dl[c]);
      m[c] = add_u(hn[c], mul(hk, d[c]));
      hv[c] = add(hv0[c], m[c]);
    }
    df dx[3], dv[3];
    const Series o = series_increments(xx, hv, mhh, wide, far, dx, dv);
    r3s = o.r3s;
    ri2s = o.ri2s;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      hn[c] = add(m[c], dv[c]);
      dl[c] = add(dl[c], dx[c]);
    }
    ph = o.P;
    qh = o.Q;
    uh = o.U;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const float oh = __shfl_xor_sync(FULL, dl[c].h, 1), ol = __shfl_xor_sync(FULL, dl[c].l, 1);
      const df t = two_sum(oh, -dl[c].h), e = two_sum(d0[c].h, t.h);
      d[c] = fast_two_sum(e.h, __fadd_rn(e.l, __fadd_rn(t.l, __fadd_rn(__fsub_rn(ol, dl[c].l), d0[c].l))));
    }
    RUN_KICK(i + 1 == M ? fM : 0.0f);
  }

#pragma unroll
  for (int c = 0; c < 3; ++c) { S.hn[c] = hn[c]; S.dl[c] = dl[c]; S.d[c] = d[c]; }
  S.hk = hk; S.r3s = r3s; S.ri2s = ri2s; S.r2 = r2; S.r = r; S.r3 = r3; S.yp = yp;
  S.ph = ph; S.qh = qh; S.uh = uh;
}

// The Kepler solver on a lane's anchors, called and not inlined: inlined, its registers are taken from
// the sub-steps that never reach it.
static __device__ __noinline__ int kepler_anchors(PairTab *T, int odd, double mu, double h) {
  double x[3], v[3];
#pragma unroll
  for (int c = 0; c < 3; ++c) { x[c] = T->X0[c][odd]; v[c] = T->V0[c][odd]; }
  const int st = kepler_drift(mu, h, x[0], x[1], x[2], v[0], v[1], v[2]);
  __syncwarp();
#pragma unroll
  for (int c = 0; c < 3; ++c) { T->X0[c][odd] = x[c]; T->V0[c][odd] = v[c]; }
  return st;
}

// Runs the sub-steps of levels >= k with F_{k-1} = {q}, from the opening of a sub-step at level
// k.  x, v: this lane's body (even lanes a, odd lanes b); G, ea, eb: the group's table and units.  Returns 0 when level k has finished (k is
// then k - 1), 1 when the pair may be in contact at the next check, or the scaled state does not
// fit (k is that check's level; the general path takes the sub-step), 2 when the sub-step budget
// ran out.
__device__ __forceinline__ int pair_run(const Dev &D, const GroupCtx &C, int lane, double *hs, int *cs,
                                        PairTab *T, const GroupTab *G, int ea, int eb, double (&x)[3],
                                        double (&v)[3], double gA, double gB,
                                        double pR0sq, double piR0, double pRcut, int &kio, int &plev_io,
                                        long long &substeps_io, int &deepest_io) {
  const int odd = lane & 1;
  const DiskDesc *dp = C.dp;
  const int M = C.M, max_depth = C.max_depth, k0 = kio;
  const long long max_sub = C.max_substeps;

  const int et = -2 * ea - eb;                          // scale of G m h
  // (a short visit is mostly this: entries of one pair only, and no level above k0 - 1)
  for (int L = k0 - 1 + lane; L < SYM_MAX_LEVELS + 2; L += 32) {
    const double h = dp->hk[L], hh = 0.5 * h, fa = gB * hh, fb = gA * hh;
    const df ta = split(scale2(fa, et)), tb = split(scale2(fb, et));
    const df tc = split(scale2(fa * h, et + eb - ea)), td = split(scale2(fb * h, et + eb - ea));
    const df tr = split(scale2(pR0sq * dp->ck2[L], -2 * ea)), tA = split(scale2(2.0 * piR0 * dp->invdc[L], ea));
    T->ga[L] = make_float2(ta.h, ta.l);
    T->gb[L] = make_float2(tb.h, tb.l);
    T->ha[L] = make_float2(tc.h, tc.l);
    T->hb[L] = make_float2(td.h, td.l);
    T->R2[L] = make_float2(tr.h, tr.l);
    T->A[L] = make_float2(tA.h, tA.l);
  }
  __syncwarp();
  {
    // the scaled quantities that must be normal FP32 numbers, with room for their products
    const float hm = fabsf(G->h[k0].x), mm = fabsf(G->mh[k0].x), rr = T->R2[k0].x;
    const bool fits = hm > 1e-18f && hm < 1e12f && mm > 1e-28f && mm < 1e12f && rr > 1e-24f && rr < 1e12f &&
                      fabsf(T->ga[k0].x) < 1e12f && fabsf(T->gb[k0].x) < 1e12f && abs(ea) < 400 && abs(eb) < 400;
    if (!fits) return 1;
  }
  const float cut = f32_trunc(scale2(pRcut, -2 * ea)) * 1.000001f;   // not below the contact prefilter
  const float rcut = cut > 0.0f ? cut * rsqrt_seed(cut) * 1.000001f : 0.0f;

#pragma unroll
  for (int c = 0; c < 3; ++c) { T->X0[c][odd] = scale2(x[c], -ea); T->V0[c][odd] = scale2(v[c], -eb); }
  __syncwarp();
  df x0[3], v0[3], d0[3], dl[3], nu[3], hv0[3];
  float dv0[3], vsum = 0.0f;
  df r3s = mk(0.0f, 0.0f);                 // 1/r^3 of this lane's body from the sun
  float ri2s = 0.0f;                       // 1/r^2, FP32
  float t_el = 0.0f, t_lim = 0.0f;         // time since the anchor, and its limit
  int n_el = 0;                            // sub-steps since the anchor
  bool fresh = false;                      // r3s belongs to the current position
  bool order2 = false;                     // the last drift was of order 2

  long long substeps = substeps_io;
  int deepest = max(deepest_io, kio), plev = plev_io;
  int j = k0, cj = cs[j];

  // constants of the current level
  df h, mh, gg, R2j, R2n, R2p;
  df Ap, Bp;                               // of zone j - 1
  float hf, Rj, Rp, kmax;
  auto set_level = [&]() {
    h = ld(G->h[j]); mh = ld(G->mh[j]); gg = ld(odd ? T->gb[j] : T->ga[j]);
    R2p = ld(T->R2[j - 1]); R2j = ld(T->R2[j]); R2n = ld(T->R2[j + 1]);
    Ap = ld(T->A[j - 1]); Bp = ld(G->B[j - 1]);
    hf = h.h;
    Rj = R2j.h > 0.0f ? R2j.h * rsqrt_seed(R2j.h) * 1.000001f : 0.0f;   // not below R_j
    Rp = R2p.h > 0.0f ? R2p.h * rsqrt_seed(R2p.h) * 0.999999f : 0.0f;   // not above R_{j-1}
    // h times what one opening kick changes |dv| by at most, with the two of level j - 1 (r >= R_j)
    kmax = 2.0f * (float)(M + 1) * fabsf(hf) * (fabsf(T->ga[j].x) + fabsf(T->gb[j].x)) / R2j.h;
#pragma unroll
    for (int c = 0; c < 3; ++c) hv0[c] = renorm(mul(h, v0[c]));
  };
  auto sun = [&]() {                       // r3s, ri2s at the current position
    df xx[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) xx[c] = add(x0[c], dl[c]);
    const df_root q = root_fine(norm2(xx));
    r3s = inverse_cube(q);
    ri2s = q.t.h;
    fresh = true;
  };
  // anchor at X0, V0; offsets zero
  auto anchor = [&]() {
    float xs = 0.0f, vs = 0.0f, va = 0.0f;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      x0[c] = split(T->X0[c][odd]);
      v0[c] = split(T->V0[c][odd]);
      d0[c] = split(T->X0[c][odd ^ 1] - T->X0[c][odd]);
      dv0[c] = (__shfl_xor_sync(FULL, v0[c].h, 1) - v0[c].h) + (__shfl_xor_sync(FULL, v0[c].l, 1) - v0[c].l);
      dl[c] = nu[c] = mk(0.0f, 0.0f);
      xs = fmaf(x0[c].h, x0[c].h, xs);
      vs = fmaf(v0[c].h, v0[c].h, vs);
      va += fabsf(v0[c].h);
      hv0[c] = renorm(mul(h, v0[c]));
    }
    vsum = va + __shfl_xor_sync(FULL, va, 1);
    const float xa = xs * rsqrt_seed(xs);
    const float tl = 0.015625f * xa * rsqrt_seed(fmaxf(vs, 1e-30f));    // 2^-6 |x| / |v|
    t_lim = fminf(tl, __shfl_xor_sync(FULL, tl, 1));
    t_el = 0.0f;
    n_el = 0;
    sun();
  };
  auto absorb = [&]() {                    // the offsets into the anchors
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const double xa = (T->X0[c][odd] + f32_to_f64(dl[c].l)) + f32_to_f64(dl[c].h);
      const double va = (T->V0[c][odd] + f32_to_f64(nu[c].l)) + f32_to_f64(nu[c].h);
      __syncwarp();
      T->X0[c][odd] = xa;
      T->V0[c][odd] = va;
    }
    __syncwarp();
  };

  // the pair at the current positions: separation, r, r^-3, and yp = g - 1/2 of zone zc (the
  // transition zone [R_{zc+1}, R_zc) r lies in)
  df r = mk(0.0f, 0.0f), r2 = mk(0.0f, 0.0f), r3 = mk(0.0f, 0.0f), yp = mk(0.0f, 0.0f);
  df d[3];
  int zc = -1;
  auto separate = [&]() {
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const float oh = __shfl_xor_sync(FULL, dl[c].h, 1), ol = __shfl_xor_sync(FULL, dl[c].l, 1);
      const df t = two_sum(oh, -dl[c].h), u = two_sum(d0[c].h, t.h);
      d[c] = fast_two_sum(u.h, __fadd_rn(u.l, __fadd_rn(t.l, __fadd_rn(__fsub_rn(ol, dl[c].l), d0[c].l))));
    }
  };
  auto geometry = [&]() {
    separate();
    r2 = norm2(d);
    const df_root q = root(r2);
    r = root_of(r2, q);
    r3 = inverse_cube(q);
  };
  auto absorb_if_due = [&]() {
    if (n_el >= ANCHOR_N || t_el > (order2 ? 0.03125f * t_lim : t_lim)) {
      absorb();
      anchor();
    }
  };

  set_level();      // hv0 follows with the anchor
  anchor();
#pragma unroll
  for (int c = 0; c < 3; ++c) d[c] = mk(0.0f, 0.0f);

  bool moved = true, closing = false, pend = false;
  int rc = 0;
  df hc = mk(0.0f, 0.0f);                          // the kick due at this position is hc d
  float k1 = 0.0f;                                 // less k1 d: the velocity the check sees
  for (;;) {
    // ---- the force at level j
    if (moved) {
      geometry();
      zc = -1;
      moved = false;
    }
    bool fl = less(r2, R2j);
    {
      {
        const bool zero = r2.h < R2n.h || !(r2.h < R2p.h);     // w_j = 0 outside [R_{j+1}, R_{j-1})
        const int z = fl ? j : j - 1;
        if (zc != z && !zero) {
          yp = zone_odd(r, ld(T->A[z]), ld(G->B[z]));
          zc = z;
        }
        // w_j = g_j inside R_j, 1 - g_{j-1} outside
        const df w = from(0.5f, mk(fl ? -yp.h : yp.h, fl ? -yp.l : yp.l));
        hc = mul(w, mul(r3, gg));
        hc.h = zero ? 0.0f : hc.h;
        hc.l = zero ? 0.0f : hc.l;
      }
      // ---- end of a sub-step at level j: the closing kick is hc d
      if (closing) {
        if (++cj >= M) {
#pragma unroll
          for (int c = 0; c < 3; ++c) nu[c] = add(nu[c], mul(hc, d[c]));
          --j;
          if (j < k0) break;
          cj = cs[j];
          set_level();
          continue;
        }
        closing = false;
        pend = true;
      }
      // ---- opening of the next sub-step at level j
      if (r2.h < cut || substeps >= max_sub) {
        if (pend) {
#pragma unroll
          for (int c = 0; c < 3; ++c) nu[c] = add(nu[c], mul(hc, d[c]));
        }
        if (r2.h < cut) rc = 1;
        else { ++substeps; rc = 2; }
        break;
      }
      absorb_if_due();
      ++substeps;
      k1 = hc.h;
      if (pend) hc = mk(2.0f * hc.h, 2.0f * hc.l);
    }
    float hdv = 0.0f, ph = 0.0f, uh = 0.0f, qh = 0.0f, so = 1.0f;
    bool far = false;
    if (!fl) {
      // conservative FP32 test that the pair stays outside R_j: |d| - |dv| h > R_j, with relative
      // margins of 2^-15 and 2^-22 of the velocities, far above the FP32 rounding
      float s2 = 0.0f, sa = vsum, rv = 0.0f, vv = 0.0f;
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        const float nh = __fmaf_rn(hc.h, d[c].h, nu[c].h);
        const float uf = __fmaf_rn(-k1, d[c].h, nh);
        const float uo = __shfl_xor_sync(FULL, uf, 1);
        const float du = dv0[c] + (uo - uf);
        s2 = fmaf(du, du, s2);
        sa += fabsf(uo) + fabsf(uf);
        const float vf = v0[c].h + nh;
        rv = fmaf(x0[c].h + dl[c].h, vf, rv);
        vv = fmaf(vf, vf, vv);
      }
      const float mg = 1.0f + 3.0517578e-5f;
      const float dvm = s2 * rsqrt_seed(fmaxf(s2, 1e-30f)) * mg + sa * 2.3841858e-7f;
      hdv = dvm * fabsf(hf) * mg;
      far = r.h * (1.0f - 3.0517578e-5f) > (Rj + dvm * hf * mg) * mg;
      // s = h^2 max(u, p^2, |q|) in FP32 (r3s may lag behind by the drifts since the anchor: a few
      // per cent of s at most)
      uh = mh.h * r3s.h;
      ph = rv * ri2s * hf;
      qh = fmaf(vv * ri2s * hf, hf, -uh);
      so = fmaxf(fmaxf(fabsf(uh), ph * ph), fabsf(qh));
      so = fmaxf(so, __shfl_xor_sync(FULL, so, 1));        // of both bodies
      order2 = so < 5e-13f;
      if (__builtin_expect(!far, 0)) {
        // minimum distance of the straight-line relative motion over [0, h] below R_j (division-free)
        double e[3], u[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          e[c] = f32_to_f64(d[c].h) + f32_to_f64(d[c].l);
          double vc = (T->V0[c][odd] + f32_to_f64(nu[c].l)) + f32_to_f64(nu[c].h);
          if (pend) vc = fma(0.5 * (f32_to_f64(hc.h) + f32_to_f64(hc.l)), e[c], vc);
          u[c] = __shfl_xor_sync(FULL, vc, 1) - vc;
        }
        const double e2 = fma(e[2], e[2], fma(e[1], e[1], e[0] * e[0]));
        const double er = fma(e[2], u[2], fma(e[1], u[1], e[0] * u[0]));
        const double u2 = fma(u[2], u[2], fma(u[1], u[1], u[0] * u[0]));
        const double hd = scale2(dp->hk[j], eb - ea), Rd = scale2(pR0sq * dp->ck2[j], -2 * ea);
        if (e2 < Rd) fl = true;
        else if (er < 0.0) {
          if (-er < hd * u2) fl = fma(e2, u2, -er * er) < Rd * u2;
          else fl = fma(hd, fma(hd, u2, 2.0 * er), e2) < Rd;
        }
        fl = __any_sync(FULL, fl) != 0;
      }
    }
    pend = false;
    if (__builtin_expect(fl, 0)) {                 // the pair is in F_j
      plev = j;
      if (j + 1 <= max_depth) {
#pragma unroll
        for (int c = 0; c < 3; ++c) nu[c] = add(nu[c], mul(hc, d[c]));
        cs[j] = cj;
        ++j;
        deepest = max(deepest, j);
        hs[j] = dp->hk[j];
        cj = 0;
        set_level();
        continue;
      }
      if (lane == 0) set_status(&D.stat[C.d], SYMBA_E_DEPTH);
      so = 1.0f;
    } else {
      plev = j - 1;
    }
    if (__builtin_expect(so <= 1.28e-4f, 1)) {
      // ---- A run of sub-steps of level j by the series.  When the pair is between R_j and R_{j-1} it is
      // in F_{j-1} and not in F_j, and every level below j - 1 has weight zero there.  So when the M
      // sub-steps of level j are over, level j - 1 (and any that end with it) ends and starts again, and
      // the kicks at that position add up to two of level j, weight 1 - g, and two of level j - 1, M times
      // longer, weight g.  One test clears the next M sub-steps at once: in them |d| cannot change by more
      // than M times h |dv| and what the kicks and the sun's tide can add to it; the sub-steps themselves
      // then have no decision left.  Without that clearance the run is this one sub-step.
      // Velocities and kicks in a run are times h.
      const float fM = (float)M;
      auto clear = [&](float speed, float u) {             // speed: h |dv| here; u: u h^2
        const float need = fM * (speed + fM * (kmax + 4.0f * fabsf(u) * Rp)) * 1.0001f;
        return r.h * 0.9999f > fmaxf(Rj, rcut) + need && r.h * 1.0001f + need < Rp;
      };
      // A run's kick takes G m h^2 / 2 as one number: below 2^-100 its low part is lost (pairs closer than about
      // 2^-27 of their distance from the sun), and the sub-steps are taken one by one, kick and h apart.
      const df gh = ld(odd ? T->hb[j] : T->ha[j]);
      const bool whole = fabsf(gh.h) > 7.8886091e-31f || gg.h == 0.0f;
      const bool run = far && substeps + M < max_sub && __all_sync(FULL, whole && clear(hdv, uh));
      int end = run ? M : cj + 1;
      substeps += end - 1 - cj;                            // (this one is counted)
      if (order2 && !fresh) sun();
      const bool wide = so >= 1e-8f, beyond = so > 2.0e-6f;
      Run S;
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        S.x0[c] = x0[c]; S.d0[c] = d0[c]; S.hv0[c] = hv0[c];
        S.hn[c] = renorm(mul(h, nu[c])); S.dl[c] = dl[c]; S.d[c] = d[c];
      }
      S.hk = mul(hc, h);
      S.Ap = Ap; S.Bp = Bp; S.r3s = r3s; S.ri2s = ri2s;
      for (;;) {
        if (order2) run_order2(S, gh, mh, cj, end, M);
        else run_series(S, gh, mh, cj, end, M, wide, beyond);
        t_el = fmaf((float)(end - cj), fabsf(hf), t_el);
        n_el += end - cj;
        cj = end - 1;
        if (!run) break;
        int up = 1;                                        // levels that end and start again here
        while (j - up >= k0 && cs[j - up] + 1 >= M) ++up;
        if (j - up < k0 || n_el > ANCHOR_N || t_el > (order2 ? 0.03125f * t_lim : t_lim) || substeps + M + up >= max_sub)
          break;
        // h |dv| with the opening kick of level j (within kmax of what the test there sees)
        float s2 = 0.0f, sa = vsum * fabsf(hf);
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          const float uf = fmaf(S.hk.h, S.d[c].h, S.hn[c].h), uo = __shfl_xor_sync(FULL, uf, 1);
          const float du = fmaf(hf, dv0[c], uo - uf);
          s2 = fmaf(du, du, s2);
          sa += fabsf(uo) + fabsf(uf);
        }
        r = S.r;
        const float so1 = fmaxf(fmaxf(fabsf(S.uh), S.ph * S.ph), fabsf(S.qh));
        const float hdv1 = s2 * rsqrt_seed(fmaxf(s2, 1e-36f)) * 1.0001f + sa * 2.3841858e-7f;
        if (!__all_sync(FULL, clear(hdv1, S.uh) && so1 < (order2 ? 5e-13f : (beyond ? 1.28e-4f : (wide ? 2.0e-6f : 1e-8f))))) break;
        const int t = cs[j - up] + 1;
        __syncwarp();
        for (int i = 1; i < up; ++i) cs[j - i] = 0;
        cs[j - up] = t;
        __syncwarp();
        cj = 0;
        substeps += up + M;                                // the levels below, and the M of level j
      }
      const df rh = ld(G->rh[j]);
#pragma unroll
      for (int c = 0; c < 3; ++c) { nu[c] = renorm(mul(rh, S.hn[c])); dl[c] = S.dl[c]; d[c] = S.d[c]; }
      r3s = S.r3s; ri2s = S.ri2s; r2 = S.r2; r = S.r; r3 = S.r3; yp = S.yp;
      fresh = order2;
      zc = run ? j - 1 : -1;
    } else {
      // longer intervals: the FP64 Kepler solver
#pragma unroll
      for (int c = 0; c < 3; ++c) nu[c] = add(nu[c], mul(hc, d[c]));
      absorb();
      const int st = kepler_anchors(T, odd, scale2(C.mu, -ea - 2 * eb), scale2(dp->hk[j], eb - ea));
      if (st != SYMBA_OK && lane < 2) set_status(&D.stat[C.d], st);
      __syncwarp();
      order2 = false;
      anchor();
      moved = true;
    }
    closing = true;
  }
  if (j >= k0) cs[j] = cj;
  absorb();
#pragma unroll
  for (int c = 0; c < 3; ++c) { x[c] = scale2(T->X0[c][odd], ea); v[c] = scale2(T->V0[c][odd], eb); }
  __syncwarp();
  kio = j;
  substeps_io = substeps;
  deepest_io = deepest;
  plev_io = plev;
  return rc;
}
