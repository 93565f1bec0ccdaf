// Levels >= k0 of a group's recursion while F_{k0-1} holds at most 32 pairs of at most 32 bodies
// (included by k_recur.cu): lane a holds body a, lane q holds pair q.  The whole of a small group runs
// here (k0 = 1), and a large group once it has come down to that size; F_{k-1} of one pair goes on to
// pair_path.cuh.
//
// A sub-step costs what its FP64 instructions cost, 64 cycles of the warp each however many lanes
// hold a body.  So it uses the arithmetic of the pair path: positions and velocities are FP64 anchors,
// X0 and V0, plus double-float offsets, dl and nu; separations are exact differences of the anchors
// plus differences of the offsets; forces, kicks and series drifts are formed in double-float, and
// FP64 is left to anchoring, to the rare check near a threshold, to mergers and to intervals too long
// for the series.  Pairs read their bodies, and bodies their pairs' forces, with warp shuffles; F_{k-1}
// and F_k are ballot masks and a body's pairs a bitmask, so no list is stored or partitioned.  Forces
// add up in pair-list order.
//
// Recursion of one step, before (FP64 in registers or in the view) and now: two binaries in one group
// (5,460 sub-steps with both, 16,384 with one) 70 -> 46 ms, three bodies in a hierarchy 12.5 -> 5.0,
// two binaries in a group of 42 bodies 117 -> 45; 260 disks of 500 to 4,000 bodies 4.3 times as fast
// (geometric mean, with the single-pair path's share).

// The group's units, |x| ~ 2^ea and |v| ~ 2^eb, and whether its quantities are normal FP32 numbers in them,
// with room for their products, at every level down to max_depth (h_k falls by M per level, R_k by the shell
// ratio).  At the deepest:
//   R_{k+1}: the force of level k is used from there on, and r^-3, times G m, stays below 2^125;
//   G m h/2: not below 2^-100, from where on its low part would be lost;
//   h: not below 2^-70, so that h times what FP64 still adds to v (2^-53) is a normal number.
// (The sun's mu h^2 may leave the range: what it then moves v by is below 2^-63 per sub-step.)
struct GroupScale {
  int ea, eb;
  bool fits;
};
__device__ GroupScale group_scale(const GView &S, const GroupCtx &C, int lane) {
  auto hi = [](double t) { return (unsigned)__double2hiint(t) & 0x7FFFFFFFu; };
  auto top = [&](double t) { return (int)(hi(t) >> 20) - 1023; };
  unsigned mx = 0u, mv = 0u, mg = 0u, lg = 0x7FFFFFFFu;
  for (int a = lane; a < C.mcnt; a += 32) {
    mx = max(mx, max(hi(S.x[a]), max(hi(S.y[a]), hi(S.z[a]))));
    mv = max(mv, max(hi(S.vx[a]), max(hi(S.vy[a]), hi(S.vz[a]))));
    mg = max(mg, hi(S.gm[a]));
    if (hi(S.gm[a])) lg = min(lg, hi(S.gm[a]));
  }
  GroupScale g;
  g.ea = (int)(__reduce_max_sync(FULL, mx) >> 20) - 1023;
  g.eb = (int)(__reduce_max_sync(FULL, mv) >> 20) - 1023;
  // a state at rest takes the circular speed's scale
  if (g.eb < -900) g.eb = ((((__double2hiint(C.mu) >> 20) & 0x7FF) - 1023) - g.ea) / 2;
  bool ok = abs(g.ea) < 400 && abs(g.eb) < 400;
  const int et = -g.ea - 2 * g.eb, eg = (int)(__reduce_max_sync(FULL, mg) >> 20) - 1023 + et;
  const int el = (int)(__reduce_min_sync(FULL, lg) >> 20) - 1023 + et;        // (large where no body has mass)
  const int eh = top(C.dp->hk[C.max_depth]) + g.eb - g.ea;
  const float h = fabsf(f32_trunc(scale2(C.dp->hk[1], g.eb - g.ea))), mh = fabsf(f32_trunc(scale2(C.mu, et))) * h * h;
  ok = ok && h < 1e12f && mh > 1e-28f && mh < 1e12f && eg < 38 && eh >= -70 && el + eh - 1 >= -100;
  for (int q = lane; q < C.pcnt; q += 32) {
    const int er = top(S.R0[q] * C.dp->ck[C.max_depth + 1]) - g.ea;
    ok = ok && 3 * -er + max(eg, 0) <= 124 && f32_trunc(scale2(S.R0[q], -g.ea)) < 1e6f;
  }
  g.fits = __all_sync(FULL, ok) != 0;
  return g;
}

__device__ void group_table(GroupTab *G, const GroupCtx &C, const GroupScale &g, int lane) {
  const DiskDesc *dp = C.dp;
  for (int L = lane; L < SYM_MAX_LEVELS + 2; L += 32) {
    const int Ln = min(L + 1, SYM_MAX_LEVELS + 1);
    const double h = scale2(dp->hk[L], g.eb - g.ea), i2 = 2.0 * dp->invdc[L];
    const df th = split(h), ti = split(recip_fp64(h)), tm = split(scale2(C.mu, -g.ea - 2 * g.eb) * (h * h));
    const df ta = split(i2), tb = split(fma(-dp->ck[Ln], i2, -1.0)), tc = split(dp->ck2[L]);
    G->h[L] = make_float2(th.h, th.l);
    G->rh[L] = make_float2(ti.h, ti.l);
    G->mh[L] = make_float2(tm.h, tm.l);
    G->A[L] = make_float2(ta.h, ta.l);
    G->B[L] = make_float2(tb.h, tb.l);
    G->c2[L] = make_float2(tc.h, tc.l);
  }
  __syncwarp();
}

#define SH(v, src) __shfl_sync(FULL, (v), (src))
__device__ __forceinline__ df shf(df a, int src) { return mk(SH(a.h, src), SH(a.l, src)); }

__device__ __forceinline__ bool contact_regs(double xa, double ya, double za, double xb, double yb,
                                             double zb, double ra, double rb) {
  const double dx = __dsub_rn(xb, xa), dy = __dsub_rn(yb, ya), dz = __dsub_rn(zb, za);
  const double r2 = __dadd_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)), __dmul_rn(dz, dz));
  const double Rc = __dadd_rn(ra, rb);
  return r2 < __dmul_rn(Rc, Rc);
}

__device__ __forceinline__ bool predicate_regs(double dx, double dy, double dz, double r2, double dvx,
                                               double dvy, double dvz, double R2, double h) {
  if (lt_nn(r2, R2)) return true;
  const double vr = fma(dz, dvz, fma(dy, dvy, dx * dvx));
  if (!is_neg(vr)) return false;
  const double v2 = fma(dvz, dvz, fma(dvy, dvy, dvx * dvx));
  if (lt_nn(neg(vr), h * v2)) return lt_nn(fma(r2, v2, -vr * vr), R2 * v2);
  const double e = fma(h, fma(h, v2, 2.0 * vr), r2);
  return is_neg(e) || lt_nn(e, R2);
}

// one body's state in a member slot of the group's view
struct Body {
  double x[3], v[3], m, gm, rad, rh;
};
__device__ __forceinline__ void body_load(const GView &S, int a, Body &b) {
  b.x[0] = S.x[a]; b.x[1] = S.y[a]; b.x[2] = S.z[a];
  b.v[0] = S.vx[a]; b.v[1] = S.vy[a]; b.v[2] = S.vz[a];
  b.m = S.m[a]; b.gm = S.gm[a]; b.rad = S.rad[a]; b.rh = S.rh[a];
}
__device__ __forceinline__ void body_store(const GView &S, int a, const Body &b) {
  S.x[a] = b.x[0]; S.y[a] = b.x[1]; S.z[a] = b.x[2];
  S.vx[a] = b.v[0]; S.vy[a] = b.v[1]; S.vz[a] = b.v[2];
  S.m[a] = b.m; S.gm[a] = b.gm; S.rad[a] = b.rad; S.rh[a] = b.rh;
}

// the Kepler solver on a body in the view, called and not inlined (as kepler_anchors())
static __device__ __noinline__ int kepler_slot(const GView &S, int a, double mu, double h) {
  double x = S.x[a], y = S.y[a], z = S.z[a], vx = S.vx[a], vy = S.vy[a], vz = S.vz[a];
  const int st = kepler_drift(mu, h, x, y, z, vx, vy, vz);
  S.x[a] = x; S.y[a] = y; S.z[a] = z;
  S.vx[a] = vx; S.vy[a] = vy; S.vz[a] = vz;
  return st;
}

// Runs level k0 of the group to its end, from the opening of a sub-step there: bodies mperm[0..nm),
// pairs perm[0..np) of the view.  Returns false when the sub-step budget ran out; *merged_any: bodies
// merged (critical radii of pairs outside this call are then out of date).
__device__ __forceinline__ bool small_levels(const Dev &D, const GroupCtx &C, const GView &S, const GroupScale &gs,
                                             int lane, int nm, int np, double *hs, int *cs, PairTab *T, GroupTab *G,
                                             int k0, long long &substeps, int &deepest, bool *merged_any) {
  const DiskDesc *dp = C.dp;
  const int ea = gs.ea, eb = gs.eb;
  const bool ism = lane < nm, isp = lane < np;
  const int slot = ism ? S.mperm[lane] : 0, qs = isp ? S.perm[lane] : 0;
  if (ism) S.mtmp[slot] = lane;
  __syncwarp();
  const int ia = isp ? S.mtmp[S.pa[qs]] : 0, ib = isp ? S.mtmp[S.pb[qs]] : 0;
  int lev = isp ? S.lev[qs] : -1;
  Body b;
  auto clear_body = [&]() {
    b.m = b.gm = b.rad = b.rh = 0.0;
#pragma unroll
    for (int c = 0; c < 3; ++c) b.x[c] = b.v[c] = 0.0;
  };
  if (ism) body_load(S, slot, b);
  else clear_body();
  unsigned am = __ballot_sync(FULL, ism && S.alive[slot]);   // bodies alive
  unsigned im = 0u, jm = 0u;
  for (int q = 0; q < np; ++q) {
    if (SH(ia, q) == lane) im |= 1u << q;
    if (SH(ib, q) == lane) jm |= 1u << q;
  }
  const unsigned adjm = ism ? (im | jm) : 0u;

  // per-pair constants in the scaled units: R_0^2, 1/R_0, contact prefilter, G m of both bodies
  df R2, iR, gA, gB;
  float cut;
  auto pair_consts = [&]() {
    const double R0 = isp ? S.R0[qs] : 0.0;
    const double Rc = SH(b.rad, ia) + SH(b.rad, ib);
    const double ga = SH(b.gm, ia), gb = SH(b.gm, ib);
    R2 = split(scale2(R0 * R0, -2 * ea));
    iR = split(scale2(isp ? S.invR0[qs] : 0.0, ea));
    cut = f32_trunc(scale2(1.0000001 * (Rc * Rc), -2 * ea)) * 1.000001f;
    gA = split(scale2(ga, -ea - 2 * eb));
    gB = split(scale2(gb, -ea - 2 * eb));
  };
  pair_consts();

  df x0[3], v0[3], dl[3], nu[3];           // body: anchor and offsets
  df d0[3], d[3], r2, r, r3;               // pair: separation of the anchors, separation, r^2, r, r^-3
  float dv0[3], vsum = 0.0f;               // pair: velocity difference and sum of the anchors' |v|
  df acc[3];                               // body: sum of its pairs' accelerations
  float t_el = 0.0f, t_lim = 0.0f;         // time since the anchor, and its limit
  int n_el = 0;                            // drifts since the anchor
  bool anchored = false, placed = false;   // anchors, separations belong to the state

  auto clear = [&]() {
    const df z = mk(0.0f, 0.0f);
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      x0[c] = v0[c] = dl[c] = nu[c] = d0[c] = d[c] = acc[c] = z;
      dv0[c] = 0.0f;
    }
    r2 = r = r3 = z;
    vsum = t_el = t_lim = 0.0f;
    n_el = 0;
  };
  clear();
  auto absorb = [&]() {                    // the offsets into the FP64 state
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      b.x[c] = (b.x[c] + scale2(f32_to_f64(dl[c].l), ea)) + scale2(f32_to_f64(dl[c].h), ea);
      b.v[c] = (b.v[c] + scale2(f32_to_f64(nu[c].l), eb)) + scale2(f32_to_f64(nu[c].h), eb);
      dl[c] = nu[c] = mk(0.0f, 0.0f);
    }
    anchored = placed = false;
  };
  auto anchor = [&]() {
    float xs = 0.0f, vs = 0.0f, va = 0.0f;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      x0[c] = split(scale2(b.x[c], -ea));
      v0[c] = split(scale2(b.v[c], -eb));
      d0[c] = split(scale2(SH(b.x[c], ib) - SH(b.x[c], ia), -ea));
      const df fa = shf(v0[c], ia), fb = shf(v0[c], ib);
      dv0[c] = (fb.h - fa.h) + (fb.l - fa.l);
      xs = fmaf(x0[c].h, x0[c].h, xs);
      vs = fmaf(v0[c].h, v0[c].h, vs);
      va += fabsf(v0[c].h);
    }
    vsum = SH(va, ia) + SH(va, ib);
    const float tl = 0.015625f * xs * rsqrt_seed(fmaxf(xs, 1e-30f)) * rsqrt_seed(fmaxf(vs, 1e-30f));   // 2^-6 |x| / |v|
    t_lim = __uint_as_float(__reduce_min_sync(FULL, (am >> lane) & 1u ? __float_as_uint(tl) : 0x7F000000u));
    t_el = 0.0f;
    n_el = 0;
    anchored = true;
    placed = false;
  };
  auto place = [&]() {                     // separations at the current positions
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const df fa = shf(dl[c], ia), fb = shf(dl[c], ib);
      const df t = two_sum(fb.h, -fa.h), u = two_sum(d0[c].h, t.h);
      d[c] = fast_two_sum(u.h, __fadd_rn(u.l, __fadd_rn(t.l, __fadd_rn(__fsub_rn(fb.l, fa.l), d0[c].l))));
    }
    r2 = norm2(d);
    const df_root q = root(r2);
    r = root_of(r2, q);
    r3 = inverse_cube(q);
    placed = true;
  };
  auto active = [&](int k) { return isp && lev >= k - 1 && ((am >> ia) & (am >> ib) & 1u); };

  // the level-k share of every F_{k-1} force, summed per body
  auto forces = [&](int k) {
    df K[3];
    {
      const df Rk = renorm(mul(R2, ld(G->c2[k])));
      const bool in = less(r2, Rk);
      // w_k = g_k inside R_k, 1 - g_{k-1} outside; zero outside [R_{k+1}, R_{k-1})
      const bool zero = !active(k) || r2.h < mul(R2, ld(G->c2[k + 1])).h || !(r2.h < mul(R2, ld(G->c2[k - 1])).h);
      const int z = in ? k : k - 1;
      const df rho = renorm(mul(r, iR));
      df w;
      if (C.l == 3) {
        const df yp = zone_odd(rho, ld(G->A[z]), ld(G->B[z]));
        w = from(0.5f, mk(in ? -yp.h : yp.h, in ? -yp.l : yp.l));
      } else {
        const double g = partition_fn(((f32_to_f64(rho.h) + f32_to_f64(rho.l)) - dp->ck[z + 1]) * dp->invdc[z], C.l);
        w = split(in ? g : 1.0 - g);
      }
      const df s = mul(w, r3);
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        K[c] = mul(s, d[c]);
        if (zero) K[c] = mk(0.0f, 0.0f);
      }
    }
    const unsigned Lm = __ballot_sync(FULL, isp && lev >= k - 1);
    unsigned mine = adjm & Lm;
    const int iters = __reduce_max_sync(FULL, (unsigned)__popc(mine));
#pragma unroll
    for (int c = 0; c < 3; ++c) acc[c] = mk(0.0f, 0.0f);
    for (int it = 0; it < iters; ++it) {
      const int q = mine ? (__ffs(mine) - 1) : lane;
      const df ga = shf(gA, q), gb = shf(gB, q);
      const bool first = (im >> q) & 1u;
      df f = first ? gb : neg(ga);
      if (!mine) f = mk(0.0f, 0.0f);
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        const df t = mul(f, shf(K[c], q));
        if (mine) acc[c] = add(acc[c], t);
      }
      mine &= mine - 1u;
    }
  };
  auto kick = [&](int k) {                 // by h_k / 2
    const df h = ld(G->h[k]), hh = mk(0.5f * h.h, 0.5f * h.l);
#pragma unroll
    for (int c = 0; c < 3; ++c) nu[c] = add(nu[c], mul(hh, acc[c]));
  };

  // (iii): the bodies of F_{k-1} in no F_k pair (or all of them) drift h_k
  auto drift = [&](int k, bool all) {
    const unsigned Lm = __ballot_sync(FULL, isp && lev >= k - 1);
    const unsigned Fm = __ballot_sync(FULL, isp && lev >= k);
    const bool go = ((am >> lane) & 1u) && (adjm & Lm) != 0u && (all || (adjm & Fm) == 0u);
    if (!__any_sync(FULL, go)) return;
    const df h = ld(G->h[k]), mh = ld(G->mh[k]), ih = ld(G->rh[k]);
    float rv = 0.0f, vv = 0.0f, rr = 0.0f;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const float xf = x0[c].h + dl[c].h, vf = h.h * (v0[c].h + nu[c].h);
      rr = fmaf(xf, xf, rr);
      rv = fmaf(xf, vf, rv);
      vv = fmaf(vf, vf, vv);
    }
    const float y = rsqrt_seed(rr), y2 = y * y, uf = mh.h * y2 * y, pf = rv * y2, qf = fmaf(vv, y2, -uf);
    const float sl = fmaxf(fmaxf(fabsf(uf), pf * pf), fabsf(qf));   // s of drift_series()
    const float so = __uint_as_float(__reduce_max_sync(FULL, go ? __float_as_uint(sl) : 0u));
    if (!(so <= 1.28e-4f)) {               // the FP64 Kepler solver
      absorb();
      if (go) {
        body_store(S, slot, b);
        const int st = kepler_slot(S, slot, C.mu, dp->hk[k]);
        if (st != SYMBA_OK) set_status(&D.stat[C.d], st);
        body_load(S, slot, b);
      }
      __syncwarp();
      return;
    }
    if (go) {
      df xx[3], hv[3], dx[3], dv[3];
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        xx[c] = add(x0[c], dl[c]);
        hv[c] = mul(h, add(v0[c], nu[c]));
      }
      series_increments(xx, hv, mh, so >= 1e-8f, so > 2.0e-6f, dx, dv);
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        dl[c] = add(dl[c], dx[c]);
        nu[c] = add(nu[c], mul(ih, dv[c]));
      }
    }
    __syncwarp();
    n_el += 1;
    t_el += fabsf(h.h);
  };

  // (i) in double-float; returns whether F_k is non-empty
  auto check = [&](int k) -> bool {
    const bool act = active(k);
    const df Rk = renorm(mul(R2, ld(G->c2[k])));
    bool fl = act && less(r2, Rk);
    const float Rj = Rk.h > 0.0f ? Rk.h * rsqrt_seed(Rk.h) * 1.000001f : 0.0f;   // not below R_k
    // conservative FP32 test that the pair stays outside R_k over h (pair_path.cuh)
    float s2 = 0.0f, sa = vsum;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const float ua = SH(nu[c].h, ia), ub = SH(nu[c].h, ib), du = dv0[c] + (ub - ua);
      s2 = fmaf(du, du, s2);
      sa += fabsf(ua) + fabsf(ub);
    }
    const float mg = 1.0f + 3.0517578e-5f;
    const float dvm = s2 * rsqrt_seed(fmaxf(s2, 1e-30f)) * mg + sa * 2.3841858e-7f;
    const bool far = r.h * (1.0f - 3.0517578e-5f) > (Rj + dvm * fabsf(G->h[k].x) * mg) * mg;
    const bool near = act && !fl && !far;
    if (__any_sync(FULL, near)) {
      double e[3], u[3];
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        const double vt = (scale2(b.v[c], -eb) + f32_to_f64(nu[c].l)) + f32_to_f64(nu[c].h);
        u[c] = SH(vt, ib) - SH(vt, ia);
        e[c] = f32_to_f64(d[c].h) + f32_to_f64(d[c].l);
      }
      if (near) {
        const double R0 = S.R0[qs];
        fl = predicate_regs(e[0], e[1], e[2], fma(e[2], e[2], fma(e[1], e[1], e[0] * e[0])), u[0], u[1], u[2],
                            scale2(R0 * R0 * dp->ck2[k], -2 * ea), scale2(dp->hk[k], eb - ea));
      }
    }
    if (isp && lev >= k - 1) lev = fl ? k : k - 1;
    return __any_sync(FULL, fl) != 0;
  };

  // (i) with a pair that may be in contact: the pairs one by one in list order, on the FP64 state
  auto check_contacts = [&](int k, double h) -> bool {
    bool any = false, nonempty = false;
    for (int q = 0; q < np; ++q) {
      if (SH(lev, q) < k - 1) continue;
      const int a_ = SH(ia, q), b_ = SH(ib, q);
      bool fl = false;
      if ((am >> a_) & (am >> b_) & 1u) {
        double xa[3], xb[3], va[3], vb[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          xa[c] = SH(b.x[c], a_); xb[c] = SH(b.x[c], b_);
          va[c] = SH(b.v[c], a_); vb[c] = SH(b.v[c], b_);
        }
        const double ra = SH(b.rad, a_), rb = SH(b.rad, b_), ma = SH(b.m, a_), mb = SH(b.m, b_), rha = SH(b.rh, a_);
        if (contact_regs(xa[0], xa[1], xa[2], xb[0], xb[1], xb[2], ra, rb)) {
          const double Mt = __dadd_rn(ma, mb);
          if (lane == a_) {
            if (Mt > 0.0) {
#pragma unroll
              for (int c = 0; c < 3; ++c) {
                b.x[c] = __ddiv_rn(__dadd_rn(__dmul_rn(ma, xa[c]), __dmul_rn(mb, xb[c])), Mt);
                b.v[c] = __ddiv_rn(__dadd_rn(__dmul_rn(ma, va[c]), __dmul_rn(mb, vb[c])), Mt);
              }
            }
            b.rad = cbrt_rn(__dadd_rn(__dmul_rn(__dmul_rn(ra, ra), ra), __dmul_rn(__dmul_rn(rb, rb), rb)));
            if (ma > 0.0) b.rh = __dmul_rn(rha, cbrt_rn(__ddiv_rn(Mt, ma)));
            b.m = Mt;
            b.gm = __dmul_rn(C.G, Mt);
          }
          if (lane == b_) b.m = b.gm = b.rad = b.rh = 0.0;
          if (lane == 0) atomicAdd(&D.stat[C.d].merges, 1ull);
          am &= ~(1u << b_);
          any = true;
          // critical radii follow the new body
          const double R0 = __dmul_rn(C.lam, __dadd_rn(SH(b.rh, ia), SH(b.rh, ib)));
          if (isp) {
            S.R0[qs] = R0;
            S.invR0[qs] = R0 > 0.0 ? 1.0 / R0 : 0.0;
          }
          __syncwarp();
        } else {
          const double R0q = S.R0[SH(qs, q)], dx = xb[0] - xa[0], dy = xb[1] - xa[1], dz = xb[2] - xa[2];
          fl = predicate_regs(dx, dy, dz, fma(dz, dz, fma(dy, dy, dx * dx)), vb[0] - va[0], vb[1] - va[1], vb[2] - va[2],
                              R0q * R0q * dp->ck2[k], h);
        }
      }
      if (lane == q) lev = fl ? k : k - 1;
      nonempty |= fl;
    }
    if (any) {
      pair_consts();
      *merged_any = true;
    }
    return nonempty;
  };

  int k = k0, forces_at = -1;
  bool start = true, done = true;
  for (;;) {
    if (start) {
      // a single pair below this level: the single-pair path
      const unsigned Lm = __ballot_sync(FULL, isp && lev >= k - 1);
      if (C.l == 3 && __popc(Lm) == 1) {
        const int q = __ffs(Lm) - 1;
        const int a_ = SH(ia, q), b_ = SH(ib, q);
        if ((am >> a_) & (am >> b_) & 1u) {
          // the state waits in the view: pair_run() needs the registers
          absorb();
          if (ism) body_store(S, slot, b);
          const int src = SH(slot, (lane & 1) ? b_ : a_);
          const int q_ = SH(qs, q), oa = SH(slot, a_), ob = SH(slot, b_);
          __syncwarp();
          double px[3] = {S.x[src], S.y[src], S.z[src]}, pv[3] = {S.vx[src], S.vy[src], S.vz[src]};
          const double R0 = S.R0[q_], Rc = S.rad[oa] + S.rad[ob];
          int plev = SH(lev, q);
          const long long sub0 = substeps;
          const int rc = pair_run(D, C, lane, hs, cs, T, G, ea, eb, px, pv, S.gm[oa], S.gm[ob], R0 * R0, S.invR0[q_],
                                  1.0000001 * (Rc * Rc), k, plev, substeps, deepest);
          if (lane == 0) atomicAdd(&D.stat[C.d].pair_substeps, (unsigned long long)(substeps - sub0));
          if (lane < 2) {
            S.x[src] = px[0]; S.y[src] = px[1]; S.z[src] = px[2];
            S.vx[src] = pv[0]; S.vy[src] = pv[1]; S.vz[src] = pv[2];
          }
          __syncwarp();
          // nothing but the view and the pair marks is kept over the call
          if (ism) body_load(S, slot, b);
          else clear_body();
          clear();
          pair_consts();
          if (lane == q) lev = plev;
          forces_at = -1;
          if (rc == 2) { done = false; break; }
          if (rc == 0) {                   // level k + 1 finished: continue with the closing kick of k
            if (k < k0) break;
            start = false;
            continue;
          }
          // rc == 1: a contact may be due; this sub-step is taken here
        }
      }
      ++substeps;
      if (substeps > C.max_substeps) { done = false; break; }
      deepest = max(deepest, k);
      if (n_el >= ANCHOR_N || t_el > t_lim) absorb();
    } else {
      placed = false;
      forces_at = -1;
    }
    bool fk = false, checked = !start;
    for (;;) {
      if (!anchored) anchor();
      if (!placed) place();
      if (checked) break;
      checked = true;
      if (!__any_sync(FULL, active(k) && r2.h < cut)) {
        fk = check(k);
        break;
      }
      absorb();
      const unsigned before = am;
      fk = check_contacts(k, dp->hk[k]);
      if (am != before) forces_at = -1;
    }
    if (forces_at != k) { forces(k); forces_at = k; }
    kick(k);
    if (start) {
      const bool deeper = fk && (k + 1 <= C.max_depth);
      if (fk && !deeper && lane == 0) set_status(&D.stat[C.d], SYMBA_E_DEPTH);
      drift(k, fk && !deeper);
      if (deeper) {
        // (the pairs of F_k have not moved: their separations hold unless the anchors did)
        ++k;
        hs[k] = dp->hk[k];
        cs[k] = 0;
        continue;
      }
      start = false;
      continue;
    }
    if (++cs[k] < C.M) { start = true; continue; }
    --k;
    if (k < k0) break;
  }
  absorb();
  if (ism) {
    body_store(S, slot, b);
    S.alive[slot] = (am >> lane) & 1u;
  }
  if (isp) S.lev[qs] = lev;
  __syncwarp();
  return done;
}
