// The right-angled-trapezoid pair kick (Sec. 2): every pair i < N_m, j > i once, both
// reactions accumulated, no atomics.
//
// Work decomposition.  Indices are cut into 32-blocks; tile (I, J), I <= J, over the column
// blocks that hold massive bodies, holds the pairs of block I (rows) with block J (columns): the
// trapezoid becomes a rectangle of off-diagonal tiles plus the diagonal tiles of the triangle.
// Tiles are grouped into macro-tiles of 4 row blocks (a 128-body quad q) by SYM_MACRO_COLS column
// blocks (column group p, p >= 4q / SYM_MACRO_COLS), all macro-tiles of all systems in one flat
// list that persistent CTAs consume from a counter (the fold of the triangle into a rectangle, done
// by a work queue instead of index arithmetic).
//
// One CTA per macro-tile: a warp keeps row particle I*32 + l in lane l and sweeps the macro's column
// blocks in turn; in each tile lane l meets column (l + s) mod 32 at step s (32 steps; 16 on a
// diagonal tile, where each unordered pair is met once).  The column sums rotate through the lanes
// by warp shuffle (the mixed path rotates the bodies with them).  The row accumulators run on across
// the macro-tile's tiles; row and column sums of the CTA's warps are added in shared memory in warp
// order and written once per macro-tile.  Both kinds of partials are summed later in a fixed order:
// the result does not depend on scheduling, on how many macro-tiles a CTA takes per grab, or on
// which other systems share the launch.
//
// FP64 systems form the pair force in double-float (df32.cuh) on the FP32 pipe, which GB300 runs at
// 62x the FP64 rate.  Separations come from coordinates cut on grids common to a macro-tile, exact
// to 2^-61 of its extent; r^-3, the products and a macro-tile's sums carry 46 to 48 bits, which lies below
// the rounding of v += (tau/2) a while a kick is a small part of v (a body of 1e-3 m0 at 1 AU and
// tau = 0.5 yr: 1/300); where it is not, and where the macro-tile's extent would cost digits, the
// macro-tile is taken in FP64 (see "how far the double-float form may go").  Against an 80-bit kick the
// new v is as close as FP64 pairs bring it.
//   10,000 bodies, per kick: 1.48 ms with 16.5 FP64 instructions per pair (FP64 pipe 90 % busy) ->
//   0.50-0.57 ms with ~275 warp instructions per 32 pairs (60 % of the issue slots; four barriers per
//   macro-tile take most of the rest); 3.1 ms when every macro-tile is taken in FP64.  1,000 bodies
//   0.160 -> 0.019 ms, 100 bodies 0.065 -> 0.018 ms (see k_trap_df and launch_trap for the small systems).
//
// Kick 1 also runs the close-encounter check (Sec. 2) of every pair: a conservative FP32
// prefilter (|d| - tau |dv| against R_0 with rounding margins) and, for the rare pairs that pass,
// the exact FP64 predicate, identical operation for operation to the definition; flagged pairs
// are appended to the system's pair list and weighted by g_0(r).  Kick 2 weights the same
// flagged pairs, found through the group each particle belongs to.
#include "df32.cuh"
#include "internal.cuh"

#define FULL 0xffffffffu

struct TileCtx {
  int off, n, nm, pair_base, pair_cap, l;
  double dt, lam, c0, c1;
};

__device__ __forceinline__ TileCtx load_ctx(const DiskDesc *dp) {
  TileCtx c;
  c.off = dp->off; c.n = dp->n; c.nm = dp->nm;
  c.pair_base = dp->pair_base; c.pair_cap = dp->pair_cap; c.l = dp->l;
  c.dt = dp->dt; c.lam = dp->hill_scale; c.c0 = dp->ck[0]; c.c1 = dp->ck[1];
  return c;
}

__device__ __forceinline__ double g0_weight(const TileCtx &c, double R0, double r) {
  const double Rk = R0 * c.c0, Rk1 = R0 * c.c1;
  return partition_fn((r - Rk1) / (Rk - Rk1), c.l);
}

// level-0 weight of a pair by the encounter predicate: g_0(r) when it is flagged, else 1
__device__ __forceinline__ double flagged_weight(const Dev &D, const TileCtx &c, int lo, int hi) {
  const double ex = __dsub_rn(D.x[hi], D.x[lo]), ey = __dsub_rn(D.y[hi], D.y[lo]), ez = __dsub_rn(D.z[hi], D.z[lo]);
  const double evx = __dsub_rn(D.vx[hi], D.vx[lo]), evy = __dsub_rn(D.vy[hi], D.vy[lo]),
               evz = __dsub_rn(D.vz[hi], D.vz[lo]);
  const double R0 = __dmul_rn(c.lam, __dadd_rn(D.rh[lo], D.rh[hi]));
  if (!encounter_exact(ex, ey, ez, evx, evy, evz, R0, c.dt)) return 1.0;
  return g0_weight(c, R0, __dsqrt_rn(__dadd_rn(__dadd_rn(__dmul_rn(ex, ex), __dmul_rn(ey, ey)), __dmul_rn(ez, ez))));
}

// Binary search of (lo, hi) in the sorted pair list of a group.
__device__ __forceinline__ bool group_has_pair(const Dev &D, int g, int lo, int hi) {
  int a = D.g_poff[g], b = a + D.g_pcnt[g];
  while (a < b) {
    const int m = (a + b) >> 1;
    const int mi = D.gpi[m], mj = D.gpj[m];
    if (mi < lo || (mi == lo && mj < hi)) a = m + 1; else b = m;
  }
  return a < D.g_poff[g] + D.g_pcnt[g] && D.gpi[a] == lo && D.gpj[a] == hi;
}


// partial slots of macro-tile m: rows [w][component][lane], then columns [k][component][lane]
__device__ __forceinline__ size_t part_row(int m, int w) { return (size_t)m * SYM_MACRO_PART + w * 96; }
__device__ __forceinline__ size_t part_col(int m, int k) { return (size_t)m * SYM_MACRO_PART + 384 + k * 96; }
#define MC SYM_MACRO_COLS
__device__ __forceinline__ df ld2(const float2 &v) { return mk(v.x, v.y); }

// ---- FP64 systems: the pair arithmetic in double-float --------------------------------------------
// A coordinate as three FP32 numbers on grids common to a tile: x = a + b + c with a a multiple of
// 2^(E - 21), b in [0, 2^(E - 21)) of 2^(E - 41), c in [0, 2^(E - 41)) of 2^(E - 61), for |x| < 2^(E + 1).
// Differences of a, of b and of c are exact, so a separation keeps every digit that matters down to
// 2^-61 of the tile's extent in that component (FP64 positions of that size are multiples of 2^-52).
// Values are scaled by 2^-kex.
__device__ __forceinline__ void on_grid(double x, int E, int kex, float &a, float &b, float &c) {
  const long long bits = __double_as_longlong(x);
  const int e = (int)((bits >> 52) & 0x7FF) - 1023;
  const unsigned long long man = (bits & 0xFFFFFFFFFFFFFll) | (1ll << 52);
  const int sh = 9 - (E - e);
  unsigned long long u = sh >= 0 ? man << (sh & 63) : man >> min(-sh, 63);
  if (e == -1023) u = 0ull;
  const long long X = bits < 0 ? -(long long)u : (long long)u;       // x 2^(61 - E)
  const float sa = __int_as_float((E - kex - 21 + 127) << 23);
  a = __int2float_rn((int)(X >> 40)) * sa;
  b = __int2float_rn((int)((X >> 20) & 0xFFFFF)) * (sa * 9.5367432e-7f);                   // 2^-20
  c = __int2float_rn((int)(X & 0xFFFFF)) * (sa * 9.0949470e-13f);                          // 2^-40
}
// exponent of the grid of a component: that of its largest |x| (hi: the largest high word), not below
// 2^-60 of the largest of the three
__device__ __forceinline__ int grid_exp(int hi, int kex) { return max((hi >> 20) - 1023, kex - 60); }
__device__ __forceinline__ df separation(float aj, float bj, float cj, float ai, float bi, float ci) {
  const df t = fast_two_sum(__fsub_rn(aj, ai), __fsub_rn(bj, bi));   // |da| >= |db| or da = 0
  return fast_two_sum(t.h, __fadd_rn(t.l, __fsub_rn(cj, ci)));
}
// sum += t, the sum's low part collecting errors (48 bits of the sum)
__device__ __forceinline__ void accumulate(df &sum, df t) {
  const df s = two_sum(sum.h, t.h);
  sum.h = s.h;
  sum.l = __fadd_rn(sum.l, __fadd_rn(s.l, t.l));
}

// ---- how far the double-float form may go
// Positions are scaled by 2^-kex and G m by 2^-keg, the largest of the macro-tile (of the field chunk), so
// neither what lies elsewhere in the system nor how far it has spread since set-up matters.  What is lost:
// the arithmetic leaves an error of about 2^-46 of a pair's force s d, s = G m / r^3, and the grid moves a
// separation by up to sqrt(3) 2^-61, which changes the force by up to 4 sqrt(3) 2^-61 s < 2^-58 s.  Every
// body's sum of s (r + GRID_TERM) is kept beside its force, and the macro-tile is taken again in FP64
// (macro_general) when 2^-46 of it, times tau/2, may exceed 2^-54 |v| of a body -- half of what the rounding
// of v loses anyway -- or when a force left the FP32 range.  So kicks above 2^-8 |v| (a body of 1e-3 m0 five
// mutual Hill radii away, tau a tenth of the period) keep FP64's digits, and a body far from the rest
// (ejected, or parked) costs the macro-tiles it is in time and not accuracy: for pairs 0.05 AU apart in a
// disk of 10 AU the double-float force is off by 2e-16 of itself, and with a body of the macro-tile at
// 1e8 AU by 1.5e-9.
#define GRID_TERM 2.4414062e-4f          // 2^-12
struct Units {
  int kex, keg;
  bool fits;             // the exponents leave room for the scaled arithmetic
};
__device__ __forceinline__ int top_exp(int hi) { return (hi >> 20) - 1023; }
// from the high words of the largest |x|, |y|, |z|, G m and the smallest G m > 0
__device__ __forceinline__ Units units_of(int hx, int hy, int hz, int gmax, int gmin) {
  Units u;
  u.kex = top_exp(max(hx, max(hy, hz)));
  u.keg = gmax ? top_exp(gmax) : 0;
  // (a G m below 2^-80 of the largest would lose its low part)
  u.fits = abs(u.kex) <= 250 && abs(u.keg) <= 250 && (gmax == 0 || top_exp(gmin) >= u.keg - 80);
  return u;
}
// Largest sum of s (r + GRID_TERM) (scaled) allowed for a body: 2^-8 |v| / (tau/2) over the square root of the
// number of such sums (their errors are independent), rounded down to a power of two.  hv: high word of
// the body's largest |v| component.
__device__ __forceinline__ float error_room(int hv, double dt, const Units &u, int nsum) {
  const int eh = top_exp(__double2hiint(dt) & 0x7FFFFFFF);          // tau/2 < 2^eh
  const int n = top_exp(hv) - 8 - eh + 2 * u.kex - u.keg - (33 - __clz(nsum)) / 2;
  return n < -126 ? 0.0f : __int_as_float(min(n + 127, 254) << 23);
}

// the row side of one warp: row particle I*32 + lane, its data and its accumulators
struct RowDF {
  int pi;
  bool live, row;          // a live body; live and massive (a row of the trapezoid)
  float x[3][3];           // a, b, c of each component
  df ngm;                  // -G m, scaled
  float xf, yf, zf, vxf, vyf, vzf, lam, sig;   // kick 1: FP32 prefilter copies
  int gid;                 // kick 2: encounter group
  df acc[3];               // carried across the macro-tile's column blocks
  float lost;              // sum of s (r + GRID_TERM)
};

// a column body in shared memory: {x: a b c, y: a} {y: b c, z: a b} {z: c, G m: h l, group}
struct ColDF {
  float4 q[3];
};

template <int MODE>
__device__ __forceinline__ void row_load_df(const Dev &D, const TileCtx &c, const int *E, const Units &u, int I, int lane,
                                            RowDF &r) {
  r.pi = I * 32 + lane;
  const int li = r.pi - c.off;
  r.live = li < c.n && D.alive[r.pi];
  r.row = r.live && li < c.nm;
  const double p[3] = {D.x[r.pi], D.y[r.pi], D.z[r.pi]};
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    on_grid(r.live ? p[k] : 0.0, E[k], u.kex, r.x[k][0], r.x[k][1], r.x[k][2]);
    r.acc[k] = mk(0.0f, 0.0f);
  }
  r.lost = 0.0f;
  r.ngm = neg(split(scale2(D.gm[r.pi], -u.keg)));
  r.xf = r.yf = r.zf = r.vxf = r.vyf = r.vzf = r.lam = r.sig = 0.f;
  r.gid = -1;
  if (MODE == 1) {
    r.xf = D.xf[r.pi]; r.yf = D.yf[r.pi]; r.zf = D.zf[r.pi];
    r.vxf = D.vxf[r.pi]; r.vyf = D.vyf[r.pi]; r.vzf = D.vzf[r.pi];
    r.lam = D.lamf[r.pi]; r.sig = D.sigf[r.pi];
  } else {
    r.gid = D.gid[r.pi];
  }
}

// s w for the level-0 weight of a flagged pair (zero also where r^-3 left the FP32 range)
__device__ __forceinline__ df weighted(df s, double w) { return w == 0.0 ? mk(0.0f, 0.0f) : mul(s, split(w)); }

// Steps [t0, t1) of one 32 x 32 tile (rows of block I, columns of block J >= I, 32 steps; 16 on the
// diagonal): at step t lane l meets column (l + t + o) mod 32 (o = 1 on the diagonal), whose
// column-side sums travel with it from lane to lane.  The row side goes into r.acc, the column side
// into out[component][column].
template <int MODE>
__device__ __forceinline__ void tile_steps_df(const Dev &D, const TileCtx &c, int sys, RowDF &r, int I, int J, int lane,
                                              int t0, int t1, const ColDF *col, const float4 (*cf)[2],
                                              unsigned mlive, unsigned mmass, float2 (*out)[32], float *out_lost) {
  const bool diag = I == J;
  const int o = diag ? 1 : 0;
  const float tauf = __double2float_ru(c.dt);
  df ca[3] = {mk(0.0f, 0.0f), mk(0.0f, 0.0f), mk(0.0f, 0.0f)};
  float lost = 0.0f;
#pragma unroll 1
  for (int t = t0; t < t1; ++t) {
    const int cj = (lane + t + o) & 31;
    const int jid = J * 32 + cj;
    const bool jl = (mlive >> cj) & 1u, jm = (mmass >> cj) & 1u;
    const float4 q0 = col[cj].q[0], q1 = col[cj].q[1], q2 = col[cj].q[2];
    bool valid;
    if (!diag) {
      valid = r.row && jl;
    } else {
      valid = (jid > r.pi) ? (r.row && jl) : (r.live && jm);
      if (t == 15 && lane >= 16) valid = false;  // pair {l, l+16} belongs to lane l < 16
    }
    const df d[3] = {separation(q0.x, q0.y, q0.z, r.x[0][0], r.x[0][1], r.x[0][2]),
                     separation(q0.w, q1.x, q1.y, r.x[1][0], r.x[1][1], r.x[1][2]),
                     separation(q1.z, q1.w, q2.x, r.x[2][0], r.x[2][1], r.x[2][2])};
    const df r2 = norm2(d);
    const df_root rt = root(r2);
    const float reach = fminf(fmaf(r2.h, rt.y, GRID_TERM), 8.0f);     // (8 where r = 0: a pair left out)
    const df r3 = inverse_cube(rt);
    df sj = mul(mk(q2.y, q2.z), r3);
    df si = mul(r.ngm, r3);             // the column side's -G m_i / r^3
    if (MODE == 1) {
      const float4 fa = cf[cj][0], fb = cf[cj][1];
      const float dxf = fa.x - r.xf, dyf = fa.y - r.yf, dzf = fa.z - r.zf;
      const float r2f = fmaf(dzf, dzf, fmaf(dyf, dyf, dxf * dxf));
      const float dvxf = fa.w - r.vxf, dvyf = fb.x - r.vyf, dvzf = fb.y - r.vzf;
      const float vmag = sqrtf(fmaf(dvzf, dvzf, fmaf(dvyf, dvyf, dvxf * dvxf)));
      const float Bf = fmaf(tauf, vmag, r.lam + fb.z) * 1.0000039f + 1.9073486e-6f * (r.sig + fb.w);
      const bool cand = valid && !(r2f > Bf * Bf);
      if (__any_sync(FULL, cand)) {
        if (cand) {
          const int lo = min(r.pi, jid), hi = max(r.pi, jid);
          const double ex = __dsub_rn(D.x[hi], D.x[lo]), ey = __dsub_rn(D.y[hi], D.y[lo]),
                       ez = __dsub_rn(D.z[hi], D.z[lo]);
          const double evx = __dsub_rn(D.vx[hi], D.vx[lo]), evy = __dsub_rn(D.vy[hi], D.vy[lo]),
                       evz = __dsub_rn(D.vz[hi], D.vz[lo]);
          const double R0 = __dmul_rn(c.lam, __dadd_rn(D.rh[lo], D.rh[hi]));
          if (encounter_exact(ex, ey, ez, evx, evy, evz, R0, c.dt)) {
            const int k = atomicAdd(&D.stat[sys].npairs, 1);
            if (k < c.pair_cap) {
              D.raw_i[c.pair_base + k] = lo;
              D.raw_j[c.pair_base + k] = hi;
            }
            const double er2 = __dadd_rn(__dadd_rn(__dmul_rn(ex, ex), __dmul_rn(ey, ey)), __dmul_rn(ez, ez));
            const double w = g0_weight(c, R0, __dsqrt_rn(er2));
            sj = weighted(sj, w);
            si = weighted(si, w);
          }
        }
        __syncwarp();
      }
    } else {
      if (r.gid >= 0 && r.gid == __float_as_int(q2.w) && valid) {
        const int lo = min(r.pi, jid), hi = max(r.pi, jid);
        if (group_has_pair(D, r.gid, lo, hi)) {
          const double R0 = __dmul_rn(c.lam, __dadd_rn(D.rh[lo], D.rh[hi]));
          const double ex = D.x[hi] - D.x[lo], ey = D.y[hi] - D.y[lo], ez = D.z[hi] - D.z[lo];
          const double w = g0_weight(c, R0, sqrt(fma(ez, ez, fma(ey, ey, ex * ex))));
          sj = weighted(sj, w);
          si = weighted(si, w);
        }
      }
    }
    sj.h = valid ? sj.h : 0.0f; sj.l = valid ? sj.l : 0.0f;
    si.h = valid ? si.h : 0.0f; si.l = valid ? si.l : 0.0f;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      accumulate(r.acc[k], mul(sj, d[k]));
      accumulate(ca[k], mul(si, d[k]));
    }
    r.lost = fmaf(fabsf(sj.h), reach, r.lost);
    lost = fmaf(fabsf(si.h), reach, lost);
    if (t + 1 < t1) {
      const int src = (lane + 1) & 31;
      lost = __shfl_sync(FULL, lost, src);
#pragma unroll
      for (int k = 0; k < 3; ++k) ca[k] = mk(__shfl_sync(FULL, ca[k].h, src), __shfl_sync(FULL, ca[k].l, src));
    }
  }
  const int last = (lane + t1 - 1 + o) & 31;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const df q = t1 > t0 ? renorm(ca[k]) : ca[k];
    out[k][last] = make_float2(q.h, q.l);
  }
  out_lost[last] = lost;
}

// The macro-tile again in FP64 (its encounters are in the pair list already): the same warps, quarters and
// order, sums into the same slots.  For the rare macro-tile, so bodies are read where they lie.
template <int MODE>
static __device__ __noinline__ void macro_general(const Dev &D, const int4 mt, const ColDF (*col)[32], const float4 (*cf)[32][2],
                                                  const unsigned *mlive, const unsigned *mmass, double (*rowbuf)[3][32],
                                                  double (*colbuf)[MC][3][32]) {
  const TileCtx c = load_ctx(&D.disks[mt.x]);
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, ws = w >> 2, I = mt.y + (w & 3), pi = I * 32 + lane;
  const bool has_row = I < mt.w;
  const int q = has_row ? pi : c.off, li = pi - c.off;
  const bool live = has_row && li < c.n && D.alive[q], row = live && li < c.nm;
  const double x = D.x[q], y = D.y[q], z = D.z[q], ngm = -D.gm[q];
  const float tauf = __double2float_ru(c.dt);
  double ra[3] = {0.0, 0.0, 0.0};
  for (int k = 0; k < MC; ++k) {
    const int J = mt.z + k;
    const bool diag = I == J, any = has_row && J < mt.w && J >= I;
    const int len = any ? (diag ? 4 : 8) : 0, o = diag ? 1 : 0;
    double ca[3] = {0.0, 0.0, 0.0};
    for (int t = len * ws; t < len * ws + len; ++t) {
      const int cj = (lane + t + o) & 31, jid = J * 32 + cj;
      const bool jl = (mlive[k] >> cj) & 1u, jm = (mmass[k] >> cj) & 1u;
      bool valid = diag ? (jid > pi ? (row && jl) : (live && jm)) : (row && jl);
      if (diag && t == 15 && lane >= 16) valid = false;
      const double dx = D.x[jid] - x, dy = D.y[jid] - y, dz = D.z[jid] - z;
      const double r2 = fma(dz, dz, fma(dy, dy, dx * dx));
      const double ri = rsqrt_fp64(r2), r3 = ri * ri * ri;
      double wt = 1.0;
      if (valid) {
        const int lo = min(pi, jid), hi = max(pi, jid);
        if (MODE == 1) {
          const float4 fa = cf[k][cj][0], fb = cf[k][cj][1];
          const float dxf = fa.x - D.xf[pi], dyf = fa.y - D.yf[pi], dzf = fa.z - D.zf[pi];
          const float r2f = fmaf(dzf, dzf, fmaf(dyf, dyf, dxf * dxf));
          const float dvxf = fa.w - D.vxf[pi], dvyf = fb.x - D.vyf[pi], dvzf = fb.y - D.vzf[pi];
          const float vmag = sqrtf(fmaf(dvzf, dvzf, fmaf(dvyf, dvyf, dvxf * dvxf)));
          const float Bf = fmaf(tauf, vmag, D.lamf[pi] + fb.z) * 1.0000039f + 1.9073486e-6f * (D.sigf[pi] + fb.w);
          if (!(r2f > Bf * Bf)) wt = flagged_weight(D, c, lo, hi);
        } else if (D.gid[pi] >= 0 && D.gid[pi] == __float_as_int(col[k][cj].q[2].w) && group_has_pair(D, D.gid[pi], lo, hi)) {
          wt = g0_weight(c, __dmul_rn(c.lam, __dadd_rn(D.rh[lo], D.rh[hi])), sqrt(r2));
        }
      }
      const double sj = valid && wt != 0.0 ? D.gm[jid] * r3 * wt : 0.0, si = valid && wt != 0.0 ? ngm * r3 * wt : 0.0;
      ra[0] = fma(sj, dx, ra[0]); ra[1] = fma(sj, dy, ra[1]); ra[2] = fma(sj, dz, ra[2]);
      ca[0] = fma(si, dx, ca[0]); ca[1] = fma(si, dy, ca[1]); ca[2] = fma(si, dz, ca[2]);
      if (t + 1 < len * ws + len) {
        const int src = (lane + 1) & 31;
        for (int e = 0; e < 3; ++e) ca[e] = __shfl_sync(FULL, ca[e], src);
      }
    }
    const int last = (lane + len * ws + len - 1 + o) & 31;
    for (int e = 0; e < 3; ++e) colbuf[w][k][e][len ? last : lane] = ca[e];
  }
  for (int e = 0; e < 3; ++e) rowbuf[w][e][lane] = ra[e];
}

// Mixed precision (FP32 pair path): the relative displacement is formed from the two-float split
// x = xf + xl of each FP64 position, (xf_j - xf_i) + (xl_j - xl_i) -- RN32 of the FP64 difference
// or a neighbouring float for every pair the level-0 weight does not zero; r^-3 from the FP32
// rsqrt plus one Newton step; both sides accumulated in FP32 with Kahan compensation and written
// as (sum, compensation) pairs that the reduction carries into FP64.  The encounter check is the
// same FP64 decision as in the FP64 path.
__device__ __forceinline__ void kahan(float &s, float &c, float term) {
  const float y = term - c;
  const float t = s + y;
  c = (t - s) - y;
  s = t;
}

struct RowMixed {
  int pi;
  bool live, row;
  float xh, yh, zh, xl, yl, zl, gm;
  float vxf, vyf, vzf, lam, sig;   // kick 1 prefilter
  int gid;                         // kick 2
  float sx, sy, sz, cx, cy, cz;    // Kahan sums of the row side, carried across the macro-tile
};

template <int MODE>
__device__ __forceinline__ void row_load_mixed(const Dev &D, const TileCtx &c, int I, int lane, RowMixed &r) {
  r.pi = I * 32 + lane;
  const int li = r.pi - c.off;
  r.live = li < c.n && D.alive[r.pi];
  r.row = r.live && li < c.nm;
  r.xh = D.xf[r.pi]; r.yh = D.yf[r.pi]; r.zh = D.zf[r.pi];
  r.xl = D.xl[r.pi]; r.yl = D.yl[r.pi]; r.zl = D.zl[r.pi];
  r.gm = D.gmf[r.pi];
  r.vxf = r.vyf = r.vzf = r.lam = r.sig = 0.f;
  r.gid = -1;
  if (MODE == 1) {
    r.vxf = D.vxf[r.pi]; r.vyf = D.vyf[r.pi]; r.vzf = D.vzf[r.pi]; r.lam = D.lamf[r.pi]; r.sig = D.sigf[r.pi];
  } else {
    r.gid = D.gid[r.pi];
  }
  r.sx = r.sy = r.sz = r.cx = r.cy = r.cz = 0.f;
}

// one tile; the column side comes back as Kahan pairs (s, c) per component, zero on a diagonal
template <int MODE>
__device__ __forceinline__ void tile_sweep_mixed(const Dev &D, const TileCtx &c, int sys, RowMixed &r,
                                                 int I, int J, int lane, float2 &ox, float2 &oy, float2 &oz) {
  const bool diag = I == J;
  int jid = J * 32 + lane;
  const int lj0 = jid - c.off;
  const bool live_j0 = lj0 < c.n && D.alive[jid];
  int jflags = (live_j0 ? 1 : 0) | ((live_j0 && lj0 < c.nm) ? 2 : 0);
  float xhj = D.xf[jid], yhj = D.yf[jid], zhj = D.zf[jid];
  float xlj = D.xl[jid], ylj = D.yl[jid], zlj = D.zl[jid];
  float gmj = D.gmf[jid];
  float sxj = 0.f, syj = 0.f, szj = 0.f, cxj = 0.f, cyj = 0.f, czj = 0.f;
  float vxfj = 0.f, vyfj = 0.f, vzfj = 0.f, lamj = 0.f, sigj = 0.f;
  int gidj = -1;
  if (MODE == 1) {
    vxfj = D.vxf[jid]; vyfj = D.vyf[jid]; vzfj = D.vzf[jid]; lamj = D.lamf[jid]; sigj = D.sigf[jid];
  } else {
    gidj = D.gid[jid];
  }
  const float tauf = __double2float_ru(c.dt);

  auto rotate = [&]() {
    const int src = (lane + 1) & 31;
    xhj = __shfl_sync(FULL, xhj, src); yhj = __shfl_sync(FULL, yhj, src); zhj = __shfl_sync(FULL, zhj, src);
    xlj = __shfl_sync(FULL, xlj, src); ylj = __shfl_sync(FULL, ylj, src); zlj = __shfl_sync(FULL, zlj, src);
    gmj = __shfl_sync(FULL, gmj, src);
    sxj = __shfl_sync(FULL, sxj, src); syj = __shfl_sync(FULL, syj, src); szj = __shfl_sync(FULL, szj, src);
    cxj = __shfl_sync(FULL, cxj, src); cyj = __shfl_sync(FULL, cyj, src); czj = __shfl_sync(FULL, czj, src);
    jid = __shfl_sync(FULL, jid, src); jflags = __shfl_sync(FULL, jflags, src);
    if (MODE == 1) {
      vxfj = __shfl_sync(FULL, vxfj, src); vyfj = __shfl_sync(FULL, vyfj, src);
      vzfj = __shfl_sync(FULL, vzfj, src); lamj = __shfl_sync(FULL, lamj, src);
      sigj = __shfl_sync(FULL, sigj, src);
    } else {
      gidj = __shfl_sync(FULL, gidj, src);
    }
  };

  const int nsteps = diag ? 16 : 32;
  if (diag) rotate();
#pragma unroll 1
  for (int s = 0; s < nsteps; ++s) {
    bool valid;
    if (!diag) {
      valid = r.row && (jflags & 1);
    } else {
      valid = (jid > r.pi) ? (r.row && (jflags & 1)) : (r.live && (jflags & 2));
      if (s == 15 && lane >= 16) valid = false;
    }
    const float dx = (xhj - r.xh) + (xlj - r.xl);
    const float dy = (yhj - r.yh) + (ylj - r.yl);
    const float dz = (zhj - r.zh) + (zlj - r.zl);
    const float r2 = fmaf(dz, dz, fmaf(dy, dy, dx * dx));
    float ri;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(ri) : "f"(r2));
    ri = ri * fmaf(-0.5f * r2, ri * ri, 1.5f);
    const float s3 = ri * ri * ri;
    float sj = gmj * s3, si = r.gm * s3;
    if (MODE == 1) {
      const float dvxf = vxfj - r.vxf, dvyf = vyfj - r.vyf, dvzf = vzfj - r.vzf;
      const float vmag = sqrtf(fmaf(dvzf, dvzf, fmaf(dvyf, dvyf, dvxf * dvxf)));
      const float Bf = fmaf(tauf, vmag, r.lam + lamj) * 1.0000039f + 1.9073486e-6f * (r.sig + sigj);
      const bool cand = valid && !(r2 > Bf * Bf * 1.0000153f);
      if (__any_sync(FULL, cand)) {
        if (cand) {
          const int lo = min(r.pi, jid), hi = max(r.pi, jid);
          const double ex = __dsub_rn(D.x[hi], D.x[lo]), ey = __dsub_rn(D.y[hi], D.y[lo]),
                       ez = __dsub_rn(D.z[hi], D.z[lo]);
          const double evx = __dsub_rn(D.vx[hi], D.vx[lo]), evy = __dsub_rn(D.vy[hi], D.vy[lo]),
                       evz = __dsub_rn(D.vz[hi], D.vz[lo]);
          const double R0 = __dmul_rn(c.lam, __dadd_rn(D.rh[lo], D.rh[hi]));
          if (encounter_exact(ex, ey, ez, evx, evy, evz, R0, c.dt)) {
            const int k = atomicAdd(&D.stat[sys].npairs, 1);
            if (k < c.pair_cap) {
              D.raw_i[c.pair_base + k] = lo;
              D.raw_j[c.pair_base + k] = hi;
            }
            const double er2 = __dadd_rn(__dadd_rn(__dmul_rn(ex, ex), __dmul_rn(ey, ey)), __dmul_rn(ez, ez));
            const float w = (float)g0_weight(c, R0, __dsqrt_rn(er2));
            sj *= w;
            si *= w;
          }
        }
      }
    } else {
      if (r.gid >= 0 && r.gid == gidj && valid) {
        const int lo = min(r.pi, jid), hi = max(r.pi, jid);
        if (group_has_pair(D, r.gid, lo, hi)) {
          const double R0 = __dmul_rn(c.lam, __dadd_rn(D.rh[lo], D.rh[hi]));
          const double ex = D.x[hi] - D.x[lo], ey = D.y[hi] - D.y[lo], ez = D.z[hi] - D.z[lo];
          const float w = (float)g0_weight(c, R0, sqrt(fma(ez, ez, fma(ey, ey, ex * ex))));
          sj *= w;
          si *= w;
        }
      }
    }
    if (!valid) { sj = 0.f; si = 0.f; }
    kahan(r.sx, r.cx, sj * dx); kahan(r.sy, r.cy, sj * dy); kahan(r.sz, r.cz, sj * dz);
    kahan(sxj, cxj, -si * dx); kahan(syj, cyj, -si * dy); kahan(szj, czj, -si * dz);
    if (!diag || s + 1 < nsteps) rotate();
  }
  if (diag) {
    const int src = (lane + 16) & 31;
    const float hx = __shfl_sync(FULL, sxj, src), hy = __shfl_sync(FULL, syj, src), hz = __shfl_sync(FULL, szj, src);
    const float kx = __shfl_sync(FULL, cxj, src), ky = __shfl_sync(FULL, cyj, src), kz = __shfl_sync(FULL, czj, src);
    kahan(r.sx, r.cx, hx); kahan(r.sx, r.cx, -kx);
    kahan(r.sy, r.cy, hy); kahan(r.sy, r.cy, -ky);
    kahan(r.sz, r.cz, hz); kahan(r.sz, r.cz, -kz);
    ox = make_float2(0.f, 0.f); oy = ox; oz = ox;
  } else {
    ox = make_float2(sxj, cxj); oy = make_float2(syj, cyj); oz = make_float2(szj, czj);
  }
}

// One CTA per macro-tile.  The macro-tile list entry is {system, first row block, first column block,
// end of the system's massive blocks}; the CTA's rows are blocks I0 .. I0 + 3 and its columns J0 ..
// J0 + SYM_MACRO_COLS - 1, without those below a row (the triangle) or past the massive blocks.  Rows
// and columns are written once per macro-tile, summed over warps in warp order through shared memory.
//
// FP64 systems: sixteen warps; warp w takes row block I0 + w % 4 and a quarter, w / 4, of the steps of
// each of its tiles, so that a system of a few blocks (one macro-tile per 128 x 64 bodies) still fills
// the SM it runs on: the 1,000-body disk has 80 macro-tiles for 152 SMs.
template <int MODE>
__global__ void __launch_bounds__(512) k_trap_df(const __grid_constant__ Dev D) {
  __shared__ ColDF col[MC][32];
  __shared__ float4 cf[MC][32][2];              // kick 1: xf, yf, zf, vxf | vyf, vzf, lambda, sigma
  __shared__ float2 rowbuf[16][3][32];          // [warp][component][lane]
  __shared__ float2 colbuf[16][MC][3][32];
  __shared__ float rowlost[16][32], collost[16][MC][32];
  __shared__ int s_max[4], s_min;               // high words of the largest |x|, |y|, |z|, G m; smallest G m > 0
  __shared__ int s_v[4 + MC][32];               // of each body's largest |v| component; -1: no live body
  __shared__ unsigned s_live[MC], s_mass[MC];
  __shared__ int s_item;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, wr = w & 3, ws = w >> 2;
  const int nmac = D.ntiles_total;
  const int S = D.seg_len;
  int *counter = &D.work[MODE - 1];
  if (threadIdx.x == 0) { s_item = atomicAdd(counter, 1); s_min = 0x7FFFFFFF; }
  if (threadIdx.x < 4) s_max[threadIdx.x] = 0;
  __syncthreads();
  int m0 = s_item * S;
  while (m0 < nmac) {
    const int m1 = min(m0 + S, nmac);
    for (int m = m0; m < m1; ++m) {
      const int4 mt = D.tiles[m];
      const TileCtx c = load_ctx(&D.disks[mt.x]);
      // the units and grids: largest |x|, component by component, and G m of the macro-tile's live bodies
      if (w < 4 + MC) {
        const int b = w < 4 ? mt.y + w : mt.z + (w - 4);
        const int p = b * 32 + lane;
        const bool in = b < mt.w && p - c.off < c.n && D.alive[p];
        const double *xs[4] = {D.x, D.y, D.z, D.gm};
        auto hi = [&](const double *a) { return in ? __double2hiint(a[p]) & 0x7FFFFFFF : 0; };
        s_v[w][lane] = in ? max(hi(D.vx), max(hi(D.vy), hi(D.vz))) : -1;
        int h = 0;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          h = hi(xs[k]);
          const int top = __reduce_max_sync(FULL, h);
          if (lane == 0) atomicMax(&s_max[k], top);
        }
        const int low = __reduce_min_sync(FULL, h ? h : 0x7FFFFFFF);
        if (lane == 0) atomicMin(&s_min, low);
      }
      __syncthreads();
      const Units u = units_of(s_max[0], s_max[1], s_max[2], s_max[3], s_min);
      const int E[3] = {grid_exp(s_max[0], u.kex), grid_exp(s_max[1], u.kex), grid_exp(s_max[2], u.kex)};
      if (w >= 16 - MC) {                       // the last warps stage the column blocks
        const int k = w - (16 - MC), b = mt.z + k, j = b * 32 + lane;
        const bool in = b < mt.w, live = in && j - c.off < c.n && D.alive[j];
        const unsigned ml = __ballot_sync(FULL, live), mm = __ballot_sync(FULL, live && j - c.off < c.nm);
        if (lane == 0) { s_live[k] = ml; s_mass[k] = mm; }
        if (in) {
          float g[3][3];
          const double p[3] = {D.x[j], D.y[j], D.z[j]};
#pragma unroll
          for (int q = 0; q < 3; ++q) on_grid(live ? p[q] : 0.0, E[q], u.kex, g[q][0], g[q][1], g[q][2]);
          const df gm = split(scale2(D.gm[j], -u.keg));
          col[k][lane].q[0] = make_float4(g[0][0], g[0][1], g[0][2], g[1][0]);
          col[k][lane].q[1] = make_float4(g[1][1], g[1][2], g[2][0], g[2][1]);
          col[k][lane].q[2] = make_float4(g[2][2], gm.h, gm.l, __int_as_float(MODE == 2 ? D.gid[j] : -1));
          if (MODE == 1) {
            cf[k][lane][0] = make_float4(D.xf[j], D.yf[j], D.zf[j], D.vxf[j]);
            cf[k][lane][1] = make_float4(D.vyf[j], D.vzf[j], D.lamf[j], D.sigf[j]);
          }
        }
      }
      const int I = mt.y + wr;
      const bool has_row = I < mt.w;
      RowDF r;
      if (has_row) row_load_df<MODE>(D, c, E, u, I, lane, r);
      __syncthreads();
#pragma unroll 1
      for (int k = 0; k < MC; ++k) {
        const int J = mt.z + k;
        if (has_row && J < mt.w && J >= I) {
          const int q = I == J ? 4 : 8;         // a quarter of 16 or 32 steps
          tile_steps_df<MODE>(D, c, mt.x, r, I, J, lane, q * ws, q * ws + q, col[k], cf[k], s_live[k], s_mass[k],
                              colbuf[w][k], collost[w][k]);
        } else {
#pragma unroll
          for (int q = 0; q < 3; ++q) colbuf[w][k][q][lane] = make_float2(0.0f, 0.0f);
          collost[w][k][lane] = 0.0f;
        }
      }
#pragma unroll
      for (int q = 0; q < 3; ++q) {
        const df a = has_row ? renorm(r.acc[q]) : mk(0.0f, 0.0f);
        rowbuf[w][q][lane] = make_float2(a.h, a.l);
      }
      rowlost[w][lane] = has_row ? r.lost : 0.0f;
      // the next item is taken while the sums are formed (everyone has read s_item)
      if (threadIdx.x < 4) s_max[threadIdx.x] = 0;
      if (threadIdx.x == 0) {
        s_min = 0x7FFFFFFF;
        if (m + 1 == m1) s_item = atomicAdd(counter, 1);
      }
      __syncthreads();
      double *part = D.part + (size_t)m * SYM_MACRO_PART;
      bool general = !u.fits;
      for (int i = threadIdx.x; i < SYM_MACRO_PART; i += 512) {     // [4 rows, MC columns][component][lane]
        const int blk = i / 96, q = (i / 32) % 3, l = i & 31;
        if (q == 0 && s_v[blk][l] >= 0) {
          float lost = 0.0f;
          if (blk < 4) {
#pragma unroll
            for (int v = 0; v < 4; ++v) lost += rowlost[4 * v + blk][l];
          } else {
#pragma unroll
            for (int v = 0; v < 16; ++v) lost += collost[v][blk - 4][l];
          }
          const int ng = (mt.w - (c.off >> 5) + MC - 1) / MC;       // at most ng + 1 sums for a body
          if (!(lost <= error_room(s_v[blk][l], c.dt, u, ng + 1))) general = true;
        }
        df a = mk(0.0f, 0.0f);
        if (blk < 4) {
#pragma unroll
          for (int v = 0; v < 4; ++v) accumulate(a, ld2(rowbuf[4 * v + blk][q][l]));
        } else {
#pragma unroll 4
          for (int v = 0; v < 16; ++v) accumulate(a, ld2(colbuf[v][blk - 4][q][l]));
        }
        part[i] = kick_value(a, u.keg - 2 * u.kex);
      }
      if (__syncthreads_or(general)) {          // (and the buffers are free)
        auto rows = reinterpret_cast<double (*)[3][32]>(rowbuf);
        auto cols = reinterpret_cast<double (*)[MC][3][32]>(colbuf);
        macro_general<MODE>(D, mt, col, cf, s_live, s_mass, rows, cols);
        __syncthreads();
        for (int i = threadIdx.x; i < SYM_MACRO_PART; i += 512) {
          const int blk = i / 96, q = (i / 32) % 3, l = i & 31;
          double a = 0.0;
          for (int v = blk < 4 ? blk : 0; v < 16; v += blk < 4 ? 4 : 1) a += blk < 4 ? rows[v][q][l] : cols[v][blk - 4][q][l];
          part[i] = a;
        }
        __syncthreads();
      }
    }
    m0 = s_item * S;
  }
}

template <int MODE>
__global__ void __launch_bounds__(128) k_trap_mixed(Dev D) {
  __shared__ float2 colbuf[4][MC][3][32];
  __shared__ int s_item;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int nmac = D.ntiles_total;
  const int S = D.seg_len;
  int *counter = &D.work[MODE - 1];
  float2 *part = reinterpret_cast<float2 *>(D.part);
  if (threadIdx.x == 0) s_item = atomicAdd(counter, 1);
  __syncthreads();
  int m0 = s_item * S;
  while (m0 < nmac) {
    const int m1 = min(m0 + S, nmac);
    for (int m = m0; m < m1; ++m) {
      const int4 mt = D.tiles[m];
      const TileCtx c = load_ctx(&D.disks[mt.x]);
      const int I = mt.y + w;
      const bool has_row = I < mt.w;
      RowMixed r;
      if (has_row) row_load_mixed<MODE>(D, c, I, lane, r);
#pragma unroll 1
      for (int k = 0; k < MC; ++k) {
        const int J = mt.z + k;
        float2 ox = make_float2(0.f, 0.f), oy = ox, oz = ox;
        if (has_row && J < mt.w && J >= I) tile_sweep_mixed<MODE>(D, c, mt.x, r, I, J, lane, ox, oy, oz);
        colbuf[w][k][0][lane] = ox; colbuf[w][k][1][lane] = oy; colbuf[w][k][2][lane] = oz;
      }
      float2 *rowp = part + part_row(m, w) + lane;
      const float2 z = make_float2(0.f, 0.f);
      rowp[0] = has_row ? make_float2(r.sx, r.cx) : z;
      rowp[32] = has_row ? make_float2(r.sy, r.cy) : z;
      rowp[64] = has_row ? make_float2(r.sz, r.cz) : z;
      __syncthreads();
      if (w < MC) {
        float2 *colp = part + part_col(m, w) + lane;
#pragma unroll
        for (int q = 0; q < 3; ++q) {
          float s = 0.f, cc = 0.f;
#pragma unroll
          for (int v = 0; v < 4; ++v) {
            const float2 t = colbuf[v][w][q][lane];
            kahan(s, cc, t.x);
            kahan(s, cc, -t.y);
          }
          colp[32 * q] = make_float2(s, cc);
        }
      }
      if (m + 1 == m1 && threadIdx.x == 0) s_item = atomicAdd(counter, 1);
      __syncthreads();
    }
    m0 = s_item * S;
  }
}

// kick CTAs per multiprocessor a schedule may ask for
int trap_blocks_per_sm(int precision) {
  if (precision != SYMBA_PRECISION_MIXED) return 4;
  int nb = 0;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_trap_mixed<1>, 128, 0);
  return nb > 8 ? 8 : (nb > 0 ? nb : 1);
}

// resident CTAs per multiprocessor, the schedule a pool starts with
int trap_blocks_default(int precision) {
  if (precision == SYMBA_PRECISION_MIXED) return trap_blocks_per_sm(precision);
  int nb = 0;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_trap_df<1>, 512, 0);
  return nb > 4 ? 4 : (nb > 0 ? nb : 1);
}

// No more CTAs than work items: with more, several on one SM could take an item each while other SMs
// had none (80 macro-tiles of the 1,000-body disk for 608 CTAs).
void launch_trap(const Dev &D, const LaunchCfg &L, int mode, int precision, cudaStream_t s) {
  if (D.ntiles_total <= 0) return;
  const int items = (D.ntiles_total + D.seg_len - 1) / D.seg_len;
  const int blocks = L.trap_blocks < items ? L.trap_blocks : items;
  if (precision == SYMBA_PRECISION_MIXED) {
    if (mode == 1) k_trap_mixed<1><<<blocks, 128, 0, s>>>(D);
    else k_trap_mixed<2><<<blocks, 128, 0, s>>>(D);
  } else {
    if (mode == 1) k_trap_df<1><<<blocks, 512, 0, s>>>(D);
    else k_trap_df<2><<<blocks, 512, 0, s>>>(D);
  }
}

// ---------------------------------------------------------------------------------------------
// The field rectangle (Sec. 2: field particles interact only with massive bodies).  The
// trapezoid's tiles cover the column blocks that hold massive bodies; every block of field
// particles beyond them is one row of the rectangle N_m x N_field: lane l owns field particle
// b*32 + l, the system's massive bodies stream through a per-warp shared-memory chunk of 32 (one
// coalesced load, then broadcast reads), and only the field particle's side is accumulated -- a
// massless body exerts no force, so the massive side and the per-tile partials of the trapezoid are
// not needed.  FP64 systems: four warps take every fourth chunk each and their sums are added in
// warp order; mixed: one warp takes all, in ascending order.  So the result does not depend on the
// launch or on other systems.  The kick v += (tau/2) a is applied at the end (the reduction skips
// these blocks).  Kick 1 runs the same
// fused encounter check as the tiles (FP32 prefilter, exact FP64 predicate, pair emission,
// g_0 weight); kick 2 weights the flagged pairs through the groups.
// ---------------------------------------------------------------------------------------------
struct FieldSrc {                              // mixed precision
  float xf, yf, zf, xl, yl, zl, gmf;           // FP32 copies, low parts, G m
  float vxf, vyf, vzf, lam, sig;               // kick 1 prefilter
  int id, ok, gid;
};

// stage massive bodies [c0, c0 + 32) of the system into the warp's chunk
template <int MODE>
__device__ __forceinline__ void stage_sources(const Dev &D, const TileCtx &c, int c0, int lane, FieldSrc *src) {
  const int li = c0 + lane;
  FieldSrc s;
  const int p = c.off + li;
  s.id = p;
  s.ok = (li < c.nm && D.alive[p]) ? 1 : 0;
  const int q = s.ok ? p : c.off;               // a valid address for the loads below
  s.xf = D.xf[q]; s.yf = D.yf[q]; s.zf = D.zf[q];
  s.xl = D.xl[q]; s.yl = D.yl[q]; s.zl = D.zl[q]; s.gmf = D.gmf[q];
  s.vxf = 0.f; s.vyf = 0.f; s.vzf = 0.f; s.lam = 0.f; s.sig = 0.f;
  if (MODE == 1) {
    s.vxf = D.vxf[q]; s.vyf = D.vyf[q]; s.vzf = D.vzf[q]; s.lam = D.lamf[q]; s.sig = D.sigf[q];
  }
  s.gid = MODE == 2 ? D.gid[q] : -1;
  src[lane] = s;
}

// the FP64 predicate of pair (i massive, p field) and, when flagged, its pair-list entry and
// level-0 weight (1 when not flagged)
__device__ __forceinline__ double field_check(const Dev &D, const TileCtx &c, int sys, int i, int p) {
  const double ex = __dsub_rn(D.x[p], D.x[i]), ey = __dsub_rn(D.y[p], D.y[i]), ez = __dsub_rn(D.z[p], D.z[i]);
  const double evx = __dsub_rn(D.vx[p], D.vx[i]), evy = __dsub_rn(D.vy[p], D.vy[i]),
               evz = __dsub_rn(D.vz[p], D.vz[i]);
  const double R0 = __dmul_rn(c.lam, __dadd_rn(D.rh[i], D.rh[p]));
  if (!encounter_exact(ex, ey, ez, evx, evy, evz, R0, c.dt)) return 1.0;
  const int k = atomicAdd(&D.stat[sys].npairs, 1);
  if (k < c.pair_cap) {
    D.raw_i[c.pair_base + k] = i;
    D.raw_j[c.pair_base + k] = p;
  }
  const double er2 = __dadd_rn(__dadd_rn(__dmul_rn(ex, ex), __dmul_rn(ey, ey)), __dmul_rn(ez, ez));
  return g0_weight(c, R0, __dsqrt_rn(er2));
}

// FP64 systems, in double-float as the tiles, with units of each chunk's own: one CTA per field block, its
// four warps each taking every fourth chunk of 32 massive bodies; a chunk's sum joins the warp's in FP64, the
// four sums are added in warp order.  A chunk where a particle's error may exceed its share of the rounding
// of v (as in the tiles) is taken again in FP64, bodies read where they lie:
template <int MODE>
static __device__ __noinline__ double3 field_chunk_general(const Dev &D, int sys, int p, bool live, int c0, const float4 (*cf)[2]) {
  const TileCtx c = load_ctx(&D.disks[sys]);
  const float tauf = __double2float_ru(c.dt);
  const double x = D.x[p], y = D.y[p], z = D.z[p];
  const int cnt = min(32, c.nm - c0);
  double3 a = make_double3(0.0, 0.0, 0.0);
  for (int s = 0; s < cnt; ++s) {
    const int id = c.off + c0 + s;
    const bool valid = live && D.alive[id];
    const double dx = D.x[id] - x, dy = D.y[id] - y, dz = D.z[id] - z;
    const double r2 = fma(dz, dz, fma(dy, dy, dx * dx));
    const double ri = rsqrt_fp64(r2);
    double wt = 1.0;
    if (valid && MODE == 1) {
      const float4 fa = cf[s][0], fq = cf[s][1];
      const float dxf = fa.x - D.xf[p], dyf = fa.y - D.yf[p], dzf = fa.z - D.zf[p];
      const float r2f = fmaf(dzf, dzf, fmaf(dyf, dyf, dxf * dxf));
      const float dvxf = fa.w - D.vxf[p], dvyf = fq.x - D.vyf[p], dvzf = fq.y - D.vzf[p];
      const float vmag = sqrtf(fmaf(dvzf, dvzf, fmaf(dvyf, dvyf, dvxf * dvxf)));
      const float Bf = fmaf(tauf, vmag, fq.z + D.lamf[p]) * 1.0000039f + 1.9073486e-6f * (fq.w + D.sigf[p]);
      if (!(r2f > Bf * Bf)) wt = flagged_weight(D, c, id, p);
    } else if (valid && D.gid[p] >= 0 && D.gid[p] == D.gid[id] && group_has_pair(D, D.gid[p], id, p)) {
      wt = g0_weight(c, __dmul_rn(c.lam, __dadd_rn(D.rh[id], D.rh[p])), sqrt(r2));
    }
    const double sp = valid && wt != 0.0 ? D.gm[id] * (ri * ri * ri) * wt : 0.0;
    a.x = fma(sp, dx, a.x); a.y = fma(sp, dy, a.y); a.z = fma(sp, dz, a.z);
  }
  return a;
}

template <int MODE>
__global__ void __launch_bounds__(128) k_field_df(const __grid_constant__ Dev D) {
  __shared__ ColDF col[4][32];
  __shared__ float4 cf[4][32][2];
  __shared__ int sid[4][32];
  __shared__ double sums[4][3][32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int2 fb = D.fblk[blockIdx.x];            // {system, global block}
  const TileCtx c = load_ctx(&D.disks[fb.x]);
  const int p = fb.y * 32 + lane;
  const int lp = p - c.off;
  const bool live = lp < c.n && D.alive[p];
  const double xp[3] = {D.x[p], D.y[p], D.z[p]};
  int top[3];
#pragma unroll
  for (int k = 0; k < 3; ++k)
    top[k] = (int)__reduce_max_sync(FULL, live ? (unsigned)__double2hiint(xp[k]) & 0x7FFFFFFFu : 0u);
  auto hi = [](double a) { return __double2hiint(a) & 0x7FFFFFFF; };
  const int hv = max(hi(D.vx[p]), max(hi(D.vy[p]), hi(D.vz[p])));
  const float xfp = D.xf[p], yfp = D.yf[p], zfp = D.zf[p];
  float vxfp = 0.f, vyfp = 0.f, vzfp = 0.f, lamp = 0.f, sigp = 0.f;
  int gidp = -1;
  if (MODE == 1) {
    vxfp = D.vxf[p]; vyfp = D.vyf[p]; vzfp = D.vzf[p]; lamp = D.lamf[p]; sigp = D.sigf[p];
  } else {
    gidp = D.gid[p];
  }
  const float tauf = __double2float_ru(c.dt);
  double tot[3] = {0.0, 0.0, 0.0};
  for (int c0 = 32 * w; c0 < c.nm; c0 += 128) {
    const int li = c0 + lane, j = c.off + li;
    const bool ok = li < c.nm && D.alive[j];
    const int jq = ok ? j : c.off;                // a valid address for the loads below
    const double xj[3] = {D.x[jq], D.y[jq], D.z[jq]};
    float g[3][3], gp[3][3];
    int t[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) t[k] = max(top[k], __reduce_max_sync(FULL, ok ? hi(xj[k]) : 0));
    const int hg = ok ? hi(D.gm[jq]) : 0;
    const Units u = units_of(t[0], t[1], t[2], __reduce_max_sync(FULL, hg), __reduce_min_sync(FULL, hg ? hg : 0x7FFFFFFF));
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const int E = grid_exp(t[k], u.kex);
      on_grid(ok ? xj[k] : 0.0, E, u.kex, g[k][0], g[k][1], g[k][2]);
      on_grid(live ? xp[k] : 0.0, E, u.kex, gp[k][0], gp[k][1], gp[k][2]);
    }
    const df gm = split(scale2(D.gm[jq], -u.keg));
    df acc[3] = {mk(0.0f, 0.0f), mk(0.0f, 0.0f), mk(0.0f, 0.0f)};
    float lost = 0.0f;
    __syncwarp();
    col[w][lane].q[0] = make_float4(g[0][0], g[0][1], g[0][2], g[1][0]);
    col[w][lane].q[1] = make_float4(g[1][1], g[1][2], g[2][0], g[2][1]);
    col[w][lane].q[2] = make_float4(g[2][2], gm.h, gm.l, __int_as_float(MODE == 2 ? D.gid[jq] : -1));
    sid[w][lane] = ok ? j : -1;
    if (MODE == 1) {
      cf[w][lane][0] = make_float4(D.xf[jq], D.yf[jq], D.zf[jq], D.vxf[jq]);
      cf[w][lane][1] = make_float4(D.vyf[jq], D.vzf[jq], D.lamf[jq], D.sigf[jq]);
    }
    __syncwarp();
    const int cnt = min(32, c.nm - c0);
#pragma unroll 1
    for (int s = 0; s < cnt; ++s) {
      const float4 q0 = col[w][s].q[0], q1 = col[w][s].q[1], q2 = col[w][s].q[2];
      const int id = sid[w][s];
      const bool valid = live && id >= 0;
      const df d[3] = {separation(q0.x, q0.y, q0.z, gp[0][0], gp[0][1], gp[0][2]),
                       separation(q0.w, q1.x, q1.y, gp[1][0], gp[1][1], gp[1][2]),
                       separation(q1.z, q1.w, q2.x, gp[2][0], gp[2][1], gp[2][2])};
      const df r2 = norm2(d);
      const df_root rt = root(r2);
      df sp = mul(mk(q2.y, q2.z), inverse_cube(rt));
      if (MODE == 1) {
        const float4 fa = cf[w][s][0], fq = cf[w][s][1];
        const float dxf = fa.x - xfp, dyf = fa.y - yfp, dzf = fa.z - zfp;
        const float r2f = fmaf(dzf, dzf, fmaf(dyf, dyf, dxf * dxf));
        const float dvxf = fa.w - vxfp, dvyf = fq.x - vyfp, dvzf = fq.y - vzfp;
        const float vmag = sqrtf(fmaf(dvzf, dvzf, fmaf(dvyf, dvyf, dvxf * dvxf)));
        const float Bf = fmaf(tauf, vmag, fq.z + lamp) * 1.0000039f + 1.9073486e-6f * (fq.w + sigp);
        const bool cand = valid && !(r2f > Bf * Bf);
        if (__any_sync(FULL, cand)) {
          if (cand) {
            const double wt = field_check(D, c, fb.x, id, p);
            if (wt != 1.0) sp = weighted(sp, wt);
          }
          __syncwarp();
        }
      } else if (gidp >= 0 && gidp == __float_as_int(q2.w) && valid) {
        if (group_has_pair(D, gidp, id, p)) {
          const double R0 = __dmul_rn(c.lam, __dadd_rn(D.rh[id], D.rh[p]));
          const double ex = D.x[p] - D.x[id], ey = D.y[p] - D.y[id], ez = D.z[p] - D.z[id];
          sp = weighted(sp, g0_weight(c, R0, sqrt(fma(ez, ez, fma(ey, ey, ex * ex)))));
        }
      }
      sp.h = valid ? sp.h : 0.0f;
      sp.l = valid ? sp.l : 0.0f;
#pragma unroll
      for (int k = 0; k < 3; ++k) accumulate(acc[k], mul(sp, d[k]));
      lost = fmaf(fabsf(sp.h), fminf(fmaf(r2.h, rt.y, GRID_TERM), 8.0f), lost);
    }
    const bool good = u.fits && (!live || lost <= error_room(hv, c.dt, u, (c.nm + 31) / 32));
    if (__all_sync(FULL, good)) {
#pragma unroll
      for (int k = 0; k < 3; ++k) tot[k] += kick_value(acc[k], u.keg - 2 * u.kex);
    } else {
      const double3 a = field_chunk_general<MODE>(D, fb.x, p, live, c0, cf[w]);
      tot[0] += a.x; tot[1] += a.y; tot[2] += a.z;
    }
  }
#pragma unroll
  for (int k = 0; k < 3; ++k) sums[w][k][lane] = tot[k];
  __syncthreads();
  if (w < 3 && live) {                           // warp w adds component w
    const double a = (sums[0][w][lane] + sums[1][w][lane]) + (sums[2][w][lane] + sums[3][w][lane]);
    double *vel = w == 0 ? D.vx : (w == 1 ? D.vy : D.vz);
    vel[p] = __dadd_rn(vel[p], __dmul_rn(0.5 * c.dt, a));
  }
}

// Mixed precision: the same rectangle with the FP32 pair arithmetic of tile_mixed (two-float
// displacement, FP32 rsqrt and one Newton step, Kahan-compensated FP32 sums carried into FP64
// once); the encounter check is the FP64 one.
template <int MODE>
__global__ void __launch_bounds__(128) k_field_mixed(Dev D) {
  __shared__ FieldSrc chunk[4][32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int e = blockIdx.x * 4 + w;
  if (e >= D.nfblk) return;
  const int2 fb = D.fblk[e];
  const TileCtx c = load_ctx(&D.disks[fb.x]);
  FieldSrc *src = chunk[w];
  const int p = fb.y * 32 + lane;
  const int lp = p - c.off;
  const bool live = lp < c.n && D.alive[p];
  const float xhp = D.xf[p], yhp = D.yf[p], zhp = D.zf[p];
  const float xlp = D.xl[p], ylp = D.yl[p], zlp = D.zl[p];
  float vxfp = 0.f, vyfp = 0.f, vzfp = 0.f, lamp = 0.f, sigp = 0.f;
  int gidp = -1;
  if (MODE == 1) {
    vxfp = D.vxf[p]; vyfp = D.vyf[p]; vzfp = D.vzf[p]; lamp = D.lamf[p]; sigp = D.sigf[p];
  } else {
    gidp = D.gid[p];
  }
  const float tauf = __double2float_ru(c.dt);
  float sx = 0.f, sy = 0.f, sz = 0.f, cx = 0.f, cy = 0.f, cz = 0.f;
  for (int c0 = 0; c0 < c.nm; c0 += 32) {
    __syncwarp();
    stage_sources<MODE>(D, c, c0, lane, src);
    __syncwarp();
    const int cnt = min(32, c.nm - c0);
#pragma unroll 1
    for (int s = 0; s < cnt; ++s) {
      const FieldSrc &q = src[s];
      const bool valid = live && q.ok;
      const float dx = (q.xf - xhp) + (q.xl - xlp);
      const float dy = (q.yf - yhp) + (q.yl - ylp);
      const float dz = (q.zf - zhp) + (q.zl - zlp);
      const float r2 = fmaf(dz, dz, fmaf(dy, dy, dx * dx));
      float ri;
      asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(ri) : "f"(r2));
      ri = ri * fmaf(-0.5f * r2, ri * ri, 1.5f);
      float sp = q.gmf * (ri * ri * ri);
      if (MODE == 1) {
        const float dvxf = q.vxf - vxfp, dvyf = q.vyf - vyfp, dvzf = q.vzf - vzfp;
        const float vmag = sqrtf(fmaf(dvzf, dvzf, fmaf(dvyf, dvyf, dvxf * dvxf)));
        const float Bf = fmaf(tauf, vmag, q.lam + lamp) * 1.0000039f + 1.9073486e-6f * (q.sig + sigp);
        const bool cand = valid && !(r2 > Bf * Bf * 1.0000153f);
        if (__any_sync(FULL, cand)) {
          if (cand) sp *= (float)field_check(D, c, fb.x, q.id, p);
        }
      } else if (gidp >= 0 && gidp == q.gid && valid) {
        if (group_has_pair(D, gidp, q.id, p)) {
          const double R0 = __dmul_rn(c.lam, __dadd_rn(D.rh[q.id], D.rh[p]));
          const double ex = D.x[p] - D.x[q.id], ey = D.y[p] - D.y[q.id], ez = D.z[p] - D.z[q.id];
          sp *= (float)g0_weight(c, R0, sqrt(fma(ez, ez, fma(ey, ey, ex * ex))));
        }
      }
      if (!valid) sp = 0.f;
      kahan(sx, cx, sp * dx); kahan(sy, cy, sp * dy); kahan(sz, cz, sp * dz);
    }
  }
  if (live) {
    const double h = 0.5 * c.dt;
    D.vx[p] = fma(h, (double)sx - (double)cx, D.vx[p]);
    D.vy[p] = fma(h, (double)sy - (double)cy, D.vy[p]);
    D.vz[p] = fma(h, (double)sz - (double)cz, D.vz[p]);
  }
}

void launch_field(const Dev &D, int mode, int precision, cudaStream_t s) {
  if (D.nfblk <= 0) return;
  if (precision == SYMBA_PRECISION_MIXED) {
    const int blocks = (D.nfblk + 3) / 4;
    if (mode == 1) k_field_mixed<1><<<blocks, 128, 0, s>>>(D);
    else k_field_mixed<2><<<blocks, 128, 0, s>>>(D);
  } else {
    if (mode == 1) k_field_df<1><<<D.nfblk, 128, 0, s>>>(D);
    else k_field_df<2><<<D.nfblk, 128, 0, s>>>(D);
  }
}
