// Double-float evaluation of two Nystrom entries of one target (adjacent
// sources j, j + 1) with omega r >= 20, in packed FP32 pairs (pair32.cuh): used
// by the true-residual matvecs (matvec_df.cu).
//
// A double-float d2 is an unevaluated sum h + l of two FP32 values, here for
// both sources at once.  Products and sums use error-free transformations
// (TwoProd with fma, TwoSum, FastTwoSum where the larger operand is known); the
// low part is renormalised only where it would cost accuracy (before it is
// multiplied on at full weight), so a product takes 4 operations and a sum 8
// instead of 7 and 11.
//
//  * Coordinates are stored times omega in three parts, x = h + m + l: h on the
//    grid 2^(e - 23) where every omega |x|, omega |y| < 2^e, m the rest on the grid
//    2^(e - 47), so that the differences of both are exact, and l what is left.
//  * The phase omega r - pi/4 is reduced by a multiple of 2 pi / 1024 in one step:
//    J C1 (C1 the FP32 2 pi / 1024) subtracts exactly by fma, because the result is
//    a multiple of 2^-31 below 2^-8; the rest of the constant follows as J C2, J C3.
//    A table in shared memory holds sine and cosine of J 2 pi / 1024 - pi / 4; with
//    |d| <= pi / 1024, sin d - d needs FP32 only (2e-6 d) and cos d - 1 two terms.
//  * Hankel's asymptotic expansion (A&S 9.2.5, 9.2.9, 9.2.10) carries its leading
//    terms in double-float and the small corrections in FP32: for omega r >= 64
//    four terms of P and Q; pairs with 20 <= omega r < 64 (next to the band) are
//    redone one by one with seven and their first corrections in double-float.
//    The dropped terms are below 1e-13.
#pragma once

#include "pair32.cuh"

constexpr float kXD = 20.0f;   // asymptotic expansion for omega r >= 20
// Short series (small terms in FP32) from here on: at 48 the products were off by up
// to 1.3 times as much as with full series (2.5e-13 against 2.1e-13, ellipse n = 592),
// at 64 by less than those (1.2e-13) for 0.6 to 1.6 % more time.
constexpr float kXS = 64.0f;
constexpr int kDfTab = 1024;   // (sin h, l, cos h, l) of 2 pi j / 1024 - pi / 4

// ---------------------------------------------------------------------------
// scalar double-float (drains, running sums, the 20 <= omega r < 64 series)
// ---------------------------------------------------------------------------
struct df {
  float h, l;
};
__device__ __forceinline__ df quick(float a, float b) {
  const float s = a + b;
  return {s, b - (s - a)};
}
__device__ __forceinline__ df dadd(df a, df b) {
  const float s = a.h + b.h;
  const float v = s - a.h;
  const float e = (a.h - (s - v)) + (b.h - v) + a.l + b.l;
  return quick(s, e);
}
__device__ __forceinline__ df dneg(df a) { return {-a.h, -a.l}; }
__device__ __forceinline__ df dsub(df a, df b) { return dadd(a, dneg(b)); }
__device__ __forceinline__ df dmul(df a, df b) {
  const float p = a.h * b.h;
  float e = fmaf(a.h, b.h, -p);
  e = fmaf(a.h, b.l, e);
  e = fmaf(a.l, b.h, e);
  return quick(p, e);
}
__device__ __forceinline__ df dmulf(df a, float b) {
  const float p = a.h * b;
  float e = fmaf(a.h, b, -p);
  e = fmaf(a.l, b, e);
  return quick(p, e);
}
__host__ __device__ __forceinline__ df dmake(double v) {
  const float h = (float)v;
  return {h, (float)(v - (double)h)};
}

// packed double-float, one of its two lanes
__device__ __forceinline__ df lane0(d2 a) { return {a.h.x, a.l.x}; }
__device__ __forceinline__ df lane1(d2 a) { return {a.h.y, a.l.y}; }

// x = omega r, t = 1 / x and ra = x^(-1/2), j_m and y_m with J_m = c0 ra j_m,
// Y_m = c0 ra y_m (c0 = sqrt(2 / pi)), dx, dy = omega (z_i - z_j)
struct df_hankel2 {
  d2 dx, dy, t, ra, j0, y0, j1, y1;
};

// one source with 20 <= omega r < 64 (t = 1/x, sine and cosine of the phase):
// terms up to t^14 (P) and t^15 (Q), the first omitted one below 1e-14 at x =
// 20; the t^2 term of P and the t^3 term of Q (up to 2e-4 and 1e-5 there) in
// double-float
__device__ __forceinline__ void df_near_series(df t, df sn, df cs, df& j0, df& y0, df& j1,
                                               df& y1) {
  const df u2 = dmul(t, t), u3 = dmul(u2, t);
  const float u = u2.h;
  const float p0 = u * u * (0.112152099609375f + u * (-0.5725014209747314f +
                   u * (6.074042001273483f + u * (-110.01714026924674f +
                   u * (3038.090510922384f + u * -118838.42625678325f)))));
  const float p1 = u * u * (-0.144195556640625f + u * (0.6765925884246826f +
                   u * (-6.883914268109947f + u * (121.59789187653587f +
                   u * (-3302.2722944808525f + u * 127641.2726461746f)))));
  const float q0 = u3.h * u * (-0.22710800170898438f + u * (1.7277275025844574f +
                   u * (-24.380529699556064f + u * (551.3358961220206f +
                   u * (-18257.755474293175f + u * 832859.3040162893f)))));
  const float q1 = u3.h * u * (0.2775764465332031f + u * (-1.993531733751297f +
                   u * (27.248827311268542f + u * (-603.8440767050702f +
                   u * (19718.37591223663f + u * -890297.8767070678f)))));
  df P0 = dadd({1.0f, 0.f}, dmulf(u2, -0.0703125f));
  P0 = quick(P0.h, P0.l + p0);
  df P1 = dadd({1.0f, 0.f}, dmulf(u2, 0.1171875f));
  P1 = quick(P1.h, P1.l + p1);
  df Q0 = dadd({-0.125f * t.h, -0.125f * t.l}, dmulf(u3, 0.0732421875f));
  Q0 = quick(Q0.h, Q0.l + q0);
  df Q1 = dadd(dmulf(t, 0.375f), dmulf(u3, -0.1025390625f));
  Q1 = quick(Q1.h, Q1.l + q1);
  j0 = dsub(dmul(P0, cs), dmul(Q0, sn));
  y0 = dadd(dmul(P0, sn), dmul(Q0, cs));
  j1 = dadd(dmul(P1, sn), dmul(Q1, cs));
  y1 = dsub(dmul(Q1, sn), dmul(P1, cs));
}

// a + p a.h + q b, |p a.h|, |q b| << 1: one of the four combinations of P = 1 +
// p, Q = q with sine and cosine, normalised
__device__ __forceinline__ d2 df_combine(d2 a, float2 p, d2 q, d2 b) {
  const float2 m = mul2(q.h, b.h);
  float2 e = fma2(q.h, b.h, neg2(m));
  e = fma2(q.h, b.l, e);
  e = fma2(q.l, b.h, e);
  const d2 s = two_sum(a.h, m);
  return fast_sum(s.h, fma2(p, a.h, add2(s.l, add2(a.l, e))));
}

// (tx, ty) the target's coordinates in three parts each, s0, s1, s2 the
// sources' negated ones by pairs: (xh xh' xm xm'), (xl xl' yh yh'), (ym ym' yl yl')
__device__ __forceinline__ df_hankel2 hankel_df2(float3 tx, float3 ty, float4 s0, float4 s1,
                                                 float4 s2, const float4* __restrict__ tab) {
  df_hankel2 H;
  {
    const d2 x = fast_sum(add2(f2(tx.x), lo2(s0)), add2(f2(tx.y), hi2(s0)));   // exact parts
    const d2 y = fast_sum(add2(f2(ty.x), hi2(s1)), add2(f2(ty.y), lo2(s2)));
    H.dx = {x.h, add2(x.l, add2(f2(tx.z), lo2(s1)))};
    H.dy = {y.h, add2(y.l, add2(f2(ty.z), hi2(s2)))};
  }
  // x^2
  const float2 px = mul2(H.dx.h, H.dx.h), py = mul2(H.dy.h, H.dy.h);
  const float2 ex = fma2(add2(H.dx.h, H.dx.h), H.dx.l, fma2(H.dx.h, H.dx.h, neg2(px)));
  const float2 ey = fma2(add2(H.dy.h, H.dy.h), H.dy.l, fma2(H.dy.h, H.dy.h, neg2(py)));
  const d2 xs = two_sum(px, py);
  const float2 xl = add2(xs.l, add2(ex, ey));
  // x = r + c: r = x^2 y with y ~ 1/x (one Newton step on the special-function
  // unit's value, so that x^2 - r^2 needs few bits), c = (x^2 - r^2) y / 2
  const float2 ya = make_float2(rsqrt_sfu(xs.h.x), rsqrt_sfu(xs.h.y));
  const float2 y = mul2(ya, fma2(mul2(mul2(xs.h, f2(-0.5f)), ya), ya, f2(1.5f)));
  const float2 r = mul2(xs.h, y);
  const float2 er = add2(fma2(neg2(r), r, xs.h), xl);
  const d2 x = fast_sum(r, mul2(er, mul2(y, f2(0.5f))));
  // t = 1 / x = y (1 + e + e^2), e = 1 - x y
  {
    const float2 e = fma2(neg2(x.l), y, fma2(neg2(x.h), y, f2(1.0f)));
    H.t = fast_sum(y, mul2(fma2(e, e, e), y));
  }
  // ra = x^(-1/2) = z (1 + e/2 + 3 e^2 / 8), e = 1 - x z^2
  {
    const float2 z = make_float2(rsqrt_sfu(x.h.x), rsqrt_sfu(x.h.y));
    const float2 zz = mul2(z, z), ze = fma2(z, z, neg2(zz)), nx = neg2(x.h);
    float2 e = fma2(nx, zz, f2(1.0f));
    e = fma2(nx, ze, e);
    e = fma2(neg2(x.l), zz, e);
    H.ra = fast_sum(z, mul2(mul2(e, fma2(e, f2(0.375f), f2(0.5f))), z));
  }
  // phase
  d2 sn, cs;
  {
    constexpr float C1 = 0.006135923322290182f, C2 = -1.7074761049507003e-10f,
                    C3 = -6.699705117210476e-18f;
    const float2 u = mul2(x.h, f2(162.97466172610083f));   // 1024 / (2 pi)
    const int k0 = __float2int_rn(u.x), k1 = __float2int_rn(u.y);
    const float2 J = make_float2((float)k0, (float)k1);
    const float4 t0 = tab[k0 & (kDfTab - 1)], t1 = tab[k1 & (kDfTab - 1)];
    const float2 nJ = neg2(J);
    const float2 d1 = fma2(nJ, f2(C1), x.h);               // exact
    const float2 p = mul2(nJ, f2(C2));
    const float2 pe = fma2(nJ, f2(C3), fma2(nJ, f2(C2), neg2(p)));
    const d2 ds = two_sum(d1, p);
    const d2 d = fast_sum(ds.h, add2(ds.l, add2(x.l, pe)));
    // sin d = (d.h, sl), cos d - 1 = (ch, cl)
    const float2 z = mul2(d.h, d.h);
    const float2 sl = fma2(mul2(d.h, z), fma2(z, f2(1.0f / 120.0f), f2(-1.0f / 6.0f)), d.l);
    const float2 zl = fma2(add2(d.h, d.h), d.l, fma2(d.h, d.h, neg2(z)));
    const float2 ch = mul2(z, f2(-0.5f));
    const float2 cl = fma2(mul2(z, z), f2(1.0f / 24.0f), mul2(zl, f2(-0.5f)));
    // table angle plus d: S + (C sin d + S (cos d - 1)), the bracket with its
    // rounding error (|S (cos d - 1)| <= |C sin d| or that is zero)
    const float2 Sh = make_float2(t0.x, t1.x), Sl = make_float2(t0.y, t1.y);
    const float2 Ch = make_float2(t0.z, t1.z), Cl = make_float2(t0.w, t1.w);
    auto turn = [&](float2 Ah, float2 Al, float2 Bh, float2 Bl) {   // A + B sin d + A (cos d - 1)
      const float2 q0 = mul2(Bh, d.h);
      const float2 q = fma2(Ah, ch, q0);
      float2 e = fma2(Ah, ch, sub2(q0, q));
      e = add2(e, fma2(Bh, d.h, neg2(q0)));
      e = fma2(Bh, sl, e);
      e = fma2(Bl, d.h, e);
      e = fma2(Ah, cl, e);
      e = fma2(Al, ch, e);
      const d2 s = fast_sum(Ah, q);
      return d2{s.h, add2(s.l, add2(Al, e))};
    };
    sn = turn(Sh, Sl, Ch, Cl);
    cs = turn(Ch, Cl, neg2(Sh), neg2(Sl));
  }
  // x >= 64: terms up to t^8 (P) and t^7 (Q), the corrections in FP32 (t^2 with
  // the lo part of t: its FP32 error, times the 0.07 t^2 term, stays below 3e-12
  // of P)
  const float2 th = H.t.h;
  const float2 u = fma2(th, th, mul2(add2(th, th), H.t.l));
  const float2 p0 = mul2(u, fma2(u, fma2(u, fma2(u, f2(6.074042001273483f), f2(-0.5725014209747314f)),
                                         f2(0.112152099609375f)), f2(-0.0703125f)));
  const float2 p1 = mul2(u, fma2(u, fma2(u, fma2(u, f2(-6.883914268109947f), f2(0.6765925884246826f)),
                                         f2(-0.144195556640625f)), f2(0.1171875f)));
  const float2 tu = mul2(th, u);
  const float2 q0 = fma2(u, fma2(u, f2(1.7277275025844574f), f2(-0.22710800170898438f)),
                         f2(0.0732421875f));
  const float2 q1 = fma2(u, fma2(u, f2(-1.993531733751297f), f2(0.2775764465332031f)),
                         f2(-0.1025390625f));
  d2 Q0, Q1;
  Q0.h = mul2(th, f2(-0.125f));
  Q0.l = fma2(tu, q0, mul2(H.t.l, f2(-0.125f)));
  Q1.h = mul2(th, f2(0.375f));
  Q1.l = fma2(tu, q1, fma2(H.t.l, f2(0.375f), fma2(th, f2(0.375f), neg2(Q1.h))));
  H.j0 = df_combine(cs, p0, dd_neg(Q0), sn);
  H.y0 = df_combine(sn, p0, Q0, cs);
  H.j1 = df_combine(sn, p1, Q1, cs);
  H.y1 = dd_neg(df_combine(cs, p1, dd_neg(Q1), sn));
  if (fminf(x.h.x, x.h.y) < kXS) {
    df j0, y0, j1, y1;
    if (x.h.x < kXS) {
      df_near_series(lane0(H.t), lane0(sn), lane0(cs), j0, y0, j1, y1);
      H.j0.h.x = j0.h, H.j0.l.x = j0.l, H.y0.h.x = y0.h, H.y0.l.x = y0.l;
      H.j1.h.x = j1.h, H.j1.l.x = j1.l, H.y1.h.x = y1.h, H.y1.l.x = y1.l;
    }
    if (x.h.y < kXS) {
      df_near_series(lane1(H.t), lane1(sn), lane1(cs), j0, y0, j1, y1);
      H.j0.h.y = j0.h, H.j0.l.y = j0.l, H.y0.h.y = y0.h, H.y0.l.y = y0.l;
      H.j1.h.y = j1.h, H.j1.l.y = j1.l, H.y1.h.y = y1.h, H.y1.l.y = y1.l;
    }
  }
  return H;
}

// Per-node double-float data, built by df_prepare:
//  tgt  2 float4 per node: omega (x, y) in three parts each, (h, m, l, 0)
//  tq   float4 per node (hard): omega nu / |z'| as (x h, x l, y h, y l)
//  src  6 float4 per pair of nodes j, j + 1: the negated coordinates as above,
//       then the factors (a h h', a l l'), (b h h', b l l'), (c h h', c l l')
//       with hq = h / 4, nu the unnormalised normal, |z'| the speed:
//       soft (a, b) = omega hq c0 nu, c = hq c0 eta |z'|;
//       hard (a, b) = (omega / eta) nu / |z'|, c = hq c0 |z'|
//  w    2 n entries by i - j + n: Kress weights / (pi h) of j and j + 1 (h h' l l')
struct df_nodes {
  const float4 *tgt, *tq, *src, *w, *tab;
};

// Entries of two far pairs, target (tx, ty, tq), sources from sp:
//   OP_SOFT (eq. 1): A = c ra, B = (a, b).(dx, dy) ra / x,
//                    re = A j0 - B w1, im = A w0 + B j1
//   OP_S:  S' = -i S of eq. 2:  re = A j0, im = A w0
//   OP_C:  C = -D' + kn S', D = tq.(dx, dy) A / x, kn = tq.(a, b) = (omega^2 / eta)
//          n_i . n_j:  re = kn A j0 - D w1, im = kn A w0 + D j1
//   OP_SC: both (S' in re, im; C in re2, im2)
// with w0 = y0 + wk j0, w1 = y1 + wk j1 (see pair32.cuh).
struct df_entry2 {
  d2 re, im, re2, im2;
};

template <int OP>
__device__ __forceinline__ df_entry2 entry_df2(float3 tx, float3 ty, float4 tq,
                                               const float4* __restrict__ sp, float4 w,
                                               const float4* __restrict__ tab) {
  const df_hankel2 H = hankel_df2(tx, ty, __ldg(sp), __ldg(sp + 1), __ldg(sp + 2), tab);
  const float4 fa = __ldg(sp + 3), fb = __ldg(sp + 4), fc = __ldg(sp + 5);
  const d2 a = {lo2(fa), hi2(fa)}, b = {lo2(fb), hi2(fb)}, c = {lo2(fc), hi2(fc)};
  const d2 wk = {lo2(w), hi2(w)};
  df_entry2 e;
  const d2 A = dd_mul(c, H.ra);
  const d2 w0 = dd_norm(dd_add(H.y0, dd_mul(wk, H.j0)));
  if constexpr (OP == OP_SOFT) {
    const d2 w1 = dd_norm(dd_add(H.y1, dd_mul(wk, H.j1)));
    const d2 p = dd_add(dd_mul(H.dx, a), dd_mul(H.dy, b));
    const d2 B = dd_mul(p, dd_mul(H.t, H.ra));
    e.re = dd_norm(dd_add(dd_mul(A, H.j0), dd_neg(dd_mul(B, w1))));
    e.im = dd_norm(dd_add(dd_mul(A, w0), dd_mul(B, H.j1)));
  } else {
    const d2 sr = dd_mul(A, H.j0), si = dd_mul(A, w0);
    if constexpr (OP == OP_S || OP == OP_SC) {
      e.re = dd_norm(sr);
      e.im = dd_norm(si);
    }
    if constexpr (OP == OP_C || OP == OP_SC) {
      const d2 w1 = dd_norm(dd_add(H.y1, dd_mul(wk, H.j1)));
      const d2 ux = {f2(tq.x), f2(tq.y)}, uy = {f2(tq.z), f2(tq.w)};
      const d2 p = dd_add(dd_mul(H.dx, ux), dd_mul(H.dy, uy));
      const d2 D = dd_mul(p, dd_mul(H.t, A));
      const d2 kn = dd_add(dd_mul(ux, a), dd_mul(uy, b));
      const d2 cr = dd_norm(dd_add(dd_mul(kn, sr), dd_neg(dd_mul(D, w1))));
      const d2 ci = dd_norm(dd_add(dd_mul(kn, si), dd_mul(D, H.j1)));
      if constexpr (OP == OP_C) {
        e.re = cr;
        e.im = ci;
      } else {
        e.re2 = cr;
        e.im2 = ci;
      }
    }
  }
  return e;
}
