// FP32 evaluation of one Nystrom entry pair with omega r >= kX0 (shared by the
// fused matrix-free matvec and the stored-matrix assembly).  See the header
// comment of matvec_fp32.cu for the two-float phase and the asymptotic
// Hankel expansion (A&S 9.2.5, 9.2.9, 9.2.10).
#pragma once
#include "packed32.cuh"

// FP32 geometry of an operator: coordinates times omega as hi/lo pairs,
// unnormalised normal, speed.
// Stored in one buffer: 8 n floats xh, xl, yh, yl, nx, ny, sp, w32 (Kress
// table); then, for the fused tensor-core kernel, starting on 16-byte boundaries:
//   n float4 coordinates      (omega x hi, lo, omega y hi, lo)
//   n float4 source factors   (omega hq c0 nu1, omega hq c0 nu2, hq c0 eta |z'|, hq c0 |z'|)
//   n float4 target factors   2 omega (nu1, nu2) / |z'|, 0, 0
//   2 n + 8 float2: the Kress table twice over divided by pi h, entry
//   k = i - j + n holding the weights of sources j and j + 1,
//   (w_{k mod n}, w_{(k - 1) mod n}) / (pi h), then zeros
//   n float4 source coordinates by pairs j, j + 1 (n is even), negated:
//   (-xh_j, -xh_j+1, -xl_j, -xl_j+1), (-yh_j, ..)
//   n float4 source factors by pairs, (a_j, a_j+1, b_j, b_j+1), (c_j, c_j+1, 0, 0):
//   soft a, b = 2 omega hq c0 nu, c = hq c0 eta |z'|; hard a, b = (omega / (2 eta))
//   nu / |z'|, c = hq c0 |z'|
// (the entries of pairs carry 1 / (2 x) in the place of 1 / x)
// with hq = h / 4 and c0 = sqrt(2 / pi) (nu = unnormalised normal, |z'| = speed).
struct geo32 {
  float *xh, *xl, *yh, *yl, *nx, *ny, *sp;
};

inline size_t geo32_pack_offset(int n) { return ((size_t)8 * n + 3) & ~size_t(3); }
inline size_t geo32_wk_offset(int n) { return geo32_pack_offset(n) + (size_t)12 * n; }
inline size_t geo32_pair_offset(int n) {
  return (geo32_wk_offset(n) + (size_t)4 * n + 16 + 3) & ~size_t(3);
}
// (+ 256 floats of slack: the fused kernel copies whole 32-source tiles)
inline size_t geo32_floats(int n) { return geo32_pair_offset(n) + (size_t)8 * n + 256; }

// the last float: bit pattern of the largest |x|, |y| over the nodes
inline size_t geo32_bound_offset(int n) { return geo32_floats(n) - 1; }

inline geo32 geo32_at(float* base, int n) {
  return geo32{base, base + n, base + 2 * n, base + 3 * n, base + 4 * n, base + 5 * n,
               base + 6 * n};
}

// omega (FP32), eta, h = 2 pi / n: the operator constants of the generic
// entries (the phase comes from the omega-scaled coordinates)
struct omega32 {
  float wh, eta, h;
};

constexpr float kX0 = 16.0f;  // asymptotic expansion used for omega r >= kX0

// Cody-Waite split of 2 pi: C1 has 10 significant bits
constexpr float kC1 = 6.28125f;
constexpr float kC2 = 0.0019353071693331003f;
constexpr float kC3 = 1.0253131677018246e-11f;
constexpr float kPi4H = 0.7853981852531433f;
constexpr float kPi4L = -2.1855695031547384e-08f;
constexpr float kInv2Pi = 0.15915493667125702f;
constexpr float kSqrt2OverPi = 0.7978845834732056f;
constexpr float kInv4Pi = 0.07957747154594767f;

// Special-function-unit approximations without subnormal handling: their
// arguments here are >= 16 (square roots) or reduced phases, never subnormal
__device__ __forceinline__ float rsqrt_sfu(float x) {
  float y;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ void sincos_sfu(float x, float* s, float* c) {
  asm("sin.approx.ftz.f32 %0, %1;" : "=f"(*s) : "f"(x));
  asm("cos.approx.ftz.f32 %0, %1;" : "=f"(*c) : "f"(x));
}

// Distance and phase of one pair with omega r >= kX0.  Coordinates are scaled
// by omega, so the distance of two nodes is the Hankel argument x = omega r
// itself, and split as hi + lo with the hi parts on a grid coarse enough that
// the difference of two of them and the sum of the two squared differences
// are exact in FP32 (geometry set-up).  Then x^2 = H + C with H = dxh^2 + dyh^2
// exact and the lo-part terms C = dxl (2 dxh + dxl) + dyl (2 dyh + dyl) in
// FP32; x^2 and x are carried as two-float numbers (error-free
// transformations built from fmaf), and chi = x - pi/4 is reduced modulo 2 pi
// with a three-part Cody-Waite constant.  Phase error ~2^(e - 33) rad when
// omega |z| < 2^e (6.5e-7 rad at most for the kite at omega = 2048).
struct pair_phase {
  float dx, dy;   // omega (z_i - z_j)
  float xinv;     // 1 / (omega r)
  float ra;       // (omega r)^(-1/2)
  float s, c;     // sin, cos of omega r - pi / 4
};

__device__ __forceinline__ pair_phase pair_phase32(float txh, float txl, float tyh, float tyl,
                                                   float sxh, float sxl, float syh, float syl) {
  pair_phase f;
  const float dxh = txh - sxh, dxl = txl - sxl;   // dxh, dyh exact
  const float dyh = tyh - syh, dyl = tyl - syl;
  const float H = fmaf(dxh, dxh, dyh * dyh);      // exact
  const float C = fmaf(dxl, fmaf(2.0f, dxh, dxl), dyl * fmaf(2.0f, dyh, dyl));
  // x^2 = H + C as two-float (TwoSum)
  const float x2 = H + C;
  const float bv = x2 - H;
  const float x2l = (H - (x2 - bv)) + (C - bv);
  const float xinv = rsqrt_sfu(x2);
  const float xh = x2 * xinv;
  // x lo, less the lo part of the pi/4 split
  const float xl4 = fmaf(fmaf(-xh, xh, x2) + x2l, 0.5f * xinv, -kPi4L);
  // chi = x - pi/4 reduced to [-pi, pi]
  const float k = rintf(fmaf(xh, kInv2Pi, -0.125f));
  float chi = fmaf(-k, kC1, xh);
  chi = fmaf(-k, kC2, chi);
  chi = fmaf(-k, kC3, chi - kPi4H) + xl4;
  sincos_sfu(chi, &f.s, &f.c);
  f.dx = dxh + dxl;
  f.dy = dyh + dyl;
  f.xinv = xinv;
  f.ra = rsqrt_sfu(xh);
  return f;
}

// The same distance and phase to the accuracy of the stored and the fused
// tensor-core kernels, whose entries reach the tensor cores as bf16 hi + lo pairs (2^-17
// relative): the lo part of x comes from H - xh^2 (one fma, of the size of C)
// plus C instead of from the exact sum H + C, the Cody-Waite constant has two
// parts (the third, k C3, is 1.6e-12 omega r rad) and the lo part of pi/4 is
// dropped (2.2e-8 rad).  Phase error a few 1e-7 rad for the kite at
// omega = 2048.
__device__ __forceinline__ pair_phase pair_phase32_tc(float txh, float txl, float tyh, float tyl,
                                                      float sxh, float sxl, float syh, float syl) {
  pair_phase f;
  const float dxh = txh - sxh, dxl = txl - sxl;   // dxh, dyh exact
  const float dyh = tyh - syh, dyl = tyl - syl;
  const float H = fmaf(dxh, dxh, dyh * dyh);      // exact
  const float C = fmaf(dxl, fmaf(2.0f, dxh, dxl), dyl * fmaf(2.0f, dyh, dyl));
  const float x2 = H + C;
  const float xinv = rsqrt_sfu(x2);
  const float xh = x2 * xinv;
  const float xl = (fmaf(-xh, xh, H) + C) * (0.5f * xinv);
  const float k = rintf(fmaf(xh, kInv2Pi, -0.125f));
  float chi = fmaf(-k, kC1, xh);                  // exact
  chi = fmaf(-k, kC2, chi);
  chi = (chi - kPi4H) + xl;
  sincos_sfu(chi, &f.s, &f.c);
  f.dx = dxh + dxl;
  f.dy = dyh + dyl;
  f.xinv = xinv;
  f.ra = rsqrt_sfu(xh);
  return f;
}

// Hankel's asymptotic expansion for x >= kX0 (t = 1/x), three terms of each
// of P and Q (A&S 9.2.9, 9.2.10), without the common factor c0 x^(-1/2):
// J_m = c0 ra j_m, Y_m = c0 ra y_m.  The remainder is below the first omitted
// term (A&S 9.2.10 remark), < 4.1e-8 for x >= 16: under one FP32 ulp.
__device__ __forceinline__ void hankel_asym32(float ti, float s, float c, float& j0, float& y0,
                                              float& j1, float& y1) {
  const float t2 = ti * ti;
  const float P0 = fmaf(t2, fmaf(t2, 0.112152099609375f, -0.0703125f), 1.0f);
  const float Q0 = ti * fmaf(t2, fmaf(t2, -0.22710800170898438f, 0.0732421875f), -0.125f);
  const float P1 = fmaf(t2, fmaf(t2, -0.144195556640625f, 0.1171875f), 1.0f);
  const float Q1 = ti * fmaf(t2, fmaf(t2, 0.2775764465332031f, -0.1025390625f), 0.375f);
  j0 = fmaf(P0, c, -Q0 * s);
  y0 = fmaf(P0, s, Q0 * c);
  j1 = fmaf(P1, s, Q1 * c);
  y1 = fmaf(Q1, s, -P1 * c);
}

// Two terms of each of P and Q (the stored operators): the remainder
// is below the first omitted term, < 2.2e-6 relative for x >= 16 and
// < 1.4e-8 for x >= 64, near the bf16 hi + lo split's 2^-17.
__device__ __forceinline__ void hankel_asym32_tc(float ti, float s, float c, float& j0, float& y0,
                                                 float& j1, float& y1) {
  const float t2 = ti * ti;
  const float P0 = fmaf(t2, -0.0703125f, 1.0f);
  const float Q0 = ti * fmaf(t2, 0.0732421875f, -0.125f);
  const float P1 = fmaf(t2, 0.1171875f, 1.0f);
  const float Q1 = ti * fmaf(t2, -0.1025390625f, 0.375f);
  j0 = fmaf(P0, c, -Q0 * s);
  y0 = fmaf(P0, s, Q0 * c);
  j1 = fmaf(P1, s, Q1 * c);
  y1 = fmaf(Q1, s, -P1 * c);
}

// Entries of one pair with omega r >= kX0 (outside the band).
// (xh, xl, yh, yl) of target i and source j; returns soft a, hard (a = S, b = D').
template <int BC>
__device__ __forceinline__ void pair_entries_fp32(const omega32& P, float txh, float txl,
                                                  float tyh, float tyl, float tnx, float tny,
                                                  float tsp, float sxh, float sxl, float syh,
                                                  float syl, float snx, float sny, float ssp,
                                                  float w, float2& a, float2& b) {
  const pair_phase f = pair_phase32(txh, txl, tyh, tyl, sxh, sxl, syh, syl);
  float j0, y0, j1, y1;
  hankel_asym32(f.xinv, f.s, f.c, j0, y0, j1, y1);
  const float amp = kSqrt2OverPi * f.ra;
  const float J0 = amp * j0, Y0 = amp * y0, J1 = amp * j1, Y1 = amp * y1;
  const float omega = P.wh;
  const float hq = 0.25f * P.h;
  if constexpr (BC == 0) {
    const float cc = (f.dx * snx + f.dy * sny) * f.xinv;
    const float es = P.eta * ssp;
    const float oc = omega * cc;
    a.x = hq * (es * J0 - oc * Y1) - w * kInv4Pi * oc * J1;
    a.y = hq * (oc * J1 + es * Y0) + w * kInv4Pi * es * J0;
  } else {
    a.x = -hq * Y0 * ssp - w * kInv4Pi * J0 * ssp;
    a.y = hq * J0 * ssp;
    const float cp = -(f.dx * tnx + f.dy * tny) * f.xinv * ssp / tsp;
    const float oc = omega * cp;
    b.x = -hq * oc * Y1 - w * kInv4Pi * oc * J1;
    b.y = hq * oc * J1;
  }
}

// The sound-soft entry with the per-node factors folded in, to the accuracy of
// the operators' bf16 hi + lo planes (phase and series above): tg, sc = target
// and source coordinates, sq = source factors, wk = Kress weight / (pi h); see
// the packed layout above.  With A = hq c0 eta |z'_j| ra and B = omega hq c0
// (nu_j . (z_i - z_j)) ra / r,
//   re = A j0 - B (y1 + wk j1),      im = B j1 + A (y0 + wk j0)
__device__ __forceinline__ float2 entry_folded32(float4 tg, float4 sc, float4 sq, float wk) {
  const pair_phase f = pair_phase32_tc(tg.x, tg.y, tg.z, tg.w, sc.x, sc.y, sc.z, sc.w);
  float j0, y0, j1, y1;
  hankel_asym32_tc(f.xinv, f.s, f.c, j0, y0, j1, y1);
  const float A = sq.z * f.ra;
  const float B = fmaf(f.dx, sq.x, f.dy * sq.y) * (f.xinv * f.ra);
  return make_float2(fmaf(A, j0, -B * fmaf(wk, j1, y1)), fmaf(B, j1, A * fmaf(wk, j0, y0)));
}

// ---------------------------------------------------------------------------
// Two entries of one target at once (the adjacent sources j, j + 1), in packed
// FP32 pairs: add, mul and fma on float2 issue once for two lanes of
// arithmetic (measured: the same 121 lane-ops per clock and SM as scalar FMAs
// at half the issue slots); the producers of the fused kernel were bound by issue
// slots with scalar ones and are by the FMA pipe now.  Signs sit in the per-node
// data and in the constants where they can.
// ---------------------------------------------------------------------------

// as pair_phase, for the two sources
struct pair_phase2 {
  float2 dx, dy, half, ra, chi;   // half = 1 / (2 x), chi = x - pi/4 less a multiple of 2 pi
};

// pair_phase32_tc for both sources: t0, t1 the target's (xh, xh, xl, xl), (yh,
// ..), s0, s1 the sources' negated coordinates by pairs.  k is rounded by adding
// and subtracting 1.5 2^23 (k < 2^14), -pi/4 joins the lo part of x.
__device__ __forceinline__ pair_phase2 phase32_pair(float4 t0, float4 t1, float4 s0, float4 s1) {
  pair_phase2 f;
  const float2 dxh = add2(lo2(t0), lo2(s0)), dxl = add2(hi2(t0), hi2(s0));   // dxh, dyh exact
  const float2 dyh = add2(lo2(t1), lo2(s1)), dyl = add2(hi2(t1), hi2(s1));
  const float2 H = fma2(dxh, dxh, mul2(dyh, dyh));                           // exact
  f.dx = add2(dxh, dxl);
  f.dy = add2(dyh, dyl);
  const float2 C = fma2(dxl, add2(dxh, f.dx), mul2(dyl, add2(dyh, f.dy)));
  const float2 x2 = add2(H, C);
  const float2 xinv = make_float2(rsqrt_sfu(x2.x), rsqrt_sfu(x2.y));
  const float2 xh = mul2(x2, xinv);
  f.ra = make_float2(rsqrt_sfu(xh.x), rsqrt_sfu(xh.y));
  const float2 e = add2(fma2(neg2(xh), xh, H), C);                // x^2 - xh^2
  f.half = mul2(xinv, f2(0.5f));
  const float2 xl = fma2(e, f.half, f2(-kPi4H));                             // x lo - pi/4
  const float2 kr = add2(fma2(xh, f2(kInv2Pi), f2(-0.125f)), f2(12582912.0f));
  const float2 k = add2(kr, f2(-12582912.0f));
  f.chi = add2(fma2(k, f2(-kC2), fma2(k, f2(-kC1), xh)), xl);                // first fma exact
  return f;
}

// H_nu(x) = c0 ra m_nu exp(i (chi + psi_nu - nu pi / 2)) of both sources, as
// modulus and phase (A&S 9.2.28, 9.2.29: two terms each): j0 = m0 c0, w0 = y0 + wk
// j0 = m0 u0, j1 = m1 s1, w1 = y1 + wk j1 = m1 u1.  m1 = 1 + 3 t^2 / 16 - 0.193 t^4 ..
// takes psi_1 / t = 3/8 - 0.164 t^2 times t^2 / 2, which costs nothing and holds -0.082
// of the third term: at omega r = 16 the entries are off by 1.6e-6 of H0 and 1.7e-6 of
// H1 (two terms of P and Q: 1.7e-6 and 2.2e-6; m1 with two terms 2.9e-6, with three
// 3.5e-7 and 4 % more time for the kite).  Everything is in u = t^2 / 4 and h = t / 2,
// which the phase needs anyway; the factors of two sit in the node data.  Two more
// sines and cosines on the special-function unit than with P and Q, but six packed
// instructions of 52 fewer on the FMA pipe, which bounds the fused kernel: kite n =
// 32768, 64 right-hand sides 2.51 -> 2.45 ms.
struct hankel_pair {
  float2 m0, m1, c0, u0, s1, u1;
};
__device__ __forceinline__ hankel_pair hankel32_pair(const pair_phase2& f, float2 wk) {
  const float2 u = mul2(f.half, f.half);   // t^2 / 4
  const float2 q1 = fma2(u, f2(-21.0f / 16.0f), f2(0.75f));
  const float2 a0 = fma2(f.half, fma2(u, f2(25.0f / 48.0f), f2(-0.25f)), f.chi);
  const float2 a1 = fma2(f.half, q1, f.chi);
  hankel_pair h;
  float2 s0, c1;
  sincos_sfu(a0.x, &s0.x, &h.c0.x);
  sincos_sfu(a0.y, &s0.y, &h.c0.y);
  sincos_sfu(a1.x, &h.s1.x, &c1.x);
  sincos_sfu(a1.y, &h.s1.y, &c1.y);
  h.m0 = fma2(u, f2(-0.25f), f2(1.0f));
  h.m1 = fma2(u, q1, f2(1.0f));
  h.u0 = fma2(wk, h.c0, s0);
  h.u1 = fma2(wk, h.s1, neg2(c1));
  return h;
}

// Operators of the fused kernel: the sound-soft one (eq. 1); of the sound-hard
// one (eq. 2, Maue's identity summed over the pairs) S' = -i S, applied to u =
// d/ds x, and C = -D' - i (omega^2 / eta) (n_i . n_j) S, applied to x; or both
// from one phase.  With A = c ra, B (soft) = (a, b).(dx, dy) ra / (2 x), D =
// (tq).(dx, dy) A / (2 x), kn = tq.(a, b) = (omega^2 / eta) n_i . n_j:
//   soft: re = A j0 - B w1,           im = A w0 + B j1
//   S':   re = A j0,                  im = A w0
//   C:    re = kn A j0 - D w1,        im = kn A w0 + D j1
enum { OP_SOFT = 0, OP_S = 1, OP_C = 2, OP_SC = 3 };

struct entry_pair {
  float2 re, im;     // soft, S' or C
  float2 re2, im2;   // OP_SC: C (the first is S')
};

// tq = (tx, tx, ty, ty) target factors 2 omega nu / |z'| (hard), s2, s3 the source
// factors by pairs
template <int OP>
__device__ __forceinline__ entry_pair finish32_pair(const pair_phase2& f, float4 tq, float4 s2,
                                                    float2 sc, float2 wk) {
  const hankel_pair h = hankel32_pair(f, wk);
  const float2 A = mul2(sc, f.ra), A0 = mul2(A, h.m0);
  entry_pair e;
  if constexpr (OP == OP_SOFT) {
    const float2 B = mul2(fma2(f.dx, lo2(s2), mul2(f.dy, hi2(s2))),
                          mul2(h.m1, mul2(f.half, f.ra)));
    e.re = fma2(A0, h.c0, mul2(neg2(B), h.u1));
    e.im = fma2(A0, h.u0, mul2(B, h.s1));
  } else {
    const float2 sr = mul2(A0, h.c0), si = mul2(A0, h.u0);
    if constexpr (OP == OP_S || OP == OP_SC) {
      e.re = sr;
      e.im = si;
    }
    if constexpr (OP == OP_C || OP == OP_SC) {
      const float2 D = mul2(fma2(f.dx, lo2(tq), mul2(f.dy, hi2(tq))),
                            mul2(h.m1, mul2(f.half, A)));
      const float2 kn = fma2(lo2(tq), lo2(s2), mul2(hi2(tq), hi2(s2)));
      const float2 cr = fma2(kn, sr, mul2(neg2(D), h.u1));
      const float2 ci = fma2(kn, si, mul2(D, h.s1));
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
