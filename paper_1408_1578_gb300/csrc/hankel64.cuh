// FP64 Bessel functions J0, Y0, J1, Y1 (the Hankel functions H_nu^(1) = J_nu + i Y_nu
// of G(x, y) = (i/4) H0^(1)(omega |x - y|), paper Section 1), written from
// published methods and tested against mpmath at 40 digits through the field of one
// node (tests/test_parity_fp64_values.py):
//
//  x >= 20: Hankel's asymptotic expansion as modulus and phase (Abramowitz & Stegun
//           9.2.28, 9.2.29): H_nu^(1)(x) = sqrt(2/(pi x)) m exp(i theta) with
//           m = 1 + O(x^-2), theta = x - (nu/2 + 1/4) pi + O(1/x).  Eleven terms
//           of each reach double precision for x >= 20; fewer do further out
//           (eight from 32, five from 64).
//  x <  20: J0 and g = Y0 - (2/pi) ln(x/2) J0, both entire, from their Taylor
//           polynomials about the nearest multiple of 1/2 (degree 13: the next
//           term is below 1e-18), with J1 = -J0' and Y1 = -Y0' from the same
//           coefficients.  The coefficients are made once per operator, from
//           the values at the centres by the recurrence of Bessel's equation.
//
// GB300 issues one FP64 instruction for every 64 FP32 ones (measured 1.7
// lanes per clock and SM, latency 64 clocks), so a pair costs what its FP64
// instructions cost and nothing else: shared square roots and reciprocals
// (Newton's method from the special-function unit's estimate, which runs off
// the FP64 pipe), one table look-up for sine and cosine, per-node factors.  What
// is small is kept off the FP64 pipe: everything that is added to the table's
// sine and cosine is below 0.03, so that packed FP32 double-floats give it, and
// FP64 numbers are taken apart and joined with integer instructions.
// About 38 FP64 instructions per far pair of the sound-hard operator; 70 with the
// series and the rotation in FP64, 150 with the library's sqrt, division and
// sincos besides.  Measured (GB300), series in FP64 -> here: circle n = 1024, one
// right-hand side 138 -> 96 us; star n = 4096, 16, sound hard 3.2 -> 2.22 ms; field of
// 16 densities at 20000 points 10.9 -> 6.8 ms.  Values emulated on the
// CPU against quadruple precision, rms over 20 < x < 50000: 3.8e-17 .. 6.3e-17 times
// amp (FP64 series 6.5e-17 .. 7.4e-17).  Whole entries on the GPU, with their factors
// and the distance: rms 1.1 to 1.2 2^-53 for H0, 1.8 to 1.9 for H1 from x = 20 on, 1.2
// to 3 below (FP64 series and Miller's recurrence 1.5, 1.5 and 1 to 6).
#pragma once

#include "internal.h"
#include "packed32.cuh"

namespace h64 {

// H_nu^(1)(x) = sqrt(2/(pi x)) m exp(i (x - (nu/2 + 1/4) pi + psi)), t = 1 / x:
//   m = 1 + sum_k kMod[k-1] t^2k, psi = sum_k kPsi[k-1] t^(2k-1)
// lane x: nu = 0, lane y: nu = 1.  From the series of m^2 (A&S 9.2.28), its
// square root, and psi' = 1 / m^2 - 1 term by term.
constexpr int kFarTerms = 11;
static __constant__ float2 kMod[kFarTerms] = {
    {-0.0625f, 0.1875f}, {0.103515625f, -0.193359375f}, {-0.5428466796875f, 0.8052978515625f},
    {5.848699569702148f, -7.739953994750977f}, {-106.8867939710617f, 132.76182425022125f},
    {2968.1429378427565f, -3543.303665366024f}, {-116538.47969683609f, 135394.22856918094f},
    {6148451.462878801f, -7003141.574752433f}, {-419670939.1557855f, 470832610.30922693f},
    {35988758012.12494f, -39896618143.18781f}, {-3787947157068.18f, 4158798688522.596f}};
static __constant__ float2 kPsi[kFarTerms] = {
    {-0.125f, 0.375f}, {0.06510416666666667f, -0.1640625f}, {-0.2095703125f, 0.3708984375f},
    {1.6380658830915178f, -2.3693978445870534f}, {-23.475127749972874f, 30.624011993408203f},
    {535.640519510616f, -659.185221823779f}, {-17837.279688947478f, 21156.314045527808f},
    {816737.8421910767f, -944346.6095480548f}, {-49232732.339998595f, 55869739.657019265f},
    {3779795380.667541f, -4228159535.534621f}, {-360101552365.56555f, 398251272117.5241f}};
// what the FP32 numbers leave of the first four
static __constant__ float2 kModL[4] = {{0.0f, 0.0f}, {0.0f, 0.0f}, {0.0f, 0.0f}, {0.0f, 0.0f}};
static __constant__ float2 kPsiL[4] = {{0.0f, 0.0f}, {2.48352687e-09f, 0.0f}, {5.96046448e-09f, 1.1920929e-08f}, {-5.10896955e-08f, 3.4059797e-08f}};

constexpr int kTrig = 1024;                     // table of sin, cos (2 pi j / kTrig - pi / 4),
                                                // then both as double-floats (h, l, h, l)
constexpr double kTrigInv = 162.97466172610083;  // kTrig / (2 pi)
constexpr double kTrigC1 = 0.006135923151542565;   // 2 pi / kTrig as a double ..
constexpr float kTrigC2 = 3.898171832519376e-17f;  // .. and what is left, divided by it
constexpr double kC0Inv = 1.2533141373155003;    // sqrt(pi / 2)
constexpr double kTwoOverPi = 0.6366197723675814;
constexpr double kGamma = 0.57721566490153286061;

constexpr int kNear = 41;    // Taylor centres 0, 1/2, .. 20
constexpr int kTaylor = 14;  // coefficients per centre
// tables of one operator: kTrig entries of sine and cosine, then kNear x kTaylor
// coefficients (J0, g) of the Taylor polynomials
constexpr int kTableDouble2 = 2 * kTrig + kNear * kTaylor;

// J0, J0', g, g' at x = 1/2, 1, .. 20 (50-digit mpmath values, rounded)
static __constant__ double kCentre[kNear - 1][4] = {
    {0.9384698072408129, -0.2422684576748739, 0.3837206630761735, 0.06276333632264228},
    {0.7651976865579666, -0.4400505857449335, 0.42591666583395205, 0.09989119410083765},
    {0.5118276717359181, -0.5579365079100996, 0.4761871397786934, 0.09289943931699093},
    {0.22389077914123567, -0.5767248077568734, 0.5103756726497451, 0.035765783114890606},
    {-0.048383776468198, -0.49709410246427405, 0.5049436426264904, -0.06298131686132265},
    {-0.26005195490193345, -0.3390589585259365, 0.44397646823618026, -0.18196937868409993},
    {-0.3801277399872634, -0.1373775273623272, 0.3244471935858393, -0.29210400696416305},
    {-0.39714980986384735, 0.06604332802354913, 0.15831003397457788, -0.3638603737983707},
    {-0.32054250898512143, 0.23106043192337064, -0.029223588992998203, -0.37493575504464993},
    {-0.1775967713143383, 0.32757913759146523, -0.20492031426082816, -0.31633716446784677},
    {-0.006843869417819197, 0.34143821542904335, -0.33507310578484045, -0.19533755611589018},
    {0.15064525725099692, 0.27668385812756563, -0.39355572157911856, -0.034485835361334524},
    {0.2600946055816064, 0.15384130140997185, -0.36840574231975065, 0.13318161592165007},
    {0.3000792705195556, 0.004682823482345833, -0.26527306762627273, 0.27164161375754337},
    {0.2663396578803784, -0.1352484275797055, -0.10679979090525553, 0.3503264857896045},
    {0.1716508071375539, -0.23463634685391463, 0.07203237398964119, 0.35147744933337655},
    {0.041939251842934504, -0.2731219636740537, 0.2315732989459774, 0.2746103886203401},
    {-0.09033361118287614, -0.24531178657332528, 0.3364334263659793, 0.13696748969726463},
    {-0.19392874768742235, -0.16126443075752986, 0.36357740815861234, -0.03021867416605251},
    {-0.24593576445134835, -0.04347274616886144, 0.3076569509141883, -0.18881649155483307},
    {-0.23664819446234714, 0.07885001422733148, 0.18228984521023106, -0.30259500834210773},
    {-0.1711903004071961, 0.17678529895672151, 0.016941459192461213, -0.34565888278147905},
    {-0.06765394811166522, 0.22837862066532347, -0.14989435198578846, -0.30851411481576235},
    {0.047689310796833535, 0.2234471044906276, -0.2796350551956371, -0.20031007642517237},
    {0.1468840547004211, 0.16548380461475973, -0.3425777047419778, -0.0467054243268109},
    {0.20692610237706782, 0.07031805212177837, -0.324786445264353, 0.11615524306696424},
    {0.21498916588040082, -0.03804929208600142, -0.23127511110741492, 0.25013939951728476},
    {0.17107347611045867, -0.13337515469879324, -0.08473408780156279, 0.324091436894338},
    {0.08754486801037623, -0.19342946359604696, 0.07989514451932415, 0.32114099361157245},
    {-0.014224472826780772, -0.20510403861352275, 0.22371041284948062, 0.24262258645672033},
    {-0.10923065090005017, -0.16721318035174715, 0.313038179095388, 0.10767960019907366},
    {-0.1748990739836292, -0.09039717566130419, 0.3273447700078386, -0.051347145272925325},
    {-0.19638069293686103, 0.005764213735631227, 0.2639997323225998, -0.19664254287178853},
    {-0.16985425215118355, 0.09766849275778065, 0.13877366721484735, -0.293908674606601},
    {-0.10311039822868592, 0.1634199694257549, -0.018029913016757566, -0.32048232366449525},
    {-0.013355805721984111, 0.18799488548806959, -0.16887010384015153, -0.2706493758460295},
    {0.0771648214225547, 0.16663364001001604, -0.2779402007239245, -0.15690064422514974},
    {0.1466294396596512, 0.10570143114240926, -0.3196714782905203, -0.0068459712359973755},
    {0.17885382704017289, 0.02087707014809752, -0.28474568336143846, 0.1434588929665195},
    {0.16702466434058316, -0.06683312417585005, -0.1821960479628176, 0.2581638059585272},
};

// 1 / sqrt(a) to about one unit in the last place: the special-function
// unit's estimate (relative error e0 < 2^-18), then one step of Halley's
// iteration, y (1 + e/2 + 3 e^2 / 8) with e = 1 - a y^2 (error ~ e0^3)
__device__ __forceinline__ double rsqrt_newton(double a) {
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(a));
  const double e = fma(-(a * y), y, 1.0);
  return fma(e * y, fma(e, 0.375, 0.5), y);
}

// J0 = c0 amp j0, Y0 = c0 amp y0, J1 = c0 amp j1, Y1 = c0 amp y1 with c0 =
// sqrt(2 / (pi omega)), which the callers' per-node factors take
struct values {
  double amp, j0, y0, j1, y1;
};

// ---- FP64 numbers taken apart and put together on the integer units

// FP32 number of the leading 24 bits of v (positive, in the FP32 range)
__device__ __forceinline__ float leading(unsigned hi, unsigned lo) {
  return __uint_as_float((hi - 0x38000000u) << 3 | lo >> 29);
}
// v = h + l, v positive and below 2^127; zero below 2^-126
__device__ __forceinline__ void split(double v, float& h, float& l) {
  const unsigned hi = __double2hiint(v), lo = __double2loint(v);
  const bool in = hi >= 0x38100000u;
  h = in ? leading(hi, lo) : 0.0f;
  // 29 bits of weight 2^(e - 1075)
  l = (float)(int)(lo & 0x1fffffff) * __int_as_float(max((int)(hi >> 20) - 948, 0) << 23);
}
// h + l in FP64, |l| <= 2^-24 |h| (2^-127 for h = 0)
__device__ __forceinline__ double join(float h, float l) {
  const unsigned b = __float_as_uint(h), m = b & 0x7fffffff;
  // l in units of h's last place in FP64, its sign against h's
  const unsigned s = (306u - max(m >> 23, 52u)) << 23 | (b & 0x80000000u);
  int u = __float2int_rn(l * __uint_as_float(s));
  if (u < 0 && (m & 0x7fffff) == 0) u *= 2;   // below a power of two places are half as large
  const unsigned long long v =
      ((unsigned long long)((m >> 3) + 0x38000000u) << 32 | m << 29) + (long long)u;
  return __hiloint2double((int)((unsigned)(v >> 32) | (b & 0x80000000u)), (int)(unsigned)v);
}

// distance r, 1 / r and q = r^(-1/2) from r^2
struct polar {
  double r, rinv, q;
};
// One Newton step of third order for r2^(-1/4) gives all three: y from the
// special-function unit (|e| < 2^-18 for e = 1 - r2 y^4), q = y (1 + e / 4 + 5
// e^2 / 32), whose second factor, less 1, takes a double-float; 8 FP64
// instructions where separate steps for 1 / r and x^(-1/2) take 13.  The plain
// functions take what is outside FP32's range.
__device__ __forceinline__ polar distance(double r2) {
  polar p;
  const unsigned hi = __double2hiint(r2);
  if (hi - 0x38700000u < 0x0f000000u) {   // 2^-120 <= r2 < 2^120
    float y = leading(hi, __double2loint(r2));
    asm("sqrt.approx.ftz.f32 %0, %0;" : "+f"(y));
    asm("rsqrt.approx.ftz.f32 %0, %0;" : "+f"(y));
    const float s0 = y * y;
    const double s = join(s0, fmaf(y, y, -s0));            // y^2, exact
    const double w = fma(-(r2 * s), s, 1.0) + 0x1.8p-17;   // e in units of 2^-69
    const unsigned wl = __double2loint(w);
    const int wh = __double2hiint(w) - 0x3ee80000;
    const float eh = (float)(int)__funnelshift_l(wl, wh, 5) * 0x1p-42f;
    const float el = (float)(int)(wl & 0x7ffffff) * 0x1p-69f;
    const float gh = 0.25f * eh, gl = fmaf(0.15625f * eh, eh, 0.25f * el);
    const float yg = y * gh, c = fmaf(y, gl, fmaf(y, gh, -yg)), h = yg + c;
    p.q = join(y, 0.0f) + join(h, c - (h - yg));
    p.rinv = p.q * p.q;
    const double r0 = r2 * p.rinv;
    const double half = __hiloint2double(__double2hiint(p.rinv) - 0x00100000, __double2loint(p.rinv));
    p.r = fma(fma(-r0, r0, r2), half, r0);
  } else {
    p.r = sqrt(r2);
    p.rinv = 1.0 / p.r;
    p.q = sqrt(p.rinv);
  }
  return p;
}

// c_1 + t2 (c_2 + .. + t2 c_N): terms 1 .. D in double-float, the others in FP32
template <int N, int D>
__device__ __forceinline__ d2 far_series(d2 t2, const float2* c, const float2* cl) {
  float2 f = c[N - 1];
#pragma unroll
  for (int k = N - 2; k >= D; --k) f = fma2(f, t2.h, c[k]);
  d2 v = {mul2(t2.h, f), f2(0.0f)};
#pragma unroll
  for (int k = D - 1; k >= 0; --k) {
    if (k < D - 1) v = dd_mul(t2, v);
    const d2 s = fast_sum(c[k], v.h);
    v = {s.h, add2(s.l, add2(v.l, cl[k]))};
  }
  return v;
}

// x >= 20, t = 1 / x.  The angle x + psi = j 2 pi / kTrig + (d + psi), the table
// holding sine and cosine S, C of the first part less pi / 4, and
// |d + psi| < 0.023: with alpha = m cos(d + psi) - 1 and beta = m sin(d + psi)
//   m cos = C + (C alpha - S beta),  m sin = S + (S alpha + C beta)
// where the brackets are small: double-floats (2^-46) leave 2^-52 of the sum, far
// below the x 2^-53 that the rounding of x itself moves it by.  Both orders
// run in the lanes of packed FP32 pairs (about 130 instructions, the time of
// three FP64 ones); FP64 are the reduction of x and the four last additions.
__device__ __forceinline__ values far(double x, double t, double amp, const double2* __restrict__ tab) {
  float th, tl;
  split(t, th, tl);
  const d2 T = {f2(th), f2(tl)}, t2 = dd_mul(T, T);
  // further out fewer terms matter, and fewer in double-float: the rounding and
  // the dropped terms stay below 2^-53
  d2 psi, mod;
  const int xh = __double2hiint(x);
  if (xh >= 0x40500000) {          // 64
    psi = far_series<5, 2>(t2, kPsi, kPsiL);
    mod = far_series<5, 2>(t2, kMod, kModL);
  } else if (xh >= 0x40400000) {   // 32
    psi = far_series<8, 3>(t2, kPsi, kPsiL);
    mod = far_series<8, 3>(t2, kMod, kModL);
  } else {
    psi = far_series<kFarTerms, 4>(t2, kPsi, kPsiL);
    mod = far_series<kFarTerms, 4>(t2, kMod, kModL);
  }
  psi = dd_mul(T, psi);
  mod = dd_mul(t2, mod);
  // x = j 2 pi / kTrig + d, |d| <= pi / kTrig < 2^-8, d in units of 2^-59
  constexpr double magic = 6755399441055744.0;   // 1.5 2^52
  const double u = fma(x, kTrigInv, magic);
  const int j = __double2loint(u) & (kTrig - 1);
  const double w = fma(-(u - magic), kTrigC1, x) + 0x1.8p-7;
  const unsigned wl = __double2loint(w);
  const int wh = __double2hiint(w) - 0x3f880000;
  const float dh = (float)(int)__funnelshift_l(wl, wh, 5) * 0x1p-32f;
  const float dl = fmaf((float)(int)(wl & 0x7ffffff), 0x1p-59f,
                        -(leading(__double2hiint(x), __double2loint(x)) * kTrigC2));
  const double2 sc = __ldg(tab + 2 * j);
  const float4 scf = __ldg(reinterpret_cast<const float4*>(tab) + 2 * j + 1);
  // e = d + psi, q = e^2, y = sin(e) / e - 1, c = cos(e) - 1
  d2 e = two_sum(f2(dh), psi.h);
  e.l = add2(e.l, add2(f2(dl), psi.l));
  e = dd_norm(e);
  const d2 q = dd_norm(dd_mul(e, e));
  d2 y = fast_sum(f2(-1.0f / 6.0f), mul2(q.h, fma2(q.h, f2(-1.0f / 5040.0f), f2(1.0f / 120.0f))));
  y.l = add2(y.l, f2(4.967053731282552e-09f));     // 1 / 6 in FP32 less 1 / 6
  y = dd_mul(q, y);
  d2 c = fast_sum(f2(1.0f / 24.0f), mul2(q.h, f2(-1.0f / 720.0f)));
  c.l = add2(c.l, f2(-1.241763432820638e-09f));    // 1 / 24 less that in FP32
  c = dd_mul(q, c);
  const d2 c2 = fast_sum(f2(-0.5f), c.h);
  c = dd_mul(q, {c2.h, add2(c2.l, c.l)});
  // times m = 1 + mod
  d2 m = fast_sum(f2(1.0f), mod.h);
  m.l = add2(m.l, mod.l);
  const d2 alpha = dd_add(dd_mul(c, m), mod), em = dd_mul(e, m), ey = dd_mul(em, y);
  d2 beta = fast_sum(em.h, ey.h);
  beta.l = add2(beta.l, add2(em.l, ey.l));
  const d2 S = {f2(scf.x), f2(scf.y)}, C = {f2(scf.z), f2(scf.w)};
  const d2 re = dd_norm(dd_add(dd_mul(C, alpha), dd_neg(dd_mul(S, beta))));
  const d2 im = dd_norm(dd_add(dd_mul(S, alpha), dd_mul(C, beta)));
  values v;
  v.amp = amp;
  v.j0 = sc.y + join(re.h.x, re.l.x);
  v.y0 = sc.x + join(im.h.x, im.l.x);
  // chi_1 = chi - pi/2: cos chi_1 = sin, sin chi_1 = -cos
  v.j1 = sc.x + join(im.h.y, im.l.y);
  v.y1 = -(sc.y + join(re.h.y, re.l.y));
  return v;
}

// 0 < x < 20, t = 1 / x: Taylor polynomials about c = k / 2, k nearest 2 x,
// Horner's scheme for each value and derivative.  A NaN with its sign set (a field
// point that is not a number) also comes here; as an integer it is -2^31, which
// must not address the table.
__device__ __forceinline__ values taylor(double x, double t, double amp, const double2* __restrict__ tab) {
  const int k = min(max(__double2int_rn(2.0 * x), 0), kNear - 1);
  const double d = fma((double)k, -0.5, x);
  const double2* a = tab + 2 * kTrig + k * kTaylor;
  double2 q = __ldg(a + kTaylor - 1);
  double J = q.x, G = q.y, dJ = 0.0, dG = 0.0;
#pragma unroll
  for (int m = kTaylor - 2; m >= 0; --m) {
    q = __ldg(a + m);
    dJ = fma(dJ, d, J);
    dG = fma(dG, d, G);
    J = fma(J, d, q.x);
    G = fma(G, d, q.y);
  }
  const double lg = log(0.5 * x);
  values v;
  v.amp = amp;
  v.j0 = J;
  v.j1 = -dJ;
  v.y0 = fma(kTwoOverPi * lg, J, G);
  v.y1 = -fma(kTwoOverPi, fma(lg, dJ, J * t), dG);
  return v;
}

// x = omega r > 0, t = 1 / x, q = r^(-1/2), near = sqrt(pi omega / 2)
__device__ __forceinline__ values bessel01(double x, double t, double q, double near,
                                           const double2* __restrict__ tab) {
  return __double2hiint(x) >= 0x40340000 ? far(x, t, q, tab) : taylor(x, t, near, tab);   // 20
}

// tables of one operator (see kTableDouble2): thread j of the first kTrig
// makes one sine / cosine pair, then one thread per Taylor centre
__device__ __forceinline__ void fill_tables(int j, double2* __restrict__ tab) {
  if (j < kTrig) {
    double s, c;
    sincospi(2.0 * j / kTrig - 0.25, &s, &c);
    tab[2 * j] = make_double2(s, c);
    const float sh = (float)s, ch = (float)c;
    reinterpret_cast<float4*>(tab)[2 * j + 1] =
        make_float4(sh, (float)(s - (double)sh), ch, (float)(c - (double)ch));
  } else if (j < kTrig + kNear) {
    const int k = j - kTrig;
    double2* a = tab + 2 * kTrig + k * kTaylor;
    double J[kTaylor + 1], G[kTaylor + 1];
    if (k == 0) {
      // J0 = sum (-x^2/4)^m / (m!)^2,
      // g = (2/pi) [gamma J0 + sum (-1)^(m+1) H_m (x^2/4)^m / (m!)^2] (A&S 9.1.13)
      double f = 1.0, H = 0.0;
      for (int m = 0; 2 * m < kTaylor; ++m) {
        if (m) {
          f *= -0.25 / ((double)m * m);
          H += 1.0 / m;
        }
        J[2 * m] = f;
        G[2 * m] = kTwoOverPi * f * (kGamma - H);
        J[2 * m + 1] = G[2 * m + 1] = 0.0;
      }
    } else {
      const double c = 0.5 * k;
      J[0] = kCentre[k - 1][0];
      J[1] = kCentre[k - 1][1];
      G[0] = kCentre[k - 1][2];
      G[1] = kCentre[k - 1][3];
      // x y'' + y' + x y = 0 for J0, = -(4/pi) J0' for g, coefficient of d^m
      for (int m = 0; m + 2 < kTaylor; ++m) {
        const double f = 1.0 / (c * (m + 2) * (m + 1));
        const double q = (double)(m + 1) * (m + 1);
        J[m + 2] = -f * (q * J[m + 1] + c * J[m] + (m ? J[m - 1] : 0.0));
        G[m + 2] = -f * (q * G[m + 1] + c * G[m] + (m ? G[m - 1] : 0.0) +
                         2.0 * kTwoOverPi * (m + 1) * J[m + 1]);
      }
    }
    for (int m = 0; m < kTaylor; ++m) a[m] = make_double2(J[m], G[m]);
  }
}

// hq c0 and sqrt(pi omega / 2) of the folded entries below
__host__ __device__ __forceinline__ double pair_factor(double omega, double h) {
  return 0.25 * 0.7978845608028654 * h / sqrt(omega);
}
__host__ __device__ __forceinline__ double near_amp(double omega) { return kC0Inv * sqrt(omega); }

}  // namespace h64

// Nystrom entries of one off-diagonal pair (i != j) in FP64, (dx, dy) =
// z_i - z_j, with the per-node factors folded in (hq = h / 4, c0 =
// sqrt(2 / (pi omega)), nu the unnormalised normal, |z'| the speed, wk = Kress weight
// / (pi h); h64::values' amp is r^(-1/2)):
//   soft (eq. 1):  sx, sy = omega hq c0 nu_j,  se = hq c0 eta |z'_j|;  A = se amp,
//                  B = ((dx, dy) . (sx, sy)) amp / r
//                  re = A j0 - B (y1 + wk j1),  im = B j1 + A (y0 + wk j0)
//   hard (eq. 2):  se = hq c0 |z'_j|, tx, ty = omega nu_i / |z'_i|;  A = se amp,
//                  D = ((dx, dy) . (tx, ty)) A / r
//                  S  = -A (y0 + wk j0) + i A j0,  D' = D (y1 + wk j1) - i D j1
// omega_inv = 1 / omega, near = sqrt(pi omega / 2), tab = the operator's tables.  KRESS false: no Kress term
// (points off the curve).
template <int BC, bool KRESS = true>
__device__ __forceinline__ void pair_folded_fp64(double dx, double dy, double omega,
                                                 double omega_inv, double near, double fx, double fy,
                                                 double se, double wk, const double2* __restrict__ tab,
                                                 double2& a, double2& b) {
  const h64::polar d = h64::distance(fma(dx, dx, dy * dy));
  const h64::values v = h64::bessel01(omega * d.r, omega_inv * d.rinv, d.q, near, tab);
  const double A = se * v.amp;
  const double w0 = KRESS ? fma(wk, v.j0, v.y0) : v.y0, w1 = KRESS ? fma(wk, v.j1, v.y1) : v.y1;
  const double p = fma(dx, fx, dy * fy);
  if constexpr (BC == 0) {
    const double B = p * (d.rinv * v.amp);
    a = make_double2(fma(A, v.j0, -(B * w1)), fma(B, v.j1, A * w0));
    b = make_double2(0.0, 0.0);
  } else {
    const double D = p * (d.rinv * A);
    a = make_double2(-(A * w0), A * v.j0);
    b = make_double2(D * w1, -(D * v.j1));
  }
}

// The same entries from plain node data (set-up kernels): wk = Kress weight
// w_{(i-j) mod n} / (pi h).
//   soft:  a = h K + w K1 for K = L - i eta M (eq. 1)
//   hard:  a = S_ij = h M + w M1, b = D'_ij = h L' + w L'1 (eq. 2)
// The operator's constants come ready: per entry their root and quotients cost as
// much as the entry.
struct pair_consts {
  double omega, omega_inv, near, f, eta;
};
__host__ __device__ __forceinline__ pair_consts make_pair_consts(double omega, double eta,
                                                                 double h) {
  return {omega, 1.0 / omega, h64::near_amp(omega), h64::pair_factor(omega, h), eta};
}
template <int BC>
__device__ __forceinline__ void pair_entries_fp64(double dx, double dy, const pair_consts& c,
                                                  double wk, double nxj, double nyj, double sj,
                                                  double nxi, double nyi, double si,
                                                  const double2* __restrict__ tab, double2& a,
                                                  double2& b) {
  const double m = BC == 0 ? c.omega * c.f : c.omega / si;
  pair_folded_fp64<BC>(dx, dy, c.omega, c.omega_inv, c.near, m * (BC == 0 ? nxj : nxi),
                       m * (BC == 0 ? nyj : nyi), c.f * sj * (BC == 0 ? c.eta : 1.0), wk, tab, a, b);
}

// C_ij = -D'_ij - i (omega^2 / eta) (n_i . n_j) S_ij, the operator that the
// sound-hard sums apply to x (n the unit normals; i == j: the diagonal entries)
__device__ __forceinline__ double2 hard_combined(const geom_dev& g, double omega, double eta, int i,
                                                 int j, double2 S, double2 Dp) {
  const double k = omega * omega / eta / (g.sp[i] * g.sp[j]) *
                   fma(g.nx[i], g.nx[j], g.ny[i] * g.ny[j]);
  return make_double2(fma(k, S.y, -Dp.x), -fma(k, S.x, Dp.y));
}
