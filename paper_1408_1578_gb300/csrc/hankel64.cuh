// FP64 Bessel functions J0, Y0, J1, Y1 (the Hankel functions H_nu^(1) = J_nu + i Y_nu
// of G(x, y) = (i/4) H0^(1)(omega |x - y|), paper Section 1), written from
// published methods and tested against scipy / mpmath values:
//
//  x >= 20: Hankel's asymptotic expansion (Abramowitz & Stegun 9.2.5, 9.2.9,
//           9.2.10):  H_nu^(1)(x) = sqrt(2/(pi x)) (P + i Q) exp(i chi),
//           chi = x - (nu/2 + 1/4) pi,  P = sum_k (-1)^k a_2k x^-2k,
//           Q = sum_k (-1)^k a_(2k+1) x^-(2k+1),
//           a_k(nu) = prod_{m=1..k} (4 nu^2 - (2m-1)^2) / (8^k k!).
//           Twenty-one terms reach double precision for x >= 20; fewer do
//           further out (thirteen from 40, nine from 100, six from 400).
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
// the FP64 pipe), one table look-up for sine and cosine, per-node factors.
// About 70 FP64 instructions per far pair; 150 with the library's sqrt,
// division and sincos and the full series everywhere.
#pragma once

#include "internal.h"

namespace h64 {

// a_k(nu) of the asymptotic expansion with the alternating sign folded in
static __constant__ double kP0[11] = {1.0, -0.0703125, 0.112152099609375, -0.5725014209747314,
                               6.074042001273483, -110.01714026924674, 3038.090510922384,
                               -118838.42625678325, 6252951.493434797, -425939216.5047669,
                               36468400807.06556};
static __constant__ double kQ0[10] = {-0.125, 0.0732421875, -0.22710800170898438, 1.7277275025844574,
                               -24.380529699556064, 551.3358961220206, -18257.755474293175,
                               832859.3040162893, -50069589.531988926, 3836255180.2304335};
static __constant__ double kP1[11] = {1.0, 0.1171875, -0.144195556640625, 0.6765925884246826,
                               -6.883914268109947, 121.59789187653587, -3302.2722944808525,
                               127641.2726461746, -6656367.718817688, 450278600.3050393,
                               -38338575207.427895};
static __constant__ double kQ1[10] = {0.375, -0.1025390625, 0.2775764465332031, -1.993531733751297,
                               27.248827311268542, -603.8440767050702, 19718.37591223663,
                               -890297.8767070678, 53104110.10968523, -4043620325.107754};

constexpr int kTrig = 1024;                     // table of sin, cos (2 pi j / kTrig - pi / 4)
constexpr double kTrigInv = 162.97466172610083;  // kTrig / (2 pi)
constexpr double kTrigC1 = 0.006135923151542565, kTrigC2 = 2.391888279584674e-19;  // 2 pi / kTrig
constexpr double kC0Inv = 1.2533141373155003;    // sqrt(pi / 2)
constexpr double kTwoOverPi = 0.6366197723675814;
constexpr double kGamma = 0.57721566490153286061;

constexpr int kNear = 41;    // Taylor centres 0, 1/2, .. 20
constexpr int kTaylor = 14;  // coefficients per centre
// tables of one operator: kTrig (sin, cos) pairs, then kNear x kTaylor
// coefficients (J0, g) of the Taylor polynomials
constexpr int kTableDouble2 = kTrig + kNear * kTaylor;

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

// distance r = sqrt(r2) and 1 / r.  The plain functions take the arguments
// near the ends of the exponent range, where the estimate flushes to zero.
__device__ __forceinline__ void distance(double r2, double& r, double& rinv) {
  const unsigned hi = (unsigned)__double2hiint(r2);
  if (hi - 0x02000000u < 0x7c000000u) {   // 2^-991 < r2 < 2^993
    rinv = rsqrt_newton(r2);
    const double r0 = r2 * rinv;
    const double half = __hiloint2double(__double2hiint(rinv) - 0x00100000, __double2loint(rinv));
    r = fma(fma(-r0, r0, r2), half, r0);
  } else {
    r = sqrt(r2);
    rinv = 1.0 / r;
  }
}

// J0 = amp j0, Y0 = amp y0, J1 = amp j1, Y1 = amp y1, with c0 = sqrt(2/pi)
// left out of amp: J = c0 amp j
struct values {
  double amp, j0, y0, j1, y1;
};

template <int NP, int NQ>
__device__ __forceinline__ void series(double t2, double& P0, double& P1, double& Q0, double& Q1) {
  P0 = kP0[NP];
  P1 = kP1[NP];
  Q0 = kQ0[NQ];
  Q1 = kQ1[NQ];
#pragma unroll
  for (int k = NP - 1; k >= 0; --k) {
    P0 = fma(P0, t2, kP0[k]);
    P1 = fma(P1, t2, kP1[k]);
  }
#pragma unroll
  for (int k = NQ - 1; k >= 0; --k) {
    Q0 = fma(Q0, t2, kQ0[k]);
    Q1 = fma(Q1, t2, kQ1[k]);
  }
}

// x >= 20, t = 1 / x
__device__ __forceinline__ values asymptotic(double x, double t, const double2* __restrict__ tab) {
  const double t2 = t * t;
  double P0, P1, Q0, Q1;
  // number of terms by the size of x (its high word, off the FP64 pipe), so
  // that the first dropped one is below 2^-55 of the sum; the lanes of a
  // warp hold neighbouring sources and mostly agree
  const int xh = __double2hiint(x);
  if (xh >= 0x40790000)        // 400
    series<3, 2>(t2, P0, P1, Q0, Q1);
  else if (xh >= 0x40590000)   // 100
    series<4, 4>(t2, P0, P1, Q0, Q1);
  else if (xh >= 0x40440000)   // 40
    series<6, 6>(t2, P0, P1, Q0, Q1);
  else
    series<10, 9>(t2, P0, P1, Q0, Q1);
  Q0 *= t;
  Q1 *= t;
  // x = j 2 pi / kTrig + d; the table holds sine and cosine of the first part
  // less pi / 4, and |d| <= pi / kTrig needs two terms of each series
  // (remainders < 4e-22 and < 2e-18)
  constexpr double magic = 6755399441055744.0;   // 1.5 2^52
  const double u = fma(x, kTrigInv, magic);
  const int j = __double2loint(u) & (kTrig - 1);
  const double jd = u - magic;
  double d = fma(-jd, kTrigC1, x);
  d = fma(-jd, kTrigC2, d);
  const double2 sc = __ldg(tab + j);
  const double d2 = d * d;
  const double sd = fma(d * d2, fma(d2, 1.0 / 120.0, -1.0 / 6.0), d);
  const double cm = d2 * fma(d2, 1.0 / 24.0, -0.5);            // cos d - 1
  const double s = fma(sc.y, sd, fma(sc.x, cm, sc.x));
  const double c = fma(-sc.x, sd, fma(sc.y, cm, sc.y));
  values v;
  v.amp = rsqrt_newton(x);
  v.j0 = fma(P0, c, -(Q0 * s));
  v.y0 = fma(P0, s, Q0 * c);
  // chi_1 = chi - pi/2: cos chi_1 = s, sin chi_1 = -c
  v.j1 = fma(P1, s, Q1 * c);
  v.y1 = fma(Q1, s, -(P1 * c));
  return v;
}

// 0 < x < 20, t = 1 / x: Taylor polynomials about c = k / 2, k nearest 2 x,
// Horner's scheme for each value and derivative
__device__ __forceinline__ values taylor(double x, double t, const double2* __restrict__ tab) {
  const int k = __double2int_rn(2.0 * x);
  const double d = fma((double)k, -0.5, x);
  const double2* a = tab + kTrig + k * kTaylor;
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
  v.amp = kC0Inv;
  v.j0 = J;
  v.j1 = -dJ;
  v.y0 = fma(kTwoOverPi * lg, J, G);
  v.y1 = -fma(kTwoOverPi, fma(lg, dJ, J * t), dG);
  return v;
}

// x > 0, t = 1 / x
__device__ __forceinline__ values bessel01(double x, double t, const double2* __restrict__ tab) {
  return __double2hiint(x) >= 0x40340000 ? asymptotic(x, t, tab) : taylor(x, t, tab);   // 20
}

// tables of one operator (see kTableDouble2): thread j of the first kTrig
// makes one sine / cosine pair, then one thread per Taylor centre
__device__ __forceinline__ void fill_tables(int j, double2* __restrict__ tab) {
  if (j < kTrig) {
    double s, c;
    sincospi(2.0 * j / kTrig - 0.25, &s, &c);
    tab[j] = make_double2(s, c);
  } else if (j < kTrig + kNear) {
    const int k = j - kTrig;
    double2* a = tab + kTrig + k * kTaylor;
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

}  // namespace h64

// Nystrom entries of one off-diagonal pair (i != j) in FP64, (dx, dy) =
// z_i - z_j, with the per-node factors folded in (hq = h / 4, c0 =
// sqrt(2/pi), nu the unnormalised normal, |z'| the speed, wk = Kress weight
// / (pi h); h64::values' amp is x^(-1/2)):
//   soft (eq. 1):  sx, sy = omega hq c0 nu_j,  se = hq c0 eta |z'_j|;  A = se amp,
//                  B = ((dx, dy) . (sx, sy)) amp / r
//                  re = A j0 - B (y1 + wk j1),  im = B j1 + A (y0 + wk j0)
//   hard (eq. 2):  se = hq c0 |z'_j|, tx, ty = omega nu_i / |z'_i|;  A = se amp,
//                  D = ((dx, dy) . (tx, ty)) A / r
//                  S  = -A (y0 + wk j0) + i A j0,  D' = D (y1 + wk j1) - i D j1
// omega_inv = 1 / omega, tab = the operator's tables.  KRESS false: no Kress term
// (points off the curve).
template <int BC, bool KRESS = true>
__device__ __forceinline__ void pair_folded_fp64(double dx, double dy, double omega,
                                                 double omega_inv, double fx, double fy, double se,
                                                 double wk, const double2* __restrict__ tab,
                                                 double2& a, double2& b) {
  double r, rinv;
  h64::distance(fma(dx, dx, dy * dy), r, rinv);
  const h64::values v = h64::bessel01(omega * r, omega_inv * rinv, tab);
  const double A = se * v.amp;
  const double w0 = KRESS ? fma(wk, v.j0, v.y0) : v.y0, w1 = KRESS ? fma(wk, v.j1, v.y1) : v.y1;
  const double p = fma(dx, fx, dy * fy);
  if constexpr (BC == 0) {
    const double B = p * (rinv * v.amp);
    a = make_double2(fma(A, v.j0, -(B * w1)), fma(B, v.j1, A * w0));
    b = make_double2(0.0, 0.0);
  } else {
    const double D = p * (rinv * A);
    a = make_double2(-(A * w0), A * v.j0);
    b = make_double2(D * w1, -(D * v.j1));
  }
}

// The same entries from plain node data (set-up kernels): w = Kress table
// entry w_{(i-j) mod n}, h = 2 pi / n.
//   soft:  a = h K + w K1 for K = L - i eta M (eq. 1)
//   hard:  a = S_ij = h M + w M1, b = D'_ij = h L' + w L'1 (eq. 2)
template <int BC>
__device__ __forceinline__ void pair_entries_fp64(double dx, double dy, double omega, double eta,
                                                  double h, double w, double nxj, double nyj,
                                                  double sj, double nxi, double nyi, double si,
                                                  const double2* __restrict__ tab, double2& a,
                                                  double2& b) {
  constexpr double c0q = 0.25 * 0.7978845608028654;   // c0 / 4
  const double f = c0q * h, wk = w / (CFIE_PI * h);
  if constexpr (BC == 0)
    pair_folded_fp64<0>(dx, dy, omega, 1.0 / omega, omega * f * nxj, omega * f * nyj, f * eta * sj,
                        wk, tab, a, b);
  else
    pair_folded_fp64<1>(dx, dy, omega, 1.0 / omega, omega * nxi / si, omega * nyi / si, f * sj, wk,
                        tab, a, b);
}

// C_ij = -D'_ij - i (omega^2 / eta) (n_i . n_j) S_ij, the operator that the
// sound-hard sums apply to x (n the unit normals; i == j: the diagonal entries)
__device__ __forceinline__ double2 hard_combined(const geom_dev& g, double omega, double eta, int i,
                                                 int j, double2 S, double2 Dp) {
  const double k = omega * omega / eta / (g.sp[i] * g.sp[j]) *
                   fma(g.nx[i], g.nx[j], g.ny[i] * g.ny[j]);
  return make_double2(fma(k, S.y, -Dp.x), -fma(k, S.x, Dp.y));
}
