// FP64 matrix-free Nystrom matvec (the plain FP64 comparison form) and the
// spectral tangential derivative used by Maue's identity.
//
// Operators (paper, Section 1): soft  A = 1/2 I + D - i eta S        (eq. 1)
//                               hard  A = 1/2 I - D' + N / (i eta)   (eq. 2)
// Per pair (i != j), r = |z_i - z_j|, x = omega r, s_j = |z'_j|, h = 2 pi / n,
// w = w_{(i-j) mod n} (Kress table):
//   soft:  A_ij = h K_ij + w K1_ij,  K = L - i eta M, K1 = L1 - i eta M1 with
//          L  = (i omega/4) H1(x) c,      L1 = -(omega/4pi) J1(x) c,  c = (z_i - z_j).nu~_j / r
//          M  = (i/4) H0(x) s_j,          M1 = -(1/4pi) J0(x) s_j
//   hard:  S_ij  = h M_ij + w M1_ij
//          D'_ij = h L'_ij + w L'1_ij with c' = (z_j - z_i).nu~_i / r * s_j / s_i
//          A x = 1/2 x - D' x + (1/(i eta)) [ (1/s) Dt S (1/s) Dt x
//                                            + omega^2 (n1 S (n1 x) + n2 S (n2 x)) ]
//          (Maue's identity; Dt = spectral derivative, Nyquist mode zeroed),
//          summed as two operators over the same pairs: S on u = (1/s) Dt x, and
//          C on x, C_ij = -D'_ij - i (omega^2 / eta) (n_i . n_j) S_ij, because
//          n1 S n1 + n2 S n2 has the entries (n_i . n_j) S_ij (four multiply-adds
//          per right-hand side and pair fewer than S on three vectors and D')
// Diagonal entries come precomputed (geometry.cu).
//
// Kernels: k_pair_sym (both entries of a pair of nodes at once) for a few
// right-hand sides, else sums64.cuh (entries shared by a block of columns, sums on
// the integer units).
// In both of them source ranges are split across CTAs when the rows alone do
// not fill the GPU; the per-split partial sums go to a scratch buffer and a
// second kernel adds them in a fixed order (deterministic results) and applies
// the hard-path epilogue.
//
// Bound: the FP64 pipe (one instruction of a warp per 64 clocks and
// scheduler): per pair about 38 instructions for the entry (hankel64.cuh).
// Measured (GB300): circle n = 1024, 1 right-hand side 1120 -> 96 us; star n =
// 4096, 16 right-hand sides, sound hard 15.8 -> 2.25 ms.
#include <algorithm>
#include <mutex>
#include <string>

#include <cuda.h>

#include "internal.h"
#include "hankel64.cuh"
#include "sums64.cuh"

namespace {

__device__ __forceinline__ double2 cmad(double2 acc, double2 a, double2 b) {
  acc.x = fma(a.x, b.x, acc.x);
  acc.x = fma(-a.y, b.y, acc.x);
  acc.y = fma(a.x, b.y, acc.y);
  acc.y = fma(a.y, b.x, acc.y);
  return acc;
}

// A few right-hand sides: each pair of nodes once for both of its entries.
// (i, j) and (j, i) share the distance, the Hankel values and the Kress weight,
// about 27 of the 38 FP64 instructions of an entry; what then remains per entry
// is its normal and speed factors, the multiply-adds and two additions of the
// reduction over the rows of the transposed product.
//
// A warp owns 32 rows (one per lane, sums in registers) and walks units of 8
// sources: row blocks I and J = I + d (mod the number of blocks), d = 0 .. half
// of it, cover every pair of blocks once; d = 0 takes its pairs in both orders.
// The transposed sums of SB sources are reduced across the warp together (16
// values: 16 additions instead of 80) and go out by (d, j), each written by one
// warp; the direct sums by (split, i): the layout of the block kernel's split
// partial sums with splits + nblk / 2 entries.
// Measured (GB300, kite), against the block kernel, which takes up to four columns
// in the same time: sound soft, one right-hand side n = 512 86 -> 69 us, n = 4096 1.39
// -> 0.97 ms, n = 16384 18.8 -> 14.3 ms, two 18.8 -> 16.5 ms; sound hard, one n = 4096
// 1.71 -> 1.38 ms.
template <int BC, int R>
__global__ void __launch_bounds__(32)
k_pair_sym(int n, int nblk, double omega, double omega_inv, double near, double eta_inv, double nf,
           double sf, int units_per_warp, int splits, geom_dev g, const double* __restrict__ wks,
           const double2* __restrict__ diag, const double2* __restrict__ xin,
           const double2* __restrict__ uin, int nrhs, double2* __restrict__ part) {
  constexpr int NO = BC ? 2 : 1;
  constexpr int SB = 8 / (R * NO);     // sources whose transposed sums are reduced together
  const int lane = threadIdx.x, I = blockIdx.x, i = 32 * I + lane;
  const bool ok = i < n;
  const int dmax = nblk / 2, units = 4 * (dmax + 1), nsp = splits + dmax;
  // node data of a row or a source: coordinates, folded normal (soft nf nu;
  // hard omega nu / |z'|), folded speed; densities of every output
  auto normal = [&](int k, double& ax, double& ay) {
    const double m = BC ? omega / g.sp[k] : nf;
    ax = m * g.nx[k];
    ay = m * g.ny[k];
  };
  // rows past n sit far away and contribute nothing
  double tx = 1e3 * (lane + 2), ty = 1e3, tfx = 0.0, tfy = 0.0, te = 0.0;
  double2 xi[R][NO], acc[R][NO];
#pragma unroll
  for (int r = 0; r < R; ++r)
#pragma unroll
    for (int o = 0; o < NO; ++o) xi[r][o] = acc[r][o] = make_double2(0.0, 0.0);
  if (ok) {
    tx = g.x[i];
    ty = g.y[i];
    normal(i, tfx, tfy);
    te = sf * g.sp[i];
#pragma unroll
    for (int r = 0; r < R; ++r)
      if (r < nrhs) {
        xi[r][NO - 1] = xin[(size_t)r * n + i];
        if (BC) xi[r][0] = uin[(size_t)r * n + i];
      }
  }
  const int u1 = min(units, (int)(blockIdx.y + 1) * units_per_warp);
  for (int u = blockIdx.y * units_per_warp; u < u1; ++u) {
    const int d = u >> 2;
    int J = I + d;
    if (J >= nblk) J -= nblk;
    const int jb = 32 * J + 8 * (u & 3);
    // an even number of blocks meets its opposite pairs twice: the second time
    // only writes the zeros that the reduction reads
    const bool skip = d > 0 && 2 * d == nblk && I >= d;
    // lanes 8 q .. 8 q + 7 hold the eight sources
    const int jl = jb + (lane & 7);
    double sx = 0.0, sy = 0.0, sfx = 0.0, sfy = 0.0, se = 0.0;
    double2 xj[R][NO];
#pragma unroll
    for (int r = 0; r < R; ++r)
#pragma unroll
      for (int o = 0; o < NO; ++o) xj[r][o] = make_double2(0.0, 0.0);
    if (!skip && jl < n) {
      sx = g.x[jl];
      sy = g.y[jl];
      normal(jl, sfx, sfy);
      se = sf * g.sp[jl];
#pragma unroll
      for (int r = 0; r < R; ++r)
        if (r < nrhs) {
          xj[r][NO - 1] = xin[(size_t)r * n + jl];
          if (BC) xj[r][0] = uin[(size_t)r * n + jl];
        }
    }
#pragma unroll 1
    for (int s0 = 0; s0 < 8; s0 += SB) {
      double v[16];
#pragma unroll
      for (int k = 0; k < 16; ++k) v[k] = 0.0;
#pragma unroll
      for (int b = 0; b < SB; ++b) {
        const int s = s0 + b, j = jb + s;
        if (skip || j >= n) continue;            // uniform
        auto from = [&](double a) { return __shfl_sync(0xffffffffu, a, s); };
        const double qx = from(sx), qy = from(sy), qfx = from(sfx), qfy = from(sfy), qe = from(se);
        double2 q[R][NO];
#pragma unroll
        for (int r = 0; r < R; ++r)
#pragma unroll
          for (int o = 0; o < NO; ++o) q[r][o] = make_double2(from(xj[r][o].x), from(xj[r][o].y));
        int di = i - j;
        if (di < 0) di += n;
        const double wk = ok ? wks[di] : 0.0;
        const double dx = tx - qx, dy = ty - qy;
        const h64::polar p = h64::distance(fma(dx, dx, dy * dy));
        const h64::values h = h64::bessel01(omega * p.r, omega_inv * p.rinv, p.q, near, g.tab);
        const double w0 = fma(wk, h.j0, h.y0), w1 = fma(wk, h.j1, h.y1);
        const double ra = p.rinv * h.amp;
        // entries from the receiving node's and the sending node's factors
        double2 e[NO], et[NO];
        if constexpr (BC == 0) {
          const double A = qe * h.amp, B = fma(dx, qfx, dy * qfy) * ra;
          e[0] = make_double2(fma(A, h.j0, -(B * w1)), fma(B, h.j1, A * w0));
          const double At = te * h.amp, Bt = -(fma(dx, tfx, dy * tfy) * ra);
          et[0] = make_double2(fma(At, h.j0, -(Bt * w1)), fma(Bt, h.j1, At * w0));
        } else {
          const double kn = fma(tfx, qfx, tfy * qfy) * eta_inv;
          const double j0a = h.j0 * h.amp, w0a = w0 * h.amp, w1a = w1 * ra, j1a = h.j1 * ra;
          const double D = fma(dx, tfx, dy * tfy) * qe;
          e[0] = make_double2(-(qe * w0a), qe * j0a);
          e[NO - 1] = make_double2(fma(kn, e[0].y, -(D * w1a)), fma(-kn, e[0].x, D * j1a));
          const double Dt = -(fma(dx, qfx, dy * qfy) * te);
          et[0] = make_double2(-(te * w0a), te * j0a);
          et[NO - 1] = make_double2(fma(kn, et[0].y, -(Dt * w1a)), fma(-kn, et[0].x, Dt * j1a));
        }
        if (d == 0 && i == j) {
          e[0] = BC ? diag[2 * i] : diag[i];
          if constexpr (BC == 1) {
            // C_ii = -D'_ii - i (omega^2 / eta) S_ii
            const double k = omega * omega * eta_inv;
            const double2 D = diag[2 * i + 1];
            e[NO - 1] = make_double2(fma(k, e[0].y, -D.x), -fma(k, e[0].x, D.y));
          }
        }
#pragma unroll
        for (int r = 0; r < R; ++r)
#pragma unroll
          for (int o = 0; o < NO; ++o) {
            acc[r][o] = cmad(acc[r][o], e[o], q[r][o]);
            if (d > 0 && ok) {
              const double2 t = cmad(make_double2(0.0, 0.0), et[o], xi[r][o]);
              const int k = 2 * ((b * R + r) * NO + o);
              v[k] = t.x;
              v[k + 1] = t.y;
            }
          }
      }
      if (d == 0) continue;
      // value k ends in the lanes whose bits 4 .. 1 are k, then bit 0 joins
#pragma unroll
      for (int w = 8, o = 16; w >= 1; w /= 2, o /= 2) {
        const bool up = lane & o;
#pragma unroll
        for (int k = 0; k < w; ++k) {
          const double mine = up ? v[k + w] : v[k], other = up ? v[k] : v[k + w];
          v[k] = mine + __shfl_xor_sync(0xffffffffu, other, o);
        }
      }
      v[0] += __shfl_xor_sync(0xffffffffu, v[0], 1);
      const int k = lane >> 1, o = (k >> 1) % NO, r = (k >> 1) / NO % R, b = (k >> 1) / (NO * R);
      const int j = jb + s0 + b;
      if (!(lane & 1) && j < n && r < nrhs)
        reinterpret_cast<double*>(
            part + (((size_t)o * nsp + splits + d - 1) * nrhs + r) * n + j)[k & 1] = v[0];
    }
  }
  if (!ok) return;
#pragma unroll
  for (int r = 0; r < R; ++r)
    if (r < nrhs)
#pragma unroll
      for (int o = 0; o < NO; ++o)
        part[(((size_t)o * nsp + blockIdx.y) * nrhs + r) * n + i] = acc[r][o];
}

// Sum split partials in a fixed order: four threads per element take every
// fourth split, then two shuffles join them.  Soft: y = sum.  Hard: t = S u,
// y = 1/2 x + C x.
template <int BC>
__global__ void __launch_bounds__(256)
k_reduce_fp64(size_t tot, int splits, const double2* __restrict__ part,
              const double2* __restrict__ x, double2* __restrict__ t_out,
              double2* __restrict__ y) {
  // element by lane % 8, split group by lane / 8: eight neighbouring
  // elements are one 128-byte line
  const int lane = threadIdx.x & 31, g = lane >> 3;
  const size_t e = ((size_t)blockIdx.x * 256 + threadIdx.x) / 32 * 8 + (lane & 7);
  double2 s[BC ? 2 : 1];
#pragma unroll
  for (int o = 0; o < (BC ? 2 : 1); ++o) {
    double2 v = make_double2(0.0, 0.0);
    if (e < tot) {
#pragma unroll 4
      for (int sp = g; sp < splits; sp += 4) {
        const double2 p = part[((size_t)o * splits + sp) * tot + e];
        v.x += p.x;
        v.y += p.y;
      }
    }
    for (int k = 8; k < 32; k *= 2) {
      v.x += __shfl_xor_sync(0xffffffffu, v.x, k);
      v.y += __shfl_xor_sync(0xffffffffu, v.y, k);
    }
    s[o] = v;
  }
  if (e >= tot || g) return;
  if (BC == 0) {
    y[e] = s[0];
  } else {
    const double2 xv = x[e], c = s[BC ? 1 : 0];
    y[e] = make_double2(fma(0.5, xv.x, c.x), fma(0.5, xv.y, c.y));
    t_out[e] = s[0];
  }
}

// out[k][i] = base[k][i] + (scale / s_i) sum_j c_{(i-j) mod n} in[k][j]
// (spectral derivative as a circulant; c_d = (-1)^d cot(pi d / n) / 2)
constexpr int SPT = 256;
__global__ void __launch_bounds__(SPT)
k_spectral_fp64(int n, const double* __restrict__ ct, const double* __restrict__ sp,
                const double2* __restrict__ in, const double2* __restrict__ base, double2 scale,
                double2* __restrict__ out) {
  __shared__ double2 xs[SPT];
  const int i = blockIdx.x * SPT + threadIdx.x;
  const int k = blockIdx.y;
  const double2* ink = in + (size_t)k * n;
  double2 acc = make_double2(0.0, 0.0);
  for (int j0 = 0; j0 < n; j0 += SPT) {
    __syncthreads();
    int jj = j0 + threadIdx.x;
    xs[threadIdx.x] = jj < n ? ink[jj] : make_double2(0.0, 0.0);
    __syncthreads();
    if (i < n) {
      int jn = min(SPT, n - j0);
      int idx = i - j0;
      if (idx < 0) idx += n;
      for (int q = 0; q < jn; ++q) {
        double c = ct[idx];
        acc.x = fma(c, xs[q].x, acc.x);
        acc.y = fma(c, xs[q].y, acc.y);
        idx = idx == 0 ? n - 1 : idx - 1;
      }
    }
  }
  if (i < n) {
    double inv = 1.0 / sp[i];
    double2 sc = make_double2(scale.x * inv, scale.y * inv);
    double2 v = make_double2(sc.x * acc.x - sc.y * acc.y, sc.x * acc.y + sc.y * acc.x);
    if (base) {
      double2 b = base[(size_t)k * n + i];
      v.x += b.x;
      v.y += b.y;
    }
    out[(size_t)k * n + i] = v;
  }
}

// How one product is cut: right-hand sides per CTA, targets per CTA, source
// splits.  Two or three CTAs fit an SM; 16 per SM fill their waves (640 CTAs of
// star n = 4096, 16 right-hand sides, sound hard, left the FP64 pipe idle 20 %
// of the time).  Problems of fewer 64 x 32 tiles than eight per SM take
// 32-target tiles.
// k_pair_sym takes one or two sums per entry (sound soft: right-hand sides, sound
// hard: two each), and three or four up to n = 2048, where its smaller units fill the
// GPU better (four right-hand sides, n = 1024 159 -> 131 us, 2048 386 -> 414 kite and
// 394 -> 375 circle; further up the reduction of each sum over the rows costs more
// than the shared evaluation saves: n = 3072 807 -> 826 us, 8192 4.96 -> 5.37 ms, sound
// hard, two, 3072 1078 -> 1088 us, 8192 6.02 -> 6.37 ms).  From n = 400 on: below, the
// block kernel has at most one tile per SM (kite n = 384, one right-hand side 57
// against 52 us).  And while its partial sums, one per block distance, stay within
// 512 MB (or the caller's scratch): n = 46000 for one sound-soft right-hand side.
struct pair_plan {
  int sym;                  // 0, or the right-hand sides of k_pair_sym (1, 2, 4)
  int rbt, ti, splits, tps;
  int parts;                // partial sums per output and element
};

pair_plan plan_pair(int n, int nrhs, int hard, int device, size_t max_parts) {
  pair_plan p{};
  int sms = 152;
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device);
  const size_t vec = sizeof(double2) * (hard ? 2 : 1) * (size_t)n * nrhs;
  const int sums = nrhs * (hard ? 2 : 1);
  if (n >= 400 && (sums <= 2 || (sums <= 4 && n <= 2048))) {
    const int nblk = (n + 31) / 32, units = 4 * (nblk / 2 + 1);
    const int want = (32 * sms + nblk - 1) / nblk;       // about 32 warps per SM
    p.tps = (units + std::min(units, want) - 1) / std::min(units, want);
    p.splits = (units + p.tps - 1) / p.tps;
    p.parts = p.splits + nblk / 2;
    if ((size_t)p.parts <= max_parts && p.parts * vec <= (size_t)512 << 20) {
      p.sym = nrhs <= 2 ? nrhs : 4;
      return p;
    }
  }
  p.rbt = sums64::block_width(nrhs, hard);
  const int rhsblocks = (nrhs + p.rbt - 1) / p.rbt, ntiles = (n + sums64::TJ - 1) / sums64::TJ;
  p.ti = sums64::block_rows(p.rbt, hard);
  if ((long long)((n + 63) / 64) * ntiles * rhsblocks < 8LL * sms) p.ti = 32;
  const int rows = (n + p.ti - 1) / p.ti * rhsblocks;
  const int target = 16 * sms;   // several waves of the two or three CTAs that fit an SM
  p.splits = std::max<int>(1, std::min<size_t>(std::min<size_t>(ntiles, max_parts),
                                               (target + rows - 1) / rows));
  p.tps = (ntiles + p.splits - 1) / p.splits;
  p.splits = p.parts = (ntiles + p.tps - 1) / p.tps;
  return p;
}

template <int BC, int R>
void launch_sym(cfie_op* op, const pair_plan& p, const double2* x, const double2* u, int nrhs,
                double2* part) {
  const int n = op->n, nblk = (n + 31) / 32;
  const double f = h64::pair_factor(op->omega, op->h);   // hq c0
  prof_scope ps(op->ctx, CFIE_K_MATVEC_FP64);
  k_pair_sym<BC, R><<<dim3(nblk, p.splits), 32, 0, op->ctx->stream>>>(
      n, nblk, op->omega, 1.0 / op->omega, h64::near_amp(op->omega), 1.0 / op->eta, op->omega * f, BC ? f : f * op->eta,
      p.tps, p.splits, op->g, op->wtab.as<double>() + n, op->diag.as<double2>(), x, u, nrhs, part);
  CFIE_CHECK_LAUNCH();
}

// partial sums of every output, then their reduction (soft: into y; hard: t = S
// u and y = 1/2 x + C x)
template <int BC>
void run_pair(cfie_op* op, const pair_plan& p, const double2* x, const double2* u, int nrhs,
              double2* part, double2* t, double2* y) {
  if (p.sym == 1)
    launch_sym<BC, 1>(op, p, x, u, nrhs, part);
  else if (p.sym == 2)
    launch_sym<BC, 2>(op, p, x, u, nrhs, part);
  else if (BC == 0 && p.sym == 4)
    launch_sym<0, 4>(op, p, x, u, nrhs, part);
  else {
    const double f = h64::pair_factor(op->omega, op->h);   // hq c0
    prof_scope ps(op->ctx, CFIE_K_MATVEC_FP64);
    sums64::block_args a{};
    a.n = a.rows = op->n;
    a.nrhs = nrhs;
    a.splits = p.splits;
    a.tiles_per_split = p.tps;
    a.omega = op->omega;
    a.omega_inv = 1.0 / op->omega;
    a.near = h64::near_amp(op->omega);
    a.nf = op->omega * f;
    a.sf = BC ? f : f * op->eta;
    a.eta_inv = 1.0 / op->eta;
    a.g = op->g;
    a.wks = op->wtab.as<double>() + op->n;
    a.diag = op->diag.as<double2>();
    a.x = x;
    a.u = u;
    a.out = part;
    sums64::run_block<BC>(a, p.ti, p.rbt, op->ctx->stream);
  }
  reduce_fp64(op, part, p.parts, x, t, y, nrhs);
}

}  // namespace

// out = base + scale (1/|z'|) d/dt in: by FFT (O(n log n) per column); the
// allocation-free variant below keeps the circulant kernel
void spectral_apply(cfie_op* op, const double2* in, double2* out, const double2* base,
                    double2 scale, int nrhs) {
  spectral_fft64(op, in, out, base, scale, nrhs);
}

void reduce_fp64(cfie_op* op, const double2* part, int splits, const double2* x, double2* t,
                 double2* y, int nrhs) {
  const size_t tot = (size_t)op->n * nrhs;
  const unsigned blocks = (unsigned)((tot + 63) / 64);
  if (op->bc == CFIE_SOUND_HARD)
    k_reduce_fp64<1><<<blocks, 256, 0, op->ctx->stream>>>(tot, splits, part, x, t, y);
  else
    k_reduce_fp64<0><<<blocks, 256, 0, op->ctx->stream>>>(tot, splits, part, x, t, y);
  CFIE_CHECK_LAUNCH();
}

void matvec_fp64(cfie_op* op, const double2* x, double2* y, int nrhs) {
  const bool hard = op->bc == CFIE_SOUND_HARD;
  const pair_plan p = plan_pair(op->n, nrhs, hard, op->ctx->device, 1 << 20);
  const size_t tot = (size_t)op->n * nrhs;
  op->partial.reserve(sizeof(double2) * (hard ? 2 : 1) * (size_t)p.parts * tot);
  double2* part = op->partial.as<double2>();
  if (!hard) {
    run_pair<0>(op, p, x, nullptr, nrhs, part, nullptr, y);
    op->partial.trim();
    return;
  }
  op->tmp1.reserve(sizeof(double2) * tot);
  op->tmp2.reserve(sizeof(double2) * tot);
  double2* u = op->tmp1.as<double2>();
  double2* t = op->tmp2.as<double2>();
  // u = (1/s) Dt x
  spectral_apply(op, x, u, nullptr, make_double2(1.0, 0.0), nrhs);
  run_pair<1>(op, p, x, u, nrhs, part, t, y);
  op->partial.trim();
  // y += (1/(i eta)) (1/s) Dt t
  spectral_apply(op, t, y, y, make_double2(0.0, -1.0 / op->eta), nrhs);
}

// ---------------------------------------------------------------------------
// Allocation-free variant of the FP64 matvec (cfie_apply_fp64_static).
//
// The split-source partial sums (and, for the sound-hard operator, the two
// derivative vectors) live in one file-scope device array instead of buffers
// the operator grows with cudaMalloc.  Every GPU that loads the library holds
// this array until the process exits.  Its device address is looked up once
// per device (cudaGetSymbolAddress, with that device current) on the first
// call there, and again if the device's context has been replaced since;
// host code never hands the array's name itself to a kernel.
// Each call overwrites every scratch element it later reads, so nothing has to
// start at zero; calls that overlap on the GPU share the array and race.
// ---------------------------------------------------------------------------
namespace {

constexpr size_t kStaticScratchBytes = size_t(32) << 20;  // 32 MiB
constexpr int kMaxDevices = 64;

static __device__ __align__(256) unsigned char g_static_scratch[kStaticScratchBytes];

// The address is cached per device together with the device's current CUDA
// context: a context torn down and created again (cudaDeviceReset) reloads the
// module, so a cached address from the old context is looked up afresh.
using ctx_get_fn = CUresult (*)(CUcontext*);
ctx_get_fn driver_ctx_get_current() {
  static ctx_get_fn fn = [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q{};
    if (cudaGetDriverEntryPointByVersion("cuCtxGetCurrent", &p, 12000, cudaEnableDefault, &q) !=
            cudaSuccess ||
        q != cudaDriverEntryPointSuccess)
      p = nullptr;
    return reinterpret_cast<ctx_get_fn>(p);
  }();
  return fn;
}

std::mutex g_static_mu;
void* g_static_addr[kMaxDevices] = {};
CUcontext g_static_ctx[kMaxDevices] = {};

void* static_scratch_address(int device) {
  if (device < 0 || device >= kMaxDevices)
    throw cfie_error(CFIE_EINVAL, "device index out of range for the static scratch table");
  ctx_get_fn get = driver_ctx_get_current();
  CUcontext cur = nullptr;
  if (!get || get(&cur) != CUDA_SUCCESS || !cur)
    throw cfie_error(CFIE_ECUDA, "cuCtxGetCurrent: no current CUDA context for the static scratch");
  std::lock_guard<std::mutex> lock(g_static_mu);
  if (!g_static_addr[device] || g_static_ctx[device] != cur) {
    void* p = nullptr;
    cudaError_t e = cudaGetSymbolAddress(&p, g_static_scratch);
    if (e != cudaSuccess || !p)
      throw cfie_error(CFIE_ECUDA, std::string("cudaGetSymbolAddress(static scratch): ") +
                                       cudaGetErrorString(e));
    g_static_addr[device] = p;
    g_static_ctx[device] = cur;
  }
  return g_static_addr[device];
}

}  // namespace

size_t static_scratch_capacity() { return kStaticScratchBytes; }

void matvec_fp64_static(cfie_op* op, const double2* x, double2* y, int nrhs) {
  const int n = op->n;
  const bool hard = op->bc == CFIE_SOUND_HARD;
  const size_t tot = (size_t)n * nrhs;
  const size_t vec_bytes = sizeof(double2) * tot;
  const size_t fixed = hard ? 2 * vec_bytes : 0;          // u and t
  const size_t per_split = sizeof(double2) * (hard ? 2 : 1) * tot;
  // the documented limit (16 and 96 bytes per element; the hard form now uses
  // 64 of them)
  const size_t need = (hard ? 6 : 1) * vec_bytes;
  if (need > kStaticScratchBytes)
    throw cfie_error(CFIE_EINVAL,
                     "cfie_apply_fp64_static: n * nrhs too large for the 32 MiB static scratch "
                     "(needs " + std::to_string(need) + " bytes)");
  // device address of the array on the context's (current) device
  unsigned char* base = static_cast<unsigned char*>(static_scratch_address(op->ctx->device));
  const size_t fit = (kStaticScratchBytes - fixed) / per_split;
  const pair_plan p = plan_pair(n, nrhs, hard, op->ctx->device, fit);
  double2* part = reinterpret_cast<double2*>(base + fixed);
  if (!hard) {
    run_pair<0>(op, p, x, nullptr, nrhs, part, nullptr, y);
    return;
  }
  double2* u = reinterpret_cast<double2*>(base);
  double2* t = reinterpret_cast<double2*>(base + vec_bytes);
  cudaStream_t st = op->ctx->stream;
  const dim3 sgrid((n + SPT - 1) / SPT, nrhs);
  k_spectral_fp64<<<sgrid, SPT, 0, st>>>(n, op->ctab.as<double>(), op->g.sp, x, nullptr,
                                          make_double2(1.0, 0.0), u);
  CFIE_CHECK_LAUNCH();
  run_pair<1>(op, p, x, u, nrhs, part, t, y);
  k_spectral_fp64<<<sgrid, SPT, 0, st>>>(n, op->ctab.as<double>(), op->g.sp, t, y,
                                          make_double2(0.0, -1.0 / op->eta), y);
  CFIE_CHECK_LAUNCH();
}
