// Off-surface scattered field from the boundary density (step after the solve;
// Section 1 of the paper evaluates u through a boundary integral without
// writing it out).  Representations whose boundary limits give eq. 1 and
// eq. 2 through the jump relations (outward normal):
//
//     sound soft:  u(x) = (D q)(x) - i eta (S q)(x)
//     sound hard:  u(x) = -(S q)(x) + (D q)(x) / (i eta)
//
//     (S q)(x) = h sum_j (i/4) H0(omega r_j) |z'_j| q_j
//     (D q)(x) = h sum_j (i/4) omega H1(omega r_j) ((x - z_j) . nu~_j / r_j) q_j
//
// discretised by the plain trapezoidal rule (spectrally accurate a few node
// spacings away from the curve), FP64 throughout with the library's own
// Hankel evaluation.  Up to four densities: one thread per (point, quarter of
// the sources), sources staged in shared memory a tile at a time, the quarters
// added at the end.  More: the block kernel of sums64.cuh.
//
// Bound: the FP64 pipe, about 36 instructions per kernel value, which the
// densities of a block share.  When the points alone do not fill the GPU the
// sources are split across CTAs and a second kernel adds the splits in a fixed
// order.
// Measured (GB300): 16 densities of n = 4096 nodes at 20000 points, sound hard,
// 70.2 -> 7.4 ms.
#include <algorithm>

#include "hankel64.cuh"
#include "internal.h"
#include "sums64.cuh"

namespace {

constexpr int FPT = 64;      // points per CTA
constexpr int FSPL = 4;      // source quarters (threads per point)
constexpr int FNT = FPT * FSPL;
constexpr int FTJ = 128;     // sources per shared-memory tile

// out: u, or with several splits the partial sums [split][density][point]
template <int BC, int FRB>
__global__ void __launch_bounds__(FNT)
k_field(int n, int npts, int nrhs, int tiles_per_split, double omega, double eta, double h,
        geom_dev g, const double2* __restrict__ pts, const double2* __restrict__ q,
        double2* __restrict__ out) {
  __shared__ double sx[FTJ], sy[FTJ], sfx[FTJ], sfy[FTJ], se[FTJ];
  // densities of the tile during the loop, the quarters' sums after it
  constexpr int BUF = FTJ * FRB > FSPL * FPT ? FTJ * FRB : FSPL * FPT;
  __shared__ double2 buf[BUF];
  double2 (*sq)[FRB] = reinterpret_cast<double2 (*)[FRB]>(buf);
  const int tid = threadIdx.x;
  const int pl = tid % FPT, quarter = tid / FPT;
  const int p = blockIdx.x * FPT + pl;
  const int rn = min(FRB, nrhs);
  const int j_begin = blockIdx.z * tiles_per_split * FTJ;
  const int j_end = min(n, j_begin + tiles_per_split * FTJ);
  const double f = 0.25 * 0.7978845608028654 * h;   // h c0 / 4
  const double nf = BC == 0 ? omega * f : omega * f / eta, sf = BC == 0 ? eta * f : f;
  const double omega_inv = 1.0 / omega;
  const double2 xp = p < npts ? pts[p] : make_double2(0.0, 0.0);
  double2 acc[FRB];
#pragma unroll
  for (int k = 0; k < FRB; ++k) acc[k] = make_double2(0.0, 0.0);
  for (int j0 = j_begin; j0 < j_end; j0 += FTJ) {
    __syncthreads();
    for (int e = tid; e < FTJ; e += FNT) {
      const int j = j0 + e;
      const bool ok = j < n;
      sx[e] = ok ? g.x[j] : 0.0;
      sy[e] = ok ? g.y[j] : 0.0;
      sfx[e] = ok ? nf * g.nx[j] : 0.0;
      sfy[e] = ok ? nf * g.ny[j] : 0.0;
      se[e] = ok ? sf * g.sp[j] : 0.0;
    }
    for (int e = tid; e < FTJ * FRB; e += FNT) {
      const int jl = e / FRB, k = e % FRB, j = j0 + jl;
      sq[jl][k] = (j < n && k < rn) ? q[(size_t)k * n + j] : make_double2(0.0, 0.0);
    }
    __syncthreads();
    if (p >= npts) continue;
    const int jn = min(FTJ, j_end - j0);
    for (int jl = quarter; jl < jn; jl += FSPL) {
      const double dx = xp.x - sx[jl], dy = xp.y - sy[jl];
      double r, rinv;
      h64::distance(fma(dx, dx, dy * dy), r, rinv);
      const h64::values v = h64::bessel01(omega * r, omega_inv * rinv, g.tab);
      // h times the kernel, H = J + i Y:  S = (i/4) H0 |z'|, D = (i/4) omega H1
      // (x - z) . nu~ / r, soft D - i eta S, hard -S + D / (i eta)
      const double A = se[jl] * v.amp;
      const double B = fma(dx, sfx[jl], dy * sfy[jl]) * (rinv * v.amp);
      const double2 c = BC == 0 ? make_double2(fma(A, v.j0, -(B * v.y1)), fma(A, v.y0, B * v.j1))
                                : make_double2(fma(A, v.y0, B * v.j1), fma(B, v.y1, -(A * v.j0)));
#pragma unroll
      for (int k = 0; k < FRB; ++k) {
        const double2 qq = sq[jl][k];
        acc[k].x = fma(c.x, qq.x, acc[k].x);
        acc[k].x = fma(-c.y, qq.y, acc[k].x);
        acc[k].y = fma(c.x, qq.y, acc[k].y);
        acc[k].y = fma(c.y, qq.x, acc[k].y);
      }
    }
  }
  double2* dst = out + (size_t)blockIdx.z * nrhs * npts;
#pragma unroll
  for (int k = 0; k < FRB; ++k) {
    __syncthreads();   // the buffer's last readers are done
    if (k >= rn) continue;
    buf[tid] = acc[k];
    __syncthreads();
    if (quarter == 0 && p < npts) {
      double2 s = buf[pl];
      for (int t = 1; t < FSPL; ++t) {
        s.x += buf[t * FPT + pl].x;
        s.y += buf[t * FPT + pl].y;
      }
      dst[(size_t)k * npts + p] = s;
    }
  }
}

__global__ void k_field_sum(size_t tot, int splits, const double2* __restrict__ part,
                            double2* __restrict__ u) {
  const size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= tot) return;
  double2 s = part[e];
#pragma unroll 4
  for (int k = 1; k < splits; ++k) {
    const double2 v = part[(size_t)k * tot + e];
    s.x += v.x;
    s.y += v.y;
  }
  u[e] = s;
}

// about 16 CTAs per SM (two fit, so that the last of several waves is a small
// part): source splits of `tiles` tiles for `ctas` CTAs without, with no more
// partial sums than 256 MB, and each one's tiles
void split_sources(cfie_op* op, size_t tot, int tiles, long long ctas, int& splits, int& tps) {
  int sms = 152;
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, op->ctx->device);
  long long s = std::max<long long>(1, (16LL * sms + ctas - 1) / ctas);
  s = std::min<long long>(s, std::min<long long>(tiles, std::max<size_t>(1, ((size_t)1 << 24) / tot)));
  tps = (int)((tiles + s - 1) / s);
  splits = (tiles + tps - 1) / tps;
}

// where the partial sums of several splits go, and their sum
double2* field_partials(cfie_op* op, size_t tot, int splits, double2* u) {
  if (splits == 1) return u;
  op->partial.reserve(sizeof(double2) * tot * splits);
  return op->partial.as<double2>();
}
void sum_splits(cfie_op* op, size_t tot, int splits, const double2* part, double2* u) {
  if (splits == 1) return;
  k_field_sum<<<(unsigned)((tot + 255) / 256), 256, 0, op->ctx->stream>>>(tot, splits, part, u);
  CFIE_CHECK_LAUNCH();
}

template <int BC, int FRB>
void launch_field(cfie_op* op, const double2* q, int nrhs, int npts, const double2* pts,
                  double2* u) {
  const int n = op->n, px = (npts + FPT - 1) / FPT;
  const size_t tot = (size_t)nrhs * npts;
  int splits, tps;
  split_sources(op, tot, (n + FTJ - 1) / FTJ, px, splits, tps);
  double2* out = field_partials(op, tot, splits, u);
  k_field<BC, FRB><<<dim3(px, 1, splits), FNT, 0, op->ctx->stream>>>(
      n, npts, nrhs, tps, op->omega, op->eta, op->h, op->g, pts, q, out);
  CFIE_CHECK_LAUNCH();
  sum_splits(op, tot, splits, out, u);
}

// five and more densities: entries shared by up to 64, sums on the integer units
void launch_block_field(cfie_op* op, bool hard, const double2* q, int nrhs, int npts,
                        const double2* pts, double2* u) {
  const double f = 0.25 * 0.7978845608028654 * op->h;   // h c0 / 4
  const int width = sums64::block_width(nrhs, false), ti = sums64::block_rows(width, false);
  const size_t tot = (size_t)nrhs * npts;
  sums64::block_args a{};
  split_sources(op, tot, (op->n + sums64::TJ - 1) / sums64::TJ,
                (long long)((npts + ti - 1) / ti) * ((nrhs + width - 1) / width), a.splits,
                a.tiles_per_split);
  a.n = op->n;
  a.rows = npts;
  a.nrhs = nrhs;
  a.rotate = hard;   // -S + D / (i eta) = -i (D / eta - i S)
  a.omega = op->omega;
  a.omega_inv = 1.0 / op->omega;
  a.nf = hard ? op->omega * f / op->eta : op->omega * f;
  a.sf = hard ? f : op->eta * f;
  a.g = op->g;
  a.pts = pts;
  a.x = q;
  a.out = field_partials(op, tot, a.splits, u);
  sums64::run_block<sums64::FIELD>(a, ti, width, op->ctx->stream);
  sum_splits(op, tot, a.splits, a.out, u);
}

template <int BC>
void field_bc(cfie_op* op, const double2* q, int nrhs, int npts, const double2* pts, double2* u) {
  if (nrhs > 4)
    launch_block_field(op, BC == 1, q, nrhs, npts, pts, u);
  else if (nrhs == 1)
    launch_field<BC, 1>(op, q, nrhs, npts, pts, u);
  else if (nrhs == 2)
    launch_field<BC, 2>(op, q, nrhs, npts, pts, u);
  else
    launch_field<BC, 4>(op, q, nrhs, npts, pts, u);
}

}  // namespace

void field_eval(cfie_op* op, const double2* q, int nrhs, int npts, const double2* pts,
                double2* u) {
  if (op->bc == CFIE_SOUND_SOFT)
    field_bc<0>(op, q, nrhs, npts, pts, u);
  else
    field_bc<1>(op, q, nrhs, npts, pts, u);
}
