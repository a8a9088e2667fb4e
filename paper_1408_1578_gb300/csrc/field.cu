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
// Hankel evaluation: the block kernel of sums64.cuh.
//
// Bound: the FP64 pipe, about 31 instructions per kernel value, which the
// densities of a block share.  When the points alone do not fill the GPU the
// sources are split across CTAs and a second kernel adds the splits in a fixed
// order.
// Measured (GB300): 16 densities of n = 4096 nodes at 20000 points, sound hard,
// 70.2 -> 6.8 ms.
#include <algorithm>

#include "hankel64.cuh"
#include "internal.h"
#include "sums64.cuh"

namespace {

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

}  // namespace

void field_eval(cfie_op* op, const double2* q, int nrhs, int npts, const double2* pts,
                double2* u) {
  const bool hard = op->bc == CFIE_SOUND_HARD;
  const double f = h64::pair_factor(op->omega, op->h);   // h c0 / 4
  const int width = sums64::block_width(nrhs, false), ti = sums64::block_rows(width, false);
  const int tiles = (op->n + sums64::TJ - 1) / sums64::TJ;
  const size_t tot = (size_t)nrhs * npts;
  // about 16 CTAs per SM (two fit, so that the last of several waves is a small
  // part), as many splits of the sources as that takes (no more partial sums
  // than 256 MB)
  int sms = 152;
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, op->ctx->device);
  const long long ctas = (long long)((npts + ti - 1) / ti) * ((nrhs + width - 1) / width);
  long long splits = std::max<long long>(1, (16LL * sms + ctas - 1) / ctas);
  splits = std::min<long long>(splits, std::min<long long>(tiles, std::max<size_t>(1, ((size_t)1 << 24) / tot)));
  sums64::block_args a{};
  a.tiles_per_split = (int)((tiles + splits - 1) / splits);
  a.splits = (tiles + a.tiles_per_split - 1) / a.tiles_per_split;
  a.n = op->n;
  a.rows = npts;
  a.nrhs = nrhs;
  a.rotate = hard;   // -S + D / (i eta) = -i (D / eta - i S)
  a.omega = op->omega;
  a.omega_inv = 1.0 / op->omega;
  a.near = h64::near_amp(op->omega);
  a.nf = hard ? op->omega * f / op->eta : op->omega * f;
  a.sf = hard ? f : op->eta * f;
  a.g = op->g;
  a.pts = pts;
  a.x = q;
  a.out = u;
  if (a.splits > 1) {
    op->partial.reserve(sizeof(double2) * tot * a.splits);
    a.out = op->partial.as<double2>();
  }
  sums64::run_block<sums64::FIELD>(a, ti, width, op->ctx->stream);
  if (a.splits > 1) {
    k_field_sum<<<(unsigned)((tot + 255) / 256), 256, 0, op->ctx->stream>>>(tot, a.splits, a.out, u);
    CFIE_CHECK_LAUNCH();
    op->partial.trim();
  }
}
