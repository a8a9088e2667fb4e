// Sums of FP64 kernel entries over a block of right-hand sides, on the integer
// units: y_r(i) = sum_j K_ij x_r(j).
//
// GB300 has 1.7 lanes of FP64 multiply-add per clock and SM, and 25 of 32 x 32
// -> 64-bit integer multiply-add.  An entry takes about 40 FP64 instructions
// (hankel64.cuh); its sums took 4 more per right-hand side, twice that for the
// sound-hard operator's two.  Here a tile of 32 sources works in fixed point:
// the 32 entries of a row share the exponent of the largest of them, the 32
// densities of a column share theirs, each number is rounded to 57 bits and a
// sign below it and kept as two 29-bit limbs.  Three integer multiply-adds
// (high x high, the two mixed products) give a real product, the tile's sums
// stay below 2^63, and at its end one conversion and one FP64 multiply-add take
// each of them to the FP64 accumulator.  Within a tile an addend is off by
// at most 2^-56 of the largest entry times the largest density, and
// additions are exact, where FP64 rounds each to 2^-53 of the sum so far.
// Measured (GB300): star n = 4096, 16 right-hand sides, sound hard, 6.2 -> 3.2 ms;
// 16 densities at 20000 points 20.7 -> 10.9 ms.
//
// So an addend loses what lies between the largest entry times the largest
// density and itself, which is at most the smaller of the two ranges: where a row's
// entries in a tile range over more than 2^kSpread and so does a column of
// densities, the row's sums of that tile are FP64 multiply-adds with the entries as
// they were evaluated.  So they are in a tile with a value that fixed point does not
// hold (infinities, NaN, exponents beyond 2^+-420).
//
// Layout: a CTA owns TI rows and walks its range of source tiles.  It evaluates
// the TI x 32 block of entries into shared memory (one warp per row, lanes over
// sources: the row's exponent is one reduction), then thread (row, group)
// contracts its row with RBT / RG of the columns.
#pragma once
#include "hankel64.cuh"
#include "internal.h"

namespace sums64 {

constexpr int TJ = 32;
enum { SOFT = 0, HARD = 1, FIELD = 2 };

// a number v < 2^(E - 1022), E a biased exponent, as v 2^(1079 - E) = hi 2^29 + lo
// rounded to the nearest integer (|hi|, |lo| <= 2^28)
__device__ __forceinline__ void to_limbs(double v, int E, int& hi, int& lo) {
  const int h = __double2hiint(v), e = (h >> 20) & 0x7ff;
  unsigned long long m =
      ((unsigned long long)((h & 0xfffff) | 0x100000) << 32 | (unsigned)__double2loint(v)) << 5;
  m = e ? m >> min(E - e, 63) : 0;   // subnormals round to zero
  long long V = (long long)((m + 1) >> 1);
  if (h < 0) V = -V;
  hi = (int)((V + (1 << 28)) >> 29);
  lo = (int)((unsigned)V - ((unsigned)hi << 29));
}
__device__ __forceinline__ int4 to_limbs(double2 v, int E) {
  int4 q;
  to_limbs(v.x, E, q.x, q.y);
  to_limbs(v.y, E, q.z, q.w);
  return q;
}
// Range of a row's or a column's 32 values, from which the sums' form follows.  An
// addend is off by 2^-56 of the largest entry times the largest density, so with
// one of the ranges up to 2^kSpread a tile's sum is off by about 2^(kSpread - 53) of
// sum |K x| at the very worst (one small product alone), where even values leave
// 2^-56.  Random densities range wider than 2^7 in 5 of 1000 columns of a tile
// (normal) or 1 of 2000 (uniform), entries where sound hard C, or the 1 +- cos of the
// others, goes through zero.  Measured (GB300), against no limit at all: 2^7 star n
// = 4096, 16, sound hard 2.25 -> 2.25 ms, field 6.85 -> 6.85 ms; 2^6 2.28, 6.99 ms; with
// a row's smallest entry looked for only where a column ranges that wide 2.24, 6.81 ms.
constexpr int kSpread = 7;
constexpr int kRaw = 1 << 16;   // with a row's exponent: entries kept in FP64
struct tile_range {
  int e;           // exponent of the largest (zeros only: any)
  bool out, wide;  // not held in fixed point; smallest of the valid ones 2^-kSpread below
};
// (wide: whether that matters)
__device__ __forceinline__ tile_range range_of(double2 v, bool valid, bool wide) {
  const unsigned a = __double2hiint(v.x) & 0x7fffffff, b = __double2hiint(v.y) & 0x7fffffff;
  const unsigned m = max(a, b);
  const int E = (int)(__reduce_max_sync(0xffffffffu, m) >> 20);
  if (E >= 600 && E <= 1500) {
    if (wide)
      wide = E - (int)(__reduce_min_sync(0xffffffffu, valid ? m : 0xffffffffu) >> 20) > kSpread;
    return {E, false, wide};
  }
  const bool any = __any_sync(0xffffffffu, (a | b | __double2loint(v.x) | __double2loint(v.y)) != 0);
  return {E ? E : 1023, any, false};
}

// sums of products of limbs: high x high, and the mixed ones 2^29 below
struct fixed_acc {
  long long h, m;
  __device__ __forceinline__ void add(int ah, int al, int bh, int bl) {
    h += (long long)ah * bh;
    m += (long long)ah * bl;
    m += (long long)al * bh;
  }
  // scale: the high word of 2^(Ek + Ex - 2100)
  __device__ __forceinline__ void flush(double& acc, int scale) const {
    acc = fma((double)(h + ((m + (1 << 28)) >> 29)), __hiloint2double(scale, 0), acc);
  }
};

struct block_args {
  int n, rows, nrhs, splits, tiles_per_split;
  bool rotate;                         // FIELD: times -i (sound hard)
  double omega, omega_inv, near;       // near = sqrt(pi omega / 2)
  double nf, sf;                       // factors of the normal (HARD: of none) and the speed
  double eta_inv;                      // HARD
  geom_dev g;
  const double* wks;                   // Kress weights / (pi h)
  const double2 *diag, *pts, *x, *u;   // pts: FIELD; u: HARD
  double2* out;                        // [output][split][column][row]
};

template <int MODE, int TI, int RBT>
struct block_smem {
  static constexpr int NO = MODE == HARD ? 2 : 1;
  double tx[TI], ty[TI];
  // HARD: omega nu / |z'| and (omega / eta) nu / |z'|
  double tfx[NO == 2 ? TI : 1], tfy[NO == 2 ? TI : 1], tux[NO == 2 ? TI : 1], tuy[NO == 2 ? TI : 1];
  double sx[TJ], sy[TJ], sfx[TJ], sfy[TJ], se[TJ];
  double wk[TI + TJ];                    // Kress weights of the tile, by i - j
  int4 K[NO][TI][TJ + 1];                // limbs (re, im): the entries; HARD: S, C; raw rows: double2
  int4 X[NO][TJ][RBT];                   // densities; HARD: u, x
  int ek[NO][TI], ex[NO][RBT];
  int cols[NO];                          // 1: a wide column of densities, 2: one out of range
};

template <int MODE, int TI, int RBT, int RG>
__global__ void __launch_bounds__(TI* RG, 512 / (TI * RG))
k_block64(block_args p) {
  constexpr int NT = TI * RG, RQ = RBT / RG;
  constexpr int NO = MODE == HARD ? 2 : 1;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  block_smem<MODE, TI, RBT>& S = *reinterpret_cast<block_smem<MODE, TI, RBT>*>(smem_raw);
  const geom_dev& g = p.g;
  const int tid = threadIdx.x, lane = tid & 31, n = p.n;
  const int i0 = blockIdx.x * TI;
  const int rb0 = blockIdx.z * RBT;
  const int rbn = min(RBT, p.nrhs - rb0);
  const int t_begin = blockIdx.y * p.tiles_per_split;
  const int t_end = min((n + TJ - 1) / TJ, t_begin + p.tiles_per_split);

  if (tid < TI) {
    const int i = i0 + tid;
    const bool ok = i < p.rows;
    if constexpr (MODE == FIELD) {
      const double2 z = ok ? p.pts[i] : make_double2(0.0, 0.0);
      S.tx[tid] = z.x;
      S.ty[tid] = z.y;
    } else {
      S.tx[tid] = ok ? g.x[i] : 0.0;
      S.ty[tid] = ok ? g.y[i] : 0.0;
    }
    if constexpr (MODE == HARD) {
      const double inv = ok ? p.omega / g.sp[i] : 0.0;
      S.tfx[tid] = ok ? g.nx[i] * inv : 0.0;
      S.tfy[tid] = ok ? g.ny[i] * inv : 0.0;
      S.tux[tid] = S.tfx[tid] * p.eta_inv;
      S.tuy[tid] = S.tfy[tid] * p.eta_inv;
    }
  }

  if (tid < NO) S.cols[tid] = 0;

  const int row = tid % TI, rg = tid / TI;
  double2 acc[NO][RQ];
#pragma unroll
  for (int o = 0; o < NO; ++o)
#pragma unroll
    for (int q = 0; q < RQ; ++q) acc[o][q] = make_double2(0.0, 0.0);

  for (int t = t_begin; t < t_end; ++t) {
    const int j0 = t * TJ;
    __syncthreads();
    if (tid < TJ) {
      const int j = j0 + tid;
      const bool ok = j < n;
      const double sp = ok ? g.sp[j] : 1.0;
      const double m = MODE == HARD ? p.omega / sp : p.nf;
      S.sx[tid] = ok ? g.x[j] : 0.0;
      S.sy[tid] = ok ? g.y[j] : 0.0;
      S.sfx[tid] = ok ? m * g.nx[j] : 0.0;
      S.sfy[tid] = ok ? m * g.ny[j] : 0.0;
      S.se[tid] = p.sf * sp;
    }
    if constexpr (MODE != FIELD)
      for (int e = tid; e < TI + TJ - 1; e += NT) {
        int d = (i0 - j0 + e - (TJ - 1)) % n;
        if (d < 0) d += n;
        S.wk[e] = p.wks[d];
      }
    for (int c = tid / 32; c < NO * RBT; c += NT / 32) {
      const int o = c / RBT, r = c % RBT, j = j0 + lane;
      const double2* src = o == NO - 1 ? p.x : p.u;
      const double2 v = j < n && r < rbn ? src[(size_t)(rb0 + r) * n + j] : make_double2(0.0, 0.0);
      const tile_range span = range_of(v, j < n, true);
      S.X[o][lane][r] = to_limbs(v, span.e);
      if (lane == 0) {
        S.ex[o][r] = span.e;
        if (span.out || span.wide) atomicOr(&S.cols[o], span.out ? 2 : 1);
      }
    }
    __syncthreads();

    // ---- entries of the TI x TJ block
    for (int il = tid / 32; il < TI; il += NT / 32) {
      const int i = i0 + il, j = j0 + lane;
      const bool in = i < p.rows && j < n && (MODE == FIELD || i != j);
      double2 a = make_double2(0.0, 0.0), b = a;
      if (in)
        pair_folded_fp64<MODE == HARD, MODE != FIELD>(
            S.tx[il] - S.sx[lane], S.ty[il] - S.sy[lane], p.omega, p.omega_inv, p.near,
            MODE == HARD ? S.tfx[il] : S.sfx[lane], MODE == HARD ? S.tfy[il] : S.sfy[lane],
            S.se[lane], MODE == FIELD ? 0.0 : S.wk[il - lane + TJ - 1], g.tab, a, b);
      if (MODE == FIELD && p.rotate) a = make_double2(a.y, -a.x);
      auto keep = [&](int o, double2 v) {
        const int c = S.cols[o];
        const tile_range span = range_of(v, in, c == 1);
        const bool raw = span.out || (c & 2) || span.wide;
        int4 q;
        if (raw)
          q = make_int4(__double2loint(v.x), __double2hiint(v.x), __double2loint(v.y),
                        __double2hiint(v.y));
        else
          q = to_limbs(v, span.e);
        S.K[o][il][lane] = q;
        if (lane == 0) S.ek[o][il] = raw ? span.e | kRaw : span.e;
      };
      keep(0, a);
      if constexpr (MODE == HARD) {
        // C = -D' - i (omega^2 / eta) (n_i . n_j) S
        const double k = fma(S.tux[il], S.sfx[lane], S.tuy[il] * S.sfy[lane]);
        keep(NO - 1, make_double2(fma(k, a.y, -b.x), -fma(k, a.x, b.y)));
      }
    }

    // ---- contraction
    __syncthreads();
    if (tid < NO) S.cols[tid] = 0;
    const int self = MODE == FIELD ? -1 : i0 + row - j0;   // the diagonal entry's source
    if (MODE != FIELD && self >= 0 && self < TJ && i0 + row < n) {
      // in FP64: sound soft it holds the 1/2 of the identity, whose exponent would
      // take twelve bits from the other entries of the tile
      const int i = i0 + row;
      double2 d[NO];
      d[0] = MODE == HARD ? p.diag[2 * i] : p.diag[i];
      if constexpr (MODE == HARD) {
        // C_ii = -D'_ii - i (omega^2 / eta) S_ii
        const double k = p.omega * p.omega * p.eta_inv;
        const double2 D = p.diag[2 * i + 1];
        d[NO - 1] = make_double2(fma(k, d[0].y, -D.x), -fma(k, d[0].x, D.y));
      }
#pragma unroll
      for (int o = 0; o < NO; ++o) {
        const double2* src = o == NO - 1 ? p.x : p.u;
#pragma unroll
        for (int q = 0; q < RQ; ++q) {
          const int r = rg + RG * q;
          if (r >= rbn) continue;
          const double2 v = src[(size_t)(rb0 + r) * n + i];
          acc[o][q].x = fma(-d[o].y, v.y, fma(d[o].x, v.x, acc[o][q].x));
          acc[o][q].y = fma(d[o].y, v.x, fma(d[o].x, v.y, acc[o][q].y));
        }
      }
    }
    fixed_acc re[NO][RQ], im[NO][RQ];
#pragma unroll
    for (int o = 0; o < NO; ++o)
#pragma unroll
      for (int q = 0; q < RQ; ++q) re[o][q] = im[o][q] = fixed_acc{0, 0};
#pragma unroll 2
    for (int jl = 0; jl < TJ; ++jl)
#pragma unroll
      for (int o = 0; o < NO; ++o) {
        const int4 k = S.K[o][row][jl];
#pragma unroll
        for (int q = 0; q < RQ; ++q) {
          const int4 v = S.X[o][jl][rg + RG * q];
          re[o][q].add(k.x, k.y, v.x, v.y);
          re[o][q].add(-k.z, -k.w, v.z, v.w);
          im[o][q].add(k.x, k.y, v.z, v.w);
          im[o][q].add(k.z, k.w, v.x, v.y);
        }
      }
#pragma unroll
    for (int o = 0; o < NO; ++o) {
      const int ek = S.ek[o][row];
      if (!(ek & kRaw)) {
#pragma unroll
        for (int q = 0; q < RQ; ++q) {
          const int scale = (ek + S.ex[o][rg + RG * q] - 1077) << 20;
          re[o][q].flush(acc[o][q].x, scale);
          im[o][q].flush(acc[o][q].y, scale);
        }
        continue;
      }
      // the row's entries are in FP64, the sums above meaningless
      const double2* src = o == NO - 1 ? p.x : p.u;
#pragma unroll 1
      for (int jl = 0; jl < min(TJ, n - j0); ++jl) {
        if (jl == self) continue;
        const int4 k = S.K[o][row][jl];
        const double kr = __hiloint2double(k.y, k.x), ki = __hiloint2double(k.w, k.z);
#pragma unroll
        for (int q = 0; q < RQ; ++q) {
          const int r = rg + RG * q;
          if (r >= rbn) continue;
          const double2 v = src[(size_t)(rb0 + r) * n + j0 + jl];
          acc[o][q].x = fma(-ki, v.y, fma(kr, v.x, acc[o][q].x));
          acc[o][q].y = fma(ki, v.x, fma(kr, v.y, acc[o][q].y));
        }
      }
    }
  }

  const int i = i0 + row;
  if (i >= p.rows) return;
#pragma unroll
  for (int q = 0; q < RQ; ++q) {
    const int r = rg + RG * q;
    if (r < rbn)
#pragma unroll
      for (int o = 0; o < NO; ++o)
        p.out[(((size_t)o * p.splits + blockIdx.y) * p.nrhs + rb0 + r) * p.rows + i] = acc[o][q];
  }
}

template <int MODE, int TI, int RBT, int RG>
void launch_block(const block_args& p, cudaStream_t stream) {
  const size_t smem = sizeof(block_smem<MODE, TI, RBT>);
  CFIE_CHECK_CUDA(cudaFuncSetAttribute(k_block64<MODE, TI, RBT, RG>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  const dim3 grid((p.rows + TI - 1) / TI, p.splits, (p.nrhs + RBT - 1) / RBT);
  k_block64<MODE, TI, RBT, RG><<<grid, TI * RG, smem, stream>>>(p);
  CFIE_CHECK_LAUNCH();
}

// Columns per CTA: equal blocks of at most 64 (sound hard, where a column is two
// sums: 32), each of the smallest width that has a kernel.
inline int block_width(int nrhs, bool hard) {
  const int widest = hard ? 32 : 64, blocks = (nrhs + widest - 1) / widest;
  const int per = (nrhs + blocks - 1) / blocks;
  for (int r : {4, 8, 12, 16, 24, 32, 48})
    if (per <= r) return r;
  return 64;
}
// Rows per CTA: the sums of 64 rows and 32 columns (sound hard: 16) fill the
// registers of the two CTAs that an SM holds; wider blocks have 32 rows.
inline int block_rows(int width, bool hard) { return width > (hard ? 16 : 32) ? 32 : 64; }

template <int MODE, int RBT>
void run_width(const block_args& p, int ti, cudaStream_t stream) {
  if constexpr (RBT > (MODE == HARD ? 16 : 32))
    launch_block<MODE, 32, RBT, 8>(p, stream);
  else if (ti == 32)
    launch_block<MODE, 32, RBT, 4>(p, stream);
  else
    launch_block<MODE, 64, RBT, 4>(p, stream);
}

template <int MODE>
void run_block(const block_args& p, int ti, int width, cudaStream_t stream) {
  switch (width) {
    case 4: run_width<MODE, 4>(p, ti, stream); break;
    case 8: run_width<MODE, 8>(p, ti, stream); break;
    case 12: run_width<MODE, 12>(p, ti, stream); break;
    case 16: run_width<MODE, 16>(p, ti, stream); break;
    case 24: run_width<MODE, 24>(p, ti, stream); break;
    case 32: run_width<MODE, 32>(p, ti, stream); break;
    case 48: if constexpr (MODE != HARD) run_width<MODE, 48>(p, ti, stream); break;
    default: if constexpr (MODE != HARD) run_width<MODE, 64>(p, ti, stream);
  }
}

}  // namespace sums64
