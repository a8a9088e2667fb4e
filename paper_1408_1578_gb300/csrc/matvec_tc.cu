// Matrix-free FP32 matvec with the source summation on the tensor cores.
//
// Same entries as the FP32 fused kernel (FP32 pair evaluation with two-float
// phase and Hankel asymptotics, FP64-evaluated near band), but instead of the
// register-blocked FP32 contraction the entries of each 128 x 32 tile are
// written, split as bf16 hi + lo, straight into shared memory in the tensor
// cores' 64-byte-swizzled K-major layout, and one thread issues tcgen05.mma
// against the right-hand-side block (bf16 hi / lo planes brought in by TMA):
//
//     [Yr | Yi] += Ar [Xr | Xi] + Ai [-Xi | Xr],  each product hi*hi + hi*lo + lo*hi,
//
// FP32 accumulation in tensor memory.  The sound-hard operator (eq. 2 with
// Maue's identity) is two operators over the same pairs, S on u = d/ds x and
// C = -D' - i (omega^2 / eta) (n_i . n_j) S on x (n1 S n1 + n2 S n2 has the
// entries (n_i . n_j) S_ij); a pass of up to 40 right-hand sides evaluates both from
// one phase, and where that takes more work than a pass of up to 64 for each, they
// have passes of their own (joint_passes; the operand planes of both for 64
// right-hand sides do not fit two stages of shared memory).
// Work is split stream-K: the (128-row tile, 32-source tile) pairs form one
// list and each CTA (one per SM) takes a contiguous range, cut into segments
// that end at row-tile boundaries.  Warp roles (24 warps, two of them only to fill
// the last warpgroup): 0-15 evaluate pair entries into the stage ring, 16 issues the
// TMA loads of the right-hand sides, of each tile's source geometry and of its
// Kress window, 17 issues the MMAs (double-buffered accumulators), 18-21 drain
// finished accumulators into per-segment partial sums, which a second kernel adds
// in a fixed order.  All mbarrier waits are bounded (error flag, drain, TMEM freed
// on every path).
//
// Bound: the producers' FP32 arithmetic (FMA pipe 64 % busy, its heavy half 70 %,
// ncu).  A lane keeps one target and evaluates the entries of eight adjacent sources in packed FP32
// pairs (pair32.cuh), which issue half as often as scalar instructions, four
// independent chains at a time; the sources are warp-uniform loads from a ring
// filled three tiles ahead.  Measured (GB300), kernel alone: kite n = 32768, 64
// right-hand sides 2.95 -> 2.45 ms (packed pairs in the former layout, a row
// per half warp: 2.97, bound by shared-memory cycles and by waits for the
// source loads); ellipse n = 32768, 1 right-hand side, sound hard, 4.90 (S and
// D' in two passes) -> 2.97 ms; two pairs at a time instead of four: 0.07 ms more.
#include <cuda.h>
#include <cuda_bf16.h>

#include <algorithm>
#include <climits>
#include <cstring>
#include <mutex>
#include <string>

#include "internal.h"
#include "pair32.cuh"
#include "tc_common.cuh"

namespace {

constexpr int TBM = 128;     // targets per tile (UMMA M)
constexpr int TBK = 32;      // sources per tile (32 bf16 = one 64-byte swizzle row)
// Source tiles accumulated in one tensor-memory accumulator before the epilogue
// warps add it into their running sums.  The tensor core's FP32 accumulation
// does not round to nearest: its error grows with the number of MMAs summed
// into one accumulator (~2e-8 relative per MMA), so chunks of 256 sources keep
// that bias near 2e-6 whatever n is, while the running sums and the segment
// reduction (FP32 adds, rounded to nearest) add only unbiased rounding.
constexpr int CK = 8;
constexpr int WKW = TBM + TBK + 2;   // Kress window of a tile (+ alignment slack)
// Source data (geometry, Kress window) are fetched this many tiles ahead, into
// a ring of their own: with the operand stages' ring the producers stood idle
// for the latency of these loads whenever a stage came free
constexpr int LOOK = 3;
constexpr int NPROD = 16;    // producer warps
constexpr int WTMA = NPROD, WMMA = NPROD + 1;   // then the epilogue warps
constexpr int NEPI = 4;      // epilogue warps
// six warpgroups of 128 threads: four of producers, then the other roles and
// two warps that only make the last warpgroup whole
constexpr int TNT = (NPROD + 8) * 32;
// Registers per thread: the launch has TNT x 80; the producers take 96 (their
// constants are packed pairs), the others give up what that costs (512 x 96 +
// 256 x 48 = 768 x 80)
constexpr int RLAUNCH = 80, RPRODUCER = 96, ROTHER = 48;
static_assert(NPROD * 32 * RPRODUCER + (TNT - NPROD * 32) * ROTHER <= TNT * RLAUNCH,
              "register shares exceed the launch's total");

struct tc_params {
  int n, b, ktiles;
  const float2* wext;    // Kress table / (pi h) at i - j + n, paired with the next source's
  const float4* pk;      // packed coordinates, source factors, target factors (n each)
  const float4* spk;     // source coordinates by pairs, source factors by pairs (n each)
  const float2* band;    // near entries: soft A, or S, then C
};

// v << 16 as a byte permutation: the compiler turns the shift into a multiply-add,
// on the pipe that bounds the producers (kite n = 32768 2.53 -> 2.51 ms)
__device__ __forceinline__ uint32_t shl16(uint32_t v) {
  uint32_t r;
  asm("prmt.b32 %0, %1, 0, 0x1044;" : "=r"(r) : "r"(v));
  return r;
}

// bf16 hi / lo split of eight entries of one row (adjacent sources): the packed
// words of the four planes (hi re, hi im, lo re, lo im) of each operator
template <int NO>
struct split_words {
  uint32_t v[NO][4][4];
  __device__ __forceinline__ static void split(float2 e, uint32_t& hi, uint32_t& lo) {
    const __nv_bfloat162 b = __floats2bfloat162_rn(e.x, e.y);
    hi = *reinterpret_cast<const uint32_t*>(&b);
    const float2 h = make_float2(__uint_as_float(shl16(hi)), __uint_as_float(hi & 0xffff0000u));
    const float2 d = add2(e, neg2(h));
    const __nv_bfloat162 c = __floats2bfloat162_rn(d.x, d.y);
    lo = *reinterpret_cast<const uint32_t*>(&c);
  }
  __device__ __forceinline__ void put(int p, const entry_pair& e) {
    split(e.re, v[0][0][p], v[0][2][p]);
    split(e.im, v[0][1][p], v[0][3][p]);
    if constexpr (NO == 2) {
      split(e.re2, v[1][0][p], v[1][2][p]);
      split(e.im2, v[1][1][p], v[1][3][p]);
    }
  }
  // planes `plane` bytes apart, operators four planes apart
  __device__ __forceinline__ void store(unsigned char* a, uint32_t plane) const {
#pragma unroll
    for (int o = 0; o < NO; ++o)
#pragma unroll
      for (int c = 0; c < 4; ++c)
        *reinterpret_cast<uint4*>(a + (4 * o + c) * plane) =
            make_uint4(v[o][c][0], v[o][c][1], v[o][c][2], v[o][c][3]);
  }
};

// Two entries of a tile that the near band or the end of the curve touches:
// band entries replace the far ones, rows and sources past n are zero
template <int OP>
__device__ __forceinline__ entry_pair near_pair(const tc_params& P, float4 t0, float4 t1, float4 tn,
                                                const float4* sc, const float4* sf, int i, int j) {
  entry_pair e;
  e.re = e.im = e.re2 = e.im2 = f2(0.f);
  const int n = P.n;
  if (i >= n || j >= n) return e;                    // n is even: j + 1 < n as well
  const float4 g0 = sf[0];
  e = finish32_pair<OP>(phase32_pair(t0, t1, sc[0], sc[1]), tn, g0, lo2(sf[1]), P.wext[i - j + n]);
#pragma unroll
  for (int u = 0; u < 2; ++u) {
    int d = i - j - u;
    if (d < 0) d += n;
    const int dd = d <= P.b ? d : (d >= n - P.b ? d - n : INT_MAX);
    if (dd == INT_MAX) continue;
    const size_t bw = 2 * (size_t)P.b + 1, at = (size_t)i * bw + dd + P.b;
    const float2 bv = P.band[at];                    // soft A, or S
    float2 s = bv, c = f2(0.f);
    if constexpr (OP != OP_SOFT) s = make_float2(bv.y, -bv.x);   // S' = -i S
    if constexpr (OP == OP_C || OP == OP_SC) c = P.band[(size_t)n * bw + at];
    const float2 first = OP == OP_C ? c : s;
    if (u) {
      e.re.y = first.x, e.im.y = first.y;
      e.re2.y = c.x, e.im2.y = c.y;
    } else {
      e.re.x = first.x, e.im.x = first.y;
      e.re2.x = c.x, e.im2.x = c.y;
    }
  }
  return e;
}

// operators evaluated by a pass, and the stages that fit
template <int OP>
__host__ __device__ constexpr int tc_ops() { return OP == OP_SC ? 2 : 1; }
template <int NP, int OP>
__host__ __device__ constexpr int tc_stages() { return OP == OP_SC ? 2 : 3; }

template <int NP, int OP>
struct tc_smem {
  static constexpr int NO = tc_ops<OP>(), ST = tc_stages<NP, OP>(), SD = ST + LOOK;
  __nv_bfloat16 A[ST][NO][4][TBM * TBK];    // per operator: hi_re, hi_im, lo_re, lo_im
  __nv_bfloat16 B[ST][NO][4][NP * TBK];     // per operator: B1 hi, B1 lo, B2 hi, B2 lo
  float4 src[SD][2][TBK];                   // sources by pairs: coordinates, factors
  float2 wk[SD][WKW];                       // Kress weight pairs / (pi h) of a plain tile
  uint64_t full[ST], empty[ST], sfull[SD], tfull[2], tempty[2];
  uint64_t mdone;                           // completion of every MMA issued (abort path)
  uint32_t tmem_base;
  int abort;
  int issued[ST], sissued[SD];
  int wofs[SD];                             // plain tile: window entry of (row 0, source 0); else -1
};

template <int NP, int OP>
constexpr size_t tc_smem_bytes() {
  static_assert(sizeof(tc_smem<NP, OP>) + 1024 <= 227 * 1024, "stages exceed shared memory");
  return sizeof(tc_smem<NP, OP>) + 1024;
}

// byte offset of element (row r, k) in a 64-byte-swizzled K-major tile
__device__ __forceinline__ uint32_t sw64(int r, int k) {
  return (uint32_t)(r * 64 + ((((k >> 3) ^ (r >> 1)) & 3) << 4) + (k & 7) * 2);
}

template <int NP, int OP>
__global__ void __launch_bounds__(TNT, 1)
k_fused_tc(tc_params P, const __grid_constant__ CUtensorMap tmB, const int4* __restrict__ segs,
           const int* __restrict__ cbeg, float2* __restrict__ partial, int* __restrict__ err) {
  constexpr int NR = NP / 2, NO = tc_ops<OP>(), TSTAGES = tc_stages<NP, OP>();
  constexpr int SD = TSTAGES + LOOK;
  constexpr bool HAS_TQ = OP == OP_C || OP == OP_SC;
  // per operator two accumulator buffers, then the epilogue's running sums
  // (NP columns each)
  constexpr uint32_t TMEM_COLS = 3 * NO * NP <= 256 ? 256 : 512;
  static_assert(3 * NO * NP <= 512, "accumulators exceed the tensor memory");
  constexpr uint32_t RUN = 2 * NO * NP;
  constexpr uint32_t B_BYTES = 4u * NO * NP * TBK * 2u;
  constexpr uint32_t APLANE = TBM * TBK * 2u;    // bytes of one A plane
  extern __shared__ unsigned char raw[];
  tc_smem<NP, OP>& S = smem_aligned<tc_smem<NP, OP>>(raw);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int sb = cbeg[blockIdx.x], se = cbeg[blockIdx.x + 1];
  const int n = P.n;

  if (threadIdx.x == 0) {
    for (int s = 0; s < TSTAGES; ++s) {
      mbar_init(&S.full[s], NPROD + 1);        // one arrival per producer warp + the TMA thread
      mbar_init(&S.empty[s], 1);
      S.issued[s] = -1;
    }
    for (int s = 0; s < SD; ++s) {
      mbar_init(&S.sfull[s], 1);
      S.sissued[s] = -1;
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&S.tfull[b], 1);
      mbar_init(&S.tempty[b], NEPI);
    }
    mbar_init(&S.mdone, 1);
    S.abort = 0;
    fence_mbar_init();
  }
  if (warp == WMMA) {
    tmem_alloc(&S.tmem_base, TMEM_COLS);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = S.tmem_base;

  if (warp < NPROD) {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(RPRODUCER));
    // ---- pair-entry producers.  Lane l of warp w owns row 32 (w % 4) + l of
    // the tile and the eight sources 8 (w / 4) .. + 7: the target stays in
    // registers for the whole segment, the sources are warp-uniform shared
    // loads, and the bf16 entries of a plane are one 16-byte chunk of the
    // swizzled tile, which 8 consecutive rows store without a bank conflict.
    // (A row per half warp, sources across its lanes, spent 65 % of the
    // shared-memory cycles on the strided source loads, the targets and
    // two-way conflicted stores.)
    const int row = 32 * (warp & 3) + lane, js = 8 * (warp >> 2);
    const uint32_t off = sw64(row, js);
    int it = 0;
    for (int s = sb; s < se; ++s) {
      const int4 sg = segs[s];
      const int m0 = sg.y * TBM;
      const int i = m0 + row;
      float4 t0, t1, tn;
      {
        const float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
        const float4 g = i < n ? P.pk[i] : z;
        t0 = make_float4(g.x, g.x, g.y, g.y);
        t1 = make_float4(g.z, g.z, g.w, g.w);
        const float4 q = HAS_TQ && i < n ? P.pk[2 * n + i] : z;
        tn = make_float4(q.x, q.x, q.y, q.y);
      }
      for (int k = sg.z; k < sg.w; ++k, ++it) {
        const int st = it % TSTAGES;
        const int j = k * TBK + js;                  // first of the lane's eight sources
        // exits are warp-uniform: the warp arrives on the stage barrier as one
        if (__any_sync(0xffffffffu, *(volatile int*)&S.abort)) break;
        // this tile's source geometry and Kress window (from the TMA warp),
        // and the stage's A planes (the MMAs of its previous tile are done)
        const int sl = it % SD;
        bool ok = mbar_wait_sleep<40>(&S.sfull[sl], (it / SD) & 1);
        if (ok && it >= TSTAGES) ok = mbar_wait_sleep<40>(&S.empty[st], ((it / TSTAGES) - 1) & 1);
        if (!__all_sync(0xffffffffu, ok)) {
          if (lane == 0) {
            atomicExch(err, 15);
            S.abort = 1;
          }
          break;
        }
        unsigned char* a = reinterpret_cast<unsigned char*>(S.A[st][0][0]) + off;
        const float4* sc = S.src[sl][0] + js;
        const float4* sf = S.src[sl][1] + js;
        // Plain tiles (all but ~1%, flagged by the TMA warp) skip the per-pair
        // range and band tests and take the Kress weights from the staged
        // window of the unwrapped table (entry i - j + n)
        const int wofs = S.wofs[sl];
        const float2* wq = S.wk[sl] + wofs + row - js;
        split_words<NO> w;
        entry_pair e[4];
        if (wofs >= 0) {
          // the phases (special-function ops) of the four pairs of sources
          // first, then the series and assembly, so that the chains interleave
          pair_phase2 f[4];
#pragma unroll
          for (int u = 0; u < 4; ++u) f[u] = phase32_pair(t0, t1, sc[2 * u], sc[2 * u + 1]);
#pragma unroll
          for (int u = 0; u < 4; ++u)
            e[u] = finish32_pair<OP>(f[u], tn, sf[2 * u], lo2(sf[2 * u + 1]), wq[-2 * u]);
        } else {
#pragma unroll
          for (int u = 0; u < 4; ++u)
            e[u] = near_pair<OP>(P, t0, t1, tn, sc + 2 * u, sf + 2 * u, i, j + 2 * u);
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) w.put(u, e[u]);
        w.store(a, APLANE);
        // generic-proxy writes become visible to the tensor core's async proxy;
        // the warp's writes are ordered before its one arrival by __syncwarp
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncwarp();
        if (lane == 0) mbar_arrive(&S.full[st]);
      }
      if (__any_sync(0xffffffffu, *(volatile int*)&S.abort)) break;
    }
  } else {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(ROTHER));
    if (warp == WTMA && lane == 0) {
      // ---- TMA producer of the right-hand-side planes and the source data
      asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&tmB)) : "memory");
      // Source data of the next tile of the list (segment ls, source tile lk,
      // running number lt).  A tile is plain when it holds full rows and
      // sources and no pair of the near band: d = i - j spans [dlo, dhi] there,
      // and the band is |d - t n| <= b for t = -1, 0, 1; a plain tile also gets
      // the window of the Kress table (entries dlo + n ... dhi + n) from the
      // 16-byte boundary below it.  Window bytes: WKW float2 = 1296, a multiple
      // of 16.
      int ls = sb, lt = 0, lk = sb < se ? segs[sb].z : 0;
      auto load_sources = [&] {
        if (ls >= se) return;
        const int4 sg = segs[ls];
        const int sl = lt % SD, m0 = sg.y * TBM, j0 = lk * TBK;
        const int dlo = m0 - j0 - (TBK - 1), dhi = m0 + TBM - 1 - j0;
        bool near = false;
#pragma unroll
        for (int t = -1; t <= 1; ++t) near |= (dhi >= t * n - P.b) && (dlo <= t * n + P.b);
        const bool plain = !near && m0 + TBM <= n && j0 + TBK <= n;
        S.wofs[sl] = plain ? m0 - j0 + n - ((dlo + n) & ~1) : -1;
        mbar_arrive_expect_tx(&S.sfull[sl], 2u * TBK * 16u + (plain ? WKW * 8u : 0u));
        S.sissued[sl] = (lt / SD) & 1;
        bulk_load(S.src[sl][0], P.spk + j0, TBK * 16u, &S.sfull[sl]);
        bulk_load(S.src[sl][1], P.spk + n + j0, TBK * 16u, &S.sfull[sl]);
        if (plain) bulk_load(S.wk[sl], P.wext + ((dlo + n) & ~1), WKW * 8u, &S.sfull[sl]);
        ++lt;
        if (++lk == sg.w && ++ls < se) lk = segs[ls].z;
      };
      for (int q = 0; q < LOOK; ++q) load_sources();
      int it = 0;
      for (int s = sb; s < se && !*(volatile int*)&S.abort; ++s) {
        const int4 sg = segs[s];
        for (int k = sg.z; k < sg.w; ++k, ++it) {
          const int st = it % TSTAGES;
          if (it >= TSTAGES && !mbar_wait_sleep<40>(&S.empty[st], ((it / TSTAGES) - 1) & 1)) {
            atomicExch(err, 12);
            S.abort = 1;
            break;
          }
          mbar_arrive_expect_tx(&S.full[st], B_BYTES);
          S.issued[st] = (it / TSTAGES) & 1;
#pragma unroll
          for (int p = 0; p < 4 * NO; ++p)
            tma_load_2d(S.B[st][p / 4][p % 4], &tmB, &S.full[st], k * TBK, p * NP);
          // the slot of tile it + LOOK held tile it - TSTAGES, whose MMAs, and
          // so whose producers, are done
          load_sources();
        }
      }
    }
    if (warp == WMMA && lane == 0) {
      // ---- MMA issuer: one accumulator buffer per chunk of CK source tiles
      constexpr uint32_t idesc = make_idesc(TBM, NP);
      int it = 0, cc = 0;
      for (int s = sb; s < se && !*(volatile int*)&S.abort; ++s) {
        const int4 sg = segs[s];
        for (int c0 = sg.z; c0 < sg.w; c0 += CK, ++cc) {
          const int c1 = min(sg.w, c0 + CK);
          const int tb = cc & 1, use = cc >> 1;
          if (use >= 1 && !mbar_wait_sleep<40>(&S.tempty[tb], (use - 1) & 1)) {
            atomicExch(err, 14);
            S.abort = 1;
          }
          if (*(volatile int*)&S.abort) break;
          tc_fence_after();
          for (int k = c0; k < c1; ++k, ++it) {
            const int st = it % TSTAGES;
            if (!mbar_wait_sleep<40>(&S.full[st], (it / TSTAGES) & 1)) {
              atomicExch(err, 13);
              S.abort = 1;
              break;
            }
            tc_fence_after();
#pragma unroll
            for (int o = 0; o < NO; ++o) {
              const uint32_t d = tmem + (uint32_t)((2 * o + tb) * NP);
              const uint32_t a0 = smem_u32(S.A[st][o][0]), a1 = smem_u32(S.A[st][o][1]);
              const uint32_t a2 = smem_u32(S.A[st][o][2]), a3 = smem_u32(S.A[st][o][3]);
              const uint32_t b0 = smem_u32(S.B[st][o][0]), b1 = smem_u32(S.B[st][o][1]);
              const uint32_t b2 = smem_u32(S.B[st][o][2]), b3 = smem_u32(S.B[st][o][3]);
#pragma unroll
              for (int kk = 0; kk < TBK / 16; ++kk) {
                const uint32_t off = kk * 32;
                const uint32_t acc0 = (k > c0 || kk > 0) ? 1u : 0u;
                umma_bf16(d, smem_desc_sw64(a0 + off), smem_desc_sw64(b0 + off), idesc, acc0);
                umma_bf16(d, smem_desc_sw64(a0 + off), smem_desc_sw64(b1 + off), idesc, 1u);
                umma_bf16(d, smem_desc_sw64(a2 + off), smem_desc_sw64(b0 + off), idesc, 1u);
                umma_bf16(d, smem_desc_sw64(a1 + off), smem_desc_sw64(b2 + off), idesc, 1u);
                umma_bf16(d, smem_desc_sw64(a1 + off), smem_desc_sw64(b3 + off), idesc, 1u);
                umma_bf16(d, smem_desc_sw64(a3 + off), smem_desc_sw64(b2 + off), idesc, 1u);
              }
            }
            umma_commit(&S.empty[st]);
          }
          umma_commit(&S.tfull[tb]);
        }
      }
    }
    if (warp > WMMA && warp <= WMMA + NEPI) {
    // ---- epilogue: warp w reads TMEM lanes 32 (w % 4) .. + 31, one row per
    // thread, and keeps the segment's running sums in the same lanes of the
    // last NP tensor-memory columns (FP32 adds, rounded to nearest)
    const int q = warp & 3;
    const int row = 32 * q + lane;
    const uint32_t lanes = tmem + ((uint32_t)(32 * q) << 16);
    int cc = 0;
    bool stop = false;
    for (int s = sb; s < se && !stop; ++s) {
      const int4 sg = segs[s];
      for (int c0 = sg.z; c0 < sg.w; c0 += CK, ++cc) {
        const int tb = cc & 1, use = cc >> 1;
        if (*(volatile int*)&S.abort || !mbar_wait_sleep<400>(&S.tfull[tb], use & 1)) {
          if (lane == 0) {
            atomicExch(err, 15);
            S.abort = 1;
          }
          stop = true;
          break;
        }
        __syncwarp();
        tc_fence_after();
        const bool first = c0 == sg.z;
#pragma unroll 1
        for (int o = 0; o < NO; ++o) {
          const uint32_t base = lanes + (uint32_t)((2 * o + tb) * NP);
          const uint32_t run = lanes + RUN + (uint32_t)(o * NP);
#pragma unroll 1
          for (int cb = 0; cb < NP; cb += 16) {
            float v[16];
            tmem_ld16(base + (uint32_t)cb, v);
            if (!first) {
              float r[16];
              tmem_ld16(run + (uint32_t)cb, r);
#pragma unroll
              for (int k = 0; k < 16; ++k) v[k] += r[k];
            }
            tmem_st16(run + (uint32_t)cb, v);
          }
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&S.tempty[tb]);
      }
      if (stop) break;
#pragma unroll 1
      for (int o = 0; o < NO; ++o) {
        float2* dst = partial + ((size_t)s * NO + o) * TBM * NR + row;
        const uint32_t run = lanes + RUN + (uint32_t)(o * NP);
#pragma unroll 1
        for (int cb = 0; cb + 16 <= NR; cb += 16) {
          float re[16], im[16];
          tmem_ld16(run + (uint32_t)cb, re);
          tmem_ld16(run + (uint32_t)(NR + cb), im);
#pragma unroll
          for (int k = 0; k < 16; ++k) dst[(size_t)(cb + k) * TBM] = make_float2(re[k], im[k]);
        }
        if constexpr (NR % 16) {   // NR = 40
          constexpr int cb = NR - 8;
          float re[8], im[8];
          tmem_ld8(run + (uint32_t)cb, re);
          tmem_ld8(run + (uint32_t)(NR + cb), im);
#pragma unroll
          for (int k = 0; k < 8; ++k) dst[(size_t)(cb + k) * TBM] = make_float2(re[k], im[k]);
        }
      }
    }
    }
  }
  __syncthreads();
  // after an abort, wait (bounded) for copies in flight and for every MMA
  // issued, then free TMEM
  if (*(volatile int*)&S.abort) {
    if (threadIdx.x == 0)
      for (int s = 0; s < SD; ++s) {
        if (s < TSTAGES && S.issued[s] >= 0) mbar_wait(&S.full[s], (uint32_t)S.issued[s]);
        if (S.sissued[s] >= 0) mbar_wait(&S.sfull[s], (uint32_t)S.sissued[s]);
      }
    if (warp == WMMA && lane == 0) {
      umma_commit(&S.mdone);
      mbar_wait(&S.mdone, 0);
    }
  }
  __syncthreads();
  if (warp == WMMA) {
    tc_fence_after();
    tmem_dealloc(tmem, TMEM_COLS);
  }
}

// Sums of the (one to a few) segment partials of row tile i / 128, in a fixed
// order; FP32 adds (the partials are FP32 sums of bf16 products: FP64 adds
// would buy nothing here and run at 1/64 of the FP32 rate).  Soft: y = A x.
// OP_S: t = S u = i S' u.  OP_C: y = x / 2 + C x.  OP_SC: both.
template <int OP>
__global__ void k_reduce_tc(int n, int nr, int NR, const int2* __restrict__ mt_seg,
                            const float2* __restrict__ partial, const double2* __restrict__ x,
                            float2* __restrict__ t, double2* __restrict__ y) {
  constexpr int NO = tc_ops<OP>();
  const int m = blockIdx.x, r = blockIdx.y, row = threadIdx.x;
  const int i = m * TBM + row;
  if (i >= n || r >= nr) return;
  const int2 sr = mt_seg[m];
  float2 v[NO];
#pragma unroll
  for (int o = 0; o < NO; ++o) v[o] = make_float2(0.f, 0.f);
  for (int s = sr.x; s < sr.x + sr.y; ++s) {
#pragma unroll
    for (int o = 0; o < NO; ++o) {
      const float2 p = partial[(((size_t)s * NO + o) * NR + r) * TBM + row];
      v[o].x += p.x;
      v[o].y += p.y;
    }
  }
  const size_t e = (size_t)r * n + i;
  if constexpr (OP == OP_SOFT) y[e] = make_double2(v[0].x, v[0].y);
  if constexpr (OP == OP_S || OP == OP_SC) t[e] = make_float2(-v[0].y, v[0].x);
  if constexpr (OP == OP_C || OP == OP_SC) {
    const double2 xv = x[e];
    y[e] = make_double2(fma(0.5, xv.x, (double)v[NO - 1].x), fma(0.5, xv.y, (double)v[NO - 1].y));
  }
}

// One pass for the right-hand sides r0 .. r0 + nr - 1: soft x -> y; S: u -> t;
// C: x -> y; SC: u, x -> t, y
template <int NP, int OP>
void run_fused(cfie_op* op, const double2* x, const float2* u, float2* t, double2* y, int r0,
               int nr) {
  constexpr int NR = NP / 2, NO = tc_ops<OP>();
  tc_plan& T = op->tc[OP == OP_SC ? (NP == 64 ? 2 : 3) : (NP == 64 ? 0 : 1)];
  const int n = op->n;
  cudaStream_t st = op->ctx->stream;
  const int pitch = (n + 63) / 64 * 64;
  const size_t planes = 4 * (size_t)NP * pitch;
  if (!T.built) {
    const int mtiles = (n + TBM - 1) / TBM, ktiles = (n + TBK - 1) / TBK;
    int sms = 152;
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, op->ctx->device);
    std::vector<int4> segs;
    std::vector<int> cbeg;
    std::vector<int2> mt_seg;
    streamk_segments(mtiles, ktiles, sms, segs, cbeg, mt_seg);
    T.grid = (int)cbeg.size() - 1;
    T.nsegs = (int)segs.size();
    T.mtiles = mtiles;
    T.tables.reserve(sizeof(int4) * segs.size() + sizeof(int) * cbeg.size() +
                     sizeof(int2) * mt_seg.size() + 64);
    char* tb = T.tables.as<char>();
    T.o_cbeg = (sizeof(int4) * segs.size() + 15) & ~size_t(15);
    T.o_mts = (T.o_cbeg + sizeof(int) * cbeg.size() + 15) & ~size_t(15);
    CFIE_CHECK_CUDA(cudaMemcpyAsync(tb, segs.data(), sizeof(int4) * segs.size(),
                                    cudaMemcpyHostToDevice, st));
    CFIE_CHECK_CUDA(cudaMemcpyAsync(tb + T.o_cbeg, cbeg.data(), sizeof(int) * cbeg.size(),
                                    cudaMemcpyHostToDevice, st));
    CFIE_CHECK_CUDA(cudaMemcpyAsync(tb + T.o_mts, mt_seg.data(), sizeof(int2) * mt_seg.size(),
                                    cudaMemcpyHostToDevice, st));
    T.bt.reserve(sizeof(__nv_bfloat16) * NO * planes);
    T.partial.reserve(sizeof(float2) * (size_t)T.nsegs * NO * TBM * NR);
    T.err.reserve(sizeof(int));
    CFIE_CHECK_CUDA(cudaMemsetAsync(T.err.p, 0, sizeof(int), st));
    const CUtensorMap mb = tc_make_map(T.bt.p, 4 * NO * (uint64_t)NP, (uint64_t)pitch, pitch, NP,
                                       TBK, CU_TENSOR_MAP_SWIZZLE_64B);
    std::memcpy(T.tmB, &mb, sizeof(mb));
    CFIE_CHECK_CUDA(cudaStreamSynchronize(st));
    T.built = true;
  }
  __nv_bfloat16* bt = T.bt.as<__nv_bfloat16>();
  const size_t at = (size_t)r0 * n;
  if constexpr (OP == OP_S || OP == OP_SC) prep_b_planes(op->ctx, n, pitch, NP, nr, u + at, bt);
  if constexpr (OP != OP_S)
    prep_b_planes(op->ctx, n, pitch, NP, nr, x + at, bt + (NO - 1) * planes);
  tc_params P{};
  P.n = n;
  P.b = op->band_b;
  P.ktiles = (n + TBK - 1) / TBK;
  float* base = op->geo32.as<float>();
  P.wext = reinterpret_cast<const float2*>(base + geo32_wk_offset(n));
  P.pk = reinterpret_cast<const float4*>(base + geo32_pack_offset(n));
  P.spk = reinterpret_cast<const float4*>(base + geo32_pair_offset(n));
  P.band = op->band.as<float2>();
  const size_t smem = tc_smem_bytes<NP, OP>();
  CFIE_CHECK_CUDA(cudaFuncSetAttribute(k_fused_tc<NP, OP>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  char* tb = T.tables.as<char>();
  {
    prof_scope ps(op->ctx, CFIE_K_MATVEC_FP32);
    k_fused_tc<NP, OP><<<T.grid, TNT, smem, st>>>(P, *reinterpret_cast<const CUtensorMap*>(T.tmB),
                                                  reinterpret_cast<const int4*>(tb),
                                                  reinterpret_cast<const int*>(tb + T.o_cbeg),
                                                  T.partial.as<float2>(), T.err.as<int>());
    CFIE_CHECK_LAUNCH();
  }
  k_reduce_tc<OP><<<dim3(T.mtiles, nr), TBM, 0, st>>>(
      n, nr, NR, reinterpret_cast<const int2*>(tb + T.o_mts), T.partial.as<float2>(),
      x ? x + at : nullptr, t ? t + at : nullptr, y ? y + at : nullptr);
  CFIE_CHECK_LAUNCH();
}

template <int OP>
void run_blocks(cfie_op* op, const double2* x, const float2* u, float2* t, double2* y, int nrhs) {
  for (int r0 = 0; r0 < nrhs; r0 += 64) {
    const int nr = std::min(64, nrhs - r0);
    if (nr > 32)
      run_fused<128, OP>(op, x, u, t, y, r0, nr);
    else
      run_fused<64, OP>(op, x, u, t, y, r0, nr);
  }
}

// Sound hard: passes of S and C together, 0 where each on its own is the less.  S and C
// from one phase take 1.25 to 1.3 passes of one operator, but the tensor memory and
// the stages hold 40 right-hand sides of both against 64 of one (n = 6002, 33
// right-hand sides: 405 -> 325 us with the derivatives; n = 16384, 72: 2.50 -> 1.80 ms).
int joint_passes(int nrhs) {
  const int both = (nrhs + 39) / 40, each = 2 * ((nrhs + 63) / 64);
  return 4 * both < 3 * each ? both : 0;
}

}  // namespace

int tc_passes(const cfie_op* op, int nrhs) {
  const int blocks = (nrhs + 63) / 64;
  if (op->bc == CFIE_SOUND_SOFT) return blocks;
  const int both = joint_passes(nrhs);
  return both ? both : 2 * blocks;
}

void matvec_fp32_tc(cfie_op* op, const double2* x, double2* y, int nrhs) {
  if (op->bc == CFIE_SOUND_SOFT) {
    run_blocks<OP_SOFT>(op, x, nullptr, nullptr, y, nrhs);
    return;
  }
  // sound hard: S on u = (1/|z'|) d/dt x and C on x, then the spectral
  // derivative of S u
  const size_t tot = (size_t)op->n * nrhs;
  op->xin32.reserve(sizeof(float2) * tot * 3);
  float2* u32 = op->xin32.as<float2>();
  float2* t32 = u32 + tot;
  spectral32_apply(op, x, u32, nrhs);
  if (const int both = joint_passes(nrhs)) {
    const int per = (nrhs + both - 1) / both;
    for (int r0 = 0; r0 < nrhs; r0 += per) {
      const int nr = std::min(per, nrhs - r0);
      if (nr > 32)
        run_fused<80, OP_SC>(op, x, u32, t32, y, r0, nr);
      else
        run_fused<64, OP_SC>(op, x, u32, t32, y, r0, nr);
    }
  } else {
    run_blocks<OP_S>(op, nullptr, u32, t32, nullptr, nrhs);
    run_blocks<OP_C>(op, x, nullptr, nullptr, y, nrhs);
  }
  spectral32_accumulate(op, t32, y, nrhs);
}

int tc_take_error(cfie_op* op) {
  int e = 0;
  for (auto& T : op->tc) {
    if (!T.err.p) continue;
    int v = 0;
    CFIE_CHECK_CUDA(cudaMemcpyAsync(&v, T.err.p, sizeof(int), cudaMemcpyDeviceToHost,
                                    op->ctx->stream));
    CFIE_CHECK_CUDA(cudaStreamSynchronize(op->ctx->stream));
    if (v) {
      e = v;
      CFIE_CHECK_CUDA(cudaMemsetAsync(T.err.p, 0, sizeof(int), op->ctx->stream));
    }
  }
  return e;
}
