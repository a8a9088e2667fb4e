// Restarted GMRES (Section 3 of the paper: GMRES with a relative tolerance and
// a restart length) for a set of independent problems, with the Arnoldi
// orthogonalisation, Givens rotations, Hessenberg least-squares solve and the
// solution update all in FP64 on the GPU, and mixed-precision iterative
// refinement on the outer FP64 residual for the FP32 / tensor precisions.
//
// Arnoldi step j (per problem p, V_p = [v_0 .. v_j]):
//   w = A v_j
//   classical Gram-Schmidt twice (CGS2):  h = V^H w, w -= V h   (two passes)
//   H(0:j, j) = h_1 + h_2,  H(j+1, j) = ||w||,  v_{j+1} = w / ||w||
//   rotate column j of H by the previous Givens rotations, build rotation j,
//   g(j+1) = -conj(s_j) g(j), g(j) = c_j g(j); |g(j+1)| is the residual norm.
// After a cycle: R y = g (back substitution), x += V y, then the true residual.
//
// Problems are segments of one long "super vector" of length L: problem p
// (one right-hand side of one operator) owns elements [off_p, off_p + n_p).
// For one operator with nrhs right-hand sides this is exactly the column-major
// n x nrhs layout of the C ABI; for a batch of operators the blocks of all
// operators are concatenated.  Basis vector j of every problem is the slice
// V[j * L .. (j + 1) * L), so the matvec reads it directly.  The chunked kernels
// run over a work list of (problem, chunk) items and stream V once per pass;
// per-problem quantities (H, Givens data, norms) are reduced from per-chunk
// partial sums in a fixed order by the problem's last CTA to finish.
//
// Bound: HBM (or L2, when the basis fits) for large sets, latency for small
// ones.  The chunk length (128 to 2048 elements) is chosen so that the columns of
// one operator have about two CTAs per SM (a set with several lengths takes a launch
// for each), the inner products of a small set are also split over the basis
// vectors, loads of four basis vectors are in flight at once, the four
// pairs of sums are reduced across a warp together (9 shuffles instead of 40;
// on GB300 the FP64 additions of a plain reduction cost more than the products),
// and an Arnoldi step is 5 launches instead of 9.  Measured (GB300): unrestarted
// FP64 solve of n = 1024, 30 steps, 15.2 -> 9.1 ms (490 -> 290 us a step, 227 of
// them the matvec); kite n = 8192, 64 directions, 88 steps, 34.2 -> 29.8 ms.
#include <algorithm>
#include <cmath>
#include <type_traits>
#include <vector>

#include "hankel64.cuh"
#include "internal.h"

namespace {

constexpr int AT = 256;          // threads per CTA at most
constexpr int AB = 4;            // basis vectors in flight
constexpr int MAXJ = 512;        // largest restart length

template <typename S>
__device__ __forceinline__ S warp_sum(S v) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Element type of a Krylov basis: FP64 (double2) or, for the inner solves of
// the refined precisions, FP32 (float2).
template <typename T> struct basis_t;
template <> struct basis_t<double2> {
  using S = double;
  static __device__ __forceinline__ double2 make(double a, double b) { return make_double2(a, b); }
};
template <> struct basis_t<float2> {
  using S = float;
  static __device__ __forceinline__ float2 make(double a, double b) {
    return make_float2((float)a, (float)b);
  }
  static __device__ __forceinline__ float2 make(float a, float b) { return make_float2(a, b); }
};

struct chunk_ref {
  size_t base;
  int cnt, p, slot;
};

__device__ __forceinline__ chunk_ref chunk_of(const pset_dev& ps, int item) {
  const int4 it = __ldg(reinterpret_cast<const int4*>(ps.items) + ps.first + item);
  chunk_ref r;
  r.base = (size_t)(unsigned)it.x | (size_t)(unsigned)it.y << 32;
  r.cnt = it.z;
  r.p = it.w;
  r.slot = ps.first + item;
  return r;
}

// two adjacent elements (segments and chunks have even lengths and offsets)
template <typename T> struct two { T a, b; };
__device__ __forceinline__ two<float2> load2(const float2* p) {
  const float4 v = *reinterpret_cast<const float4*>(p);
  return {make_float2(v.x, v.y), make_float2(v.z, v.w)};
}
__device__ __forceinline__ two<double2> load2(const double2* p) { return {p[0], p[1]}; }
__device__ __forceinline__ void store2(float2* p, float2 a, float2 b) {
  *reinterpret_cast<float4*>(p) = make_float4(a.x, a.y, b.x, b.y);
}
__device__ __forceinline__ void store2(double2* p, double2 a, double2 b) {
  p[0] = a;
  p[1] = b;
}

// Whether this CTA is the last of the problem's `total` to get here; all its
// earlier writes, and those of the others, are then visible to it.  The counter
// is left at zero.
__device__ __forceinline__ bool last_cta(int* counter, int total) {
  __shared__ int last;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) {
    last = atomicAdd(counter, 1) == total - 1;
    if (last) *counter = 0;
  }
  __syncthreads();
  __threadfence();
  return last != 0;
}

// h[p][jj] = V[jj]^H w, jj = 0..J: CTA (item, y) the vectors y JB .. of one chunk
// (products and the in-chunk sums in the basis precision, chunk partials FP64);
// the problem's last CTA adds the chunks and H[p][jj][col] = (first) or += h
template <typename T, int PT>
__global__ void __launch_bounds__(AT)
k_dots(int J, int JB, int m, int col, int first, const T* __restrict__ V, size_t L,
       const T* __restrict__ w, const int* __restrict__ act, pset_dev ps,
       double2* __restrict__ partial, int* __restrict__ counter, double2* __restrict__ hbuf,
       double2* __restrict__ H) {
  using S = typename basis_t<T>::S;
  extern __shared__ double2 red[];  // [JB][warps]
  const chunk_ref c = chunk_of(ps, blockIdx.x);
  if (!act[c.p]) return;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, warps = blockDim.x >> 5;
  const int j0 = blockIdx.y * JB, j1 = min(J + 1, j0 + JB);
  const int nch = ps.nch[c.p], chb = ps.chb[c.p];   // early, for the last CTA
  two<T> wr[PT];
#pragma unroll
  for (int e = 0; e < PT; ++e) {
    const int q = 2 * (e * blockDim.x + threadIdx.x);
    wr[e].a = wr[e].b = basis_t<T>::make(0.0, 0.0);
    if (q < c.cnt) wr[e] = load2(w + c.base + q);
  }
  // Two pairs per thread: an advancing pointer.  With the index of the vector in each
  // address the compiler kept half of the loads in flight there (32 registers, kite n =
  // 8192, 64 directions, 30.5 ms against 29.9), and with the pointer fewer at four pairs
  // (n = 32768: these kernels 35.9 ms a solve against 33.0).
  const T* vp = V + (size_t)j0 * L + c.base;
  for (int jj = j0; jj < j1; jj += AB, vp += AB * L) {
    two<T> v[AB][PT];
#pragma unroll
    for (int b = 0; b < AB; ++b)
#pragma unroll
      for (int e = 0; e < PT; ++e) {
        const int q = 2 * (e * blockDim.x + threadIdx.x);
        v[b][e].a = v[b][e].b = basis_t<T>::make(0.0, 0.0);
        if (q < c.cnt && jj + b < j1)
          v[b][e] = load2(PT == 2 ? vp + b * L + q : V + (size_t)(jj + b) * L + c.base + q);
      }
    S s[2 * AB];
#pragma unroll
    for (int b = 0; b < AB; ++b) {
      S re = 0, im = 0;
#pragma unroll
      for (int e = 0; e < PT; ++e) {
        const two<T> a = v[b][e];
        re = fma(a.a.x, wr[e].a.x, fma(a.a.y, wr[e].a.y, re));
        im = fma(a.a.x, wr[e].a.y, fma(-a.a.y, wr[e].a.x, im));
        re = fma(a.b.x, wr[e].b.x, fma(a.b.y, wr[e].b.y, re));
        im = fma(a.b.x, wr[e].b.y, fma(-a.b.y, wr[e].b.x, im));
      }
      s[2 * b] = re;
      s[2 * b + 1] = im;
    }
    // the 2 AB = 8 sums across the warp: halve the values and double the lanes
    // per value three times, then two plain steps; value `idx` ends in the four
    // lanes of its group
#pragma unroll
    for (int n = AB, o = 16; n >= 1; n /= 2, o /= 2) {
      const bool up = lane & o;
#pragma unroll
      for (int k = 0; k < n; ++k) {
        const S mine = up ? s[k + n] : s[k];
        const S other = up ? s[k] : s[k + n];
        s[k] = mine + __shfl_xor_sync(0xffffffffu, other, o);
      }
    }
    s[0] += __shfl_xor_sync(0xffffffffu, s[0], 2);
    s[0] += __shfl_xor_sync(0xffffffffu, s[0], 1);
    const int idx = ((lane >> 4) & 1) * 4 + ((lane >> 3) & 1) * 2 + ((lane >> 2) & 1);
    if ((lane & 3) == 0 && jj + (idx >> 1) < j1) {
      double* d = reinterpret_cast<double*>(red + (size_t)(jj - j0 + (idx >> 1)) * warps + warp);
      d[idx & 1] = (double)s[0];
    }
  }
  __syncthreads();
  for (int jj = j0 + threadIdx.x; jj < j1; jj += blockDim.x) {
    double2 t = make_double2(0.0, 0.0);
    for (int q = 0; q < warps; ++q) {
      t.x += red[(size_t)(jj - j0) * warps + q].x;
      t.y += red[(size_t)(jj - j0) * warps + q].y;
    }
    partial[(size_t)c.slot * (J + 1) + jj] = t;
  }
  if (!last_cta(counter + c.p, nch * gridDim.y)) return;
  for (int jj = threadIdx.x; jj <= J; jj += blockDim.x) {
    double2 t = make_double2(0.0, 0.0);
#pragma unroll 4
    for (int k = 0; k < nch; ++k) {
      const double2 v = __ldcg(partial + (size_t)(chb + k) * (J + 1) + jj);
      t.x += v.x;
      t.y += v.y;
    }
    hbuf[(size_t)c.p * (J + 1) + jj] = t;
    double2* hk = H + ((size_t)c.p * (m + 1) + jj) * m + col;
    if (first) {
      *hk = t;
    } else {
      hk->x += t.x;
      hk->y += t.y;
    }
  }
}

// Givens data of one cycle, per problem
struct givens_dev {
  double2* H;      // [m + 1][m]
  double* cs;      // [m]
  double2* sn;     // [m]
  double2* gv;     // [m + 1]
  double* hnorm;   // ||w||
  double* res;     // residual estimate
};

// One warp: Givens rotations on column j of H, residual estimate.  The warp
// stages the column and the previous rotations in shared memory (m + 1, m, m
// entries); lane 0 applies the rotations in order (each depends on the last).
// s2 = ||w||^2.
__device__ void givens_step(int p, int m, int j, double s2, const givens_dev& G, double2* col) {
  const int lane = threadIdx.x & 31;
  double2* ssn = col + (m + 1);
  double* scs = reinterpret_cast<double*>(ssn + m);
  double2* Hk = G.H + (size_t)p * (m + 1) * m;
  const double hn = sqrt(s2);
  for (int q = lane; q <= j; q += 32) col[q] = Hk[(size_t)q * m + j];
  for (int q = lane; q < j; q += 32) {
    scs[q] = G.cs[(size_t)p * m + q];
    ssn[q] = G.sn[(size_t)p * m + q];
  }
  __syncwarp();
  if (lane == 0) {
    G.hnorm[p] = hn;
    const double2 gj = G.gv[(size_t)p * (m + 1) + j];
    double2 a = col[0];
    for (int q = 0; q < j; ++q) {   // previous rotations [c s; -conj(s) c] on column j
      const double2 b = col[q + 1];
      const double c = scs[q];
      const double2 s = ssn[q];
      col[q] = make_double2(c * a.x + s.x * b.x - s.y * b.y, c * a.y + s.x * b.y + s.y * b.x);
      a = make_double2(-(s.x * a.x + s.y * a.y) + c * b.x, -(s.x * a.y - s.y * a.x) + c * b.y);
    }
    const double bn = hn;  // b = ||w|| is real
    double c;
    double2 s;
    const double a2 = a.x * a.x + a.y * a.y, t2 = a2 + bn * bn;
    if (bn > 0.0 && a2 > 1e-280 && t2 < 1e280) {
      // |a|, sqrt(|a|^2 + b^2) and their reciprocals from one Newton step each
      const double ra = h64::rsqrt_newton(a2), rt = h64::rsqrt_newton(t2);
      c = a2 * ra * rt;
      const double f = ra * rt * bn;       // (a/|a|) conj(b) / t
      s = make_double2(a.x * f, a.y * f);
    } else {
      const double aa = hypot(a.x, a.y);
      if (bn == 0.0) {
        c = 1.0;
        s = make_double2(0.0, 0.0);
      } else if (aa == 0.0) {
        c = 0.0;
        s = make_double2(1.0, 0.0);
      } else {
        const double t = hypot(aa, bn);
        c = aa / t;
        s = make_double2(a.x / aa * bn / t, a.y / aa * bn / t);
      }
    }
    G.cs[(size_t)p * m + j] = c;
    G.sn[(size_t)p * m + j] = s;
    col[j] = make_double2(c * a.x + s.x * bn, c * a.y + s.y * bn);
    col[j + 1] = make_double2(0.0, 0.0);
    const double2 g1 = make_double2(-(s.x * gj.x + s.y * gj.y), -(s.x * gj.y - s.y * gj.x));
    G.gv[(size_t)p * (m + 1) + j + 1] = g1;
    G.gv[(size_t)p * (m + 1) + j] = make_double2(c * gj.x, c * gj.y);
    const double g2 = g1.x * g1.x + g1.y * g1.y;
    G.res[p] = g2 > 1e-280 && g2 < 1e280 ? sqrt(g2) : hypot(g1.x, g1.y);
  }
  __syncwarp();
  for (int q = lane; q <= j + 1; q += 32) Hk[(size_t)q * m + j] = col[q];
}

// w -= sum_jj V[jj] h[p][jj] on one chunk; with GIVENS (the second pass) also
// |w|^2, and the problem's last CTA adds the chunks and does the Givens step
template <typename T, int PT, bool GIVENS>
__global__ void __launch_bounds__(AT)
k_update(int J, int m, const T* __restrict__ V, size_t L, const double2* __restrict__ hbuf,
         const int* __restrict__ act, pset_dev ps, T* __restrict__ w,
         double* __restrict__ nrm_partial, int* __restrict__ counter, givens_dev G) {
  using S = typename basis_t<T>::S;
  extern __shared__ double2 hs_raw[];   // h in the basis precision; then the Givens step's data
  T* hs = reinterpret_cast<T*>(hs_raw);
  const chunk_ref c = chunk_of(ps, blockIdx.x);
  if (!act[c.p]) return;
  for (int jj = threadIdx.x; jj <= J; jj += blockDim.x) {
    const double2 h = hbuf[(size_t)c.p * (J + 1) + jj];
    hs[jj] = basis_t<T>::make(h.x, h.y);
  }
  two<T> acc[PT];
#pragma unroll
  for (int e = 0; e < PT; ++e) {
    const int q = 2 * (e * blockDim.x + threadIdx.x);
    acc[e].a = acc[e].b = basis_t<T>::make(0.0, 0.0);
    if (q < c.cnt) acc[e] = load2(w + c.base + q);
  }
  __syncthreads();
  for (int jj = 0; jj <= J; jj += AB) {
    two<T> v[AB][PT];
#pragma unroll
    for (int b = 0; b < AB; ++b)
#pragma unroll
      for (int e = 0; e < PT; ++e) {
        const int q = 2 * (e * blockDim.x + threadIdx.x);
        v[b][e].a = v[b][e].b = basis_t<T>::make(0.0, 0.0);
        if (q < c.cnt && jj + b <= J) v[b][e] = load2(V + (size_t)(jj + b) * L + c.base + q);
      }
#pragma unroll
    for (int b = 0; b < AB; ++b) {
      if (jj + b > J) break;
      const T hh = hs[jj + b];
#pragma unroll
      for (int e = 0; e < PT; ++e) {
        const two<T> a = v[b][e];
        acc[e].a.x = fma(-a.a.x, hh.x, fma(a.a.y, hh.y, acc[e].a.x));
        acc[e].a.y = fma(-a.a.x, hh.y, fma(-a.a.y, hh.x, acc[e].a.y));
        acc[e].b.x = fma(-a.b.x, hh.x, fma(a.b.y, hh.y, acc[e].b.x));
        acc[e].b.y = fma(-a.b.x, hh.y, fma(-a.b.y, hh.x, acc[e].b.y));
      }
    }
  }
  const int nch = GIVENS ? ps.nch[c.p] : 0, chb = GIVENS ? ps.chb[c.p] : 0;
  S ss = 0;
#pragma unroll
  for (int e = 0; e < PT; ++e) {
    const int q = 2 * (e * blockDim.x + threadIdx.x);
    if (q < c.cnt) {
      store2(w + c.base + q, acc[e].a, acc[e].b);
      ss = fma(acc[e].a.x, acc[e].a.x, fma(acc[e].a.y, acc[e].a.y, ss));
      ss = fma(acc[e].b.x, acc[e].b.x, fma(acc[e].b.y, acc[e].b.y, ss));
    }
  }
  if constexpr (GIVENS) {
    __shared__ double red[AT / 32];
    const double sd = warp_sum((double)ss);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = sd;
    __syncthreads();
    if (threadIdx.x == 0) {
      double t = 0.0;
      for (int q = 0; q < (int)(blockDim.x >> 5); ++q) t += red[q];
      nrm_partial[c.slot] = t;
    }
    if (!last_cta(counter + c.p, nch)) return;
    if (threadIdx.x < 32) {
      double s2 = 0.0;
      for (int k = threadIdx.x; k < nch; k += 32) s2 += __ldcg(nrm_partial + chb + k);
      for (int o = 16; o > 0; o >>= 1) s2 += __shfl_xor_sync(0xffffffffu, s2, o);
      givens_step(c.p, m, J, s2, G, hs_raw);
    }
  }
}

// vout = w / ||w|| per problem (0 on breakdown); vin (optional) = the same
// vector in FP64, the input of the next matvec
template <typename T>
__global__ void __launch_bounds__(AT)
k_scale(const int* __restrict__ act, pset_dev ps, const double* __restrict__ hn,
        const T* __restrict__ w, T* __restrict__ vout, double2* __restrict__ vin) {
  const chunk_ref c = chunk_of(ps, blockIdx.x);
  if (!act[c.p]) return;
  const double h = hn[c.p];
  const double inv = h > 0.0 ? 1.0 / h : 0.0;
  // the multiply in the basis precision (FP64 runs at 1/64 of the FP32 rate)
  const typename basis_t<T>::S s = (typename basis_t<T>::S)inv;
#pragma unroll 4
  for (int q = threadIdx.x; q < c.cnt; q += blockDim.x) {
    {
      const T v = w[c.base + q];
      const T o = basis_t<T>::make(v.x * s, v.y * s);
      vout[c.base + q] = o;
      if (vin) vin[c.base + q] = make_double2(o.x, o.y);
    }
  }
}

// v0 = r / beta per problem (vin as in k_scale)
template <typename T>
__global__ void __launch_bounds__(AT)
k_start(const int* __restrict__ act, pset_dev ps, const double* __restrict__ beta,
        const double2* __restrict__ r, T* __restrict__ v0, double2* __restrict__ vin) {
  const chunk_ref c = chunk_of(ps, blockIdx.x);
  const double b = beta[c.p];
  const double inv = (act[c.p] && b > 0.0) ? 1.0 / b : 0.0;
#pragma unroll 4
  for (int q = threadIdx.x; q < c.cnt; q += blockDim.x) {
    {
      const double2 v = r[c.base + q];
      const T o = basis_t<T>::make(v.x * inv, v.y * inv);
      v0[c.base + q] = o;
      if (vin) vin[c.base + q] = make_double2(o.x, o.y);
    }
  }
}

// w32 = w (FP64 matvec output to the FP32 basis precision)
__global__ void __launch_bounds__(AT)
k_to32(const int* __restrict__ act, pset_dev ps, const double2* __restrict__ w,
       float2* __restrict__ w32) {
  const chunk_ref c = chunk_of(ps, blockIdx.x);
  if (!act[c.p]) return;
#pragma unroll 4
  for (int q = threadIdx.x; q < c.cnt; q += blockDim.x) {
    {
      const double2 v = w[c.base + q];
      w32[c.base + q] = make_float2((float)v.x, (float)v.y);
    }
  }
}

// g = (beta, 0, ..., 0) per problem
__global__ void k_g_init(int P, int m, const int* __restrict__ act, const double* __restrict__ beta,
                         double2* __restrict__ gv) {
  const size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= (size_t)P * (m + 1)) return;
  const int p = (int)(e / (m + 1));
  const int q = (int)(e % (m + 1));
  gv[e] = make_double2(q == 0 && act[p] ? beta[p] : 0.0, 0.0);
}

// one warp per problem: y = R^{-1} g on the leading kd x kd triangle, column by
// column from the last (each solved unknown is taken out of the rows above it,
// one row per lane; the reciprocals of the diagonal come first)
__global__ void __launch_bounds__(32)
k_lsq(int m, const int* __restrict__ kd, const double2* __restrict__ H,
      const double2* __restrict__ gv, double2* __restrict__ y) {
  extern __shared__ double2 lsh[];   // s [m], 1 / diagonal [m]
  const int p = blockIdx.x, lane = threadIdx.x;
  const int K = kd[p];
  const double2* Hk = H + (size_t)p * (m + 1) * m;
  double2* yk = y + (size_t)p * m;
  double2* s = lsh;
  double2* inv = lsh + m;
  for (int i = lane; i < K; i += 32) {
    s[i] = gv[(size_t)p * (m + 1) + i];
    const double2 d = Hk[(size_t)i * m + i];
    const double den = d.x * d.x + d.y * d.y;
    inv[i] = den > 0.0 ? make_double2(d.x / den, -d.y / den) : make_double2(0.0, 0.0);
  }
  __syncwarp();
  for (int i = K - 1; i >= 0; --i) {
    const double2 a = s[i], d = inv[i];
    const double2 yi = make_double2(a.x * d.x - a.y * d.y, a.x * d.y + a.y * d.x);
    if (lane == 0) yk[i] = yi;
    for (int q = lane; q < i; q += 32) {
      const double2 h = Hk[(size_t)q * m + i];
      s[q].x -= h.x * yi.x - h.y * yi.y;
      s[q].y -= h.x * yi.y + h.y * yi.x;
    }
    __syncwarp();
  }
}

// x += sum_{jj < kd[p]} V[jj] y[p][jj]: the sum in the basis precision (an
// FP32 basis is orthonormal to FP32 accuracy, so |sum| ~ |y| and FP32 loses
// nothing the inner solve's tolerance would notice), added to x in FP64
template <typename T, int PT>
__global__ void __launch_bounds__(AT)
k_xupdate(int m, const int* __restrict__ kd, pset_dev ps, const T* __restrict__ V, size_t L,
          const double2* __restrict__ y, double2* __restrict__ x) {
  using S = typename basis_t<T>::S;
  const chunk_ref c = chunk_of(ps, blockIdx.x);
  const int K = kd[c.p];
  if (K == 0) return;
  two<T> acc[PT];
#pragma unroll
  for (int e = 0; e < PT; ++e) acc[e].a = acc[e].b = basis_t<T>::make(0.0, 0.0);
  for (int jj = 0; jj < K; jj += AB) {
    two<T> v[AB][PT];
#pragma unroll
    for (int b = 0; b < AB; ++b)
#pragma unroll
      for (int e = 0; e < PT; ++e) {
        const int q = 2 * (e * blockDim.x + threadIdx.x);
        v[b][e].a = v[b][e].b = basis_t<T>::make(0.0, 0.0);
        if (q < c.cnt && jj + b < K) v[b][e] = load2(V + (size_t)(jj + b) * L + c.base + q);
      }
#pragma unroll
    for (int b = 0; b < AB; ++b) {
      if (jj + b >= K) break;
      const double2 yd = y[(size_t)c.p * m + jj + b];
      const S yr = (S)yd.x, yi = (S)yd.y;
#pragma unroll
      for (int e = 0; e < PT; ++e) {
        const two<T> a = v[b][e];
        acc[e].a.x = fma(a.a.x, yr, fma(-a.a.y, yi, acc[e].a.x));
        acc[e].a.y = fma(a.a.x, yi, fma(a.a.y, yr, acc[e].a.y));
        acc[e].b.x = fma(a.b.x, yr, fma(-a.b.y, yi, acc[e].b.x));
        acc[e].b.y = fma(a.b.x, yi, fma(a.b.y, yr, acc[e].b.y));
      }
    }
  }
#pragma unroll
  for (int e = 0; e < PT; ++e) {
    const int q = 2 * (e * blockDim.x + threadIdx.x);
    if (q < c.cnt) {
      const two<double2> xo = load2(x + c.base + q);
      store2(x + c.base + q,
             make_double2(xo.a.x + (double)acc[e].a.x, xo.a.y + (double)acc[e].a.y),
             make_double2(xo.b.x + (double)acc[e].b.x, xo.b.y + (double)acc[e].b.y));
    }
  }
}

// r = f - ax (ax may be null: r = f; r may be null); per-chunk ||r||^2, ||f||^2
__global__ void __launch_bounds__(AT)
k_residual(pset_dev ps, const double2* __restrict__ f, const double2* __restrict__ ax,
           double2* __restrict__ r, double* __restrict__ rr, double* __restrict__ ff) {
  const chunk_ref c = chunk_of(ps, blockIdx.x);
  double sr = 0.0, sf = 0.0;
  // pairs of elements as in the other kernels: the order of the sums is the
  // chunk's, not the CTA's
#pragma unroll 4
  for (int q = 2 * threadIdx.x; q < c.cnt; q += 2 * blockDim.x) {
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const size_t idx = c.base + q + u;
      const double2 fv = f[idx];
      double2 v = fv;
      if (ax) {
        const double2 a = ax[idx];
        v.x -= a.x;
        v.y -= a.y;
      }
      if (r) r[idx] = v;
      sr += v.x * v.x + v.y * v.y;
      sf += fv.x * fv.x + fv.y * fv.y;
    }
  }
  __shared__ double red[2][AT / 32];
  sr = warp_sum(sr);
  sf = warp_sum(sf);
  if ((threadIdx.x & 31) == 0) {
    red[0][threadIdx.x >> 5] = sr;
    red[1][threadIdx.x >> 5] = sf;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double a = 0.0, b = 0.0;
    for (int q = 0; q < (int)(blockDim.x >> 5); ++q) {
      a += red[0][q];
      b += red[1][q];
    }
    rr[c.slot] = a;
    ff[c.slot] = b;
  }
}

__global__ void k_sum_chunks(int P, pset_dev ps, const double* __restrict__ a,
                             const double* __restrict__ b, double* __restrict__ out) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= P) return;
  double s = 0.0, t = 0.0;
  for (int c = 0; c < ps.nch[p]; ++c) {
    s += a[ps.chb[p] + c];
    t += b[ps.chb[p] + c];
  }
  out[p] = sqrt(s);
  out[P + p] = sqrt(t);
}

__global__ void k_axpy(size_t len, const double2* __restrict__ d, double2* __restrict__ x) {
  const size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= len) return;
  const double2 a = x[e], b = d[e];
  x[e] = make_double2(a.x + b.x, a.y + b.y);
}

__global__ void k_zero(size_t len, double2* __restrict__ x) {
  const size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e < len) x[e] = make_double2(0.0, 0.0);
}

unsigned blocks_for(size_t len, int t = 256) { return (unsigned)((len + t - 1) / t); }

// basis elements one orthogonalisation pass of step j reads: sum over the
// active problems of (j + 1) n_p
long long arnoldi_elems(const pset& ps, const std::vector<int>& act, int j) {
  long long e = 0;
  for (int p = 0; p < ps.P; ++p)
    if (act[p]) e += (long long)(j + 1) * ps.len[p];
  return e;
}

// ---------------------------------------------------------------------------
// host driver
// ---------------------------------------------------------------------------
struct ws {
  bool f32 = false;                  // FP32 basis (inner solves of refined precisions)
  float2 *V32 = nullptr, *w32 = nullptr;
  double2* vin = nullptr;            // FP64 copy of the newest FP32 basis vector
  double2 *V, *H, *gv, *sn, *w, *hbuf, *y, *part;
  double *cs, *hn, *res, *nrmp, *rr, *ff, *norms;
  int *act, *kd, *cnt;
};

ws workspace(cudaStream_t st, krylov_ws& K, const pset& ps, int m, bool f32) {
  const int P = ps.P, Q = ps.Q;
  const size_t L = ps.L;
  if (f32) {
    K.V32.reserve(sizeof(float2) * L * (m + 1));
    K.w32.reserve(sizeof(float2) * L);
    K.vin.reserve(sizeof(double2) * L);
  } else {
    K.V.reserve(sizeof(double2) * L * (m + 1));
  }
  K.w.reserve(sizeof(double2) * L);
  K.H.reserve(sizeof(double2) * (size_t)P * (m + 1) * m);
  size_t sm = 0;
  auto take = [&](size_t bytes) {
    size_t o = sm;
    sm += (bytes + 255) & ~size_t(255);
    return o;
  };
  const size_t o_gv = take(sizeof(double2) * P * (m + 1));
  const size_t o_sn = take(sizeof(double2) * P * m);
  const size_t o_hb = take(sizeof(double2) * P * (m + 1));
  const size_t o_y = take(sizeof(double2) * P * m);
  const size_t o_part = take(sizeof(double2) * (size_t)Q * (m + 1));
  const size_t o_cs = take(sizeof(double) * P * m);
  const size_t o_hn = take(sizeof(double) * P);
  const size_t o_res = take(sizeof(double) * P);
  const size_t o_nrmp = take(sizeof(double) * Q);
  const size_t o_rr = take(sizeof(double) * Q);
  const size_t o_ff = take(sizeof(double) * Q);
  const size_t o_norms = take(sizeof(double) * 2 * P);
  const size_t o_act = take(sizeof(int) * P);
  const size_t o_kd = take(sizeof(int) * P);
  const size_t o_cnt = take(sizeof(int) * P);
  K.small.reserve(sm);
  char* b = K.small.as<char>();
  ws W;
  W.f32 = f32;
  W.V = f32 ? nullptr : K.V.as<double2>();
  W.V32 = f32 ? K.V32.as<float2>() : nullptr;
  W.w32 = f32 ? K.w32.as<float2>() : nullptr;
  W.vin = f32 ? K.vin.as<double2>() : nullptr;
  W.H = K.H.as<double2>();
  W.w = K.w.as<double2>();
  W.gv = (double2*)(b + o_gv);
  W.sn = (double2*)(b + o_sn);
  W.hbuf = (double2*)(b + o_hb);
  W.y = (double2*)(b + o_y);
  W.part = (double2*)(b + o_part);
  W.cs = (double*)(b + o_cs);
  W.hn = (double*)(b + o_hn);
  W.res = (double*)(b + o_res);
  W.nrmp = (double*)(b + o_nrmp);
  W.rr = (double*)(b + o_rr);
  W.ff = (double*)(b + o_ff);
  W.norms = (double*)(b + o_norms);
  W.act = (int*)(b + o_act);
  W.kd = (int*)(b + o_kd);
  W.cnt = (int*)(b + o_cnt);
  CFIE_CHECK_CUDA(cudaMemsetAsync(W.cnt, 0, sizeof(int) * P, st));
  if (K.host_cap < 2 * P + 8) {
    if (K.host) cudaFreeHost(K.host);
    K.host = nullptr;
    CFIE_CHECK_CUDA(cudaMallocHost(&K.host, sizeof(double) * (2 * P + 8)));
    K.host_cap = 2 * P + 8;
  }
  return W;
}

// ||r_p|| and ||f_p|| to host (synchronous); r = f - ax (ax, r may be null)
void residual_norms(cudaStream_t st, krylov_ws& K, const pset& ps, const ws& W,
                    const double2* f, const double2* ax, double2* r, std::vector<double>& rn,
                    std::vector<double>& fn) {
  const int P = ps.P;
  k_residual<<<ps.Q, ps.tb, 0, st>>>(ps.dev, f, ax, r, W.rr, W.ff);
  CFIE_CHECK_LAUNCH();
  k_sum_chunks<<<blocks_for(P, 64), 64, 0, st>>>(P, ps.dev, W.rr, W.ff, W.norms);
  CFIE_CHECK_LAUNCH();
  CFIE_CHECK_CUDA(
      cudaMemcpyAsync(K.host, W.norms, sizeof(double) * 2 * P, cudaMemcpyDeviceToHost, st));
  CFIE_CHECK_CUDA(cudaStreamSynchronize(st));
  rn.assign(K.host, K.host + P);
  fn.assign(K.host + P, K.host + 2 * P);
}

// f(items, group, pairs per thread) for the items of each chunk length
template <typename F>
void each_group(const pset& ps, F f) {
  for (const pset_group& g : ps.groups) {
    pset_dev d = ps.dev;
    d.first = g.first;
    switch (g.pairs) {
      case 1: f(d, g, std::integral_constant<int, 1>()); break;
      case 2: f(d, g, std::integral_constant<int, 2>()); break;
      default: f(d, g, std::integral_constant<int, 4>());
    }
    CFIE_CHECK_LAUNCH();
  }
}

// column j of H and the rotations: classical Gram-Schmidt twice, then the Givens
// step.  A set with fewer chunks than two per SM splits the inner products over
// the basis vectors as well.
template <typename T>
void orthogonalise(cudaStream_t st, const pset& ps, const ws& W, int m, int j, size_t L, const T* V,
                   T* w) {
  const givens_dev G{W.H, W.cs, W.sn, W.gv, W.hn, W.res};
  const int ny = std::max(1, std::min((j + AB) / AB, 304 / ps.Q));
  const int JB = std::min(256, ((j + 1 + ny - 1) / ny + AB - 1) / AB * AB);
  const size_t hs = sizeof(T) * (j + 1);
  const size_t gs = (sizeof(double2) * 2 + sizeof(double)) * m + sizeof(double2);
  for (int pass = 0; pass < 2; ++pass) {
    each_group(ps, [&](const pset_dev& d, const pset_group& g, auto pt) {
      const size_t red = sizeof(double2) * std::min(JB, j + 1) * (g.tb / 32);
      k_dots<T, decltype(pt)::value><<<dim3(g.count, (j + JB) / JB), g.tb, red, st>>>(
          j, JB, m, j, pass == 0, V, L, w, W.act, d, W.part, W.cnt, W.hbuf, W.H);
    });
    each_group(ps, [&](const pset_dev& d, const pset_group& g, auto pt) {
      constexpr int PT = decltype(pt)::value;
      if (pass == 0)
        k_update<T, PT, false>
            <<<g.count, g.tb, hs, st>>>(j, m, V, L, W.hbuf, W.act, d, w, nullptr, W.cnt, G);
      else
        k_update<T, PT, true><<<g.count, g.tb, std::max(hs, gs), st>>>(
            j, m, V, L, W.hbuf, W.act, d, w, W.nrmp, W.cnt, G);
    });
  }
}

// x += V y
template <typename T>
void add_basis(cudaStream_t st, const pset& ps, const ws& W, int m, size_t L, const T* V,
               double2* x) {
  each_group(ps, [&](const pset_dev& d, const pset_group& g, auto pt) {
    k_xupdate<T, decltype(pt)::value><<<g.count, g.tb, 0, st>>>(m, W.kd, d, V, L, W.y, x);
  });
}

// Marks the problems of an Arnoldi step's matvec for the matvec callbacks.
struct live_scope {
  std::vector<int>& v;
  live_scope(std::vector<int>& v_, const std::vector<int>& act) : v(v_) { v = act; }
  ~live_scope() { v.clear(); }
};

// One GMRES cycle: starting residual r (norms beta), basis built with the
// inner or the FP64 matvec, x += V y.  active[p] says which problems take part;
// tol[p] is the absolute residual-norm target.  Counts steps per problem.
void gmres_cycle(cudaStream_t st, cfie_ctx* ctx, krylov_ws& K, const pset& ps, const ws& W,
                 const solve_fns& fns, bool inner, const double2* r,
                 const std::vector<double>& beta, const std::vector<double>& tol,
                 const std::vector<int>& active, int m, std::vector<int>& steps_left, double2* x,
                 std::vector<int>& its, cfie_solve_stats& stats, std::vector<int>* met = nullptr) {
  const int P = ps.P;
  const size_t L = ps.L;
  std::vector<int> act = active, kd(P, 0);
  if (met) met->assign(P, 0);
  int nact = 0;
  for (int p = 0; p < P; ++p) nact += act[p];
  if (!nact) return;
  CFIE_CHECK_CUDA(cudaMemcpyAsync(W.act, act.data(), sizeof(int) * P, cudaMemcpyHostToDevice, st));
  CFIE_CHECK_CUDA(
      cudaMemcpyAsync(W.norms, beta.data(), sizeof(double) * P, cudaMemcpyHostToDevice, st));
  if (W.f32)
    k_start<float2><<<ps.Q, ps.tb, 0, st>>>(W.act, ps.dev, W.norms, r, W.V32, W.vin);
  else
    k_start<double2><<<ps.Q, ps.tb, 0, st>>>(W.act, ps.dev, W.norms, r, W.V, nullptr);
  CFIE_CHECK_LAUNCH();
  k_g_init<<<blocks_for((size_t)P * (m + 1)), 256, 0, st>>>(P, m, W.act, W.norms, W.gv);
  CFIE_CHECK_LAUNCH();
  stats.cycles++;
  for (int j = 0; j < m; ++j) {
    const double2* vj = W.f32 ? W.vin : W.V + (size_t)j * L;
    if (fns.prec) {   // right preconditioning: the operator is A P
      fns.prec(vj, K.pz.as<double2>());
      vj = K.pz.as<double2>();
    }
    {
      live_scope ls(K.live, act);
      if (inner) {
        stats.inner_matvecs++;
        fns.inner(vj, W.w);
      } else {
        stats.fp64_matvecs++;
        fns.fp64(vj, W.w);
      }
    }
    {
      prof_scope ps_(ctx, CFIE_K_ARNOLDI);
      if (W.f32) {
        k_to32<<<ps.Q, ps.tb, 0, st>>>(W.act, ps.dev, W.w, W.w32);
        CFIE_CHECK_LAUNCH();
        orthogonalise<float2>(st, ps, W, m, j, L, W.V32, W.w32);
      } else {
        orthogonalise<double2>(st, ps, W, m, j, L, W.V, W.w);
      }
      if (W.f32)
        k_scale<float2><<<ps.Q, ps.tb, 0, st>>>(W.act, ps.dev, W.hn, W.w32,
                                             W.V32 + (size_t)(j + 1) * L, W.vin);
      else
        k_scale<double2><<<ps.Q, ps.tb, 0, st>>>(W.act, ps.dev, W.hn, W.w,
                                              W.V + (size_t)(j + 1) * L, nullptr);
      CFIE_CHECK_LAUNCH();
      stats.arnoldi_elems += arnoldi_elems(ps, act, j);
    }
    CFIE_CHECK_CUDA(
        cudaMemcpyAsync(K.host, W.res, sizeof(double) * P, cudaMemcpyDeviceToHost, st));
    CFIE_CHECK_CUDA(cudaStreamSynchronize(st));
    stats.arnoldi_steps++;
    bool changed = false;
    nact = 0;
    for (int p = 0; p < P; ++p) {
      if (!act[p]) continue;
      kd[p] = j + 1;
      its[p]++;
      steps_left[p]--;
      if (K.host[p] <= tol[p] || steps_left[p] <= 0) {
        if (met && K.host[p] <= tol[p]) (*met)[p] = 1;
        act[p] = 0;
        changed = true;
      } else {
        nact++;
      }
    }
    if (!nact) break;
    if (changed)
      CFIE_CHECK_CUDA(
          cudaMemcpyAsync(W.act, act.data(), sizeof(int) * P, cudaMemcpyHostToDevice, st));
  }
  CFIE_CHECK_CUDA(cudaMemcpyAsync(W.kd, kd.data(), sizeof(int) * P, cudaMemcpyHostToDevice, st));
  k_lsq<<<P, 32, 2 * sizeof(double2) * m, st>>>(m, W.kd, W.H, W.gv, W.y);
  CFIE_CHECK_LAUNCH();
  // x += V y, or with right preconditioning x += P (V y)
  double2* xu = x;
  if (fns.prec) {
    xu = K.pz.as<double2>();
    k_zero<<<blocks_for(L), 256, 0, st>>>(L, xu);
    CFIE_CHECK_LAUNCH();
  }
  if (W.f32)
    add_basis<float2>(st, ps, W, m, L, W.V32, xu);
  else
    add_basis<double2>(st, ps, W, m, L, W.V, xu);
  if (fns.prec) {
    fns.prec(xu, K.pz2.as<double2>());
    k_axpy<<<blocks_for(L), 256, 0, st>>>(L, K.pz2.as<double2>(), x);
    CFIE_CHECK_LAUNCH();
  }
  // host vectors copied above must stay alive until the copies ran
  CFIE_CHECK_CUDA(cudaStreamSynchronize(st));
}

}  // namespace

void pset_build(pset& ps, const std::vector<size_t>& off, const std::vector<int>& len,
                const std::vector<size_t>& own, cudaStream_t st) {
  ps.P = (int)off.size();
  ps.L = 0;
  ps.len = len;
  ps.groups.clear();
  std::vector<int> nch(ps.P), chb(ps.P), ch(ps.P);
  std::vector<chunk_item> items;
  // Chunks of 2048 elements (256 threads, four pairs each), or shorter ones down to
  // 128 (64 threads, one pair) until the problem's own operator has about two per
  // SM.  What else is in the set does not change the order of a problem's sums, so
  // that a solve gives the same bits alone and in a batch.  (With the length from the
  // whole set's size a batch of 32 stars, n up to 16384, 32 directions each, takes 31 ms
  // instead of 40 for these kernels, of 174 in all; a balanced tree over units of a warp,
  // the same for every length, 30 ms, but 5 to 10 % more in small sets.)
  for (int p = 0; p < ps.P; ++p) {
    ch[p] = 2048;
    while (ch[p] > 128 && own[p] / ch[p] < 304) ch[p] /= 2;
    ps.L = std::max(ps.L, off[p] + (size_t)len[p]);
  }
  for (int c = 128; c <= 2048; c *= 2) {
    pset_group g{(int)items.size(), 0, std::min(AT, c / 2), std::max(1, c / (2 * AT))};
    for (int p = 0; p < ps.P; ++p) {
      if (ch[p] != c) continue;
      chb[p] = (int)items.size();
      for (int at = 0; at < len[p]; at += c)
        items.push_back({off[p] + (size_t)at, std::min(c, len[p] - at), p});
      nch[p] = (int)items.size() - chb[p];
    }
    g.count = (int)items.size() - g.first;
    if (!g.count) continue;
    ps.groups.push_back(g);
    ps.tb = g.tb;
  }
  ps.Q = (int)items.size();
  ps.buf.reserve(sizeof(chunk_item) * ps.Q + sizeof(int) * 2 * ps.P + 64);
  char* b = ps.buf.as<char>();
  size_t o = 0;
  auto put = [&](const void* src, size_t n) {
    CFIE_CHECK_CUDA(cudaMemcpyAsync(b + o, src, n, cudaMemcpyHostToDevice, st));
    void* at = b + o;
    o += (n + 15) & ~size_t(15);
    return at;
  };
  ps.dev.items = (const chunk_item*)put(items.data(), sizeof(chunk_item) * ps.Q);
  ps.dev.nch = (const int*)put(nch.data(), sizeof(int) * ps.P);
  ps.dev.chb = (const int*)put(chb.data(), sizeof(int) * ps.P);
  ps.dev.first = 0;
  CFIE_CHECK_CUDA(cudaStreamSynchronize(st));  // the host vectors die on return
}

void pset_uniform(pset& ps, int n, int nrhs, cudaStream_t st) {
  std::vector<size_t> off(nrhs);
  std::vector<int> len(nrhs, n);
  for (int k = 0; k < nrhs; ++k) off[k] = (size_t)k * n;
  pset_build(ps, off, len, std::vector<size_t>(nrhs, (size_t)n * nrhs), st);
}

void gmres_set(cudaStream_t st, cfie_ctx* ctx, krylov_ws& K, const pset& ps,
               const solve_fns& fns, bool refined, const double2* f, double2* x, double rtol,
               int restart, int maxit, int* iters, double* relres, cfie_status* status,
               cfie_solve_stats& stats) {
  stats = cfie_solve_stats{};
  const int P = ps.P;
  const size_t L = ps.L;
  int m = restart > 0 ? restart : maxit;
  m = std::max(1, std::min(m, std::min(maxit, MAXJ)));
  const bool f32 = refined && fns.basis32;
  stats.basis_fp32 = f32 ? 1 : 0;
  ws W = workspace(st, K, ps, m, f32);
  K.r.reserve(sizeof(double2) * L);
  if (fns.prec) {
    K.pz.reserve(sizeof(double2) * L);
    K.pz2.reserve(sizeof(double2) * L);
  }
  double2* r = K.r.as<double2>();
  double2* ax = W.w;  // matvec output scratch (free between cycles)

  std::vector<double> rn, fn, xn, dummy;
  std::vector<int> its(P, 0), steps_left(P, maxit), active(P, 1);
  // true residual of the initial guess (no matvec when x0 = 0)
  residual_norms(st, K, ps, W, x, nullptr, nullptr, xn, dummy);
  bool x_zero = true;
  for (int p = 0; p < P; ++p) x_zero = x_zero && xn[p] == 0.0;
  if (x_zero) {
    residual_norms(st, K, ps, W, f, nullptr, r, rn, fn);
  } else {
    stats.fp64_matvecs++;
    fns.fp64(x, ax);
    residual_norms(st, K, ps, W, f, ax, r, rn, fn);
  }

  if (!refined) {
    for (;;) {
      std::vector<double> tol(P);
      int nact = 0;
      for (int p = 0; p < P; ++p) {
        tol[p] = rtol * fn[p];
        active[p] = (rn[p] > tol[p] && steps_left[p] > 0) ? 1 : 0;
        nact += active[p];
      }
      if (!nact) break;
      gmres_cycle(st, ctx, K, ps, W, fns, false, r, rn, tol, active, m, steps_left, x, its,
                  stats);
      stats.fp64_matvecs++;
      fns.fp64(x, ax);
      residual_norms(st, K, ps, W, f, ax, r, rn, fn);
    }
  } else {
    // iterative refinement: inner GMRES on A d = r with the fast matvec,
    // x += d, r = f - A64 x (FP64)
    K.d.reserve(sizeof(double2) * L);
    K.rin.reserve(sizeof(double2) * L);
    double2* d = K.d.as<double2>();
    double2* rin = K.rin.as<double2>();
    const double tau_min = 1e-4;
    for (int outer = 0; outer < 12; ++outer) {
      std::vector<double> tol(P);
      int nact = 0;
      for (int p = 0; p < P; ++p) {
        active[p] = (rn[p] > rtol * fn[p] && steps_left[p] > 0) ? 1 : 0;
        nact += active[p];
        double tau = rn[p] > 0 ? 0.3 * rtol * fn[p] / rn[p] : 1.0;
        tau = std::min(0.5, std::max(tau_min, tau));
        tol[p] = tau * rn[p];
      }
      if (!nact) break;
      stats.refinements++;
      k_zero<<<blocks_for(L), 256, 0, st>>>(L, d);
      CFIE_CHECK_LAUNCH();
      std::vector<double> irn = rn, ifn;
      std::vector<int> iact = active;
      CFIE_CHECK_CUDA(cudaMemcpyAsync(rin, r, sizeof(double2) * L, cudaMemcpyDeviceToDevice, st));
      for (int cyc = 0; cyc < 64; ++cyc) {
        std::vector<int> met;
        gmres_cycle(st, ctx, K, ps, W, fns, true, rin, irn, tol, iact, m, steps_left, d, its,
                    stats, &met);
        bool all_met = true;
        for (int p = 0; p < P; ++p) all_met = all_met && (!iact[p] || met[p]);
        if (all_met) break;   // the outer FP64 residual below is the real check
        // inner true residual r - A_fast d before restarting
        stats.inner_matvecs++;
        fns.inner(d, ax);
        residual_norms(st, K, ps, W, r, ax, rin, irn, ifn);
        int left = 0;
        for (int p = 0; p < P; ++p) {
          iact[p] = active[p] && irn[p] > tol[p] && steps_left[p] > 0 ? 1 : 0;
          left += iact[p];
        }
        if (!left) break;
      }
      k_axpy<<<blocks_for(L), 256, 0, st>>>(L, d, x);
      CFIE_CHECK_LAUNCH();
      stats.fp64_matvecs++;
      fns.fp64(x, ax);
      residual_norms(st, K, ps, W, f, ax, r, rn, fn);
    }
  }
  *status = CFIE_OK;
  for (int p = 0; p < P; ++p) {
    const double rel = fn[p] > 0 ? rn[p] / fn[p] : 0.0;
    if (relres) relres[p] = rel;
    if (iters) iters[p] = its[p];
    if (!(rel <= rtol)) *status = CFIE_ENOCONV;
  }
}

void krylov_release(krylov_ws& K) {
  if (K.host) cudaFreeHost(K.host);
  K.host = nullptr;
  K.host_cap = 0;
}
