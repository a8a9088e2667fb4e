// Spectral tangential derivative of the sound-hard operator (Maue's identity,
// Section 1) by FFT: for each density column,
//
//     d/dt x = IDFT( i m' DFT(x) ),  m' = m for m < n/2, m - n for m > n/2,
//                                    0 at the Nyquist mode m = n/2,
//
// then divided by |z'| (d/ds).  This is the same operator as the circulant
// c_d = (-1)^d cot(pi d / n) / 2, at O(n log n) instead of O(n^2) per column.
// A power-of-two n is transformed directly (N = n).  A DFT of any other length
// n goes through Bluestein's chirp-z identity
//
//     X_m = conj(b_m) sum_j (x_j conj(b_j)) b_(m-j),   b_k = exp(i pi k^2 / n),
//
// a linear convolution computed with power-of-two FFTs of length N >= 2n - 1;
// the inverse DFT is conj(DFT(conj(D))) / n.  FP64 for the true residuals, FP32
// for the inner matvecs (same code, element type a template parameter).
//
// A length N = N1 N2 transform is done in two kernels (Bailey's four-step
// form, time index j = j1 N2 + j2, frequency k1 + N1 k2): N2 transforms of
// length N1 down the columns j2, times the twiddles exp(-2 pi i j2 k1 / N),
// then N1 transforms of length N2 along the rows k1.  The spectrum is left in
// that order: what it is multiplied by is stored in the same order, and the
// way back runs the steps in reverse.  So one derivative is three kernels
// (columns; rows, times i m', rows back; columns back), with Bluestein five
// (the middle one ends the first convolution and starts the second on the same
// columns).  Inside a kernel the transforms are Stockham passes of radix 8, 4
// and 2 in shared memory.
//
// Bound: launches and latency (a whole derivative moves a few MB).  Before,
// one radix-2 pass per launch (61 launches at N = 16384), or one CTA per
// column with everything in shared memory (52 passes behind barriers, 16 CTAs
// at 16 columns).  Measured (GB300), the two derivatives of one product: n =
// 4096, 16 columns, FP32 268 -> 45 us, FP64 500 -> 80 us; n = 32768, 1 column,
// FP32 500 -> 30 us; n = 6002 (N = 16384), 33 columns, FP32 470 -> 110 us.
#include <algorithm>

#include "internal.h"

namespace {

template <typename T> struct cx;
template <> struct cx<double2> {
  using S = double;
  static __device__ __forceinline__ double2 make(double a, double b) { return make_double2(a, b); }
};
template <> struct cx<float2> {
  using S = float;
  static __device__ __forceinline__ float2 make(double a, double b) {
    return make_float2((float)a, (float)b);
  }
  static __device__ __forceinline__ float2 make(float a, float b) { return make_float2(a, b); }
};

template <typename T>
__device__ __forceinline__ T cmul(T a, T b) {
  return cx<T>::make(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
template <typename T>
__device__ __forceinline__ T cmulc(T a, T b) {   // a * conj(b)
  return cx<T>::make(a.x * b.x + a.y * b.y, a.y * b.x - a.x * b.y);
}
template <typename T>
__device__ __forceinline__ T cadd(T a, T b) { return cx<T>::make(a.x + b.x, a.y + b.y); }
template <typename T>
__device__ __forceinline__ T csub(T a, T b) { return cx<T>::make(a.x - b.x, a.y - b.y); }

// twiddles exp(-2 pi i q / N), q < N, and exp(-2 pi i q / N2), q < N2 (FP64 and
// FP32 copies)
__global__ void k_twiddles(int N, int N2, double2* __restrict__ tw, float2* __restrict__ tw32,
                           double2* __restrict__ tc, float2* __restrict__ tc32) {
  const int q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= N) return;
  double s, c;
  sincospi(-2.0 * q / N, &s, &c);
  tw[q] = make_double2(c, s);
  tw32[q] = make_float2((float)c, (float)s);
  if (q % (N / N2) == 0) {
    tc[q / (N / N2)] = make_double2(c, s);
    tc32[q / (N / N2)] = make_float2((float)c, (float)s);
  }
}

// Bluestein's chirp b_k = exp(i pi (k^2 mod 2n) / n), k < n (the square reduced
// exactly in integers before the sine and cosine), its wrapped copy B[k] = b_k
// (k < n), B[N - k] = b_k (0 < k < n), zero elsewhere, and the output factors
// 1 / (n N |z'|) (direct transform: 1 / (N |z'|))
__global__ void k_chirp(int n, int N, int direct, const double* __restrict__ sp,
                        double2* __restrict__ b, float2* __restrict__ b32,
                        double2* __restrict__ B, double* __restrict__ osc) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= N) return;
  if (k < n) osc[k] = 1.0 / ((direct ? 1.0 : (double)n) * (double)N * sp[k]);
  if (direct) return;
  const long long m = k < n ? k : (k > N - n ? N - k : -1);
  double2 v = make_double2(0.0, 0.0);
  if (m >= 0) {
    const long long q = (m * m) % (2LL * n);
    double s, c;
    sincospi((double)q / n, &s, &c);
    v = make_double2(c, s);
  }
  B[k] = v;
  if (k < n) {
    b[k] = v;
    b32[k] = make_float2((float)v.x, (float)v.y);
  }
}

// discrete Fourier transforms of 2, 4 and 8 values in registers (sign -1, or +1
// when INV)
template <typename T, bool INV>
__device__ __forceinline__ T mul_i(T a) {   // a * (-i), INV: a * i
  return INV ? cx<T>::make(-a.y, a.x) : cx<T>::make(a.y, -a.x);
}
template <typename T, bool INV, int R>
__device__ __forceinline__ void dft(T* v) {
  if constexpr (R == 2) {
    const T a = v[0], b = v[1];
    v[0] = cadd(a, b);
    v[1] = csub(a, b);
  } else if constexpr (R == 4) {
    const T a = cadd(v[0], v[2]), b = csub(v[0], v[2]);
    const T c = cadd(v[1], v[3]), d = mul_i<T, INV>(csub(v[1], v[3]));
    v[0] = cadd(a, c);
    v[1] = cadd(b, d);
    v[2] = csub(a, c);
    v[3] = csub(b, d);
  } else {
    using S = typename cx<T>::S;
    T e[4] = {v[0], v[2], v[4], v[6]}, o[4] = {v[1], v[3], v[5], v[7]};
    dft<T, INV, 4>(e);
    dft<T, INV, 4>(o);
    const S h = (S)0.70710678118654752440;
    const T w1 = cx<T>::make(h, INV ? h : -h), w3 = cx<T>::make(-h, INV ? h : -h);
    o[1] = cmul(o[1], w1);
    o[2] = mul_i<T, INV>(o[2]);
    o[3] = cmul(o[3], w3);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      v[k] = cadd(e[k], o[k]);
      v[k + 4] = csub(e[k], o[k]);
    }
  }
}

// One Stockham pass of radix R over 2^lc transforms of length M in shared
// memory (element e of transform c at e es + c): m = product of the radices so
// far, butterfly (j, k), k < m, reads elements i + q M / R (i = j m + k), times
// exp(-2 pi i q k / (R m)), and writes elements R j m + k + p m.  tc: the N2
// twiddles, N2 = M ts.
template <typename T, bool INV, int R>
__device__ __forceinline__ void fft_pass(const T* __restrict__ a, T* __restrict__ o, int M, int lc,
                                         int es, int lm, const T* __restrict__ tc, int ts) {
  const int m = 1 << lm, nb = (M / R) << lc;
  const int tstep = (M / R >> lm) * ts;
  for (int b = threadIdx.x; b < nb; b += blockDim.x) {
    const int c = b & ((1 << lc) - 1), i = b >> lc;
    const int k = i & (m - 1), j = i >> lm;
    T v[R];
#pragma unroll
    for (int q = 0; q < R; ++q) v[q] = a[(i + q * (M / R)) * es + c];
    if (lm) {
#pragma unroll
      for (int q = 1; q < R; ++q) {
        const T w = __ldg(tc + q * k * tstep);
        v[q] = INV ? cmulc(v[q], w) : cmul(v[q], w);
      }
    }
    dft<T, INV, R>(v);
#pragma unroll
    for (int p = 0; p < R; ++p) o[(R * j * m + k + p * m) * es + c] = v[p];
  }
  __syncthreads();
}

// 2^lc transforms of length M = 2^lM from buffer a, b the other buffer; returns
// the one that holds the result (natural order).  The caller synchronises
// before the call.
template <typename T, bool INV>
__device__ T* fft_smem(T* a, T* b, int lM, int lc, int es, const T* __restrict__ tc, int ts) {
  const int M = 1 << lM;
  for (int lm = 0; lm < lM;) {
    const int rem = lM - lm;
    if (rem >= 5 || rem == 3) {
      fft_pass<T, INV, 8>(a, b, M, lc, es, lm, tc, ts);
      lm += 3;
    } else if (rem >= 2) {
      fft_pass<T, INV, 4>(a, b, M, lc, es, lm, tc, ts);
      lm += 2;
    } else {
      fft_pass<T, INV, 2>(a, b, M, lc, es, lm, tc, ts);
      lm += 1;
    }
    T* t = a;
    a = b;
    b = t;
  }
  return a;
}

template <typename T>
struct fft_args {
  int n, N, l1, l2, lc, direct;   // N = 2^(l1 + l2); 2^lc transforms per CTA
  const T* tw;                    // exp(-2 pi i q / N), q < N
  const T* tc;                    // exp(-2 pi i q / 2^l2)
  const T* ch;                    // chirp
  const T* bf;                    // spectrum of the wrapped chirp, [k1][k2]
  T* work;                        // [column][N]
};

// Transforms down the columns j2 = 2^lc blockIdx.x .. of density column
// blockIdx.y.  COL_IN: from x (times the chirp) to the rows; COL_RAW: the same
// from the work buffer; COL_OUT: from the rows to the output; COL_MID: from the
// rows to the time domain (the end of Bluestein's first convolution), times
// i m', and on to the rows of the second.
enum { COL_IN = 1, COL_OUT = 2, COL_MID = 3, COL_RAW = 4 };

template <typename T, int MODE, typename X, typename O>
__global__ void __launch_bounds__(256)
k_fft_cols(fft_args<T> F, const X* __restrict__ x, const double* __restrict__ osc, double2 scale,
           const O* base, O* out) {
  using S = typename cx<T>::S;
  extern __shared__ __align__(16) unsigned char raw[];
  const int N1 = 1 << F.l1, N2 = 1 << F.l2, C = 1 << F.lc, es = C + 1;
  const int col = blockIdx.y, c0 = blockIdx.x << F.lc, n = F.n;
  T* a = reinterpret_cast<T*>(raw);
  T* b = a + (size_t)N1 * es;
  T* w = F.work + (size_t)col * F.N;
  const int tot = N1 << F.lc, ts = N2 >> F.l1;
  if constexpr (MODE == COL_IN || MODE == COL_RAW) {
    for (int e = threadIdx.x; e < tot; e += blockDim.x) {
      const int c = e & (C - 1), j1 = e >> F.lc, j = j1 * N2 + c0 + c;
      T v = cx<T>::make((S)0, (S)0);
      if (MODE == COL_RAW) {
        v = w[j];
      } else if (j < n) {
        const X xv = x[(size_t)col * n + j];
        v = cx<T>::make((S)xv.x, (S)xv.y);
        if (!F.direct) v = cmulc(v, F.ch[j]);
      }
      a[j1 * es + c] = v;
    }
    __syncthreads();
  } else {
    for (int e = threadIdx.x; e < tot; e += blockDim.x) {
      const int c = e & (C - 1), k1 = e >> F.lc, j2 = c0 + c;
      a[k1 * es + c] = cmulc(w[k1 * N2 + j2], __ldg(F.tw + k1 * j2));
    }
    __syncthreads();
    T* r = fft_smem<T, true>(a, b, F.l1, F.lc, es, F.tc, ts);
    for (int e = threadIdx.x; e < tot; e += blockDim.x) {
      const int c = e & (C - 1), j1 = e >> F.lc, j = j1 * N2 + c0 + c;
      T v = r[j1 * es + c];
      if constexpr (MODE == COL_OUT) {
        // out_j = base_j + scale osc_j conj(conj(b_j) conv_j) (direct: scale osc_j v_j)
        if (j >= n) continue;
        if (!F.direct) {
          v = cmulc(v, F.ch[j]);
          v.y = -v.y;
        }
        const double f = osc[j];
        const double dx = (double)v.x * f, dy = (double)v.y * f;
        double ox = scale.x * dx - scale.y * dy, oy = scale.x * dy + scale.y * dx;
        if (base) {
          const O bv = base[(size_t)col * n + j];
          ox += (double)bv.x;
          oy += (double)bv.y;
        }
        O q;
        q.x = ox;
        q.y = oy;
        out[(size_t)col * n + j] = q;
      } else {
        // X_m = conj(b_m) conv_m; D_m = i m' X_m / N; next input conj(D_m) conj(b_m)
        T d = cx<T>::make((S)0, (S)0);
        if (j < n) {
          const T ch = F.ch[j];
          const T Xm = cmulc(v, ch);
          const S mm = (S)(2 * j < n ? j : (2 * j == n ? 0 : j - n)) / (S)F.N;
          d = cmulc(cx<T>::make(-mm * Xm.y, -mm * Xm.x), ch);
        }
        r[j1 * es + c] = d;
      }
    }
    __syncthreads();
    if (r != a) {
      b = a;
      a = r;
    }
  }
  if constexpr (MODE != COL_OUT) {
    T* r = fft_smem<T, false>(a, b, F.l1, F.lc, es, F.tc, ts);
    for (int e = threadIdx.x; e < tot; e += blockDim.x) {
      const int c = e & (C - 1), k1 = e >> F.lc, j2 = c0 + c;
      w[k1 * N2 + j2] = cmul(r[k1 * es + c], __ldg(F.tw + k1 * j2));
    }
  }
}

// rows k1 = 2^lc blockIdx.x ..: forward transform along the row, times the
// chirp's spectrum (direct: i m'), back transform; FWD_ONLY: forward alone
template <typename T, bool FWD_ONLY>
__global__ void __launch_bounds__(256) k_fft_rows(fft_args<T> F) {
  using S = typename cx<T>::S;
  extern __shared__ __align__(16) unsigned char raw[];
  const int N1 = 1 << F.l1, N2 = 1 << F.l2, C = 1 << F.lc, es = C + 1;
  const int r0 = blockIdx.x << F.lc, n = F.n;
  T* a = reinterpret_cast<T*>(raw);
  T* b = a + (size_t)N2 * es;
  T* w = F.work + (size_t)blockIdx.y * F.N + (size_t)r0 * N2;
  const int tot = N2 << F.lc;
  for (int e = threadIdx.x; e < tot; e += blockDim.x) {
    const int c = e >> F.l2, j = e & (N2 - 1);
    a[j * es + c] = w[e];
  }
  __syncthreads();
  T* r = fft_smem<T, false>(a, b, F.l2, F.lc, es, F.tc, 1);
  if constexpr (!FWD_ONLY) {
    for (int e = threadIdx.x; e < tot; e += blockDim.x) {
      const int c = e >> F.l2, k2 = e & (N2 - 1);
      T v = r[k2 * es + c];
      if (F.direct) {
        const int m = r0 + c + N1 * k2;
        const S mm = (S)(2 * m < n ? m : (2 * m == n ? 0 : m - n));
        v = cx<T>::make(-mm * v.y, mm * v.x);
      } else {
        v = cmul(v, F.bf[(size_t)(r0 + c) * N2 + k2]);
      }
      r[k2 * es + c] = v;
    }
    __syncthreads();
    r = fft_smem<T, true>(r, r == a ? b : a, F.l2, F.lc, es, F.tc, 1);
  }
  for (int e = threadIdx.x; e < tot; e += blockDim.x) {
    const int c = e >> F.l2, j = e & (N2 - 1);
    w[e] = r[j * es + c];
  }
}

unsigned nb(size_t len, int t = 256) { return (unsigned)((len + t - 1) / t); }

__global__ void k_to_f32(size_t len, const double2* __restrict__ a, float2* __restrict__ b) {
  const size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e < len) b[e] = make_float2((float)a[e].x, (float)a[e].y);
}

template <typename T>
fft_args<T> args_of(const fft_plan& F, int n, T* work) {
  fft_args<T> A{};
  A.n = n;
  A.N = F.N;
  A.l1 = F.L / 2;
  A.l2 = F.L - F.L / 2;
  A.direct = F.direct;
  if constexpr (sizeof(T) == 16) {
    A.tw = F.tw.as<double2>();
    A.tc = F.tc.as<double2>();
    A.ch = F.chirp.as<double2>();
    A.bf = F.bf.as<double2>();
  } else {
    A.tw = F.tw32.as<float2>();
    A.tc = F.tc32.as<float2>();
    A.ch = F.chirp32.as<float2>();
    A.bf = F.bf32.as<float2>();
  }
  A.work = work;
  return A;
}

// Transforms per CTA (2^lc of length 2^lM, out of 2^lOther): about 2048
// elements, at least 64 contiguous bytes per row of the columns, fewer when
// the launch would leave SMs idle.  Shared memory: two buffers, for n <= 2^20 (N <=
// 2^21) at most 2 (2^11 elements x 2) or 2 (2^10 x (4 + 1)) of 16 bytes, 160 KB;
// spectral_fft refuses what does not fit.
template <typename T>
int per_cta(int lM, int lOther, int cols, int lmin) {
  int lc = std::max(lmin, 11 - lM);
  lc = std::min(lc, lOther);
  while (lc > std::min(lmin, lOther) && ((long long)cols << (lOther - lc)) < 152) --lc;
  return lc;
}
template <typename T>
size_t smem_of(int lM, int lc) {
  return 2 * sizeof(T) * (((size_t)1 << lM) * (((size_t)1 << lc) + 1));
}
constexpr size_t kSmemMax = (size_t)200 * 1024;

// the attribute is the bound of every launch of the kernel, not this one's
// size: it is per kernel and process-wide, and operators of other sizes launch
// the same kernel from other host threads (server slots)
#define FFT_LAUNCH(kernel, grid, smem, st, ...)                                               \
  do {                                                                                        \
    CFIE_CHECK_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, \
                                         (int)kSmemMax));                                     \
    kernel<<<grid, 256, smem, st>>>(__VA_ARGS__);                                             \
    CFIE_CHECK_LAUNCH();                                                                      \
  } while (0)

// out = base + scale (1/|z'|) d/dt in, columns of length n, element type T for
// the transforms
template <typename T, typename X, typename O>
void spectral_fft(cfie_op* op, const X* in, O* out, const O* base, double2 scale, int cols) {
  fft_plan& F = op->fft;
  cudaStream_t st = op->ctx->stream;
  dbuf& wb = sizeof(T) == 16 ? F.work : F.work32;
  wb.reserve(sizeof(T) * (size_t)F.N * cols);
  fft_args<T> C = args_of<T>(F, op->n, wb.as<T>()), R = C;
  constexpr int lmin = sizeof(T) == 16 ? 2 : 3;
  C.lc = per_cta<T>(C.l1, C.l2, cols, lmin);
  R.lc = per_cta<T>(R.l2, R.l1, cols, 0);
  const dim3 gc(1u << (C.l2 - C.lc), cols), gr(1u << (R.l1 - R.lc), cols);
  const size_t sc = smem_of<T>(C.l1, C.lc), sr = smem_of<T>(R.l2, R.lc);
  CFIE_REQUIRE(std::max(sc, sr) <= kSmemMax, "spectral derivative: transform too long");
  const double* osc = F.osc.as<double>();
  prof_scope ps(op->ctx, CFIE_K_SPECTRAL);
  FFT_LAUNCH((k_fft_cols<T, COL_IN, X, O>), gc, sc, st, C, in, osc, scale, base, out);
  FFT_LAUNCH((k_fft_rows<T, false>), gr, sr, st, R);
  if (!F.direct) {
    FFT_LAUNCH((k_fft_cols<T, COL_MID, X, O>), gc, sc, st, C, in, osc, scale, base, out);
    FFT_LAUNCH((k_fft_rows<T, false>), gr, sr, st, R);
  }
  FFT_LAUNCH((k_fft_cols<T, COL_OUT, X, O>), gc, sc, st, C, in, osc, scale, base, out);
}

}  // namespace

void fft_prepare(cfie_op* op) {
  fft_plan& F = op->fft;
  const int n = op->n;
  F.direct = (n & (n - 1)) == 0;
  int N = 1, L = 0;
  while (N < (F.direct ? n : 2 * n - 1)) {
    N *= 2;
    ++L;
  }
  F.N = N;
  F.L = L;
  const int N2 = 1 << (L - L / 2);
  cudaStream_t st = op->ctx->stream;
  F.tw.reserve(sizeof(double2) * N);
  F.tw32.reserve(sizeof(float2) * N);
  F.tc.reserve(sizeof(double2) * N2);
  F.tc32.reserve(sizeof(float2) * N2);
  F.osc.reserve(sizeof(double) * n);
  k_twiddles<<<nb(N), 256, 0, st>>>(N, N2, F.tw.as<double2>(), F.tw32.as<float2>(),
                                    F.tc.as<double2>(), F.tc32.as<float2>());
  CFIE_CHECK_LAUNCH();
  if (!F.direct) {
    F.chirp.reserve(sizeof(double2) * n);
    F.chirp32.reserve(sizeof(float2) * n);
    F.bf.reserve(sizeof(double2) * N);
    F.bf32.reserve(sizeof(float2) * N);
  }
  // the wrapped chirp, then its spectrum (FP64, in place) and the FP32 copy
  k_chirp<<<nb(N), 256, 0, st>>>(n, N, F.direct, op->g.sp, F.chirp.as<double2>(),
                                 F.chirp32.as<float2>(), F.bf.as<double2>(), F.osc.as<double>());
  CFIE_CHECK_LAUNCH();
  if (F.direct) return;
  fft_args<double2> C = args_of<double2>(F, n, F.bf.as<double2>()), R = C;
  C.lc = per_cta<double2>(C.l1, C.l2, 1, 2);
  R.lc = per_cta<double2>(R.l2, R.l1, 1, 0);
  FFT_LAUNCH((k_fft_cols<double2, COL_RAW, double2, double2>), dim3(1u << (C.l2 - C.lc), 1),
             smem_of<double2>(C.l1, C.lc), st, C, nullptr, nullptr, make_double2(0.0, 0.0), nullptr,
             nullptr);
  FFT_LAUNCH((k_fft_rows<double2, true>), dim3(1u << (R.l1 - R.lc), 1),
             smem_of<double2>(R.l2, R.lc), st, R);
  k_to_f32<<<nb(N), 256, 0, st>>>(N, F.bf.as<double2>(), F.bf32.as<float2>());
  CFIE_CHECK_LAUNCH();
}

void spectral_fft64(cfie_op* op, const double2* in, double2* out, const double2* base,
                    double2 scale, int nrhs) {
  spectral_fft<double2, double2, double2>(op, in, out, base, scale, nrhs);
}

void spectral_fft32_apply(cfie_op* op, const float2* in, float2* out, int nrhs) {
  spectral_fft<float2, float2, float2>(op, in, out, nullptr, make_double2(1.0, 0.0), nrhs);
}

void spectral_fft32_apply(cfie_op* op, const double2* in, float2* out, int nrhs) {
  spectral_fft<float2, double2, float2>(op, in, out, nullptr, make_double2(1.0, 0.0), nrhs);
}

void spectral_fft32_accumulate(cfie_op* op, const float2* in, double2* y, double2 scale,
                               int nrhs) {
  spectral_fft<float2, float2, double2>(op, in, y, y, scale, nrhs);
}
