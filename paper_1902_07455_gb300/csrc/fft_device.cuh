// Batched odd-length complex FFTs of fibres staged in shared memory (FP64 double2 data in fixed point, see fft_fixed.cuh,
// or FP32 float2).
//
// Mixed-radix Stockham autosort, decimation in time.  After the stages with radices p_0..p_{s-1}
// (L = p_0...p_{s-1}), row entry c*L + f holds the length-L DFT (frequency f) of the subsequence
// x[c + (N/L) t], t = 0..L-1.  A radix-p stage with m' = N/(L p) combines p such subsequences:
//   Z'[c'][f + L q] = sum_r w_p^{q r} ( w_{Lp}^{f r} Z[c' + m' r][f] ),   q, r = 0..p-1,
// with w_M = exp(sign 2 pi i / M).  It starts from the natural order (L = 1) and ends in natural
// order (L = N), so no digit reversal is needed.  Inter-pass twiddles come from one table
// W[j] = exp(-2 pi i j / N) (w_{Lp}^{f r} = W[f r m']).  A pass of composite radix p (9, 27) does its
// p-point DFT in registers by Cooley-Tukey splitting p = P Q (index n = n1 + P n2, k = Q k1 + k2):
//   X[Q k1 + k2] = sum_{n1} w_P^{n1 k1} w_p^{n1 k2} sum_{n2} x[n1 + P n2] w_Q^{n2 k2},
// with the roots of unity of each radix in constant memory (compile-time indices, so they are
// operands of the arithmetic instructions); fewer passes through shared memory and far fewer
// instructions per point than radix-3 passes.
#pragma once

#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <mutex>

#include "common.cuh"

namespace lrfg {

constexpr int kMaxGenericRadix = 31;

// roots of unity exp(-2 pi i j / p) of the register radices, concatenated (filled once per device)
constexpr int kRootOff3 = 0, kRootOff5 = 3, kRootOff7 = 8, kRootOff9 = 15, kRootOff27 = 24, kRootCount = 51;
__constant__ float2 c_roots_f[kRootCount];
__constant__ double2 c_roots_d[kRootOff27];  // radices up to 9 (rows of one butterfly)
__constant__ int4 c_roots_x[kRootOff27];  // fixed point (fft_fixed.cuh), radices up to 9

// exp(-2 pi i j / p) in fixed point: cos 2^62 and -sin 2^62 (1 as 1 - 2^-62), each as an upper part times 2^31 and a lower
// one between -2^30 and 2^30 (2^31 - 1 for 1 itself, whose other component is 0): with both signs the lower parts leave
// room for fix_cmul's sums.
static inline int4 fixed_root(int j, int p) {
  const long double ang = 6.283185307179586476925286766559005768L * (long double)j / (long double)p;
  const long long one = (1LL << 62) - 1;
  auto upper = [](long long v) { return std::min(0x7fffffffLL, (v + (1LL << 30)) >> 31); };
  const long long x = std::min(one, (long long)llroundl(cosl(ang) * 0x1p62L)), xh = upper(x);
  const long long y = std::min(one, (long long)llroundl(-sinl(ang) * 0x1p62L)), yh = upper(y);
  return make_int4((int)xh, (int)(x - xh * (1LL << 31)), (int)yh, (int)(y - yh * (1LL << 31)));
}

// Fills this translation unit's root tables on the current device (once per device); returns the CUDA
// status of the copies.
static inline cudaError_t ensure_roots(int device) {
  static std::mutex mu;
  static unsigned long long done = 0;  // one bit per device
  std::lock_guard<std::mutex> lock(mu);
  if (device >= 0 && device < 64 && (done >> device & 1ULL)) return cudaSuccess;
  float2 hf[kRootCount];
  double2 hd[kRootOff27];
  int4 hx[kRootOff27];
  const int radix[5] = {3, 5, 7, 9, 27}, off[5] = {kRootOff3, kRootOff5, kRootOff7, kRootOff9, kRootOff27};
  const double two_pi = 6.283185307179586476925286766559;
  for (int q = 0; q < 5; ++q)
    for (int j = 0; j < radix[q]; ++j) {
      const double ang = two_pi * (double)j / (double)radix[q];
      hf[off[q] + j] = make_float2((float)std::cos(ang), (float)-std::sin(ang));
      if (radix[q] > 9) continue;
      hd[off[q] + j] = make_double2(std::cos(ang), -std::sin(ang));
      hx[off[q] + j] = fixed_root(j, radix[q]);
    }
  cudaError_t e = cudaMemcpyToSymbol(c_roots_f, hf, sizeof(hf));
  if (e == cudaSuccess) e = cudaMemcpyToSymbol(c_roots_d, hd, sizeof(hd));
  if (e == cudaSuccess) e = cudaMemcpyToSymbol(c_roots_x, hx, sizeof(hx));
  // complete before kernels on any stream (non-blocking ones included) read the tables
  if (e == cudaSuccess) e = cudaDeviceSynchronize();
  if (e == cudaSuccess && device >= 0 && device < 64) done |= 1ULL << device;
  return e;
}

// complex vector type of a real type
template <typename R> struct CplxOf;
template <> struct CplxOf<double> { using T = double2; };
template <> struct CplxOf<float> { using T = float2; };
template <typename V> struct RealOf;
template <> struct RealOf<double2> { using T = double; };
template <> struct RealOf<float2> { using T = float; };
// entries of a twiddle table: fixed point for FP64 data
template <typename V> struct TwOf { using T = V; };
template <> struct TwOf<double2> { using T = int4; };

template <typename V>
__device__ __forceinline__ V mkc(typename RealOf<V>::T x, typename RealOf<V>::T y) {
  V v;
  v.x = x;
  v.y = y;
  return v;
}
template <typename V>
__device__ __forceinline__ V cmul(V a, V b) {
  return mkc<V>(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
template <typename V>
__device__ __forceinline__ V cadd(V a, V b) { return mkc<V>(a.x + b.x, a.y + b.y); }
template <typename V>
__device__ __forceinline__ V csub(V a, V b) { return mkc<V>(a.x - b.x, a.y - b.y); }
template <typename V>
__device__ __forceinline__ V cscale(V a, typename RealOf<V>::T s) { return mkc<V>(a.x * s, a.y * s); }
// i * s * a
template <typename V>
__device__ __forceinline__ V cimul(V a, typename RealOf<V>::T s) { return mkc<V>(-a.y * s, a.x * s); }

// twiddle W[j]^(-sign): forward (sign -1) uses W, inverse (sign +1) its conjugate
template <int SIGN, typename V>
__device__ __forceinline__ V tw(const V* W, int j) {
  V w = W[j];
  if (SIGN > 0) w.y = -w.y;
  return w;
}

// One butterfly of a prime radix p > 7: inputs Z[c + m' r][f] (row offset (c + m' r) L + f), outputs Z'[c][f + L q].
template <int SIGN, typename V>
__device__ __forceinline__ void butterfly(int p, const V* __restrict__ in, V* __restrict__ out, int c, int f, int L,
                                          int mp, int N, const V* W) {
  using R = typename RealOf<V>::T;
  // direct length-p DFT with table twiddles, by the symmetric halves of the inputs
  // (see RegDFT<7>): (p - 1)^2 / 4 pairs of real-coefficient products instead of (p - 1)^2 complex ones
  V s[kMaxGenericRadix / 2 + 1], d[kMaxGenericRadix / 2 + 1];
  const int h = (p - 1) / 2;
  const V x0 = in[c * L + f];
  V sum = x0;
  for (int r = 1; r <= h; ++r) {
    V u = in[(c + r * mp) * L + f], v = in[(c + (p - r) * mp) * L + f];
    if (f) {
      u = cmul(u, tw<SIGN>(W, f * r * mp));
      v = cmul(v, tw<SIGN>(W, f * (p - r) * mp));
    }
    s[r] = cadd(u, v);
    d[r] = csub(u, v);
    sum = cadd(sum, s[r]);
  }
  const int step = N / p;
  V* o = out + c * L * p + f;
  o[0] = sum;
  for (int q = 1; q <= h; ++q) {
    V re = x0, im = mkc<V>((R)0, (R)0);
    int j = 0;
    for (int r = 1; r <= h; ++r) {
      j += q;
      if (j >= p) j -= p;
      const V w = tw<SIGN>(W, j * step);
      re = mkc<V>(re.x + w.x * s[r].x, re.y + w.x * s[r].y);
      im = mkc<V>(im.x + w.y * d[r].x, im.y + w.y * d[r].y);
    }
    o[q * L] = mkc<V>(re.x - im.y, re.y + im.x);
    o[(p - q) * L] = mkc<V>(re.x + im.y, re.y - im.x);
  }
}

// Transform `nf` rows of length pl.N (row stride ld) held in `a`, using `b` as scratch.  All threads
// of the block take part; returns the buffer that holds the result (a or b).  Ends with a barrier.
template <int P>
struct RootOff;
template <> struct RootOff<3> { static constexpr int v = kRootOff3; };
template <> struct RootOff<5> { static constexpr int v = kRootOff5; };
template <> struct RootOff<7> { static constexpr int v = kRootOff7; };
template <> struct RootOff<9> { static constexpr int v = kRootOff9; };
template <> struct RootOff<27> { static constexpr int v = kRootOff27; };

// w_P^j (forward: exp(-2 pi i j / P), inverse: its conjugate); j a compile-time constant after unrolling
template <int P, int SIGN, typename V>
__device__ __forceinline__ V root(int j) {
  V w;
  if constexpr (sizeof(V) == sizeof(double2)) w = c_roots_d[RootOff<P>::v + j % P];
  else w = c_roots_f[RootOff<P>::v + j % P];
  if (SIGN > 0) w.y = -w.y;
  return w;
}

template <int P, int SIGN, typename V>
struct RegDFT;

// Multiplications are written as multiply-adds with the additions that follow them (12 operations at p = 3).
template <int SIGN, typename V>
struct RegDFT<3, SIGN, V> {
  static __device__ __forceinline__ void run(V* x) {
    using R = typename RealOf<V>::T;
    const R s = (R)SIGN * (R)0.86602540378443864676;  // sin(2 pi / 3)
    const V t1 = cadd(x[1], x[2]), t2 = csub(x[1], x[2]);
    const R mx = fma(R(-0.5), t1.x, x[0].x), my = fma(R(-0.5), t1.y, x[0].y);
    x[0] = cadd(x[0], t1);
    x[1] = mkc<V>(fma(-s, t2.y, mx), fma(s, t2.x, my));
    x[2] = mkc<V>(fma(s, t2.y, mx), fma(-s, t2.x, my));
  }
};

template <int SIGN, typename V>
struct RegDFT<5, SIGN, V> {
  static __device__ __forceinline__ void run(V* x) {
    using R = typename RealOf<V>::T;
    const R c1 = (R)0.30901699437494742410, c2 = (R)-0.80901699437494742410;
    const R s1 = (R)0.95105651629515357212, s2 = (R)0.58778525229247312917;
    const V a1 = cadd(x[1], x[4]), b1 = csub(x[1], x[4]), a2 = cadd(x[2], x[3]), b2 = csub(x[2], x[3]);
    const V m1 = mkc<V>(fma(c2, a2.x, fma(c1, a1.x, x[0].x)), fma(c2, a2.y, fma(c1, a1.y, x[0].y)));
    const V m2 = mkc<V>(fma(c1, a2.x, fma(c2, a1.x, x[0].x)), fma(c1, a2.y, fma(c2, a1.y, x[0].y)));
    const R sa = (R)SIGN * s1, sb = (R)SIGN * s2;
    const V n1 = mkc<V>(fma(sb, b2.x, sa * b1.x), fma(sb, b2.y, sa * b1.y));
    const V n2 = mkc<V>(fma(-sa, b2.x, sb * b1.x), fma(-sa, b2.y, sb * b1.y));
    x[0] = cadd(x[0], cadd(a1, a2));
    x[1] = mkc<V>(m1.x - n1.y, m1.y + n1.x);
    x[2] = mkc<V>(m2.x - n2.y, m2.y + n2.x);
    x[3] = mkc<V>(m2.x + n2.y, m2.y - n2.x);
    x[4] = mkc<V>(m1.x + n1.y, m1.y - n1.x);
  }
};

// Prime radix by the symmetric halves of the inputs, s_r = x_r + x_{p-r} and d_r = x_r - x_{p-r}:
//   X_q, X_{p-q} = x_0 + sum_r cos(2 pi q r / p) s_r  +-  i SIGN sum_r sin(2 pi q r / p) d_r,  r, q = 1..(p-1)/2,
// real coefficients only: 36 multiply-adds and 24 additions at p = 7, against 36 complex products and as many complex
// additions (216 operations) of the direct sum.
template <int SIGN, typename V>
struct RegDFT<7, SIGN, V> {
  static __device__ __forceinline__ void run(V* x) {
    V s[4], d[4];
    const V x0 = x[0];
#pragma unroll
    for (int r = 1; r < 4; ++r) {
      s[r] = cadd(x[r], x[7 - r]);
      d[r] = csub(x[r], x[7 - r]);
    }
    x[0] = cadd(cadd(x0, s[1]), cadd(s[2], s[3]));
#pragma unroll
    for (int q = 1; q < 4; ++q) {
      V re = x0, im = mkc<V>(0, 0);
#pragma unroll
      for (int r = 1; r < 4; ++r) {
        const V w = root<7, SIGN, V>(q * r);
        re = mkc<V>(re.x + w.x * s[r].x, re.y + w.x * s[r].y);
        im = r == 1 ? mkc<V>(w.y * d[r].x, w.y * d[r].y) : mkc<V>(im.x + w.y * d[r].x, im.y + w.y * d[r].y);
      }
      x[q] = mkc<V>(re.x - im.y, re.y + im.x);
      x[7 - q] = mkc<V>(re.x + im.y, re.y - im.x);
    }
  }
};

// p = P Q in registers (see the header comment)
template <int P, int Q, int SIGN, typename V>
__device__ __forceinline__ void reg_dft_split(V* x) {
  constexpr int p = P * Q;
  V y[P][Q];
#pragma unroll
  for (int n1 = 0; n1 < P; ++n1) {
    V t[Q];
#pragma unroll
    for (int n2 = 0; n2 < Q; ++n2) t[n2] = x[n1 + P * n2];
    RegDFT<Q, SIGN, V>::run(t);
#pragma unroll
    for (int k2 = 0; k2 < Q; ++k2) y[n1][k2] = (n1 && k2) ? cmul(t[k2], root<p, SIGN, V>(n1 * k2)) : t[k2];
  }
#pragma unroll
  for (int k2 = 0; k2 < Q; ++k2) {
    V t[P];
#pragma unroll
    for (int n1 = 0; n1 < P; ++n1) t[n1] = y[n1][k2];
    RegDFT<P, SIGN, V>::run(t);
#pragma unroll
    for (int k1 = 0; k1 < P; ++k1) x[Q * k1 + k2] = t[k1];
  }
}

template <int SIGN, typename V>
struct RegDFT<9, SIGN, V> {
  static __device__ __forceinline__ void run(V* x) { reg_dft_split<3, 3, SIGN, V>(x); }
};
template <int SIGN, typename V>
struct RegDFT<27, SIGN, V> {
  static __device__ __forceinline__ void run(V* x) { reg_dft_split<3, 9, SIGN, V>(x); }
};

// x / d for 0 <= x < 2^22 and 1 <= d < 2^22 from a float reciprocal, corrected to the exact quotient
// (cheaper than the integer division sequence in the per-butterfly index arithmetic)
__device__ __forceinline__ int small_div(int x, int d, float inv) {
  int q = __float2int_rz((float)x * inv);
  const int r = x - q * d;
  if (r < 0) --q;
  else if (r >= d) ++q;
  return q;
}

}  // namespace lrfg

#include "fft_fixed.cuh"

namespace lrfg {

// One Stockham pass of register radix P over nf rows (row stride ld) from a into b.
template <int P, int SIGN, typename V>
__device__ __forceinline__ void stockham_pass(const V* __restrict__ a, V* __restrict__ b, int nf, int ld, int N,
                                              int L, const V* W) {
  const int mp = N / (L * P);
  const int nb = N / P;
  const int total = nb * nf;
  const float inv_nb = 1.0f / (float)nb, inv_L = 1.0f / (float)L;
  for (int t = threadIdx.x; t < total; t += blockDim.x) {
    const int row = small_div(t, nb, inv_nb);
    const int bt = t - row * nb;
    const int c = small_div(bt, L, inv_L);
    const int f = bt - c * L;
    const V* in = a + row * ld + c * L + f;
    V* out = b + row * ld + c * L * P + f;
    V x[P];
#pragma unroll
    for (int r = 0; r < P; ++r) x[r] = in[r * mp * L];
    if (f) {
#pragma unroll
      for (int r = 1; r < P; ++r) x[r] = cmul(x[r], tw<SIGN>(W, f * r * mp));
    }
    RegDFT<P, SIGN, V>::run(x);
#pragma unroll
    for (int q = 0; q < P; ++q) out[q * L] = x[q];
  }
}

// Transform `nf` rows of length pl.N (row stride ld) held in `a`, using `b` as scratch.  All threads
// of the block take part; returns the buffer that holds the result (a or b).  Ends with a barrier.
// (FP64 data: fft_fixed.cuh)
template <int SIGN, typename V>
__device__ V* stockham_rows(V* a, V* b, int nf, int ld, const FftPlan& pl, const typename TwOf<V>::T* W) {
  if constexpr (sizeof(V) == sizeof(double2)) {
    return fix_rows<SIGN>(a, b, nf, ld, pl, W);
  } else {
  const int N = pl.N;
  int L = 1;
  for (int s = 0; s < pl.nst; ++s) {
    const int p = pl.radix[s];
    switch (p) {
      case 3: stockham_pass<3, SIGN>(a, b, nf, ld, N, L, W); break;
      case 5: stockham_pass<5, SIGN>(a, b, nf, ld, N, L, W); break;
      case 7: stockham_pass<7, SIGN>(a, b, nf, ld, N, L, W); break;
      case 9: stockham_pass<9, SIGN>(a, b, nf, ld, N, L, W); break;
      case 27: stockham_pass<27, SIGN>(a, b, nf, ld, N, L, W); break;
      default: {
        const int mp = N / (L * p);
        const int nb = N / p;
        const int total = nb * nf;
        const float inv_nb = 1.0f / (float)nb, inv_L = 1.0f / (float)L;
        for (int t = threadIdx.x; t < total; t += blockDim.x) {
          const int row = small_div(t, nb, inv_nb);
          const int bt = t - row * nb;
          const int c = small_div(bt, L, inv_L);
          const int f = bt - c * L;
          butterfly<SIGN>(p, a + row * ld, b + row * ld, c, f, L, mp, N, W);
        }
      }
    }
    __syncthreads();
    V* tmp = a;
    a = b;
    b = tmp;
    L *= p;
  }
  return a;
  }
}

// Asynchronous global -> shared copies (cp.async, no register staging), so that a block keeps all of its
// tile's loads in flight at once; sizes 4, 8 or 16 bytes, both addresses aligned to the size.
template <int BYTES>
__device__ __forceinline__ void cp_async(void* smem, const void* gmem) {
  const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
  if (BYTES == 16) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(s), "l"(gmem) : "memory");
  } else {
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2;\n" ::"r"(s), "l"(gmem), "n"(BYTES) : "memory");
  }
}
__device__ __forceinline__ void cp_async_wait_all() {
  asm volatile("cp.async.commit_group;\n" ::: "memory");
  asm volatile("cp.async.wait_group 0;\n" ::: "memory");
}

// frequency k in Z_N of storage index n
__device__ __forceinline__ int freq_of(int n, int N) { return n <= (N - 1) / 2 ? n : n - N; }

}  // namespace lrfg
