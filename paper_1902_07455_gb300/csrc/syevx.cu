// FP64 symmetric eigensolver for the k largest eigenpairs (k = n: all of them) of a batch of matrices:
//  1. Householder tridiagonalisation  Q^T A Q = T  (Golub & Van Loan, "Matrix Computations", 4th ed.,
//     Alg. 8.3.1), reflectors kept in the columns below the diagonal;
//  2. eigenvalues of T by bisection on Sturm counts of the LDL^T recurrence (G&VL Sec. 8.4.1), one warp per
//     eigenvalue in a launch of its own;
//  3. eigenvectors of T by inverse iteration (G&VL Sec. 8.2.2) with the tridiagonal LU factorisation
//     of T - lambda I with partial pivoting (G&VL Sec. 4.3), two passes or three, and an orthonormalisation of the vectors
//     (Newton-Schulz, Cholesky of their Gram matrix, or modified Gram-Schmidt, by how far they are from orthogonal);
//  4. back-transformation by Q = H_0 .. H_{n-3}, formed beside step 2, or by the stored reflectors.
// About 4/3 n^3 + 2 k n^2 flops against ~9 n^3 per sweep (and several sweeps) for cyclic Jacobi, with the
// same absolute accuracy (eps ||A||), which is what the Gram-SVD truncation needs.
// The steps are chains of dependent FP64 operations, and on this part a warp issues one FP64 instruction per 64 cycles
// whatever its instruction-level parallelism or active lanes (an SM has four such units): each kernel is laid out to put
// few FP64 instructions on the longest of the four.  Three matrices of n = 30, k = 20 take 155 us (420 us with the same
// algorithm laid out by arithmetic alone), one of n = 60, k = 20 402 us (744), n = 135, k = 10 1.45 ms (2.3).
#include <algorithm>
#include <cfloat>
#include <cmath>

#include "ops.cuh"
#include "recip.cuh"

namespace lrfg {

constexpr int kSyevxThreads = 512;

__device__ __forceinline__ double warp_sum(double v) {
  for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffff, v, o);
  return v;
}

// Block sum: warp partials, then warp 0 alone combines them (FP64 issue slots are scarce: 2 lanes/clk/SM)
// Sum over the block of v, where only threads < nact can hold nonzero values: only their warps shuffle
// (every FP64 add of an idle warp would still cost the SM's FP64 pipe 16 cycles).  Result in red[32].
__device__ double block_reduce_sum(double v, double* red, int nact) {
  const int nwa = min((int)(blockDim.x >> 5), (nact + 31) >> 5);
  const int warp = threadIdx.x >> 5;
  if (warp < nwa) v = warp_sum(v);
  __syncthreads();
  if ((threadIdx.x & 31) == 0 && warp < nwa) red[warp] = v;
  __syncthreads();
  if (threadIdx.x < 32) {
    double s = ((int)threadIdx.x < nwa) ? red[threadIdx.x] : 0.0;
    if (nwa > 1) s = warp_sum(s);
    if (threadIdx.x == 0) red[32] = s;
  }
  __syncthreads();
  return red[32];
}

// Number of eigenvalues of the symmetric tridiagonal (d, e) below x: sign changes of the Sturm sequence
// p_0 = 1, p_1 = d_0 - x, p_{i+1} = (d_i - x) p_i - e_{i-1}^2 p_{i-1} (Barth, Martin & Wilkinson, Numer. Math.
// 9 (1967) 386-393), a zero term taking the sign opposite to its predecessor.  Division-free (FP64
// division is a long dependent chain on this part); the pair (p_{i-1}, p_i) is rescaled by exact powers of
// two every four steps to stay in range.  The caller scales T by a power of two to |T| < 1, so that four
// steps change |p| by at most a factor 3^4 (growth) or 2^-212 (cancellation) within the 2^(+-600) window.
// (the sign enters as a bit: 1 negative)
__device__ __forceinline__ unsigned sign_bit(double p, unsigned prev) {
  const unsigned hi = (unsigned)__double2hiint(p);
  return ((hi & 0x7fffffffu) | (unsigned)__double2loint(p)) == 0u ? prev ^ 1u : hi >> 31;
}

// Steps in groups of four: the coefficients first, then the recurrence, then the signs, so that the integer work on a
// result does not hold up the next FP64 instruction (a warp issues one FP64 instruction per 64 cycles on this part, and
// in order).
__device__ int sturm_count(const double* d, const double* e2, int n, double x) {
  const double up = 0x1p+600, down = 0x1p-600;
  double pm = 1.0, p = d[0] - x;
  unsigned sg = sign_bit(p, 0u);
  int c = (int)sg;
  for (int i = 1; i < n; i += 4) {
    double dv[4], ev[4], q[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int k = min(i + u, n - 1);
      dv[u] = d[k];
      ev[u] = e2[k - 1];
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const double pn = fma(dv[u] - x, p, -ev[u] * pm);
      pm = p;
      p = pn;
      q[u] = pn;
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const unsigned s = sign_bit(q[u], sg);
      if (i + u < n) {  // past the end the last step is repeated and not counted
        c += (int)(s ^ sg);
        sg = s;
      }
    }
    const int e = max((__double2hiint(p) >> 20) & 0x7ff, (__double2hiint(pm) >> 20) & 0x7ff);
    if (e > 1023 + 600 || e < 1023 - 600) {
      const double f = e > 1023 ? down : up;
      p *= f;
      pm *= f;
    }
  }
  return c;
}

// The same count in FP32 (rescaling by 2^(+-60) every step pair), used only to localise eigenvalues before the FP64
// multisection; its brackets are verified with FP64 counts.
__device__ int sturm_count_f32(const float* d, const float* e2, int n, float x) {
  const float up = 0x1p+60f, down = 0x1p-60f;
  float pm = 1.0f, p = d[0] - x;
  unsigned sg = (__float_as_uint(p) << 1) == 0u ? 1u : __float_as_uint(p) >> 31;
  int c = (int)sg;
  for (int i = 1; i < n; i += 2) {
    const int k1 = min(i + 1, n - 1);
    const float d0 = d[i] - x, d1 = d[k1] - x, e0 = -e2[i - 1], e1 = -e2[k1 - 1];
    const float q0 = fmaf(d0, p, e0 * pm), q1 = fmaf(d1, q0, e1 * p);
    unsigned s = (__float_as_uint(q0) << 1) == 0u ? sg ^ 1u : __float_as_uint(q0) >> 31;
    c += (int)(s ^ sg);
    sg = s;
    if (i + 1 < n) {
      s = (__float_as_uint(q1) << 1) == 0u ? sg ^ 1u : __float_as_uint(q1) >> 31;
      c += (int)(s ^ sg);
      sg = s;
    }
    pm = q0;
    p = q1;
    const int e = max((__float_as_int(p) >> 23) & 0xff, (__float_as_int(pm) >> 23) & 0xff);
    if (e > 127 + 60 || e < 127 - 60) {
      const float f = e > 127 ? down : up;
      p *= f;
      pm *= f;
    }
  }
  return c;
}

// LU with partial pivoting of the tridiagonal T - lam I (sub = super = e, diag d - lam).  Factors in
// dl (multipliers), dd (reciprocals of the diagonal of U), du (1st super), du2 (2nd super), piv (1 = rows
// i, i+1 swapped).  The active row is carried in registers, and both outcomes of a pivot share one reciprocal, so that
// lanes on different eigenvalues do not diverge.
__device__ __forceinline__ long long abs_bits(double x) { return __double_as_longlong(x) & 0x7fffffffffffffffLL; }

__device__ void trid_factor(const double* __restrict__ d, const double* __restrict__ e, int n, double lam, double tiny,
                            double* __restrict__ dl, double* __restrict__ dd, double* __restrict__ du,
                            double* __restrict__ du2, int* __restrict__ piv) {
  double cd = d[0] - lam, cu = n > 1 ? e[0] : 0.0, ei = cu;
  for (int i = 0; i < n - 1; ++i) {
    const double dn = d[i + 1] - lam, un = i < n - 2 ? e[i + 1] : 0.0;
    const bool sw = abs_bits(cd) < abs_bits(ei);
    if (abs_bits(cd) == 0 && !sw) cd = tiny;
    const double r = recip(sw ? ei : cd);
    const double top = sw ? dn : cu;
    const double f = (sw ? cd : ei) * r;
    dl[i] = f;
    dd[i] = r;
    du[i] = top;
    du2[i] = sw ? un : 0.0;
    piv[i] = sw ? 1 : 0;
    cd = fma(-f, top, sw ? cu : dn);
    cu = sw ? -f * un : un;
    ei = un;
  }
  if (abs_bits(cd) == 0) cd = tiny;
  dd[n - 1] = recip(cd);
}

__device__ void trid_solve(int n, const double* __restrict__ dl, const double* __restrict__ dd,
                           const double* __restrict__ du, const double* __restrict__ du2, const int* __restrict__ piv,
                           double* __restrict__ b) {
  double x = b[0];
  for (int i0 = 0; i0 < n - 1; i0 += 4) {
    double y[4], f[4], top[4];
    int sw[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int i = min(i0 + u, n - 2);
      y[u] = b[i + 1];
      f[u] = dl[i];
      sw[u] = piv[i];
    }
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (i0 + u < n - 1) {
        top[u] = sw[u] ? y[u] : x;
        x = fma(-f[u], top[u], sw[u] ? x : y[u]);
      }
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (i0 + u < n - 1) b[i0 + u] = top[u];
  }
  // back substitution, rescaling the computed tail when a term would overflow (the direction is what
  // inverse iteration needs); the test reads the exponent, off the FP64 pipe
  double y1 = x * dd[n - 1], y2 = 0.0;
  b[n - 1] = y1;
  for (int i0 = n - 2; i0 >= 0; i0 -= 4) {
    double v[4], p1[4], p2[4], r[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int i = max(i0 - u, 0);
      v[u] = b[i];
      p1[u] = du[i];
      p2[u] = du2[i];
      r[u] = dd[i];
    }
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (i0 - u >= 0) {
        double y = fma(-p1[u], y1, fma(-p2[u], y2, v[u])) * r[u];
        if (((__double2hiint(y) >> 20) & 0x7ff) > 1023 + 498) {
          for (int l = i0 - u + 1; l < n; ++l) b[l] *= 0x1p-498;
          y *= 0x1p-498;
          y1 *= 0x1p-498;
        }
        b[i0 - u] = y;
        y2 = y1;
        y1 = y;
      }
  }
}

// Gram matrix of the k vectors of Y (vector t at Y + t yst): G[t][s], s <= t, row stride k | 1.  Returns (to every
// thread) the largest |cosine| between two of them, or a value above 2 when a vector is zero or not finite; the vectors
// are then scaled to unit length (G with them).
__device__ float gram_and_normalise(double* Y, int yst, int n, int k, double* G) {
  __shared__ int s_cos;
  const int tid = threadIdx.x, nthr = blockDim.x;
  const int gst = k | 1;
  double* rs = G + (size_t)k * gst;  // k: reciprocal lengths
  if (tid == 0) s_cos = 0;
  const int np = k * (k + 1) / 2;
  auto pair = [&](int q, int& t, int& u) {
    t = (int)((sqrtf(8.0f * (float)q + 1.0f) - 1.0f) * 0.5f);
    while (t * (t + 1) / 2 > q) --t;
    while ((t + 1) * (t + 2) / 2 <= q) ++t;
    u = q - t * (t + 1) / 2;
  };
  for (int q = tid; q < np; q += nthr) {
    int t, u;
    pair(q, t, u);
    const double* a = Y + (size_t)t * yst;
    const double* b = Y + (size_t)u * yst;
    double s0 = 0.0, s1 = 0.0;
    int i = 0;
    for (; i + 1 < n; i += 2) {
      s0 = fma(a[i], b[i], s0);
      s1 = fma(a[i + 1], b[i + 1], s1);
    }
    if (i < n) s0 = fma(a[i], b[i], s0);
    G[t * gst + u] = s0 + s1;
  }
  __syncthreads();
  for (int t = tid; t < k; t += nthr) {
    const double d = G[t * gst + t];
    const bool ok = d > 0.0 && isfinite(d);
    rs[t] = ok ? recip_sqrt(d) : 0.0;
    if (!ok) s_cos = __float_as_int(3.0f);
  }
  __syncthreads();
  const bool bad = s_cos != 0;
  __syncthreads();
  if (bad) return 3.0f;
  for (int q = tid; q < np; q += nthr) {
    int t, u;
    pair(q, t, u);
    const double v = G[t * gst + u] * (rs[t] * rs[u]);
    G[t * gst + u] = v;
    if (t != u) atomicMax(&s_cos, __float_as_int(fabsf((float)v)));
  }
  for (int q = tid; q < k * n; q += nthr) {
    const int t = q / n, i = q - t * n;
    Y[(size_t)t * yst + i] *= rs[t];
  }
  __syncthreads();
  return __int_as_float(s_cos);
}

// Orthonormalises the k unit vectors of Y in order by the Cholesky factor of their Gram matrix G (as left by
// gram_and_normalise): G = L D L^T, Y <- D^-1/2 L^-1 Y, the vectors Gram-Schmidt gives, with the products spread over the
// block.  After an inverse iteration the vectors are nearly orthogonal unless eigenvalues agree to rounding, so L is close
// to the unit matrix; where a pivot falls below 1/100 the result is left to modified Gram-Schmidt (returns false, Y
// unchanged).  All threads of the block call it.
__device__ bool chol_orth(double* Y, int yst, int n, int k, double* G) {
  const int tid = threadIdx.x, nthr = blockDim.x;
  const int gst = k | 1;
  double* rs = G + (size_t)k * gst;
  // right-looking, a thread per entry below the pivot; column j keeps its unscaled entries, rs the reciprocal pivots
  for (int j = 0; j < k; ++j) {
    const double d = G[j * gst + j];
    if (!(d > 0.01)) return false;  // the same value in every thread
    const double r = recip(d);
    const int m = k - j - 1;
    for (int q = tid; q < m * m; q += nthr) {
      const int a = q / m, b = q - a * m;
      if (b <= a) {
        const int i = j + 1 + a, l = j + 1 + b;
        G[i * gst + l] = fma(-(G[i * gst + j] * r), G[l * gst + j], G[i * gst + l]);
      }
    }
    if (tid == 0) rs[j] = r;
    __syncthreads();
  }
  // Y <- L^-1 Y, eight lanes per column of Y: once row s is final its multiples leave the rows below
  const int part = tid & 7;
  for (int i0 = 0; i0 < n; i0 += nthr >> 3) {
    const int i = i0 + (tid >> 3);
    if (i0 + ((tid & ~31) >> 3) >= n) continue;  // whole warp past the columns
    const bool in = i < n;
    for (int s = 0; s < k; ++s) {
      const double ys = in ? Y[(size_t)s * yst + i] * rs[s] : 0.0;
      if (in)
        for (int t = s + 1 + part; t < k; t += 8) {
          double* y = Y + (size_t)t * yst + i;
          *y = fma(-G[t * gst + s], ys, *y);
        }
      __syncwarp();
    }
  }
  __syncthreads();
  for (int t = tid; t < k; t += nthr) rs[t] = recip_sqrt(G[t * gst + t]);
  __syncthreads();
  for (int q = tid; q < k * n; q += nthr) {
    const int t = q / n, i = q - t * n;
    Y[(size_t)t * yst + i] *= rs[t];
  }
  __syncthreads();
  return true;
}

// Power of two that brings the largest entry (bits of its upper word, over the block) near 1, so that the squares and
// products of the reduction stay in range whatever the scale of the matrix.  red: 32 ints.  All threads call it.
__device__ double range_scale(int hi_abs, int* red) {
  const int m = __reduce_max_sync(0xffffffff, hi_abs);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
  __syncthreads();
  int b = 0;
  for (int q = 0; q < (int)(blockDim.x >> 5); ++q) b = max(b, red[q]);
  const int ex = b >> 20;
  if (ex == 0) return 1.0;  // zero or denormal
  if (ex == 0x7ff) return __longlong_as_double(0x7ff8000000000000LL);  // not finite: so are all results (see K2, K3)
  return __hiloint2double(min(2046, max(1, 2046 - ex)) << 20, 0);
}

// Gershgorin interval of the tridiagonal (d, e) and the largest e_i^2, by warp 0 (lanes over the rows), left in
// red[35] (lower end), red[36] (upper end), red[37].  All threads of the block call it.
__device__ void trid_gershgorin(const double* d, const double* e, int n, double* red) {
  const int tid = threadIdx.x;
  if (tid < 32) {
    double l0 = INFINITY, h0 = -INFINITY, em = 0.0;
    for (int i = tid; i < n; i += 32) {
      const double r = (i > 0 ? fabs(e[i - 1]) : 0.0) + (i < n - 1 ? fabs(e[i]) : 0.0);
      l0 = fmin(l0, d[i] - r);
      h0 = fmax(h0, d[i] + r);
      if (i < n - 1) em = fmax(em, e[i] * e[i]);
    }
    for (int o = 16; o; o >>= 1) {
      l0 = fmin(l0, __shfl_xor_sync(0xffffffff, l0, o));
      h0 = fmax(h0, __shfl_xor_sync(0xffffffff, h0, o));
      em = fmax(em, __shfl_xor_sync(0xffffffff, em, o));
    }
    if (tid == 0) {
      red[35] = l0;
      red[36] = h0;
      red[37] = em;
    }
  }
  __syncthreads();
}

// ---- the decomposition in three launches -----------------------------------------------------------------
// K1 (one block per matrix) tridiagonalises and bounds the spectrum; K2 (one warp per wanted eigenvalue, all
// matrices) bisects; K3 (one block per matrix) runs inverse iteration, re-orthogonalises within clusters,
// back-transforms and writes the outputs.  The bisection is a chain of dependent FP64 Sturm recurrences per
// point; inside one block the k eigenvalues shared one SM's FP64 pipe (2 FMA/clk), one warp each they get one
// SM each, so every lane can take its own point (33-way multisection, about 5 bits per count instead of 2).
// Per-item global scratch (doubles): a header (active size, Gershgorin interval, largest e_i^2 and the factor back from
// the range the matrix was scaled to), d, e, beta, lam (nl each), the reflectors W (n x n, leading dimension n), the vectors Y
// (kl x nl, vector-major) and the inverse-iteration LU factors (kl x 5 nl).
constexpr int kHdr = 8;
constexpr double kTailFloor = 1e-280;  // squared length of a column tail that counts as zero (entries scaled to 1)
constexpr int kSmallEig = 96;  // sizes whose matrix fits the register kernels

__host__ __device__ inline size_t syevx_scratch_per(int nl, int kl) {
  return kHdr + 4 * (size_t)nl + (nl <= kSmallEig ? 2 : 1) * (size_t)nl * nl + (size_t)kl * nl + (size_t)kl * 5 * nl;
}

struct SyevxScratch {
  double *hdr, *d, *e, *beta, *lam, *W, *Y, *lu, *Q;
};

__device__ __forceinline__ SyevxScratch syevx_scratch(double* scratch, int nl, int kl, int item) {
  SyevxScratch g;
  g.hdr = scratch + item * syevx_scratch_per(nl, kl);
  g.d = g.hdr + kHdr;
  g.e = g.d + nl;
  g.beta = g.e + nl;
  g.lam = g.beta + nl;
  g.W = g.lam + nl;
  g.Y = g.W + (size_t)nl * nl;
  g.lu = g.Y + (size_t)kl * nl;
  g.Q = g.lu + (size_t)kl * 5 * nl;
  return g;
}

// K1 above n = 96 (n = 135: 1.60 -> 1.03 ms with the product dealt to all warps, one triangle and two multiply-adds an entry).
// nl, kl: the launch sizes (strides of the inputs and outputs).  nAg (optional): the active size of each item, the
// leading block of its matrix; the rest is zero.
__global__ void __launch_bounds__(kSyevxThreads) syevx_tri_kernel(const double* __restrict__ Ag, int nl, int kl,
                                                                  double* wg, double* Vg, int ldv, double* scratch,
                                                                  int use_smem, const int* __restrict__ nAg,
                                                                  double* work) {
  extern __shared__ __align__(16) double sm[];
  double* red = sm;            // 33 (32 partials + the result) + padding
  double* pv = red + 40;       // nl: p / w of the current reflector
  double* vv = pv + nl;        // nl: current reflector v
  double* ps = vv + nl;        // kSyevxThreads: parts of the product A22 v
  const size_t nnl = (size_t)nl * nl;
  const SyevxScratch g = syevx_scratch(scratch, nl, kl, blockIdx.x);
  double *d = g.d, *e = g.e, *beta = g.beta;  // written once per step by thread 0
  double* W = use_smem ? (ps + kSyevxThreads) : g.W;
  const int tid = threadIdx.x, nthr = blockDim.x;
  double* wout = wg + (size_t)blockIdx.x * nl;
  double* Vout = Vg + (size_t)blockIdx.x * (size_t)nl * ldv;
  // the active size: n x n, k vectors
  const int n = nAg ? max(0, min(nl, nAg[blockIdx.x])) : nl;
  const int k = min(kl, n);
  const double* A = Ag + (size_t)blockIdx.x * nnl;
  if (tid == 0) {
    add_work(work, 4.0 / 3.0 * n * (double)n * n + 4.0 * (double)k * n * n + 60.0 * k * n,
             sizeof(double) * (2.0 * n * n + (double)k * n));
    g.hdr[0] = (double)n;
  }
  for (int t = tid; t < kl; t += nthr) wout[t] = 0.0;
  for (size_t q = tid; q < (size_t)nl * kl; q += nthr) {
    const int i = (int)(q / kl), t = (int)(q - (q / kl) * kl);
    Vout[(size_t)i * ldv + t] = 0.0;
  }
  if (n == 0) return;
  // in shared memory rows have an odd stride and only the lower triangle is kept up to date
  const int ldw = use_smem ? (n | 1) : n;
  int top = 0;
  for (size_t t = tid; t < (size_t)n * n; t += nthr) {
    const size_t i = t / n, j = t - i * n;
    const double v = A[i * nl + j];
    W[i * ldw + j] = v;
    top = max(top, __double2hiint(v) & 0x7fffffff);
  }
  const double scale = range_scale(top, (int*)red);
  for (size_t t = tid; t < (size_t)n * n; t += nthr) W[t / n * ldw + t % n] *= scale;
  __syncthreads();

  // 1. tridiagonalisation
  for (int j = 0; j + 2 < n; ++j) {
    const int m = n - j - 1;
    double x0 = W[(size_t)(j + 1) * ldw + j];
    double loc = 0.0;
    for (int i = tid; i < m; i += nthr) {
      double xi = W[(size_t)(j + 1 + i) * ldw + j];
      vv[i] = xi;
      if (i > 0) loc += xi * xi;
    }
    const double tail2 = block_reduce_sum(loc, red, m);
    if (!(tail2 > kTailFloor)) {
      if (tid == 0) {
        d[j] = W[(size_t)j * ldw + j];
        e[j] = x0;
        beta[j] = 0.0;
      }
      __syncthreads();
      continue;
    }
    // the reflector's scalars once (a square root and a division are long FP64 sequences: computed by
    // every thread they would occupy the FP64 pipe for thousands of cycles)
    if (tid == 0) {
      const double s = fma(x0, x0, tail2), nrm = s * recip_sqrt(s);
      const double alpha = -copysign(nrm, x0);
      const double v0 = x0 - alpha;
      const double bb = recip(fma(fabs(x0), nrm, s));  // 2 / (v^T v)
      vv[0] = v0;
      d[j] = W[(size_t)j * ldw + j];
      e[j] = alpha;
      beta[j] = bb;
      red[34] = bb;
    }
    __syncthreads();
    const double b = red[34];
    // keep v in column j below the diagonal for the back-transformation
    for (int i = tid; i < m; i += nthr) W[(size_t)(j + 1 + i) * ldw + j] = vv[i];
    // p = b A22 v, a row per lane; the columns of a row are dealt to all warps (a warp issues one FP64 instruction per 64
    // cycles: the rows alone kept five warps busy at n = 135)
    const int warp = tid >> 5, lane = tid & 31, nw = nthr >> 5;
    const int rw = (m + 31) >> 5, parts = max(1, nw / rw), chunk = (m + parts - 1) / parts;
    for (int q = warp; q < rw * parts; q += nw) {
      const int part = q / rw, i = (q - part * rw) * 32 + lane, l1 = min(m, (part + 1) * chunk);
      if (i >= m) continue;
      const double* row = W + (size_t)(j + 1 + i) * ldw + (j + 1);  // entries l <= i
      const double* col = W + (size_t)(j + 1) * ldw + (j + 1 + i);  // the others, or all (neighbouring threads, neighbouring words)
      const int mine = use_smem ? i : -1;
      double s0 = 0.0, s1 = 0.0;
      int l = part * chunk;
      for (; l + 1 < l1; l += 2) {
        s0 = fma(l <= mine ? row[l] : col[(size_t)l * ldw], vv[l], s0);
        s1 = fma(l + 1 <= mine ? row[l + 1] : col[(size_t)(l + 1) * ldw], vv[l + 1], s1);
      }
      if (l < l1) s0 = fma(l <= mine ? row[l] : col[(size_t)l * ldw], vv[l], s0);
      (parts > 1 ? ps + part * rw * 32 : pv)[i] = parts > 1 ? s0 + s1 : b * (s0 + s1);
    }
    __syncthreads();
    double kl = 0.0;
    for (int i = tid; i < m; i += nthr) {
      if (parts > 1) {
        double p = ps[i];
        for (int q = 1; q < parts; ++q) p += ps[q * rw * 32 + i];
        pv[i] = b * p;
      }
      kl += vv[i] * pv[i];
    }
    const double K = 0.5 * b * block_reduce_sum(kl, red, m);
    for (int i = tid; i < m; i += nthr) pv[i] -= K * vv[i];
    __syncthreads();
    // A22 -= v w^T + w v^T (one warp per row)
    for (int i = warp; i < m; i += nw) {
      double* row = W + (size_t)(j + 1 + i) * ldw + (j + 1);
      const double vi = vv[i], wi = pv[i];
      const int end = use_smem ? i + 1 : m;
      for (int l = lane; l < end; l += 32) row[l] = fma(-vi, pv[l], fma(-wi, vv[l], row[l]));
    }
    __syncthreads();
  }
  if (tid == 0) {
    if (n >= 2) {
      d[n - 2] = W[(size_t)(n - 2) * ldw + (n - 2)];
      e[n - 2] = W[(size_t)(n - 1) * ldw + (n - 2)];
      if (n >= 3) beta[n - 2] = 0.0;
    }
    d[n - 1] = W[(size_t)(n - 1) * ldw + (n - 1)];
    e[n - 1] = 0.0;
    beta[n - 1] = 0.0;
  }
  __syncthreads();

  trid_gershgorin(d, e, n, red);
  if (tid == 0) {
    g.hdr[1] = red[35];
    g.hdr[2] = red[36];
    g.hdr[3] = red[37];
    g.hdr[4] = 1.0 / scale;
  }
  if (use_smem)
    for (size_t t = tid; t < (size_t)n * n; t += nthr) g.W[t] = W[t / n * ldw + t % n];
}

// K1 for n <= 32 NR: the matrix in registers, row = lane (NR rows a lane), columns dealt to TW worker warps.  A warp issues
// one FP64 instruction per 64 cycles on this part whatever its lanes or its other instructions do, and an SM has four
// such units, so a step takes as long as the unit with the most FP64 instructions on its path:
//  * warp 0 forms the reflector's scalars from the norm of x while the workers multiply: with v = x + s ||x|| e_1 the
//    product A v = A x + s ||x|| a_1 needs no finished v, and v^T A v follows from x^T A x, (A x)_1 and a_11;
//  * three workers, one per remaining unit (four at n > 32, where their share outweighs warp 0's; six halves of the
//    registers at n > 64); operands are loaded four columns ahead of the arithmetic they feed;
//  * the two columns the next step reads are updated and published first, the rest after the barrier;
//  * one square root and one reciprocal a step (recip_sqrt, recip), two barriers.
template <int NR, int TW>
__global__ void __launch_bounds__(32 * (TW + 1)) syevx_tri_small_kernel(const double* __restrict__ Ag, int nl,
                                                                             int kl, double* wg, double* Vg, int ldv,
                                                                             double* scratch,
                                                                             const int* __restrict__ nAg,
                                                                             double* work) {
  constexpr int M = 32 * NR, NC = (M + TW - 1) / TW;
  __shared__ double xs[2][M + 4 * TW], a1s[2][M + 4 * TW], ys[M], parts[TW][M], ds[M], es[M], red[40];
  __shared__ double sc[4];
  __shared__ int sred[32];
  __shared__ double2 vws[TW][M + 4 * TW];
  const SyevxScratch g = syevx_scratch(scratch, nl, kl, blockIdx.x);
  const int tid = threadIdx.x, nthr = blockDim.x, lane = tid & 31, w = (tid >> 5) - 1;
  double* wout = wg + (size_t)blockIdx.x * nl;
  double* Vout = Vg + (size_t)blockIdx.x * (size_t)nl * ldv;
  const int n = nAg ? max(0, min(nl, nAg[blockIdx.x])) : nl;
  const int k = min(kl, n);
  const double* A = Ag + (size_t)blockIdx.x * nl * nl;
  if (tid == 0) {
    add_work(work, 4.0 / 3.0 * n * (double)n * n + 4.0 * (double)k * n * n + 60.0 * k * n,
             sizeof(double) * (2.0 * n * n + (double)k * n));
    g.hdr[0] = (double)n;
  }
  for (int t = tid; t < kl; t += nthr) wout[t] = 0.0;
  for (int q = tid; q < nl * kl; q += nthr) Vout[(size_t)(q / kl) * ldv + q % kl] = 0.0;
  if (n == 0) return;
  double a[NR][NC];
  int top = 0;
  if (w >= 0) {
#pragma unroll
    for (int cc = 0; cc < NC; ++cc) {
      const int col = cc * TW + w;
#pragma unroll
      for (int r = 0; r < NR; ++r) {
        const int row = lane + 32 * r;
        a[r][cc] = row < n && col < n ? A[(size_t)col * nl + row] : 0.0;  // symmetric
        top = max(top, __double2hiint(a[r][cc]) & 0x7fffffff);
      }
    }
  }
  const double scale = range_scale(top, sred);
  if (w >= 0) {
#pragma unroll
    for (int cc = 0; cc < NC; ++cc) {
      const int col = cc * TW + w;
#pragma unroll
      for (int r = 0; r < NR; ++r) {
        a[r][cc] *= scale;
        if (col < 2) (col == 0 ? xs[0] : a1s[0])[lane + 32 * r] = a[r][cc];
      }
    }
  }
  __syncthreads();
  int par = 0;
  for (int j = 0; j + 2 < n; ++j, par ^= 1) {
    const double* x = xs[par];
    const double* a1 = a1s[par];
    double xr[NR];
#pragma unroll
    for (int r = 0; r < NR; ++r) {
      const int row = lane + 32 * r;
      xr[r] = row > j && row < n ? x[row] : 0.0;
    }
    if (w < 0) {
      double loc = 0.0;
#pragma unroll
      for (int r = 0; r < NR; ++r)
        if (lane + 32 * r != j + 1) loc = fma(xr[r], xr[r], loc);
      const double tail2 = warp_sum(loc), x0 = x[j + 1];
      double sn = 0.0, b = 0.0, alpha = x0;
      if (tail2 > kTailFloor) {
        const double s = fma(x0, x0, tail2);
        const double nrm = s * recip_sqrt(s);
        b = recip(fma(fabs(x0), nrm, s));  // 2 / (v^T v)
        sn = copysign(nrm, x0);
        alpha = -sn;
      }
      if (lane == 0) {
        sc[0] = sn;
        sc[1] = b;
        sc[3] = 0.5 * b;
        ds[j] = x[j];
        es[j] = alpha;
        g.beta[j] = b;
      }
#pragma unroll
      for (int r = 0; r < NR; ++r) {
        const int row = lane + 32 * r;
        if (row > j && row < n) g.W[(size_t)row * n + j] = row == j + 1 ? xr[r] + sn : xr[r];
      }
    } else {
      double p0[NR];
#pragma unroll
      for (int r = 0; r < NR; ++r) p0[r] = 0.0;
      // (the operands of four columns are loaded before any is used; row slots above the trailing block are skipped)
#pragma unroll
      for (int c0 = 0; c0 < NC; c0 += 4) {
        if ((c0 + 3) * TW + w <= j) continue;
        double xc[4];
#pragma unroll
        for (int u = 0; u < 4; ++u)
          if (c0 + u < NC) xc[u] = x[(c0 + u) * TW + w];
#pragma unroll
        for (int u = 0; u < 4; ++u)
          if (c0 + u < NC && (c0 + u) * TW + w > j && (c0 + u) * TW + w < n) {
#pragma unroll
            for (int r = 0; r < NR; ++r)
              if (32 * r + 31 > j) p0[r] = fma(a[r][c0 + u], xc[u], p0[r]);
          }
      }
#pragma unroll
      for (int r = 0; r < NR; ++r) parts[w][lane + 32 * r] = p0[r];
      asm volatile("bar.sync 1, %0;" ::"n"(32 * TW) : "memory");
      if (w == 0) {
        double xy = 0.0;
#pragma unroll
        for (int r = 0; r < NR; ++r) {
          const int row = lane + 32 * r;
          double y = parts[0][row] + parts[1][row];
#pragma unroll
          for (int q = 2; q < TW; ++q) y += parts[q][row];
          ys[row] = y;
          xy = fma(xr[r], y, xy);
        }
        xy = warp_sum(xy);
        if (lane == 0) sc[2] = xy;
      }
    }
    __syncthreads();
    // w = b q - K v with q = A v = y + sn a_1, K = b^2 v^T q / 2; then the next step's two columns
    double vr[NR], wr[NR];
    auto update = [&](int cc, double2 c) {
#pragma unroll
      for (int r = 0; r < NR; ++r)
        if (32 * r + 31 > j) a[r][cc] = fma(-vr[r], c.y, fma(-wr[r], c.x, a[r][cc]));
    };
    if (w >= 0) {
      const double sn = sc[0], b = sc[1];
      // v^T A v = x^T A x + 2 sn (A x)_1 + sn^2 a_11
      const double y1 = ys[j + 1];
      const double K = sc[3] * (b * fma(sn, fma(sn, a1[j + 1], y1 + y1), sc[2]));  // (b^2 alone may overflow)
#pragma unroll
      for (int r = 0; r < NR; ++r) {
        const int row = lane + 32 * r;
        const bool in = row > j && row < n;
        vr[r] = in ? (row == j + 1 ? xr[r] + sn : xr[r]) : 0.0;
        wr[r] = in ? fma(b, fma(sn, a1[row], ys[row]), -K * vr[r]) : 0.0;
        vws[w][row] = make_double2(vr[r], wr[r]);
      }
      __syncwarp();
#pragma unroll
      for (int cc = 0; cc < NC; ++cc) {
        const int col = cc * TW + w;
        if (col == j + 1 || col == j + 2) {
          update(cc, vws[w][col]);
#pragma unroll
          for (int r = 0; r < NR; ++r) (col == j + 1 ? xs[par ^ 1] : a1s[par ^ 1])[lane + 32 * r] = a[r][cc];
        }
      }
    }
    __syncthreads();
    if (w >= 0) {
#pragma unroll
      for (int c0 = 0; c0 < NC; c0 += 4) {
        if ((c0 + 3) * TW + w <= j + 2) continue;
        double2 c[4];
#pragma unroll
        for (int u = 0; u < 4; ++u)
          if (c0 + u < NC) c[u] = vws[w][(c0 + u) * TW + w];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int col = (c0 + u) * TW + w;
          if (c0 + u < NC && col > j + 2 && col < n) update(c0 + u, c[u]);
        }
      }
    }
  }
  if (tid == 0) {
    if (n >= 2) {
      ds[n - 2] = xs[par][n - 2];
      es[n - 2] = xs[par][n - 1];
      g.beta[n - 2] = 0.0;
      ds[n - 1] = a1s[par][n - 1];
    } else {
      ds[0] = xs[par][0];
    }
    es[n - 1] = 0.0;
    g.beta[n - 1] = 0.0;
  }
  __syncthreads();
  trid_gershgorin(ds, es, n, red);
  if (tid == 0) {
    g.hdr[1] = red[35];
    g.hdr[2] = red[36];
    g.hdr[3] = red[37];
    g.hdr[4] = 1.0 / scale;
  }
  for (int i = tid; i < n; i += nthr) {
    g.d[i] = ds[i];
    g.e[i] = es[i];
  }
}

// K2.  Eigenvalue t (the t-th largest) of the tridiagonal of item blockIdx.y, one block of four warps, a point of the
// multisection per thread (one warp on each of the SM's four FP64 units: 129-way rounds, 7 bits each): (a) FP32
// localisation in the Gershgorin interval in four rounds; (b) that bracket, widened, its ends the first FP64 round's
// first and last points (else the Gershgorin interval), then FP64 rounds, all on a copy of T scaled by a power of two to
// |T| in [0.5, 1) (the counts' range window), down to the absolute resolution eps ||T||: the eigenvalues of an FP64 Gram
// core carry errors of that size, and inverse iteration only needs the shift to that accuracy.
// Blocks kv .. kv + nq - 1 of an item meanwhile form Q = H_0 H_1 .. H_{n-3} (16 columns a block, eight lanes a column),
// so that K3 transforms back by one product instead of n - 2 dependent reflections.
constexpr int kBisectThreads = 128;
constexpr int kQCols = kBisectThreads / 8;

__device__ void form_q_columns(const SyevxScratch& g, int n, int c0, double* sm) {
  const int tid = threadIdx.x, gl = tid & 7, c = c0 + (tid >> 3);
  const int ld = n | 1;
  double* v = sm;                    // reflector j at v + j ld, rows j + 1 .. n - 1; beta_j at row j
  double* y = sm + (size_t)n * ld + (size_t)(tid >> 3) * ld;
  const int last = min(n - 3, c0 + kQCols - 2);  // H_j leaves e_c as it is while c <= j
  for (int q = tid; q < n * n; q += kBisectThreads) {
    const int i = q / n, j = q - i * n;
    if (j <= last && i >= j) v[j * ld + i] = i == j ? g.beta[j] : g.W[q];
  }
  for (int i = gl; i < n; i += 8) y[i] = i == c ? 1.0 : 0.0;
  __syncthreads();
  for (int j = last; j >= 0; --j) {
    const double* vj = v + j * ld;
    const double b = vj[j];
    if (b == 0.0) continue;
    // rows j + 1 .. n - 1 dealt to eight lanes
    double vr[12], yr[12], s0 = 0.0;
#pragma unroll
    for (int q = 0; q < 12; ++q) {
      const int i = j + 1 + gl + 8 * q;
      vr[q] = i < n ? vj[i] : 0.0;
      yr[q] = i < n ? y[i] : 0.0;
    }
#pragma unroll
    for (int q = 0; q < 12; ++q)
      if (j + 1 + 8 * q < n) s0 = fma(vr[q], yr[q], s0);
    for (int o = 4; o; o >>= 1) s0 += __shfl_xor_sync(0xffffffff, s0, o);
    s0 *= b;
#pragma unroll
    for (int q = 0; q < 12; ++q) {
      const int i = j + 1 + gl + 8 * q;
      if (j + 1 + 8 * q < n) {
        yr[q] = fma(-s0, vr[q], yr[q]);
        if (i < n) y[i] = yr[q];
      }
    }
    __syncwarp();
  }
  if (c < n)
    for (int i = gl; i < n; i += 8) g.Q[(size_t)i * n + c] = y[i];
}

__global__ void __launch_bounds__(kBisectThreads) syevx_bisect_kernel(int nl, int kl, int kv, double* scratch) {
  extern __shared__ __align__(16) double sm[];
  __shared__ int s_first[2][4];
  const SyevxScratch g = syevx_scratch(scratch, nl, kl, blockIdx.y);
  const int n = (int)g.hdr[0];
  const int t = blockIdx.x, tid = threadIdx.x;
  if (t >= kv) {
    const int c0 = (t - kv) * kQCols;
    if (c0 < n) form_q_columns(g, n, c0, sm);
    return;
  }
  if (t >= min(kv, n) || isnan(g.hdr[4])) return;
  const double lo = g.hdr[1], hi = g.hdr[2], emax2 = g.hdr[3];
  const double tnorm = fmax(fabs(lo), fabs(hi));
  if (tnorm == 0.0) {
    if (tid == 0) g.lam[t] = 0.0;
    return;
  }
  double* ds = sm;          // n: the scaled diagonal
  double* e2s = ds + n;     // n: the scaled e^2
  float* df = (float*)(e2s + n);  // n floats
  float* e2f = df + n;            // n floats
  int texp = 0;
  frexp(tnorm, &texp);
  const double sg = ldexp(1.0, -texp), sg2 = sg * sg;
  for (int i = tid; i < n; i += kBisectThreads) {
    const double ei = (i < n - 1) ? g.e[i] : 0.0;
    ds[i] = g.d[i] * sg;
    e2s[i] = (ei * ei) * sg2;
    df[i] = (float)ds[i];
    e2f[i] = (float)e2s[i];
  }
  __syncthreads();
  const int idx = n - 1 - t;
  int round = 0;
  // the first point (thread) whose count exceeds idx, kBisectThreads when none does
  auto first_above = [&](bool above) {
    const unsigned m = __ballot_sync(0xffffffff, above);
    if ((tid & 31) == 0) s_first[round & 1][tid >> 5] = m ? (tid & ~31) + __ffs(m) - 1 : kBisectThreads;
    __syncthreads();
    int f = kBisectThreads;
    for (int q = 3; q >= 0; --q)
      if (s_first[round & 1][q] < kBisectThreads) f = s_first[round & 1][q];
    ++round;
    return f;
  };
  const double pivmin = DBL_MIN * fmax(1.0, emax2);
  const double glo = (lo - 2.0 * DBL_EPSILON * tnorm - pivmin) * sg, ghi = (hi + 2.0 * DBL_EPSILON * tnorm + pivmin) * sg;
  float af = (float)glo, cf = (float)ghi;
  for (int it = 0; it < 4; ++it) {
    const float h = (cf - af) * (1.0f / (kBisectThreads + 1));
    const float x = af + h * (float)(tid + 1);
    const int f = first_above(sturm_count_f32(df, e2f, n, x) > idx);
    const float na = (f == 0) ? af : af + h * (float)f;
    const float nc = (f == kBisectThreads) ? cf : af + h * (float)(f + 1);
    if (!(na < nc)) break;  // FP32 resolution reached
    af = na;
    cf = nc;
  }
  const double wf = (double)cf - (double)af;
  double a = fmax(glo, (double)af - 4.0 * wf - 1e-6), c = fmin(ghi, (double)cf + 4.0 * wf + 1e-6);
  const double floor_s = DBL_EPSILON * tnorm * sg + 4.0 * pivmin * sg;
  {
    // the points a + i (c - a) / 127 with both ends: the bracket is right when the first of the points above is neither
    // the lower end nor missing
    const double h = (c - a) * (1.0 / (kBisectThreads - 1));
    const double x = tid == kBisectThreads - 1 ? c : a + h * (double)tid;
    const int f = first_above(sturm_count(ds, e2s, n, x) > idx);
    if (f == 0 || f == kBisectThreads) {
      a = glo;
      c = ghi;
    } else {
      const double na = a + h * (double)(f - 1), nc = f == kBisectThreads - 1 ? c : a + h * (double)f;
      a = na;
      c = nc;
    }
  }
  for (int it = 0; it < 40; ++it) {
    if (c - a <= 2.0 * DBL_EPSILON * fmax(fabs(a), fabs(c)) + floor_s) break;
    const double h = (c - a) * (1.0 / (kBisectThreads + 1));
    const double x = a + h * (double)(tid + 1);
    const int f = first_above(sturm_count(ds, e2s, n, x) > idx);
    const double na = (f == 0) ? a : a + h * (double)f;
    const double nc = (f == kBisectThreads) ? c : a + h * (double)(f + 1);
    if (!(na < nc)) break;
    a = na;
    c = nc;
  }
  if (tid == 0) g.lam[t] = 0.5 * (a + c) / sg;
}

// K3.  Eigenvectors of T by inverse iteration, their orthonormalisation, the back-transformation and the outputs.
// Inverse iteration takes two passes, a third when two of the vectors are still further than 1e-9 from orthogonal
// (eigenvalues closer than about 1e-12 ||T||); after each but the last they are orthonormalised only where they come
// within 0.05 of each other.  The last orthonormalisation is one Newton-Schulz step Y <- (3 I - G) Y / 2 where the vectors
// are within 1e-8 / k already (its error is the square), else by chol_orth, else by modified Gram-Schmidt.
__global__ void __launch_bounds__(kSyevxThreads) syevx_vec_kernel(int nl, int kl, int kv, double* wg, double* Vg, int ldv,
                                                                  double* scratch, int smem_flags) {
  extern __shared__ __align__(16) double sm[];
  const SyevxScratch g = syevx_scratch(scratch, nl, kl, blockIdx.x);
  const int n = (int)g.hdr[0];
  if (n == 0) return;
  if (isnan(g.hdr[4])) {
    // an entry that is not finite: the vectors' fallbacks below would make finite ones of it
    for (int t = threadIdx.x; t < min(kv, n); t += blockDim.x) wg[(size_t)blockIdx.x * nl + t] = g.hdr[4];
    for (size_t q = threadIdx.x; q < (size_t)n * min(kl, n); q += blockDim.x) {
      const size_t i = q / min(kl, n);
      Vg[(size_t)blockIdx.x * (size_t)nl * ldv + i * ldv + (q - i * min(kl, n))] = g.hdr[4];
    }
    return;
  }
  // flag 8: the tridiagonal, the reflector scalars and the eigenvalues in shared memory too
  double* d = sm;              // nl
  double* e = d + nl;          // nl
  double* beta = e + nl;       // nl
  double* lam = beta + nl;     // kl
  // the vectors, their LU factors and the reflectors (n <= kSmallEig: Q) in shared memory where they fit (flags 1, 2, 4):
  // the solves, the re-orthogonalisation and the back-transformation are dependent chains of their loads
  // strides in shared memory are odd numbers of doubles, so that the lanes of a warp walking different vectors
  // (inverse iteration: one lane per vector) or different rows (the warp sums) hit different banks
  const int npad = nl | 1;
  double* next = sm;
  if (smem_flags & 8) {
    next = lam + kl;
  } else {
    d = g.d;
    e = g.e;
    beta = g.beta;
    lam = g.lam;
  }
  const bool have_q = nl <= kSmallEig;
  double* Y = g.Y;
  double* lu = g.lu;
  double* W = have_q ? g.Q : g.W;
  if (smem_flags & 1) { Y = next; next += (size_t)kl * npad; }
  if (smem_flags & 2) { lu = next; next += (size_t)kl * 5 * npad; }
  if (smem_flags & 4) { W = next; next += (size_t)nl * npad; }
  double* G = (smem_flags & 16) ? next : nullptr;  // the Gram matrix of the vectors and k scalars
  const int k = min(kl, n);
  const int tid = threadIdx.x, nthr = blockDim.x;
  const int warp = tid >> 5, lane = tid & 31, nw = nthr >> 5;
  const int yst = (smem_flags & 1) ? npad : n;       // between vectors of Y
  const int fst = (smem_flags & 2) ? npad : n;       // between the fields of one vector's LU factors
  const int wld = (smem_flags & 4) ? npad : n;       // leading dimension of the reflectors
  double* wout = wg + (size_t)blockIdx.x * nl;
  double* Vout = Vg + (size_t)blockIdx.x * (size_t)nl * ldv;
  if (smem_flags & 8) {
    for (int i = tid; i < n; i += nthr) {
      d[i] = g.d[i];
      e[i] = g.e[i];
      beta[i] = g.beta[i];
    }
    for (int t = tid; t < k; t += nthr) lam[t] = g.lam[t];
  }
  if (smem_flags & 4) {
    const double* src = have_q ? g.Q : g.W;
    for (int t = tid; t < n * n; t += nthr) W[(t / n) * wld + t % n] = src[t];
  }
  __syncthreads();
  const double tnorm = fmax(fabs(g.hdr[1]), fabs(g.hdr[2]));
  double* Yf = Y;  // where the final vectors of T are
  int yf = yst;
  if (tnorm == 0.0) {
    // the zero matrix: eigenvalues 0, eigenvectors the unit vectors
    for (size_t q = tid; q < (size_t)k * n; q += nthr) {
      const int t = (int)(q / n), i = (int)(q - (q / n) * n);
      Y[(size_t)t * yst + i] = (i == t) ? 1.0 : 0.0;
    }
  } else {
  // separate exactly equal eigenvalues slightly so that their factorisations differ
  if (tid == 0) {
    const double sep = 10.0 * DBL_EPSILON * tnorm;
    for (int t = 1; t < k; ++t)
      if (lam[t - 1] - lam[t] < sep) lam[t] = lam[t - 1] - sep;
  }
  __syncthreads();

  // 3. inverse iteration
  const double tiny = DBL_EPSILON * fmax(tnorm, DBL_MIN);
  for (int t = tid; t < k; t += nthr) {
    double* y = Y + (size_t)t * yst;
    // deterministic start vector with entries in [0.5, 1)
    unsigned h = 2166136261u ^ (unsigned)(t * 2654435761u);
    for (int i = 0; i < n; ++i) {
      h = h * 1664525u + 1013904223u;
      y[i] = __hiloint2double(0x3fe00000 | (int)(h >> 12), (int)(h << 20));  // mantissa bits: no FP64 operation
    }
    double* f = lu + (size_t)t * 5 * fst;
    trid_factor(d, e, n, lam[t], tiny, f, f + fst, f + 2 * fst, f + 3 * fst, (int*)(f + 4 * fst));
  }
  __syncthreads();
  const double ortol = 1e-3 * tnorm;
  for (int pass = 0; pass < 3; ++pass) {
    for (int t = tid; t < k; t += nthr) {
      const double* f = lu + (size_t)t * 5 * fst;
      trid_solve(n, f, f + fst, f + 2 * fst, f + 3 * fst, (const int*)(f + 4 * fst), Y + (size_t)t * yst);
    }
    __syncthreads();
    bool last = pass == 2;
    if (G) {
      const float cos = gram_and_normalise(Y, yst, n, k, G);
      last = last || (pass == 1 && cos < 1e-9f);
      if (cos < (last ? 1e-8f / (float)k : 0.05f)) {
        if (!last) continue;
        // Newton-Schulz into the space of the LU factors: y_t - sum_{s != t} G_ts y_s / 2 (unit diagonal)
        const int gst = k | 1;
        for (int q = tid; q < k * n; q += nthr) {
          const int t = q / n, i = q - t * n;
          double s0 = 0.0, s1 = 0.0;
          for (int s = 0; s + 1 < k; s += 2) {
            s0 = fma(s == t ? 0.0 : (s < t ? G[t * gst + s] : G[s * gst + t]), Y[(size_t)s * yst + i], s0);
            s1 = fma(s + 1 == t ? 0.0 : (s + 1 < t ? G[t * gst + s + 1] : G[(s + 1) * gst + t]),
                     Y[(size_t)(s + 1) * yst + i], s1);
          }
          if ((k & 1) && t != k - 1) s0 = fma(G[(k - 1) * gst + t], Y[(size_t)(k - 1) * yst + i], s0);
          lu[q] = fma(-0.5, s0 + s1, Y[(size_t)t * yst + i]);
        }
        Yf = lu;
        yf = n;
        __syncthreads();
        break;
      }
      if (cos <= 2.0f && chol_orth(Y, yst, n, k, G)) {
        if (last) break;
        continue;
      }
      __syncthreads();
    }
    // unit lengths; after a breakdown (all-zero or overflowed solve) a unit vector, from which the re-orthogonalisation
    // and the next pass recover the direction.  Then modified Gram-Schmidt within clusters, by one warp, in descending
    // order of the eigenvalues
    for (int t = warp; t < k; t += nw) {
      double* y = Y + (size_t)t * yst;
      double s = 0.0;
      for (int i = lane; i < n; i += 32) s = fma(y[i], y[i], s);
      s = warp_sum(s);
      if (s > 0.0 && isfinite(s)) {
        s = recip_sqrt(s);
        for (int i = lane; i < n; i += 32) y[i] *= s;
      } else {
        for (int i = lane; i < n; i += 32) y[i] = (i == (t * 7 + pass) % n) ? 1.0 : 0.0;
      }
    }
    __syncthreads();
    if (tid < 32) {
      for (int t = 1; t < k; ++t) {
        double* yt = Y + (size_t)t * yst;
        bool touched = false;
        for (int s2 = t - 1; s2 >= 0 && lam[s2] - lam[t] <= ortol; --s2) {
          const double* ys = Y + (size_t)s2 * yst;
          double dp = 0.0;
          for (int i = tid; i < n; i += 32) dp += ys[i] * yt[i];
          dp = warp_sum(dp);
          for (int i = tid; i < n; i += 32) yt[i] -= dp * ys[i];
          touched = true;
        }
        if (touched) {
          double q2 = 0.0;
          for (int i = tid; i < n; i += 32) q2 += yt[i] * yt[i];
          q2 = warp_sum(q2);
          const double sc = q2 > 0.0 ? 1.0 / sqrt(q2) : 0.0;
          for (int i = tid; i < n; i += 32) yt[i] *= sc;
        }
        __syncwarp();
      }
    }
    __syncthreads();
    if (last) break;
  }
  }  // tnorm != 0
  __syncthreads();

  // outputs: eigenvalues descending, eigenvectors as the first k columns of V (leading dimension ldv)
  for (int t = tid; t < min(kv, n); t += nthr) wout[t] = (t < k ? lam[t] : g.lam[t]) * g.hdr[4];
  if (have_q && tnorm != 0.0) {
    // 4. back-transformation V = Q Y
    for (int q = tid; q < k * n; q += nthr) {
      const int i = q / k, t = q - i * k;
      const double* qi = W + (size_t)i * wld;
      const double* y = Yf + (size_t)t * yf;
      double s0 = 0.0, s1 = 0.0;
      int l = 0;
      for (; l + 1 < n; l += 2) {
        s0 = fma(qi[l], y[l], s0);
        s1 = fma(qi[l + 1], y[l + 1], s1);
      }
      if (l < n) s0 = fma(qi[l], y[l], s0);
      Vout[(size_t)i * ldv + t] = s0 + s1;
    }
    return;
  }
  if (tnorm != 0.0) {
    // x = H_0 H_1 ... H_{n-3} y, one warp per vector (the reflectors are read-only)
    for (int t = warp; t < k; t += nw) {
      double* yv = Yf + (size_t)t * yf;
      for (int j = n - 3; j >= 0; --j) {
        const double b = beta[j];
        if (b == 0.0) continue;
        const int m = n - j - 1;
        double* y = yv + (j + 1);
        double s = 0.0;
        for (int i = lane; i < m; i += 32) s += W[(size_t)(j + 1 + i) * wld + j] * y[i];
        s = b * warp_sum(s);
        for (int i = lane; i < m; i += 32) y[i] -= s * W[(size_t)(j + 1 + i) * wld + j];
        __syncwarp();
      }
    }
    __syncthreads();
  }
  for (size_t q = tid; q < (size_t)k * n; q += nthr) {
    int t = (int)(q / n), i = (int)(q - (q / n) * n);
    Vout[(size_t)i * ldv + t] = Yf[(size_t)t * yf + i];
  }
}

// k eigenvectors and kv >= k eigenvalues of every item
static void syevx_launch(lrfg_ctx* ctx, const double* A, double* w, double* V, int n, int k, int batch,
                         const int* nA, int kv = 0) {
  if (n <= 0 || batch <= 0 || k <= 0) return;
  k = std::min(k, n);
  kv = std::min(n, std::max(k, kv));
  LRFG_REQUIRE(kv < 65536 && batch < 65536, "eigensolver grid too large (k = %d, batch = %d)", k, batch);
  DBuf<double> scratch(ctx->pool, syevx_scratch_per(n, k) * batch);
  const size_t lim = (size_t)std::min(ctx->max_smem_optin, 200 * 1024);
  // K1: the register kernel up to n = 96; above, the reflectors in shared memory when they fit.  Algorithmic work at the
  // active size, counted by each block on the device
  auto tri_small = [&](auto kernel, int threads) {
    LRFG_LAUNCH(ctx, KC_EIGEN, 0.0, 0.0,
                kernel<<<batch, threads, 0, ctx->stream>>>(A, n, k, w, V, n, scratch.get(), nA,
                                                          work_counter(ctx, KC_EIGEN)));
  };
  if (n <= 32) {
    tri_small(syevx_tri_small_kernel<1, 3>, 128);
  } else if (n <= 64) {
    tri_small(syevx_tri_small_kernel<2, 4>, 160);
  } else if (n <= kSmallEig) {
    tri_small(syevx_tri_small_kernel<3, 6>, 224);
  } else {
    const size_t wbytes = sizeof(double) * (size_t)n * (n | 1);
    const size_t head1 = sizeof(double) * (40 + 2 * (size_t)n + kSyevxThreads);
    const int smem_w1 = head1 + wbytes <= (size_t)std::min(ctx->max_smem_optin, 208 * 1024) ? 1 : 0;
    const size_t smem1 = head1 + (smem_w1 ? wbytes : 0);
    LRFG_CUDA(raise_smem_limit((const void*)syevx_tri_kernel, smem1));
    LRFG_LAUNCH(ctx, KC_EIGEN, 0.0, 0.0,
                syevx_tri_kernel<<<batch, kSyevxThreads, smem1, ctx->stream>>>(A, n, k, w, V, n, scratch.get(), smem_w1,
                                                                               nA, work_counter(ctx, KC_EIGEN)));
  }
  // K2: one block per wanted eigenvalue of every item, and the blocks that form Q
  const int nq = n <= kSmallEig ? (n + kQCols - 1) / kQCols : 0;
  const size_t smem2 = sizeof(double) * std::max(3 * (size_t)n, nq ? (size_t)(n + kQCols) * (n | 1) : (size_t)0);
  LRFG_CUDA(raise_smem_limit((const void*)syevx_bisect_kernel, smem2));
  LRFG_LAUNCH(ctx, KC_EIGEN, 0.0, 0.0,
              syevx_bisect_kernel<<<dim3((unsigned)(kv + nq), (unsigned)batch), kBisectThreads, smem2, ctx->stream>>>(
                  n, k, kv, scratch.get()));
  // K3: the vectors, then their LU factors, then the reflectors in shared memory while they fit
  const size_t head3 = sizeof(double) * (3 * (size_t)n + (size_t)k);
  int flags3 = head3 <= lim ? 8 : 0;
  size_t smem3 = flags3 ? head3 : 0;
  const size_t npad = (size_t)(n | 1);  // K3's odd shared-memory strides
  const size_t parts[3] = {sizeof(double) * (size_t)k * npad, sizeof(double) * (size_t)k * 5 * npad,
                           sizeof(double) * (size_t)n * npad};
  for (int q = 0; q < 3; ++q)
    if (smem3 + parts[q] <= lim) {
      smem3 += parts[q];
      flags3 |= 1 << q;
    }
  // and the Gram matrix of the vectors' orthonormalisation
  const size_t gram3 = sizeof(double) * ((size_t)k * (k | 1) + k);
  if (smem3 + gram3 <= lim) {
    smem3 += gram3;
    flags3 |= 16;
  }
  LRFG_CUDA(raise_smem_limit((const void*)syevx_vec_kernel, smem3));
  LRFG_LAUNCH(ctx, KC_EIGEN, 0.0, 0.0,
              syevx_vec_kernel<<<batch, kSyevxThreads, smem3, ctx->stream>>>(n, k, kv, w, V, n, scratch.get(),
                                                                             flags3));
}

void syevx(lrfg_ctx* ctx, const double* A, double* w, double* V, int n, int k, int batch) {
  syevx_launch(ctx, A, w, V, n, k, batch, nullptr);
}

void syevx_values(lrfg_ctx* ctx, const double* A, double* w, double* V, int n, int k, int kv, int batch) {
  syevx_launch(ctx, A, w, V, n, k, batch, nullptr, kv);
}

void syevx_sized(lrfg_ctx* ctx, const double* A, const int* n_eff, double* w, double* V, int n, int k, int batch) {
  syevx_launch(ctx, A, w, V, n, k, batch, n_eff);
}

}  // namespace lrfg

namespace lrfg {

// ------------------------------------------------------------------------------------------------
// Factor of a (balanced) Gram matrix for the Gram-SVD: pivoted Cholesky P^T G P = L L^T (Golub & Van
// Loan Sec. 4.2, diagonal pivoting for semidefinite matrices), stopped when the largest remaining
// pivot falls below tau = 1e-16 times the largest initial diagonal (numerical rank rho).  The entries
// of an FP64 Gram matrix carry absolute errors of about eps64 times its largest diagonal, so smaller
// pivots are rounding noise: keeping them makes the basis M L^{-T} lose orthogonality in those
// directions (error ~ eps / sqrt(pivot)), dropping more loses their content (~ sqrt(pivot)).  The two
// balance near tau = eps64; an emulation of the truncations of the rank-10 solve at 243^3 (Hadamard
// products with the coefficient, exponential-sum outputs) gives relative errors against the SVD
// truncation of 4e-10..3e-9 at 1e-16, against 1.4e-8..1e-7 at 1e-20 and 7e-9..1.4e-8 at 1e-14.
// Outputs, for the orthonormal basis Q = M C P L11^{-T} of the left part M (C the balancing scaling):
//   RA  (b x b): rows i < rho hold L^T P^T (so G = RA^T RA up to the dropped Schur complement),
//   RAc (b x b): RA with column j divided by c_j (undoes the balancing in the transfer matrix),
//   Pc  (b x b): Pc[perm[l]][q] = c[perm[l]] (L11^{-1})[q][l] for l, q < rho (so Q = M Pc).
// One block per matrix; the working matrices are in shared memory when they fit.
// ------------------------------------------------------------------------------------------------
constexpr int kCholThreads = 512;

// shared-memory layout of gram_factor_kernel: bytes of the header before the two b x b work matrices
__host__ __device__ inline size_t chol_head_bytes(int b) {
  size_t bytes = sizeof(double) * (32 + 2 * (size_t)b) + sizeof(int) * (32 + 3 * (size_t)b + 2);
  return (bytes + 255) / 256 * 256;
}

// Factors of a Gram matrix with a diagonal entry that is not finite (a NaN in the data, or squares past the FP64 range): NaN
// as a whole, not the zeros of rank 0 that stopping at such a pivot would leave.  All threads of the block call it.
__device__ void gram_not_finite(int b, double* RA, double* RAc, double* Pc, int* rhog) {
  if (rhog && threadIdx.x == 0) rhog[blockIdx.x] = b;
  for (size_t t = threadIdx.x; t < (size_t)b * b; t += blockDim.x) {
    RA[t] = __longlong_as_double(0x7ff8000000000000LL);
    if (RAc) RAc[t] = RA[t];
    if (Pc) Pc[t] = RA[t];
  }
}

// Left-looking form (Golub & Van Loan Sec. 4.2.8 ordering with diagonal pivoting): pivot k takes the
// largest remaining diagonal of the Schur complement, kept as a vector, and only column k of L is formed,
// L[i][k] = (G[i][p] - sum_{l<k} L[i][l] L[p][l]) / L[p][k], for the rows not yet pivots; b rho^2 / 2
// multiply-adds up to the numerical rank instead of the b^2 rho of updating the whole trailing block.
// Column k of L is stored over column p = perm[k] of the working copy of G (that column is read only at
// this step), so L[j][l] sits at W[j][perm[l]].  The search for the next pivot runs in the same phase as
// the column (each warp over the rows it has just updated), so a pivot costs two barriers.
__global__ void __launch_bounds__(kCholThreads) gram_factor_kernel(const double* __restrict__ Gg,
                                                                   const double* __restrict__ cg, int b, double tau,
                                                                   double* RAg, double* RAcg, double* Pcg,
                                                                   int* rhog, double* scratch, int use_smem,
                                                                   double* work) {
  extern __shared__ __align__(16) double sm[];
  double* redv = sm;                   // 32 values
  double* dv = redv + 32;              // b: remaining diagonal of the Schur complement
  double* rd = dv + b;                 // b: reciprocals of the diagonal of L11
  int* redi = (int*)(rd + b);          // 32 indices
  int* perm = redi + 32;               // b: perm[k] = row of pivot k
  int* done = perm + b;                // b: 1 once a row is a pivot
  int* pos = done + b;                 // b: pivot position of a row
  int* flag = pos + b;                 // 2: rho, pivot
  const size_t bb = (size_t)b * b;
  double* W = use_smem ? (double*)((unsigned char*)sm + chol_head_bytes(b)) : scratch + (size_t)blockIdx.x * 2 * bb;
  double* Li = W + bb;                 // L11^{-1}
  const double* G = Gg + (size_t)blockIdx.x * bb;
  const double* c = cg ? cg + (size_t)blockIdx.x * b : nullptr;
  double* RA = RAg + (size_t)blockIdx.x * bb;
  double* RAc = RAcg ? RAcg + (size_t)blockIdx.x * bb : nullptr;
  double* Pc = Pcg ? Pcg + (size_t)blockIdx.x * bb : nullptr;
  const int tid = threadIdx.x, nthr = blockDim.x, lane = tid & 31, warp = tid >> 5, nw = nthr >> 5;
  for (size_t t = tid; t < bb; t += nthr) W[t] = G[t];
  double md = 0.0;
  int inf_or_nan = 0;
  for (int i = tid; i < b; i += nthr) {
    const double gi = G[(size_t)i * b + i];
    inf_or_nan |= !isfinite(gi);
    dv[i] = gi;
    done[i] = 0;
    pos[i] = b;
    perm[i] = i;
    md = fmax(md, gi);
  }
  for (int o = 16; o; o >>= 1) md = fmax(md, __shfl_xor_sync(0xffffffff, md, o));
  if (lane == 0) redv[warp] = md;
  if (__syncthreads_or(inf_or_nan)) return gram_not_finite(b, RA, RAc, Pc, rhog);
  if (tid == 0) {
    double m = 0.0;
    for (int i = 0; i < nw; ++i) m = fmax(m, redv[i]);
    redv[31] = m;
    flag[0] = b;
  }
  __syncthreads();
  const double maxd0 = redv[31];
  const int nwa = min(nw, (b + 31) >> 5);  // warps that hold rows
  // per-warp candidates for the next pivot (largest remaining diagonal; ties: smallest row) from the rows
  // this thread holds, after its own updates (two barriers per pivot)
  auto warp_candidates = [&]() {
    double best = -1.0;
    int bi = b;
    for (int i = tid; i < b; i += nthr) {
      if (done[i]) continue;
      const double v = dv[i];
      if (v > best || (v == best && i < bi)) { best = v; bi = i; }
    }
    if (warp < nwa) {
      for (int o = 16; o; o >>= 1) {
        const double ov = __shfl_xor_sync(0xffffffff, best, o);
        const int oi = __shfl_xor_sync(0xffffffff, bi, o);
        if (ov > best || (ov == best && oi < bi)) { best = ov; bi = oi; }
      }
      if (lane == 0) { redv[warp] = best; redi[warp] = bi; }
    }
  };
  warp_candidates();
  __syncthreads();
  for (int k = 0; k < b; ++k) {
    if (tid == 0) {
      double bv = -1.0;
      int bx = b;
      for (int i = 0; i < nwa; ++i)
        if (redv[i] > bv || (redv[i] == bv && redi[i] < bx)) { bv = redv[i]; bx = redi[i]; }
      if (!(bv > tau * maxd0) || !(bv > 0.0) || bx >= b) {
        flag[0] = k;
      } else {
        // the pivot's square root and reciprocal once, broadcast (see the eigensolver's reflector scalars)
        const double lkk = sqrt(bv);
        flag[1] = bx;
        done[bx] = 1;
        pos[bx] = k;
        perm[k] = bx;
        redv[29] = lkk;
        redv[30] = 1.0 / lkk;
      }
    }
    __syncthreads();
    if (flag[0] == k) break;
    const int p = flag[1];
    const double inv = redv[30];
    const double* rowp = W + (size_t)p * b;
    // column k of L for the rows that are not pivots (four independent accumulators: FP64 FMA latency)
    for (int i = tid; i < b; i += nthr) {
      if (done[i]) continue;
      const double* rowi = W + (size_t)i * b;
      double s0 = rowi[p], s1 = 0.0, s2 = 0.0, s3 = 0.0;
      int l = 0;
      for (; l + 3 < k; l += 4) {
        const int c0 = perm[l], c1 = perm[l + 1], c2 = perm[l + 2], c3 = perm[l + 3];
        s0 = fma(-rowi[c0], rowp[c0], s0);
        s1 = fma(-rowi[c1], rowp[c1], s1);
        s2 = fma(-rowi[c2], rowp[c2], s2);
        s3 = fma(-rowi[c3], rowp[c3], s3);
      }
      for (; l < k; ++l) s0 = fma(-rowi[perm[l]], rowp[perm[l]], s0);
      const double lik = ((s0 + s1) + (s2 + s3)) * inv;
      W[(size_t)i * b + p] = lik;
      dv[i] = fma(-lik, lik, dv[i]);
    }
    if (tid == 0) W[(size_t)p * b + p] = redv[29];
    warp_candidates();
    __syncthreads();
  }
  const int rho = flag[0];
  if (rhog && tid == 0) rhog[blockIdx.x] = rho;
  if (tid == 0) {
    // column q of L: (b - q - 1) rows of q multiply-adds; the triangular inverse (rho^3/6)
    double f = 0.0;
    for (int q = 0; q < rho; ++q) f += (double)(b - q - 1) * q;
    add_work(work, 2.0 * f + (Pc ? rho * (double)rho * rho / 3.0 : 0.0), sizeof(double) * 4.0 * bb);
  }
  // outputs: RA row k < rho, column j = L[j][k] for rows j that are not earlier pivots (upper triangular in
  // pivot order), RAc = RA with column j divided by c_j
  for (size_t t = tid; t < bb; t += nthr) {
    const int k = (int)(t / b), j = (int)(t - (t / b) * b);
    double v = 0.0;
    if (k < rho && pos[j] >= k) v = W[(size_t)j * b + perm[k]];
    RA[t] = v;
    if (RAc) RAc[t] = c ? v / c[j] : v;
  }
  if (!Pc) return;
  // L11^{-1} in pivot order: L11[i][l] = W[perm[i]][perm[l]]; reciprocal diagonal first, then one thread per
  // column q, forward substitution with four accumulators
  for (int i = tid; i < rho; i += nthr) rd[i] = 1.0 / W[(size_t)perm[i] * b + perm[i]];
  __syncthreads();
  for (int q = tid; q < rho; q += nthr) {
    for (int i = 0; i < q; ++i) Li[(size_t)i * b + q] = 0.0;
    for (int i = q; i < rho; ++i) {
      const double* rowi = W + (size_t)perm[i] * b;
      double s0 = (i == q) ? 1.0 : 0.0, s1 = 0.0, s2 = 0.0, s3 = 0.0;
      int l = q;
      for (; l + 3 < i; l += 4) {
        s0 = fma(-rowi[perm[l]], Li[(size_t)l * b + q], s0);
        s1 = fma(-rowi[perm[l + 1]], Li[(size_t)(l + 1) * b + q], s1);
        s2 = fma(-rowi[perm[l + 2]], Li[(size_t)(l + 2) * b + q], s2);
        s3 = fma(-rowi[perm[l + 3]], Li[(size_t)(l + 3) * b + q], s3);
      }
      for (; l < i; ++l) s0 = fma(-rowi[perm[l]], Li[(size_t)l * b + q], s0);
      Li[(size_t)i * b + q] = ((s0 + s1) + (s2 + s3)) * rd[i];
    }
  }
  __syncthreads();
  // Pc[perm[l]][q] = c[perm[l]] (L11^{-1})[q][l]
  for (size_t t = tid; t < bb; t += nthr) {
    const int r = (int)(t / b), q = (int)(t - (t / b) * b);  // Pc row r (original index), column q
    const int l = pos[r];
    const double v = (l < rho && q < rho && q >= l) ? (c ? c[r] : 1.0) * Li[(size_t)q * b + l] : 0.0;
    Pc[t] = v;
  }
}

// The same factor for b <= 32 NR with the Schur complement in registers: row = lane (NR rows a lane), columns dealt to
// CW warps (one per FP64 unit of the SM, two where the registers need it), right-looking.  Every warp holds the remaining diagonal and finds the pivot by itself with integer
// warp reductions (the bits of non-negative doubles order as integers; off the FP64 pipe), so a pivot costs one barrier,
// after the owner of the pivot's column has published it, and the chain reduction - reciprocal - two multiply-adds; the
// factor is kept as L D L^T until the end (no square root in the loop).  L11^-1 grows beside it by the same row
// operations on the unit matrix, in the shadow of that chain, instead of forward substitutions after it.
// One barrier a pivot against two, and a third of the time of the kernel above (b = 30: 105 -> 46 us).
template <int NR, int CW>
__global__ void __launch_bounds__(32 * CW) gram_factor_small_kernel(const double* __restrict__ Gg,
                                                                           const double* __restrict__ cg, int b,
                                                                           double tau, double* RAg, double* RAcg,
                                                                           double* Pcg, int* rhog, double* work) {
  constexpr int M = 32 * NR, NC = M / CW;
  extern __shared__ __align__(16) double sm[];
  double* Ls = sm;                       // b x M: column k of L (times the square root of pivot k), by rows of G
  double* rs = Ls + (size_t)b * M;       // b: 1 / sqrt(pivot)
  __shared__ int perm[M], pos[M];
  const size_t bb = (size_t)b * b;
  const double* G = Gg + blockIdx.x * bb;
  const double* c = cg ? cg + (size_t)blockIdx.x * b : nullptr;
  double* RA = RAg + blockIdx.x * bb;
  double* RAc = RAcg ? RAcg + blockIdx.x * bb : nullptr;
  double* Pc = Pcg ? Pcg + blockIdx.x * bb : nullptr;
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  double a[NR][NC], u[NR][NC], dv[NR];
  unsigned rows_done = 0, cols_done = 0;  // bit r / cc: the row / column is a pivot's
#pragma unroll
  for (int r = 0; r < NR; ++r) {
    const int row = lane + 32 * r;
    dv[r] = row < b ? G[(size_t)row * b + row] : -1.0;
    if (row >= b) rows_done |= 1u << r;
#pragma unroll
    for (int cc = 0; cc < NC; ++cc) {
      const int col = cc * CW + w;
      a[r][cc] = row < b && col < b ? G[(size_t)col * b + row] : 0.0;  // symmetric
      u[r][cc] = 0.0;
    }
  }
  for (int i = tid; i < M; i += 32 * CW) {
    perm[i] = i;
    pos[i] = b;
  }
  long long floor_bits = 0;
  int rho = b;
  bool inf_or_nan = false;  // the same in every thread
  for (int k = 0; k < b; ++k) {
    // the largest remaining diagonal (ties: the smallest row)
    double best = dv[0];
    int bi = lane;
#pragma unroll
    for (int r = 1; r < NR; ++r)
      if (__double_as_longlong(dv[r]) > __double_as_longlong(best)) {
        best = dv[r];
        bi = lane + 32 * r;
      }
    const int hi = __double2hiint(best), mh = __reduce_max_sync(0xffffffff, hi);
    const unsigned lo = hi == mh ? (unsigned)__double2loint(best) : 0u, ml = __reduce_max_sync(0xffffffff, lo);
    const int p = (int)__reduce_min_sync(0xffffffff, hi == mh && (unsigned)__double2loint(best) == ml ? (unsigned)bi : 1u << 30);
    const double piv = __hiloint2double(mh, (int)ml);
    // (positive doubles compare as integers: no FP64 comparison in the loop)
    if (k == 0) floor_bits = piv > 0.0 ? __double_as_longlong(tau * piv) : 0;
    if (mh < 0 || __double_as_longlong(piv) <= floor_bits || mh >= 0x7ff00000) {
      inf_or_nan = mh >= 0x7ff00000;
      rho = k;
      break;
    }
    const int pc = p / CW, pr = p >> 5, pl = p & 31;
    if (w == p % CW) {
#pragma unroll
      for (int cc = 0; cc < NC; ++cc)
        if (cc == pc) {
#pragma unroll
          for (int r = 0; r < NR; ++r) Ls[(size_t)k * M + lane + 32 * r] = (rows_done >> r & 1u) ? 0.0 : a[r][cc];
        }
    }
    const double inv = recip(piv);
    if (tid == 0) {
      perm[k] = p;
      pos[p] = k;
      rs[k] = piv;
    }
    __syncthreads();
    const double* col_p = Ls + (size_t)k * M;
    double t[NR];
#pragma unroll
    for (int r = 0; r < NR; ++r) {
      const bool is_p = pr == r && lane == pl;
      const double l = col_p[lane + 32 * r];
      t[r] = is_p ? 0.0 : l * inv;  // 0 for rows that are pivots already
      dv[r] = is_p || (rows_done >> r & 1u) ? -1.0 : fma(-t[r], l, dv[r]);
      if (is_p) rows_done |= 1u << r;
    }
    if (w == p % CW) cols_done |= 1u << pc;
    // four columns' operands ahead of the arithmetic they feed
#pragma unroll
    for (int c0 = 0; c0 < NC; c0 += 4) {
      if (c0 * CW + w >= b || (~cols_done >> c0 & 15u) == 0) continue;
      double lc[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) lc[q] = col_p[(c0 + q) * CW + w];
#pragma unroll
      for (int q = 0; q < 4; ++q)
        if ((c0 + q) * CW + w < b && !(cols_done >> (c0 + q) & 1u)) {
#pragma unroll
          for (int r = 0; r < NR; ++r) a[r][c0 + q] = fma(-t[r], lc[q], a[r][c0 + q]);
        }
    }
    if (Pc) {
#pragma unroll
      for (int c0 = 0; c0 < NC; c0 += 4) {
        if (c0 * CW + w > k) continue;
        double up[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const int cc = c0 + q;
          double v = u[0][cc];
#pragma unroll
          for (int r = 0; r < NR; ++r)
            if (r == pr) {
              if (cc * CW + w == k && lane == pl) u[r][cc] = 1.0;
              v = u[r][cc];
            }
          up[q] = __shfl_sync(0xffffffff, v, pl);
        }
#pragma unroll
        for (int q = 0; q < 4; ++q)
          if ((c0 + q) * CW + w <= k) {
#pragma unroll
            for (int r = 0; r < NR; ++r) u[r][c0 + q] = fma(-t[r], up[q], u[r][c0 + q]);
          }
      }
    }
  }
  __syncthreads();
  if (inf_or_nan) return gram_not_finite(b, RA, RAc, Pc, rhog);
  if (rhog && tid == 0) rhog[blockIdx.x] = rho;
  if (tid == 0) {
    // column q of L: (b - q - 1) rows of q multiply-adds; the triangular inverse (rho^3/6)
    double f = 0.0;
    for (int q = 0; q < rho; ++q) f += (double)(b - q - 1) * q;
    add_work(work, 2.0 * f + (Pc ? rho * (double)rho * rho / 3.0 : 0.0), sizeof(double) * 4.0 * bb);
  }
  for (int i = tid; i < rho; i += 32 * CW) rs[i] = recip_sqrt(rs[i]);
  __syncthreads();
  for (int t = tid; t < b * b; t += 32 * CW) {
    const int k = t / b, j = t - (t / b) * b;
    const double v = k < rho && pos[j] >= k ? Ls[(size_t)k * M + j] * rs[k] : 0.0;
    RA[t] = v;
    if (RAc) RAc[t] = c ? v / c[j] : v;
  }
  if (!Pc) return;
  __syncthreads();
  // L11^-1 in pivot order into shared memory, Ls[l][q] = (L11^-1)[q][l]: row q of the row operations is G's row perm[q]
#pragma unroll
  for (int r = 0; r < NR; ++r) {
    const int row = lane + 32 * r;
    const int q = row < b ? pos[row] : b;
    if (q < rho) {
#pragma unroll
      for (int cc = 0; cc < NC; ++cc) {
        const int l = cc * CW + w;
        if (l <= q) Ls[(size_t)l * M + q] = u[r][cc] * rs[q];
      }
    }
  }
  __syncthreads();
  // Pc[perm[l]][q] = c[perm[l]] (L11^{-1})[q][l]
  for (int t = tid; t < b * b; t += 32 * CW) {
    const int r = t / b, q = t - (t / b) * b;
    const int l = pos[r];
    Pc[t] = l < rho && q < rho && q >= l ? (c ? c[r] : 1.0) * Ls[(size_t)l * M + q] : 0.0;
  }
}

template <int NR, int CW>
static void gram_factor_small(lrfg_ctx* ctx, const double* G, const double* c, int b, int batch, double* RA, double* RAc,
                              double* Pc, int* rho, double tau) {
  const size_t smem = sizeof(double) * ((size_t)b * 32 * NR + b);
  LRFG_CUDA(raise_smem_limit((const void*)gram_factor_small_kernel<NR, CW>, smem));
  LRFG_LAUNCH(ctx, KC_CHOL, 0.0, 0.0,
              gram_factor_small_kernel<NR, CW><<<batch, 32 * CW, smem, ctx->stream>>>(
                  G, c, b, tau, RA, RAc, Pc, rho, work_counter(ctx, KC_CHOL)));
}

void gram_factor(lrfg_ctx* ctx, const double* G, const double* c, int b, int batch, double* RA, double* RAc,
                 double* Pc, int* rho, double tau) {
  if (b <= 0 || batch <= 0) return;
  if (b <= 32) return gram_factor_small<1, 4>(ctx, G, c, b, batch, RA, RAc, Pc, rho, tau);
  if (b <= 64) return gram_factor_small<2, 4>(ctx, G, c, b, batch, RA, RAc, Pc, rho, tau);
  if (b <= 96) return gram_factor_small<3, 8>(ctx, G, c, b, batch, RA, RAc, Pc, rho, tau);
  const size_t head = chol_head_bytes(b);
  const size_t full = head + sizeof(double) * 2 * (size_t)b * b;
  const int use_smem = full <= (size_t)std::min(ctx->max_smem_optin, 220 * 1024) ? 1 : 0;
  const size_t smem = use_smem ? full : head;
  DBuf<double> scratch;
  if (!use_smem) scratch = DBuf<double>(ctx->pool, (size_t)2 * b * b * batch);
  LRFG_CUDA(raise_smem_limit((const void*)gram_factor_kernel, smem));
  // algorithmic work up to the numerical rank, counted by each block on the device
  LRFG_LAUNCH(ctx, KC_CHOL, 0.0, 0.0,
              gram_factor_kernel<<<batch, kCholThreads, smem, ctx->stream>>>(G, c, b, tau, RA, RAc, Pc, rho,
                                                                               scratch.get(), use_smem,
                                                                               work_counter(ctx, KC_CHOL)));
}

}  // namespace lrfg

using namespace lrfg;

extern "C" lrfg_status lrfg_sym_eig(lrfg_ctx* ctx, const double* A, int n, int k, int batch, double* w, double* V) {
  if (!ctx) return LRFG_EINVAL;
  try {
    LRFG_CUDA(cudaSetDevice(ctx->device));
    LRFG_REQUIRE(A && w && V, "null argument");
    LRFG_REQUIRE(n >= 1 && k >= 1 && batch >= 1, "need n >= 1, k >= 1, batch >= 1 (got %d, %d, %d)", n, k, batch);
    syevx(ctx, A, w, V, n, std::min(k, n), batch);
    ctx->last_error.clear();
    return LRFG_OK;
  } catch (const Error& e) {
    ctx->last_error = e.msg;
    return e.status;
  } catch (...) {
    ctx->last_error = "unexpected internal error";
    return LRFG_ECUDA;
  }
}
