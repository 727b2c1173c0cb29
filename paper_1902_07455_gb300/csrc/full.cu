// Full-format comparison path (hot-path row a9): real <-> half-spectrum d-dimensional FFTs, the
// pointwise Fourier multipliers of the GaNi operator, and the reductions of PCG and A_eff.
//
// A grid (N_0, .., N_{d-1}) of reals has the half spectrum (N_0, .., N_{d-2}, H), H = (N_{d-1}+1)/2:
// the last axis keeps k >= 0 only (Hermitian symmetry of real fields, Sec. 2.2.1).  Forward transform:
// real-to-complex rows along the last axis (two real rows packed per complex FFT), then complex fibres
// along the other axes.  Transforms are unnormalised (Phi = |N| F_N); scalings are folded into the
// pointwise kernels.
#include <algorithm>
#include <cmath>

#include "full.cuh"

namespace lrfg {

static unsigned grid1d(lrfg_ctx* ctx, long long n) {
  long long g = (n + 255) / 256;
  long long cap = 16LL * (ctx->num_sms > 0 ? ctx->num_sms : 152);
  return (unsigned)std::max(1LL, std::min(g, cap));
}

FullGrid make_grid(int d, const int* N) {
  FullGrid g{};
  g.d = d;
  g.n_real = 1;
  for (int j = 0; j < d; ++j) { g.N[j] = N[j]; g.n_real *= N[j]; }
  g.H = (N[d - 1] + 1) / 2;
  g.rows = g.n_real / N[d - 1];
  g.n_half = g.rows * g.H;
  return g;
}

// ------------------------------------------------------------------------------------------------
// real rows -> half spectra (forward), optional pre-multiplication by a coefficient
// ------------------------------------------------------------------------------------------------
template <typename R>
__global__ void __launch_bounds__(256, 3) r2c_rows_kernel(const R* __restrict__ in, const R* __restrict__ coef, R scale,
                                                       typename CplxOf<R>::T* __restrict__ out, long long rows, int N,
                                                       int H, int TF, FftPlan pl,
                                                       const typename TwOf<typename CplxOf<R>::T>::T* __restrict__ Wg) {
  using V = typename CplxOf<R>::T;
  const float invN = 1.0f / (float)N, invH = 1.0f / (float)H;
  extern __shared__ __align__(16) unsigned char smraw_r2c[];
  V* sm = (V*)smraw_r2c;
  auto* W = reinterpret_cast<typename TwOf<V>::T*>(sm);
  V* a = sm + 2 * N;
  V* b = a + (size_t)TF * N;
  for (int j = threadIdx.x; j < N; j += blockDim.x) W[j] = Wg[j];
  const long long r0 = (long long)blockIdx.x * 2 * TF;
  const int nr = (int)min(2LL * TF, rows - r0);
  const int nrow = min(nr, TF);
  for (int t = threadIdx.x; t < nrow * N; t += blockDim.x) a[t] = mkc<V>(R(0), R(0));
  __syncthreads();
  // the tile's rows are contiguous: issue kU loads per thread before using any of them
  {
    constexpr int kU = 8;
    const R* src = in + (size_t)r0 * N;
    const R* cs = coef ? coef + (size_t)r0 * N : nullptr;
    const int total = nr * N;
    for (int base = threadIdx.x; base < total; base += kU * blockDim.x) {
      R v[kU], c[kU];
#pragma unroll
      for (int u = 0; u < kU; ++u) {
        const int t = base + u * blockDim.x;
        v[u] = t < total ? src[t] : R(0);
        c[u] = (cs && t < total) ? cs[t] : R(1);
      }
#pragma unroll
      for (int u = 0; u < kU; ++u) {
        const int t = base + u * blockDim.x;
        if (t < total) {
          const int f = small_div(t, N, invN), n = t - f * N;
          const R x = v[u] * c[u] * scale;
          if (f < TF) a[(size_t)f * N + n].x = x; else a[(size_t)(f - TF) * N + n].y = x;
        }
      }
    }
  }
  __syncthreads();
  V* Z = stockham_rows<-1>(a, b, nrow, N, pl, W);
  // split: X[k] = (Z[k] + conj Z[N-k]) / 2,  Y[k] = (Z[k] - conj Z[N-k]) / (2i)
  for (int t = threadIdx.x; t < nr * H; t += blockDim.x) {
    const int f = small_div(t, H, invH), k = t - f * H;
    int row = f < TF ? f : f - TF;
    V z = Z[(size_t)row * N + k];
    V zc = Z[(size_t)row * N + ((N - k) % N)];
    V v;
    if (f < TF) v = mkc<V>(R(0.5) * (z.x + zc.x), R(0.5) * (z.y - zc.y));
    else v = mkc<V>(R(0.5) * (z.y + zc.y), R(-0.5) * (z.x - zc.x));
    out[(size_t)(r0 + f) * H + k] = v;
  }
}

// half spectra -> real rows (inverse, unnormalised), optional post-multiplication by a coefficient
template <typename R>
__global__ void __launch_bounds__(256, 3) c2r_rows_kernel(const typename CplxOf<R>::T* __restrict__ in,
                                                       const R* __restrict__ coef, R scale, R* __restrict__ out,
                                                       long long rows, int N, int H, int TF, FftPlan pl,
                                                       const typename TwOf<typename CplxOf<R>::T>::T* __restrict__ Wg) {
  using V = typename CplxOf<R>::T;
  const float invN = 1.0f / (float)N;
  extern __shared__ __align__(16) unsigned char smraw_c2r[];
  V* sm = (V*)smraw_c2r;
  auto* W = reinterpret_cast<typename TwOf<V>::T*>(sm);
  V* a = sm + 2 * N;
  V* b = a + (size_t)TF * N;
  for (int j = threadIdx.x; j < N; j += blockDim.x) W[j] = Wg[j];
  const long long r0 = (long long)blockIdx.x * 2 * TF;
  const int nr = (int)min(2LL * TF, rows - r0);
  const int nrow = min(nr, TF);
  for (int t = threadIdx.x; t < nrow * N; t += blockDim.x) a[t] = mkc<V>(R(0), R(0));
  __syncthreads();
  // Z[k] = X[k] + i Y[k] over the full range, X[N-k] = conj X[k]; one thread per (row, k), kU (row, k)
  // pairs per thread loaded before any is used
  {
    constexpr int kU = 4;
    const int total = nrow * N;
    for (int base = threadIdx.x; base < total; base += kU * blockDim.x) {
      V x0[kU], x1[kU];
#pragma unroll
      for (int u = 0; u < kU; ++u) {
        const int t = base + u * blockDim.x;
        x0[u] = mkc<V>(R(0), R(0));
        x1[u] = mkc<V>(R(0), R(0));
        if (t < total) {
          const int row = small_div(t, N, invN), k = t - row * N;
          const int kk = k < H ? k : N - k;
          x0[u] = in[(size_t)(r0 + row) * H + kk];
          if (row + TF < nr) x1[u] = in[(size_t)(r0 + row + TF) * H + kk];
        }
      }
#pragma unroll
      for (int u = 0; u < kU; ++u) {
        const int t = base + u * blockDim.x;
        if (t < total) {
          const int row = small_div(t, N, invN), k = t - row * N;
          V p = x0[u], q = x1[u];
          if (k >= H) { p.y = -p.y; q.y = -q.y; }
          a[(size_t)row * N + k] = mkc<V>(p.x - q.y, p.y + q.x);
        }
      }
    }
  }
  __syncthreads();
  V* Z = stockham_rows<1>(a, b, nrow, N, pl, W);
  for (int t = threadIdx.x; t < nr * N; t += blockDim.x) {
    const int f = small_div(t, N, invN), n = t - f * N;
    int row = f < TF ? f : f - TF;
    V z = Z[(size_t)row * N + n];
    R v = (f < TF ? z.x : z.y) * scale;
    size_t gi = (size_t)(r0 + f) * N + n;
    if (coef) v *= coef[gi];
    out[gi] = v;
  }
}

// half spectra -> real rows -> times the coefficient -> half spectra, in one pass over the rows: the C2R pass,
// the material product and the R2C pass of the operator fused, so the real grid never goes to memory.  Both
// directions pair rows f and f + TF in one complex FFT (real and imaginary parts), so after the inverse
// transform the product acts on the two parts in place and the forward transform runs on the result as is.
// `in` and `out` may alias (a block reads all of its rows before it writes them).  H: stored frequencies of a row, at
// most (N + 1) / 2 (fewer on the double grid of the exact integration, where the others are zero and not wanted).  crows: rows
// of the coefficient, rows beyond it (a second component) starting over.
template <typename R>
__global__ void __launch_bounds__(256, 3) c2r_mul_r2c_rows_kernel(const typename CplxOf<R>::T* in,
                                                               const R* __restrict__ coef, R scale,
                                                               typename CplxOf<R>::T* out, long long rows, int N,
                                                               int H, int TF, FftPlan pl,
                                                               const typename TwOf<typename CplxOf<R>::T>::T* __restrict__ Wg,
                                                               long long crows) {
  using V = typename CplxOf<R>::T;
  const float invN = 1.0f / (float)N, invH = 1.0f / (float)H;
  extern __shared__ __align__(16) unsigned char smraw_fused[];
  V* sm = (V*)smraw_fused;
  auto* W = reinterpret_cast<typename TwOf<V>::T*>(sm);
  V* a = sm + 2 * N;
  V* b = a + (size_t)TF * N;
  for (int j = threadIdx.x; j < N; j += blockDim.x) W[j] = Wg[j];
  const long long r0 = (long long)blockIdx.x * 2 * TF;
  const int nr = (int)min(2LL * TF, rows - r0);
  const int nrow = min(nr, TF);
  // Z[k] = X[k] + i Y[k] over the full range from the two half spectra (X[N-k] = conj X[k])
  {
    constexpr int kU = 4;
    const int total = nrow * N;
    for (int base = threadIdx.x; base < total; base += kU * blockDim.x) {
      V x0[kU], x1[kU];
#pragma unroll
      for (int u = 0; u < kU; ++u) {
        const int t = base + u * blockDim.x;
        x0[u] = mkc<V>(R(0), R(0));
        x1[u] = mkc<V>(R(0), R(0));
        if (t < total) {
          const int row = small_div(t, N, invN), k = t - row * N;
          const int kk = min(k, N - k);
          if (kk < H) {
            x0[u] = in[(size_t)(r0 + row) * H + kk];
            if (row + TF < nr) x1[u] = in[(size_t)(r0 + row + TF) * H + kk];
          }
        }
      }
#pragma unroll
      for (int u = 0; u < kU; ++u) {
        const int t = base + u * blockDim.x;
        if (t < total) {
          const int row = small_div(t, N, invN), k = t - row * N;
          V p = x0[u], q = x1[u];
          if (2 * k > N) { p.y = -p.y; q.y = -q.y; }
          a[(size_t)row * N + k] = mkc<V>(p.x - q.y, p.y + q.x);
        }
      }
    }
  }
  __syncthreads();
  V* Z = stockham_rows<1>(a, b, nrow, N, pl, W);
  // the product with the coefficient on both real rows of each complex row, in place
  {
    constexpr int kU = 4;
    const int total = nrow * N;
    for (int base = threadIdx.x; base < total; base += kU * blockDim.x) {
      R ca[kU], cb[kU];
#pragma unroll
      for (int u = 0; u < kU; ++u) {
        const int t = base + u * blockDim.x;
        ca[u] = R(0);
        cb[u] = R(0);
        if (t < total) {
          const int row = small_div(t, N, invN), k = t - row * N;
          const long long ra = r0 + row, rb = ra + TF;
          ca[u] = coef[(ra < crows ? ra : ra - crows) * N + k];
          if (row + TF < nr) cb[u] = coef[(rb < crows ? rb : rb - crows) * N + k];
        }
      }
#pragma unroll
      for (int u = 0; u < kU; ++u) {
        const int t = base + u * blockDim.x;
        if (t < total) {
          const V z = Z[t];
          Z[t] = mkc<V>(z.x * scale * ca[u], z.y * scale * cb[u]);
        }
      }
    }
  }
  __syncthreads();
  V* Z2 = stockham_rows<-1>(Z, Z == a ? b : a, nrow, N, pl, W);
  // split: X[k] = (Z[k] + conj Z[N-k]) / 2,  Y[k] = (Z[k] - conj Z[N-k]) / (2i)
  for (int t = threadIdx.x; t < nr * H; t += blockDim.x) {
    const int f = small_div(t, H, invH), k = t - f * H;
    const int row = f < TF ? f : f - TF;
    const V z = Z2[(size_t)row * N + k];
    const V zc = Z2[(size_t)row * N + ((N - k) % N)];
    V v;
    if (f < TF) v = mkc<V>(R(0.5) * (z.x + zc.x), R(0.5) * (z.y - zc.y));
    else v = mkc<V>(R(0.5) * (z.y + zc.y), R(-0.5) * (z.x - zc.x));
    out[(size_t)(r0 + f) * H + k] = v;
  }
}

// ------------------------------------------------------------------------------------------------
// FP32 rows of length N = P1 P2: the fused C2R -> product -> R2C pass of the operator with the two
// register passes of fft2_fibres_kernel per direction, over a tile of 32 complex rows (real rows r0 + j
// and r0 + 32 + j in the real and imaginary parts of complex row j).  The tile lives once in shared
// memory as Z[n][j] with row stride 33 (conflict-free both along n and along j); every pass reads its
// inputs to registers, waits at a barrier and writes its outputs in place, so no second buffer is needed
// and three blocks fit an SM.  Global traffic is coalesced along each row: the half spectra in, the
// coefficient rows, the half spectra out.  `in` and `out` may alias (a block reads all its rows first).
// ------------------------------------------------------------------------------------------------
constexpr int kRowsLd = 33;

// one Stockham pass pair of the transform of the tile, in place (see the header of fft_device.cuh):
// pass 1 radix P1 (warp w = c < P2 takes x[c + P2 r]), pass 2 radix P2 with w_N^{f r} (f = w + P2 jb)
template <int SIGN, int P1, int P2>
__device__ __forceinline__ void rows2_transform(float2* Z, const float2* W, int w, int lane) {
  constexpr int N = P1 * P2;
  {
    float2 x[P1];
#pragma unroll
    for (int r = 0; r < P1; ++r) x[r] = Z[(w + P2 * r) * kRowsLd + lane];
    __syncthreads();
    RegDFT<P1, SIGN, float2>::run(x);
#pragma unroll
    for (int q = 0; q < P1; ++q) Z[(w * P1 + q) * kRowsLd + lane] = x[q];
  }
  __syncthreads();
  {
    float2 y[P1 / P2][P2];
#pragma unroll
    for (int jb = 0; jb < P1 / P2; ++jb)
#pragma unroll
      for (int r = 0; r < P2; ++r) y[jb][r] = Z[(r * P1 + w + P2 * jb) * kRowsLd + lane];
    __syncthreads();
#pragma unroll
    for (int jb = 0; jb < P1 / P2; ++jb) {
      const int f = w + P2 * jb;
#pragma unroll
      for (int r = 1; r < P2; ++r) y[jb][r] = cmul(y[jb][r], tw<SIGN>(W, f * r));
      RegDFT<P2, SIGN, float2>::run(y[jb]);
#pragma unroll
      for (int q = 0; q < P2; ++q) Z[(f + P1 * q) * kRowsLd + lane] = y[jb][q];
    }
  }
  __syncthreads();
  (void)N;
}

template <int P1, int P2>
__global__ void __launch_bounds__(32 * P2, 3) rows2_mul_kernel(const float2* in, const float* __restrict__ coef,
                                                              float scale, float2* out, long long rows,
                                                              const float2* __restrict__ Wg) {
  constexpr int N = P1 * P2, H = (N + 1) / 2, NT = 32 * P2;
  extern __shared__ __align__(16) unsigned char smraw_rows2[];
  float2* Z = (float2*)smraw_rows2;  // [N][kRowsLd]
  float2* W = Z + N * kRowsLd;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const long long r0 = (long long)blockIdx.x * 64;
  const int nr = (int)min(64LL, rows - r0);  // real rows of this tile: j < nr (real parts), 32 + j < nr (imaginary)
  for (int j = threadIdx.x; j < N; j += NT) W[j] = Wg[j];
  // Z[k] = X[k] + i Y[k] and Z[N - k] = conj X[k] + i conj Y[k] from the two half spectra
  {
    // the tile's loads in two rounds of requests (two latencies per block)
    constexpr int total = 32 * H;
    constexpr int kU = (total + 2 * NT - 1) / (2 * NT);
    for (int e0 = threadIdx.x; e0 < total; e0 += kU * NT) {
      float2 a[kU], b[kU];
#pragma unroll
      for (int u = 0; u < kU; ++u) {
        const int e = e0 + u * NT;
        const int j = e / H;
        a[u] = make_float2(0.f, 0.f);
        b[u] = make_float2(0.f, 0.f);
        if (e < total && j < nr) a[u] = in[(size_t)r0 * H + e];
        if (e < total && j + 32 < nr) b[u] = in[(size_t)(r0 + 32) * H + e];
      }
#pragma unroll
      for (int u = 0; u < kU; ++u) {
        const int e = e0 + u * NT;
        if (e < total) {
          const int j = e / H, k = e - j * H;
          Z[k * kRowsLd + j] = make_float2(a[u].x - b[u].y, a[u].y + b[u].x);
          if (k) Z[(N - k) * kRowsLd + j] = make_float2(a[u].x + b[u].y, b[u].x - a[u].y);
        }
      }
    }
  }
  __syncthreads();
  rows2_transform<1, P1, P2>(Z, W, w, lane);
  // the real rows times the coefficient: Z[n][j] = (x_j[n], x_{32+j}[n]); each thread's coefficients are
  // requested before any is used
  {
    constexpr int per = (32 * N + NT - 1) / NT;
    const float* c0 = coef + (size_t)r0 * N;
    float ca[per], cb[per];
#pragma unroll
    for (int u = 0; u < per; ++u) {
      const int e = threadIdx.x + u * NT;
      const int j = e / N;
      ca[u] = (e < 32 * N && j < nr) ? c0[e] : 0.f;
      cb[u] = (e < 32 * N && j + 32 < nr) ? c0[(size_t)32 * N + e] : 0.f;
    }
#pragma unroll
    for (int u = 0; u < per; ++u) {
      const int e = threadIdx.x + u * NT;
      if (e < 32 * N) {
        const int j = e / N, n = e - j * N;
        float2* p = Z + n * kRowsLd + j;
        const float2 z = *p;
        *p = make_float2(z.x * scale * ca[u], z.y * scale * cb[u]);
      }
    }
  }
  __syncthreads();
  rows2_transform<-1, P1, P2>(Z, W, w, lane);
  // split: X[k] = (Z[k] + conj Z[N-k]) / 2, Y[k] = (Z[k] - conj Z[N-k]) / (2i)
  {
    constexpr int total = 32 * H;
    for (int e = threadIdx.x; e < total; e += NT) {
      const int j = e / H, k = e - j * H;
      const float2 z = Z[k * kRowsLd + j];
      const float2 zc = Z[(k ? N - k : 0) * kRowsLd + j];
      if (j < nr) out[(size_t)r0 * H + e] = make_float2(0.5f * (z.x + zc.x), 0.5f * (z.y - zc.y));
      if (j + 32 < nr) out[(size_t)(r0 + 32) * H + e] = make_float2(0.5f * (z.y + zc.y), -0.5f * (z.x - zc.x));
    }
  }
}

template <typename R>
static FftPlan row_tile(lrfg_ctx* ctx, int N, long long rows, int* tf_out, size_t* smem) {
  using V = typename CplxOf<R>::T;
  // at most 72 KB for N <= 300, so that three blocks share an SM
  size_t limit = 72 * 1024;
  if (N > 300) limit = (size_t)std::min(ctx->max_smem_optin, 200 * 1024);
  long long per = 2LL * N * (long long)sizeof(V);
  long long tf = ((long long)limit - 2LL * N * (long long)sizeof(V)) / per;
  tf = std::max(1LL, std::min(tf, 32LL));
  // a tile row carries two real rows
  const FftPlan pl = choose_plan(ctx, N, sizeof(R) == sizeof(double), (rows + 1) / 2, (int)tf, tf_out);
  *smem = (size_t)(2LL * N * sizeof(V) + *tf_out * per);
  return pl;
}

template <typename R>
void full_forward(lrfg_ctx* ctx, const FullGrid& g, const R* real_in, const R* coef, R scale,
                  typename CplxOf<R>::T* half_out) {
  using V = typename CplxOf<R>::T;
  const int N = g.N[g.d - 1];
  LRFG_CUDA(ensure_roots(ctx->device));
  const auto* W = twiddle_table<R>(ctx, N);
  size_t smem;
  int TF;
  const FftPlan pl = row_tile<R>(ctx, N, g.rows, &TF, &smem);
  long long blocks = (g.rows + 2LL * TF - 1) / (2LL * TF);
  LRFG_CUDA(raise_smem_limit((const void*)r2c_rows_kernel<R>, smem));
  LRFG_LAUNCH(ctx, KC_R2C, 2.5 * N * std::log2((double)N) * (double)g.rows,
              (double)g.rows * (N * sizeof(R) * (coef ? 2 : 1) + g.H * sizeof(V)),
              r2c_rows_kernel<R><<<(unsigned)blocks, 256, smem, ctx->stream>>>(real_in, coef, scale, half_out, g.rows, N,
                                                                                g.H, TF, pl, W));
  // complex axes, innermost first
  long long inner = g.H;
  for (int ax = g.d - 2; ax >= 0; --ax) {
    long long outer = 1;
    for (int j = 0; j < ax; ++j) outer *= g.N[j];
    fft_fibres(ctx, half_out, half_out, outer, g.N[ax], inner, -1);
    inner *= g.N[ax];
  }
}

template <typename R>
void full_inverse(lrfg_ctx* ctx, const FullGrid& g, typename CplxOf<R>::T* half_inout, const R* coef, R scale,
                  R* real_out) {
  using V = typename CplxOf<R>::T;
  long long inner = g.n_half;
  for (int ax = 0; ax <= g.d - 2; ++ax) {
    inner /= g.N[ax];
    long long outer = g.n_half / (inner * g.N[ax]);
    fft_fibres(ctx, half_inout, half_inout, outer, g.N[ax], inner, 1);
  }
  const int N = g.N[g.d - 1];
  LRFG_CUDA(ensure_roots(ctx->device));
  const auto* W = twiddle_table<R>(ctx, N);
  size_t smem;
  int TF;
  const FftPlan pl = row_tile<R>(ctx, N, g.rows, &TF, &smem);
  long long blocks = (g.rows + 2LL * TF - 1) / (2LL * TF);
  LRFG_CUDA(raise_smem_limit((const void*)c2r_rows_kernel<R>, smem));
  LRFG_LAUNCH(ctx, KC_C2R, 2.5 * N * std::log2((double)N) * (double)g.rows,
              (double)g.rows * (N * sizeof(R) * (coef ? 2 : 1) + g.H * sizeof(V)),
              c2r_rows_kernel<R><<<(unsigned)blocks, 256, smem, ctx->stream>>>(half_inout, coef, scale, real_out, g.rows,
                                                                                N, g.H, TF, pl, W));
}

template <int P1, int P2>
static void rows2_launch(lrfg_ctx* ctx, const FullGrid& g, float2* half_inout, const float* coef, float scale) {
  constexpr int N = P1 * P2;
  const size_t smem = sizeof(float2) * (size_t)N * (kRowsLd + 1);
  const long long blocks = (g.rows + 63) / 64;
  LRFG_REQUIRE(blocks < (1LL << 31), "too many rows");
  const float2* W = twiddle_table<float>(ctx, N);
  LRFG_CUDA(raise_smem_limit((const void*)rows2_mul_kernel<P1, P2>, smem));
  LRFG_LAUNCH(ctx, KC_ROWS_FUSED, 5.0 * N * std::log2((double)N) * (double)g.rows,
              (double)g.rows * (2.0 * g.H * sizeof(float2) + N * sizeof(float)),
              rows2_mul_kernel<P1, P2><<<(unsigned)blocks, 32 * P2, smem, ctx->stream>>>(half_inout, coef, scale,
                                                                                        half_inout, g.rows, W));
}

template <typename R>
void full_rows_mul(lrfg_ctx* ctx, const FullGrid& g, typename CplxOf<R>::T* half_inout, const R* coef, R scale) {
  using V = typename CplxOf<R>::T;
  const int N = g.N[g.d - 1];
  if constexpr (sizeof(R) == sizeof(float)) {
    LRFG_CUDA(ensure_roots(ctx->device));
    if (N == 243) return rows2_launch<27, 9>(ctx, g, half_inout, coef, scale);
    if (N == 81) return rows2_launch<9, 9>(ctx, g, half_inout, coef, scale);
  }
  LRFG_CUDA(ensure_roots(ctx->device));
  const auto* W = twiddle_table<R>(ctx, N);
  size_t smem;
  int TF;
  const FftPlan pl = row_tile<R>(ctx, N, g.rows, &TF, &smem);
  long long blocks = (g.rows + 2LL * TF - 1) / (2LL * TF);
  LRFG_CUDA(raise_smem_limit((const void*)c2r_mul_r2c_rows_kernel<R>, smem));
  LRFG_LAUNCH(ctx, KC_ROWS_FUSED, 5.0 * N * std::log2((double)N) * (double)g.rows,
              (double)g.rows * (2.0 * g.H * sizeof(V) + N * sizeof(R)),
              c2r_mul_r2c_rows_kernel<R><<<(unsigned)blocks, 256, smem, ctx->stream>>>(
                  half_inout, coef, scale, half_inout, g.rows, N, g.H, TF, pl, W, g.rows));
}

void half_rows_mul(lrfg_ctx* ctx, long long rows, int N, int H, double2* half_inout, const double* coef, long long crows) {
  LRFG_CUDA(ensure_roots(ctx->device));
  const auto* W = twiddle_table<double>(ctx, N);
  size_t smem;
  int TF;
  const FftPlan pl = row_tile<double>(ctx, N, rows, &TF, &smem);
  const long long blocks = (rows + 2LL * TF - 1) / (2LL * TF);
  LRFG_REQUIRE(blocks < (1LL << 31), "too many rows");
  LRFG_CUDA(raise_smem_limit((const void*)c2r_mul_r2c_rows_kernel<double>, smem));
  LRFG_LAUNCH(ctx, KC_ROWS_FUSED, 5.0 * N * std::log2((double)N) * (double)rows,
              (double)rows * (2.0 * H * sizeof(double2) + N * sizeof(double)),
              c2r_mul_r2c_rows_kernel<double><<<(unsigned)blocks, 256, smem, ctx->stream>>>(
                  half_inout, coef, 1.0, half_inout, rows, N, H, TF, pl, W, crows));
}

template void full_rows_mul<double>(lrfg_ctx*, const FullGrid&, double2*, const double*, double);
template void full_rows_mul<float>(lrfg_ctx*, const FullGrid&, float2*, const float*, float);

template void full_forward<double>(lrfg_ctx*, const FullGrid&, const double*, const double*, double, double2*);
template void full_forward<float>(lrfg_ctx*, const FullGrid&, const float*, const float*, float, float2*);
template void full_inverse<double>(lrfg_ctx*, const FullGrid&, double2*, const double*, double, double*);
template void full_inverse<float>(lrfg_ctx*, const FullGrid&, float2*, const float*, float, float*);

// ------------------------------------------------------------------------------------------------
// pointwise Fourier multipliers on the half spectrum.  Launch map: blockIdx.x = row (all indices but
// the last), blockIdx.y * blockDim.x + threadIdx.x = k_last, so a thread finds its frequencies without
// per-element division.  Multipliers are formed in the storage precision R from R-rounded constants;
// 1/(k.k) comes from a table of exactly rounded reciprocals (no per-element division).
// ------------------------------------------------------------------------------------------------
struct RowMap {
  int d, N0, N1, H;
};

static RowMap rowmap(const FullGrid& g) {
  RowMap m;
  m.d = g.d;
  m.N0 = g.N[0];
  m.N1 = g.d == 3 ? g.N[1] : 1;
  m.H = g.H;
  return m;
}

static dim3 row_block(const FullGrid& g) { return dim3((unsigned)std::min(256, ((g.H + 31) / 32) * 32)); }
static dim3 row_grid(const FullGrid& g) {
  const unsigned bx = row_block(g).x;
  return dim3((unsigned)g.rows, (unsigned)((g.H + bx - 1) / bx));
}

// frequencies of (row, kl); returns false past the end of the row
__device__ __forceinline__ bool row_k(const RowMap& m, int& k0, int& k1, int& k2, size_t& t) {
  const int row = blockIdx.x;
  const int kl = blockIdx.y * blockDim.x + threadIdx.x;
  if (kl >= m.H) return false;
  if (m.d == 3) {
    const int i0 = row / m.N1, i1 = row - i0 * m.N1;
    k0 = freq_of(i0, m.N0);
    k1 = freq_of(i1, m.N1);
    k2 = kl;
  } else {
    k0 = freq_of(row, m.N0);
    k1 = kl;
    k2 = 0;
  }
  t = (size_t)row * m.H + kl;
  return true;
}

// out = in * (2 pi i k_alpha) * scale   (c2 = 2 pi scale, rounded to R)
template <typename V>
__global__ void mul_grad_kernel(const V* __restrict__ in, V* out, RowMap m, int alpha,
                                typename RealOf<V>::T c2) {
  using R = typename RealOf<V>::T;
  int k[3];
  size_t t;
  if (!row_k(m, k[0], k[1], k[2], t)) return;
  const R f = c2 * (R)k[alpha];
  const V v = in[t];
  out[t] = mkc<V>(-v.y * f, v.x * f);
}

// acc = (init ? 0 : acc) + in * (-2 pi i k_alpha) * scale; if precond, then acc /= k.k (0 at k=0)
template <typename V>
__global__ void acc_div_kernel(const V* __restrict__ in, V* acc, RowMap m, int alpha, typename RealOf<V>::T c2,
                               int init, int precond, const typename RealOf<V>::T* __restrict__ inv_kk) {
  using R = typename RealOf<V>::T;
  int k[3];
  size_t t;
  if (!row_k(m, k[0], k[1], k[2], t)) return;
  const R f = -c2 * (R)k[alpha];
  const V v = in[t];
  V r = mkc<V>(-v.y * f, v.x * f);
  if (!init) {
    const V o = acc[t];
    r.x += o.x;
    r.y += o.y;
  }
  if (precond) {
    const R s = inv_kk[k[0] * k[0] + k[1] * k[1] + k[2] * k[2]];
    r.x *= s;
    r.y *= s;
  }
  acc[t] = r;
}

template <typename V>
__global__ void precond_kernel(const V* __restrict__ in, V* out, RowMap m,
                               const typename RealOf<V>::T* __restrict__ inv_kk) {
  using R = typename RealOf<V>::T;
  int k[3];
  size_t t;
  if (!row_k(m, k[0], k[1], k[2], t)) return;
  const R s = inv_kk[k[0] * k[0] + k[1] * k[1] + k[2] * k[2]];
  const V v = in[t];
  out[t] = mkc<V>(v.x * s, v.y * s);
}

// the six distinct entries of a symmetric 3 x 3 B times a constant: (b00, b11, b22, b01, b02, b12)
template <typename R>
struct SymB {
  R b[6];
};

template <typename R>
static SymB<R> sym_b(const double* B, double c) {
  SymB<R> s;
  s.b[0] = (R)(c * B[0]);
  s.b[1] = (R)(c * B[4]);
  s.b[2] = (R)(c * B[8]);
  s.b[3] = (R)(c * B[1]);
  s.b[4] = (R)(c * B[2]);
  s.b[5] = (R)(c * B[5]);
  return s;
}

template <typename R>
__device__ __forceinline__ R quad_b(const SymB<R>& s, int k0, int k1, int k2) {
  const R x = (R)k0, y = (R)k1, z = (R)k2;
  return s.b[0] * x * x + s.b[1] * y * y + s.b[2] * z * z + (R)2 * (s.b[3] * x * y + s.b[4] * x * z + s.b[5] * y * z);
}

// acc += (c k.B k) in; then, if precond, acc /= k.k (0 at k = 0)
template <typename V>
__global__ void acc_aniso_kernel(const V* __restrict__ in, V* acc, RowMap m, SymB<typename RealOf<V>::T> sb,
                                 int precond, const typename RealOf<V>::T* __restrict__ inv_kk) {
  using R = typename RealOf<V>::T;
  int k[3];
  size_t t;
  if (!row_k(m, k[0], k[1], k[2], t)) return;
  const R q = quad_b(sb, k[0], k[1], k[2]);
  const V v = in[t];
  V r = acc[t];
  r.x += q * v.x;
  r.y += q * v.y;
  if (precond) {
    const R s = inv_kk[k[0] * k[0] + k[1] * k[1] + k[2] * k[2]];
    r.x *= s;
    r.y *= s;
  }
  acc[t] = r;
}

template <typename R> static const R* inv_table(const FullGrid& g);
template <> const double* inv_table<double>(const FullGrid& g) { return g.inv_kk64; }
template <> const float* inv_table<float>(const FullGrid& g) { return g.inv_kk32; }

__global__ void inv_table_kernel(double* t64, float* t32, int n) {
  for (int m = blockIdx.x * blockDim.x + threadIdx.x; m < n; m += gridDim.x * blockDim.x) {
    const double v = m > 0 ? 1.0 / (double)m : 0.0;
    t64[m] = v;
    t32[m] = m > 0 ? 1.0f / (float)m : 0.0f;
  }
}

void make_inv_tables(lrfg_ctx* ctx, FullGrid& g, DBuf<double>& t64, DBuf<float>& t32) {
  long long kmax = 0;
  for (int j = 0; j < g.d; ++j) kmax += (long long)((g.N[j] - 1) / 2) * ((g.N[j] - 1) / 2);
  const int n = (int)kmax + 1;
  t64 = DBuf<double>(ctx->pool, n);
  t32 = DBuf<float>(ctx->pool, n);
  LRFG_LAUNCH(ctx, KC_POINTWISE, n, 12.0 * n,
              inv_table_kernel<<<std::max(1, std::min(1024, (n + 255) / 256)), 256, 0, ctx->stream>>>(t64.get(),
                                                                                                      t32.get(), n));
  g.inv_kk64 = t64.get();
  g.inv_kk32 = t32.get();
}

static double two_pi_times(double scale) { return 6.283185307179586476925286766559 * scale; }

template <typename V>
void half_mul_grad(lrfg_ctx* ctx, const FullGrid& g, const V* in, V* out, int alpha, double scale) {
  using R = typename RealOf<V>::T;
  LRFG_LAUNCH(ctx, KC_POINTWISE, 2.0 * g.n_half, 2.0 * sizeof(V) * g.n_half,
              mul_grad_kernel<V><<<row_grid(g), row_block(g), 0, ctx->stream>>>(in, out, rowmap(g), alpha,
                                                                                 (R)two_pi_times(scale)));
}

template <typename V>
void half_acc_div(lrfg_ctx* ctx, const FullGrid& g, const V* in, V* acc, int alpha, double scale, int init,
                  int precond) {
  using R = typename RealOf<V>::T;
  LRFG_REQUIRE(!precond || inv_table<R>(g), "reciprocal table missing");
  LRFG_LAUNCH(ctx, KC_POINTWISE, 4.0 * g.n_half, (init ? 2.0 : 3.0) * sizeof(V) * g.n_half,
              acc_div_kernel<V><<<row_grid(g), row_block(g), 0, ctx->stream>>>(
                  in, acc, rowmap(g), alpha, (R)two_pi_times(scale), init, precond, inv_table<R>(g)));
}

// The complex-axis passes of the operator around its fused rows, with grad^ folded into an inverse pass and grad^* (with
// P~^-1 on the last) into a forward one.
template <typename R>
static FibreMul<R> fibre_mul(const FullGrid& g, int mode, int axis, int alpha, double scale, int init, int precond) {
  FibreMul<R> fm{};
  fm.mode = mode;
  fm.axis = axis;
  fm.alpha = alpha;
  fm.d = g.d;
  fm.N0 = g.N[0];
  fm.N1 = g.d == 3 ? g.N[1] : 1;
  fm.H = g.H;
  fm.init = init;
  fm.precond = precond;
  fm.c2 = (R)two_pi_times(scale);
  fm.inv_kk = inv_table<R>(g);
  return fm;
}

template <typename V>
void half_grad_fibres_inverse(lrfg_ctx* ctx, const FullGrid& g, const V* in, V* half, int alpha, double scale) {
  using R = typename RealOf<V>::T;
  fft_fibres_mul(ctx, in, half, fibre_mul<R>(g, 1, 0, alpha, scale, 0, 0));
  if (g.d == 3) fft_fibres(ctx, half, half, g.N[0], g.N[1], g.H, 1);
}

template <typename V>
void half_fibres_forward_div(lrfg_ctx* ctx, const FullGrid& g, V* half, V* acc, int alpha, double scale, int init,
                             int precond) {
  using R = typename RealOf<V>::T;
  if (g.d == 3) fft_fibres(ctx, half, half, g.N[0], g.N[1], g.H, -1);
  fft_fibres_mul(ctx, (const V*)half, acc, fibre_mul<R>(g, 2, 0, alpha, scale, init, precond));
}

// The whole operator on a d = 3 grid with the passes its components share.  The multipliers of axes 1 and 2 are constant
// along axis 0, so F_0^-1 v serves both components, and their divergences are summed before one F_0:
//   w1 = F_0^-1 v,  w2 = sum_{a = 1, 2} -2 pi i k_a F_1 (rows of F_1^-1 (2 pi i k_a w1)),
//   out = -2 pi i k_0 F_0 F_1 (rows of F_1^-1 F_0^-1 (2 pi i k_0 v)) + F_0 w2
// ten fibre passes instead of twelve.
template <typename R>
void full_operator_3d(lrfg_ctx* ctx, const FullGrid& g, const typename CplxOf<R>::T* v, typename CplxOf<R>::T* out,
                      const R* coef, double scale, int precond, typename CplxOf<R>::T* w0, typename CplxOf<R>::T* w1,
                      typename CplxOf<R>::T* w2) {
  using V = typename CplxOf<R>::T;
  const long long in0 = (long long)g.N[1] * g.H;
  fft_fibres_mul(ctx, v, w0, fibre_mul<R>(g, 1, 0, 0, scale, 0, 0));
  fft_fibres(ctx, (const V*)w0, w0, g.N[0], g.N[1], g.H, 1);
  full_rows_mul<R>(ctx, g, w0, coef, R(1));
  fft_fibres(ctx, (const V*)w0, w0, g.N[0], g.N[1], g.H, -1);
  fft_fibres_mul(ctx, (const V*)w0, out, fibre_mul<R>(g, 2, 0, 0, 1.0, 1, 0));
  fft_fibres(ctx, v, w1, 1, g.N[0], in0, 1);
  for (int alpha = 1; alpha <= 2; ++alpha) {
    V* h = alpha == 1 ? w0 : w1;
    fft_fibres_mul(ctx, (const V*)w1, h, fibre_mul<R>(g, 1, 1, alpha, scale, 0, 0));
    full_rows_mul<R>(ctx, g, h, coef, R(1));
    fft_fibres_mul(ctx, (const V*)h, w2, fibre_mul<R>(g, 2, 1, alpha, 1.0, alpha == 1, 0));
  }
  fft_fibres_mul(ctx, (const V*)w2, out, fibre_mul<R>(g, 2, 0, -1, 1.0, 0, precond));
}

// Operator of a d = 2 grid in FP64, both components in each of three launches: the gradient's inverse axis-0 pass of both from
// one read of v, the fused rows of both, the forward pass with the divergence summed in registers.  Small grids are bound
// by the length of a launch's dependent passes and the gaps between launches (six of 8-17 us at 63 x 63).
void full_operator_2d(lrfg_ctx* ctx, const FullGrid& g, const double2* v, double2* out, const double* coef, double scale,
                      int precond, double2* w) {
  fft_grad_2d(ctx, v, w, fibre_mul<double>(g, 1, 0, 0, scale, 0, 0));
  half_rows_mul(ctx, 2 * g.rows, g.N[1], g.H, w, coef, g.rows);
  fft_div_2d(ctx, w, out, fibre_mul<double>(g, 2, 0, 0, 1.0, 1, precond));
}

// The Ga operator (Eq. (ls_Ga_fourier)): as above with every transform between the grid's N frequencies and the double
// grid's M points.  A zero-padded spectrum is padded axis by axis inside the passes, so the fibres of frequencies outside
// the grid, zero before the inverse passes and dropped after the forward ones, are never transformed: axis 0 runs on a
// quarter of the double grid's fibres, axis 1 on half of them, and the real double grid never goes to memory.  w0: one half
// spectrum of the double grid; w1, w2: M_0 N_1 H each (d = 3).
void ga_operator(lrfg_ctx* ctx, const FullGrid& g, const FullGrid& gM, const double2* v, double2* out, const double* coef,
                 double scale, int precond, double2* w0, double2* w1, double2* w2) {
  auto fm = [&](int mode, int axis, int alpha, double sc, int init, int pc) {
    FibreMul<double> f = fibre_mul<double>(g, mode, axis, alpha, sc, init, pc);
    f.L = gM.N[axis];
    f.L0 = gM.N[0];
    return f;
  };
  const int last = gM.N[g.d - 1];
  if (g.d == 2) {
    for (int alpha = 0; alpha < 2; ++alpha) {
      fft_fibres_mul(ctx, v, w0, fm(1, 0, alpha, scale, 0, 0));
      half_rows_mul(ctx, gM.N[0], last, g.H, w0, coef, gM.N[0]);
      fft_fibres_mul(ctx, (const double2*)w0, out, fm(2, 0, alpha, 1.0, alpha == 0, alpha == 1 && precond));
    }
    return;
  }
  const long long in0 = (long long)g.N[1] * g.H, rows = (long long)gM.N[0] * gM.N[1];
  const int n1 = g.N[1], m1 = gM.N[1];
  fft_fibres_mul(ctx, v, w1, fm(1, 0, 0, scale, 0, 0));
  fft_fibres_pad(ctx, w1, w0, gM.N[0], n1, m1, g.H, 1);
  half_rows_mul(ctx, rows, last, g.H, w0, coef, rows);
  fft_fibres_pad(ctx, w0, w1, gM.N[0], n1, m1, g.H, -1);
  fft_fibres_mul(ctx, (const double2*)w1, out, fm(2, 0, 0, 1.0, 1, 0));
  fft_fibres_pad(ctx, v, w1, 1, g.N[0], gM.N[0], in0, 1);
  for (int alpha = 1; alpha <= 2; ++alpha) {
    fft_fibres_mul(ctx, (const double2*)w1, w0, fm(1, 1, alpha, scale, 0, 0));
    half_rows_mul(ctx, rows, last, g.H, w0, coef, rows);
    fft_fibres_mul(ctx, (const double2*)w0, w2, fm(2, 1, alpha, 1.0, alpha == 1, 0));
  }
  fft_fibres_mul(ctx, (const double2*)w2, out, fm(2, 0, -1, 1.0, 0, precond));
}

template void full_operator_3d<double>(lrfg_ctx*, const FullGrid&, const double2*, double2*, const double*, double, int,
                                       double2*, double2*, double2*);
template void full_operator_3d<float>(lrfg_ctx*, const FullGrid&, const float2*, float2*, const float*, double, int,
                                      float2*, float2*, float2*);

template void half_grad_fibres_inverse<double2>(lrfg_ctx*, const FullGrid&, const double2*, double2*, int, double);
template void half_grad_fibres_inverse<float2>(lrfg_ctx*, const FullGrid&, const float2*, float2*, int, double);
template void half_fibres_forward_div<double2>(lrfg_ctx*, const FullGrid&, double2*, double2*, int, double, int, int);
template void half_fibres_forward_div<float2>(lrfg_ctx*, const FullGrid&, float2*, float2*, int, double, int, int);

// ------------------------------------------------------------------------------------------------
// Ga: injection / projection between the half spectra of the grid (N) and the double grid (M = 2N - 1)
// ------------------------------------------------------------------------------------------------
__device__ __forceinline__ int wrap(int k, int n) { return k >= 0 ? k : k + n; }

// over the half spectrum of gM: the coefficient of the same frequency on g, or 0 outside Z_N
__global__ void inject_kernel(const double2* __restrict__ in, double2* __restrict__ out, RowMap mN, RowMap mM) {
  int k[3];
  size_t t;
  if (!row_k(mM, k[0], k[1], k[2], t)) return;
  const int h0 = (mN.N0 - 1) / 2, h1 = (mN.N1 - 1) / 2;
  double2 v = make_double2(0.0, 0.0);
  if (mN.d == 3) {
    if (abs(k[0]) <= h0 && abs(k[1]) <= h1 && k[2] < mN.H)
      v = in[((size_t)wrap(k[0], mN.N0) * mN.N1 + wrap(k[1], mN.N1)) * mN.H + k[2]];
  } else {
    if (abs(k[0]) <= h0 && k[1] < mN.H) v = in[(size_t)wrap(k[0], mN.N0) * mN.H + k[1]];
  }
  out[t] = v;
}

// over the half spectrum of g: the coefficient of the same frequency on gM
__global__ void project_kernel(const double2* __restrict__ in, double2* __restrict__ out, RowMap mN, RowMap mM) {
  int k[3];
  size_t t;
  if (!row_k(mN, k[0], k[1], k[2], t)) return;
  size_t tm;
  if (mN.d == 3)
    tm = ((size_t)wrap(k[0], mM.N0) * mM.N1 + wrap(k[1], mM.N1)) * mM.H + k[2];
  else
    tm = (size_t)wrap(k[0], mM.N0) * mM.H + k[1];
  out[t] = in[tm];
}

// s(m) = int over a cell of width 1/n of e^{2 pi i m t} dt = sin(pi m / n) / (pi m), 1/n at m = 0
__device__ __forceinline__ double cell_sinc(int m, int n) {
  if (m == 0) return 1.0 / n;
  const double x = 3.141592653589793238462643383279502884 * (double)m;
  return sin(x / (double)n) / x;
}

// X[m] = scale * (Phi a)(m mod N) * prod_a s(m_a) over the half spectrum of gM (Phi a from its half
// spectrum on g, by Hermitian symmetry where the last frequency wraps to a negative one)
__global__ void ga_spectrum_kernel(const double2* __restrict__ pa, double2* __restrict__ X, RowMap mN, RowMap mM,
                                   int NL, double scale) {
  int m[3];
  size_t t;
  if (!row_k(mM, m[0], m[1], m[2], t)) return;
  const int d = mN.d;
  // representatives in Z_N of m mod N, per axis
  const int n0 = mN.N0, n1 = d == 3 ? mN.N1 : NL, n2 = NL;
  int k0 = ((m[0] % n0) + n0) % n0;
  k0 = k0 <= (n0 - 1) / 2 ? k0 : k0 - n0;
  int k1 = ((m[1] % n1) + n1) % n1;
  k1 = k1 <= (n1 - 1) / 2 ? k1 : k1 - n1;
  int k2 = 0;
  if (d == 3) {
    k2 = ((m[2] % n2) + n2) % n2;
    k2 = k2 <= (n2 - 1) / 2 ? k2 : k2 - n2;
  }
  const int kl = d == 3 ? k2 : k1;  // last-axis frequency
  bool cj = false;
  if (kl < 0) {  // (Phi a)(k) = conj((Phi a)(-k)) for real a
    k0 = -k0;
    k1 = -k1;
    k2 = -k2;
    cj = true;
  }
  double2 v;
  if (d == 3)
    v = pa[((size_t)wrap(k0, n0) * mN.N1 + wrap(k1, mN.N1)) * mN.H + k2];
  else
    v = pa[(size_t)wrap(k0, n0) * mN.H + k1];
  if (cj) v.y = -v.y;
  double S = scale * cell_sinc(m[0], n0) * cell_sinc(m[1], n1);
  if (d == 3) S *= cell_sinc(m[2], n2);
  X[t] = make_double2(S * v.x, S * v.y);
}

void half_inject(lrfg_ctx* ctx, const FullGrid& g, const FullGrid& gM, const double2* in, double2* out) {
  LRFG_LAUNCH(ctx, KC_POINTWISE, 0.0, sizeof(double2) * (double)(g.n_half + gM.n_half),
              inject_kernel<<<row_grid(gM), row_block(gM), 0, ctx->stream>>>(in, out, rowmap(g), rowmap(gM)));
}

void half_project(lrfg_ctx* ctx, const FullGrid& g, const FullGrid& gM, const double2* in, double2* out) {
  LRFG_LAUNCH(ctx, KC_POINTWISE, 0.0, 2.0 * sizeof(double2) * (double)g.n_half,
              project_kernel<<<row_grid(g), row_block(g), 0, ctx->stream>>>(in, out, rowmap(g), rowmap(gM)));
}

void ga_coefficient(lrfg_ctx* ctx, const FullGrid& g, const FullGrid& gM, const double* a, double2* half_g,
                    double2* half_m, double* out) {
  full_forward<double>(ctx, g, a, nullptr, 1.0, half_g);  // Phi a on g
  const double scale = (double)g.n_real / ((double)gM.n_real * (double)gM.n_real);
  LRFG_LAUNCH(ctx, KC_POINTWISE, 20.0 * gM.n_half, sizeof(double2) * (double)(g.n_half + gM.n_half),
              ga_spectrum_kernel<<<row_grid(gM), row_block(gM), 0, ctx->stream>>>(half_g, half_m, rowmap(g), rowmap(gM),
                                                                                 g.N[g.d - 1], scale));
  full_inverse<double>(ctx, gM, half_m, nullptr, 1.0, out);  // (|N| / |M|^2) Phi*_M X
}

template <typename V>
void half_acc_aniso(lrfg_ctx* ctx, const FullGrid& g, const V* in, V* acc, const double* B, int precond) {
  using R = typename RealOf<V>::T;
  LRFG_REQUIRE(!precond || inv_table<R>(g), "reciprocal table missing");
  const double c = 4.0 * 9.869604401089358618834490999876;  // 4 pi^2
  LRFG_LAUNCH(ctx, KC_POINTWISE, 14.0 * g.n_half, 3.0 * sizeof(V) * g.n_half,
              acc_aniso_kernel<V><<<row_grid(g), row_block(g), 0, ctx->stream>>>(
                  in, acc, rowmap(g), sym_b<R>(B, c), precond, inv_table<R>(g)));
}

template <typename V>
void half_precond(lrfg_ctx* ctx, const FullGrid& g, const V* in, V* out) {
  using R = typename RealOf<V>::T;
  LRFG_REQUIRE(inv_table<R>(g), "reciprocal table missing");
  LRFG_LAUNCH(ctx, KC_POINTWISE, 2.0 * g.n_half, 2.0 * sizeof(V) * g.n_half,
              precond_kernel<V><<<row_grid(g), row_block(g), 0, ctx->stream>>>(in, out, rowmap(g), inv_table<R>(g)));
}

// ------------------------------------------------------------------------------------------------
// reductions: Hermitian-weighted inner product of half spectra, and the A_eff energy density.
// FP64 data accumulate in FP64.  FP32 data: each product is split exactly (p + e, e = fma(a, b, -p))
// and both parts are summed per thread with error-free two-sums (Knuth) in FP32, so the per-thread
// partial is accurate to ~n eps32^2 of the sum of magnitudes (FP64 class) while the work runs on the
// FP32 pipe; partials are combined in FP64.
// ------------------------------------------------------------------------------------------------
constexpr int kRedBlocks = 1216;  // 8 blocks per SM

__device__ __forceinline__ void two_sum_acc(float& s, float& c, float x) {
  const float t = s + x;
  const float bp = t - s;
  c += (s - (t - bp)) + (x - bp);
  s = t;
}

// weighted partial inner products of one thread (weight w = 1 or 2), see above
template <typename V>
struct DotAcc;
template <>
struct DotAcc<double2> {
  double s = 0.0;
  __device__ __forceinline__ void add(double2 a, double2 b, int kl) {
    s += (kl == 0 ? 1.0 : 2.0) * (a.x * b.x + a.y * b.y);
  }
  __device__ __forceinline__ double value() const { return s; }
};
template <>
struct DotAcc<float2> {
  float fs = 0.0f, fc = 0.0f;
  __device__ __forceinline__ void add(float2 a, float2 b, int kl) {
    const float w = kl == 0 ? 1.0f : 2.0f;
    const float p1 = a.x * b.x, e1 = fmaf(a.x, b.x, -p1);
    const float p2 = a.y * b.y, e2 = fmaf(a.y, b.y, -p2);
    two_sum_acc(fs, fc, w * p1);
    two_sum_acc(fs, fc, w * p2);
    fc += w * (e1 + e2);
  }
  __device__ __forceinline__ double value() const { return (double)fs + (double)fc; }
};

__device__ __forceinline__ double block_sum256(double s, double* red) {
  for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(0xffffffff, s, o);
  __syncthreads();
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
  __syncthreads();
  double v = 0.0;
  for (int i = 0; i < 8; ++i) v += red[i];
  return v;
}

// Stores this block's NV partial sums and returns true in the last block of the launch to arrive, whose every thread
// then holds the totals, summed in block order: the same bits whichever block arrives last.  The counter is zero
// between launches.  It replaces a second launch for the partials (8 us under event timing, three a CG step).
template <int NV>
__device__ bool last_block_sum(const double* mine, double* partial, unsigned int* counter, double* red, double* total) {
  __shared__ unsigned int s_last;
  if (threadIdx.x == 0) {
    for (int v = 0; v < NV; ++v) partial[(size_t)v * gridDim.x + blockIdx.x] = mine[v];
    __threadfence();
    s_last = atomicAdd(counter, 1u) == gridDim.x - 1u;
  }
  __syncthreads();
  if (!s_last) return false;
  __threadfence();
  for (int v = 0; v < NV; ++v) {
    double s = 0.0;
    for (unsigned int t = threadIdx.x; t < gridDim.x; t += 256) s += __ldcg(partial + (size_t)v * gridDim.x + t);
    total[v] = block_sum256(s, red);
  }
  if (threadIdx.x == 0) *counter = 0u;
  return true;
}

// *out = <x, y>; then, if ratio, *ratio = *aux / *out (0 when the divisor is 0): the PCG step length, formed once on the
// device
template <typename V>
__global__ void __launch_bounds__(256) half_dot_kernel(const V* __restrict__ x, const V* __restrict__ y, long long n,
                                                       int H, double* partial, unsigned int* counter, double* out,
                                                       const double* aux, double* ratio) {
  __shared__ double red[8];
  constexpr int kU = 4;  // elements' loads in flight before any is used
  DotAcc<V> acc;
  const long long stride = (long long)gridDim.x * blockDim.x;
  long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  int kl = (int)(t % H);
  const int kstep = (int)(stride % H);
  for (; t < n; t += kU * stride) {
    V a[kU], b[kU];
#pragma unroll
    for (int u = 0; u < kU; ++u) {
      const long long tu = t + u * stride;
      a[u] = tu < n ? x[tu] : mkc<V>(0, 0);
      b[u] = tu < n ? y[tu] : mkc<V>(0, 0);
    }
#pragma unroll
    for (int u = 0; u < kU; ++u) {
      acc.add(a[u], b[u], kl);
      kl += kstep;
      if (kl >= H) kl -= H;
    }
  }
  double mine[1] = {block_sum256(acc.value(), red)}, total[1];
  if (!last_block_sum<1>(mine, partial, counter, red, total)) return;
  if (threadIdx.x == 0) {
    *out = total[0];
    if (ratio) *ratio = total[0] != 0.0 ? *aux / total[0] : 0.0;
  }
}

template <typename R>
__global__ void __launch_bounds__(256) energy_kernel(const R* __restrict__ e, const R* __restrict__ a, double E,
                                                     long long n, double* partial) {
  __shared__ double red[8];
  double s = 0.0;
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < n; t += (long long)gridDim.x * blockDim.x) {
    double f = E + (double)e[t];
    s += (double)a[t] * f * f;
  }
  for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(0xffffffff, s, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    double v = 0.0;
    for (int i = 0; i < 8; ++i) v += red[i];
    partial[blockIdx.x] = v;
  }
}

// sum over the full spectrum of (k.B k) |v_k|^2 (B pre-scaled), from the half spectrum with weights 1 / 2
__global__ void __launch_bounds__(256) aniso_energy_kernel(const double2* __restrict__ v, long long n, int H, int d,
                                                           int N0, int N1, SymB<double> sb, double* partial) {
  __shared__ double red[8];
  double s = 0.0;
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < n; t += (long long)gridDim.x * blockDim.x) {
    const long long row = t / H;
    const int kl = (int)(t - row * H);
    int k0, k1, k2;
    if (d == 3) {
      const int i0 = (int)(row / N1), i1 = (int)(row - (long long)i0 * N1);
      k0 = freq_of(i0, N0);
      k1 = freq_of(i1, N1);
      k2 = kl;
    } else {
      k0 = freq_of((int)row, N0);
      k1 = kl;
      k2 = 0;
    }
    const double2 x = v[t];
    const double w = kl == 0 ? 1.0 : 2.0;
    s += w * quad_b(sb, k0, k1, k2) * (x.x * x.x + x.y * x.y);
  }
  for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(0xffffffff, s, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    double r = 0.0;
    for (int i = 0; i < 8; ++i) r += red[i];
    partial[blockIdx.x] = r;
  }
}

// *out (+)= sum of partials
__global__ void finish_sum_kernel(const double* __restrict__ partial, int n, double* out, int accumulate) {
  __shared__ double red[8];
  double s = 0.0;
  for (int t = threadIdx.x; t < n; t += blockDim.x) s += partial[t];
  const double v = block_sum256(s, red);
  if (threadIdx.x == 0) *out = accumulate ? *out + v : v;
}

// blocks of a reduction over n elements: four elements a thread, at most eight blocks per SM
static int red_blocks(long long n) { return (int)std::max(1LL, std::min<long long>(kRedBlocks, (n + 1023) / 1024)); }

template <typename V>
void half_dot(lrfg_ctx* ctx, const FullGrid& g, const V* x, const V* y, double* out_dev, const double* aux,
              double* ratio) {
  const int blocks = red_blocks(g.n_half);
  DBuf<double> partial(ctx->pool, kRedBlocks);
  LRFG_LAUNCH(ctx, KC_REDUCE, 4.0 * g.n_half, 2.0 * sizeof(V) * g.n_half,
              half_dot_kernel<V><<<blocks, 256, 0, ctx->stream>>>(x, y, g.n_half, g.H, partial.get(), ctx->splitk_cnt,
                                                                 out_dev, aux, ratio));
}

void aniso_energy_sum(lrfg_ctx* ctx, const FullGrid& g, const double2* v, const double* B, double* out_dev,
                      int accumulate) {
  DBuf<double> partial(ctx->pool, kRedBlocks);
  const double c = 4.0 * 9.869604401089358618834490999876 / (double)g.n_real;  // 4 pi^2 / |N|
  LRFG_LAUNCH(ctx, KC_REDUCE, 16.0 * g.n_half, sizeof(double2) * (double)g.n_half,
              aniso_energy_kernel<<<kRedBlocks, 256, 0, ctx->stream>>>(v, g.n_half, g.H, g.d, g.N[0],
                                                                         g.d == 3 ? g.N[1] : 1, sym_b<double>(B, c),
                                                                         partial.get()));
  LRFG_LAUNCH(ctx, KC_REDUCE, kRedBlocks, kRedBlocks * sizeof(double),
              finish_sum_kernel<<<1, 256, 0, ctx->stream>>>(partial.get(), kRedBlocks, out_dev, accumulate));
}

template <typename R>
void energy_sum(lrfg_ctx* ctx, const FullGrid& g, const R* e, const R* a, double E, double* out_dev, int accumulate) {
  DBuf<double> partial(ctx->pool, kRedBlocks);
  LRFG_LAUNCH(ctx, KC_REDUCE, 4.0 * g.n_real, 2.0 * sizeof(R) * g.n_real,
              energy_kernel<R><<<kRedBlocks, 256, 0, ctx->stream>>>(e, a, E, g.n_real, partial.get()));
  LRFG_LAUNCH(ctx, KC_REDUCE, kRedBlocks, kRedBlocks * sizeof(double),
              finish_sum_kernel<<<1, 256, 0, ctx->stream>>>(partial.get(), kRedBlocks, out_dev, accumulate));
}

// ------------------------------------------------------------------------------------------------
// PCG vector updates with device FP64 step lengths (rounded once to R).  Two passes a step, both bound by memory:
//   residual   r -= alpha q, and the inner products <z, z> and <r, z> of z = P^-1 r, which is not stored (its multiplier
//              costs one reciprocal per element); the last block forms beta;
//   direction  u += alpha p and p = P^-1 r + beta p.
// 10 vector transfers a step with the product <p, q> (2 + 3 + 5) where separate updates, products and directions took
// 15; on 243^3 in FP32 the vector part of a step went from 0.186 to 0.133 ms (the products' error-free sums bound the rest).
// ------------------------------------------------------------------------------------------------
// 1/(k.k): FP32 forms the correctly rounded reciprocal (the value of the table) without the table's scattered gather
__device__ __forceinline__ float inv_kk_of(const float*, int kk) { return kk ? __frcp_rn((float)kk) : 0.f; }
__device__ __forceinline__ double inv_kk_of(const double* t, int kk) { return t[kk]; }

// frequencies of consecutive elements of a strided walk over the half spectrum, without a division per element
struct FreqWalk {
  int kl, i0, i1, H, N0, N1, dkl, d0, d1, d;
  __device__ FreqWalk(const RowMap& m, long long t, long long stride) : H(m.H), N0(m.N0), N1(m.N1), d(m.d) {
    long long row = t / H;
    kl = (int)(t - row * H);
    i0 = (int)(row / N1);
    i1 = (int)(row - (long long)i0 * N1);
    row = stride / H;
    dkl = (int)(stride - row * H);
    d0 = (int)(row / N1);
    d1 = (int)(row - (long long)d0 * N1);
  }
  __device__ __forceinline__ int kk() const {
    const int k0 = freq_of(i0, N0), k1 = d == 3 ? freq_of(i1, N1) : 0;
    return k0 * k0 + k1 * k1 + kl * kl;
  }
  __device__ __forceinline__ void next() {
    kl += dkl;
    i1 += d1;
    i0 += d0;
    if (kl >= H) { kl -= H; ++i1; }
    if (i1 >= N1) { i1 -= N1; ++i0; }
  }
};

template <typename V>
__global__ void __launch_bounds__(256) pcg_residual_kernel(V* r, const V* __restrict__ q, long long n, RowMap m,
                                                           const double* __restrict__ alpha_dev,
                                                           const typename RealOf<V>::T* __restrict__ inv_kk,
                                                           double* partial, unsigned int* counter, double* rz,
                                                           double* zz, double* beta) {
  using R = typename RealOf<V>::T;
  __shared__ double red[8];
  constexpr int kU = 4;
  const R alpha = (R)(*alpha_dev);
  DotAcc<V> azz, arz;
  const long long stride = (long long)gridDim.x * blockDim.x;
  long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  FreqWalk w(m, t, stride);
  for (; t < n; t += kU * stride) {
    V rv[kU], qv[kU];
#pragma unroll
    for (int u = 0; u < kU; ++u) {
      const long long tu = t + u * stride;
      rv[u] = tu < n ? r[tu] : mkc<V>(0, 0);
      qv[u] = tu < n ? q[tu] : mkc<V>(0, 0);
    }
#pragma unroll
    for (int u = 0; u < kU; ++u) {
      const long long tu = t + u * stride;
      if (tu < n) {
        rv[u].x -= alpha * qv[u].x;
        rv[u].y -= alpha * qv[u].y;
        r[tu] = rv[u];
        const R s = inv_kk_of(inv_kk, w.kk());
        const V z = mkc<V>(rv[u].x * s, rv[u].y * s);
        azz.add(z, z, w.kl);
        arz.add(rv[u], z, w.kl);
      }
      w.next();
    }
  }
  double mine[2], total[2];
  mine[0] = block_sum256(azz.value(), red);
  mine[1] = block_sum256(arz.value(), red);
  if (!last_block_sum<2>(mine, partial, counter, red, total)) return;
  if (threadIdx.x == 0) {
    *zz = total[0];
    *beta = *rz != 0.0 ? total[1] / *rz : 0.0;
    *rz = total[1];
  }
}

// u += alpha p, then (unless `last`) p = P^-1 r + beta p
template <typename V>
__global__ void __launch_bounds__(256) pcg_direction_kernel(V* u, V* p, const V* __restrict__ r, long long n, RowMap m,
                                                            const double* __restrict__ alpha_dev,
                                                            const double* __restrict__ beta_dev,
                                                            const typename RealOf<V>::T* __restrict__ inv_kk, int last) {
  using R = typename RealOf<V>::T;
  constexpr int kU = 2;
  const R alpha = (R)(*alpha_dev), beta = last ? R(0) : (R)(*beta_dev);
  const long long stride = (long long)gridDim.x * blockDim.x;
  long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  FreqWalk w(m, t, stride);
  for (; t < n; t += kU * stride) {
    V uv[kU], pv[kU], rv[kU];
#pragma unroll
    for (int v = 0; v < kU; ++v) {
      const long long tu = t + v * stride;
      uv[v] = tu < n ? u[tu] : mkc<V>(0, 0);
      pv[v] = tu < n ? p[tu] : mkc<V>(0, 0);
      rv[v] = tu < n && !last ? r[tu] : mkc<V>(0, 0);
    }
#pragma unroll
    for (int v = 0; v < kU; ++v) {
      const long long tu = t + v * stride;
      if (tu < n) {
        uv[v].x += alpha * pv[v].x;
        uv[v].y += alpha * pv[v].y;
        u[tu] = uv[v];
        if (!last) {
          const R s = inv_kk_of(inv_kk, w.kk());
          p[tu] = mkc<V>(rv[v].x * s + beta * pv[v].x, rv[v].y * s + beta * pv[v].y);
        }
      }
      w.next();
    }
  }
}

template <typename V>
void pcg_residual(lrfg_ctx* ctx, const FullGrid& g, V* r, const V* q, const double* alpha, double* rz, double* zz,
                  double* beta) {
  using R = typename RealOf<V>::T;
  LRFG_REQUIRE(inv_table<R>(g), "reciprocal table missing");
  const int blocks = red_blocks(g.n_half);
  DBuf<double> partial(ctx->pool, 2 * kRedBlocks);
  LRFG_LAUNCH(ctx, KC_POINTWISE, 14.0 * g.n_half, 3.0 * sizeof(V) * g.n_half,
              pcg_residual_kernel<V><<<blocks, 256, 0, ctx->stream>>>(r, q, g.n_half, rowmap(g), alpha, inv_table<R>(g),
                                                                     partial.get(), ctx->splitk_cnt, rz, zz, beta));
}

template <typename V>
void pcg_direction(lrfg_ctx* ctx, const FullGrid& g, V* u, V* p, const V* r, const double* alpha, const double* beta,
                   bool last) {
  using R = typename RealOf<V>::T;
  LRFG_REQUIRE(inv_table<R>(g), "reciprocal table missing");
  const long long cap = 16LL * (ctx->num_sms > 0 ? ctx->num_sms : 152);
  const unsigned blocks = (unsigned)std::max(1LL, std::min<long long>(cap, (g.n_half + 511) / 512));
  LRFG_LAUNCH(ctx, KC_POINTWISE, (last ? 4.0 : 10.0) * g.n_half, (last ? 3.0 : 5.0) * sizeof(V) * g.n_half,
              pcg_direction_kernel<V><<<blocks, 256, 0, ctx->stream>>>(u, p, r, g.n_half, rowmap(g), alpha, beta,
                                                                      inv_table<R>(g), last ? 1 : 0));
}

// element-wise conversions between storage precisions (round to nearest)
__device__ __forceinline__ float cvt(double x, float*) { return (float)x; }
__device__ __forceinline__ double cvt(float x, double*) { return (double)x; }
__device__ __forceinline__ float2 cvt(double2 x, float2*) { return make_float2((float)x.x, (float)x.y); }
__device__ __forceinline__ double2 cvt(float2 x, double2*) { return make_double2((double)x.x, (double)x.y); }

template <typename A, typename B>
__global__ void convert_kernel(const A* __restrict__ in, B* out, long long n) {
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < n; t += (long long)gridDim.x * blockDim.x)
    out[t] = cvt(in[t], (B*)nullptr);
}

template <typename A, typename B>
void convert(lrfg_ctx* ctx, const A* in, B* out, long long n) {
  if (n <= 0) return;
  LRFG_LAUNCH(ctx, KC_POINTWISE, 0, (sizeof(A) + sizeof(B)) * (double)n,
              convert_kernel<A, B><<<grid1d(ctx, n), 256, 0, ctx->stream>>>(in, out, n));
}

#define LRFG_FULL_INSTANTIATE(V, R)                                                                         \
  template void half_mul_grad<V>(lrfg_ctx*, const FullGrid&, const V*, V*, int, double);                  \
  template void half_acc_div<V>(lrfg_ctx*, const FullGrid&, const V*, V*, int, double, int, int);         \
  template void half_precond<V>(lrfg_ctx*, const FullGrid&, const V*, V*);                                \
  template void half_acc_aniso<V>(lrfg_ctx*, const FullGrid&, const V*, V*, const double*, int);          \
  template void half_dot<V>(lrfg_ctx*, const FullGrid&, const V*, const V*, double*, const double*, double*); \
  template void energy_sum<R>(lrfg_ctx*, const FullGrid&, const R*, const R*, double, double*, int);      \
  template void pcg_residual<V>(lrfg_ctx*, const FullGrid&, V*, const V*, const double*, double*, double*, double*); \
  template void pcg_direction<V>(lrfg_ctx*, const FullGrid&, V*, V*, const V*, const double*, const double*, bool);
LRFG_FULL_INSTANTIATE(double2, double)
LRFG_FULL_INSTANTIATE(float2, float)
template void convert<double, float>(lrfg_ctx*, const double*, float*, long long);
template void convert<float, double>(lrfg_ctx*, const float*, double*, long long);
template void convert<double2, float2>(lrfg_ctx*, const double2*, float2*, long long);
template void convert<float2, double2>(lrfg_ctx*, const float2*, double2*, long long);

}  // namespace lrfg
