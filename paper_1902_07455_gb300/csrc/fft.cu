// Mode-wise batched FFTs of fibres (hot-path rows a1 and a2): complex fibres, and real fibres under a
// Fourier multiplier F^{-1} diag(m) F (gradient 2 pi i k, Gaussian exp(-t k^2)).
//
// A fibre is (o, :, i) of an (outer, N, inner) array; a block stages TF whole fibres in shared memory
// with coalesced loads (consecutive threads take consecutive inner indices when inner >= TF, else
// consecutive elements of one fibre), runs the Stockham passes there, and writes back the same way.
// Real fibres are packed two per complex row (x + i y): a real-symmetric multiplier maps it to
// Mx + i My, so one complex transform pair serves two real fibres.
#include <cmath>
#include <type_traits>

#include "ops.cuh"

namespace lrfg {

FftPlan make_plan(int N, int max_radix) {
  FftPlan pl{};
  pl.N = N;
  pl.nst = 0;
  int n = N;
  // register radices first (27, 9 as allowed), then 5, 7, 3, then the remaining primes (generic passes);
  // the order of the passes does not change the transform
  const int pref[] = {27, 9, 5, 7, 3};
  for (int p : pref) {
    if (p > max_radix && p > 7) continue;  // (limits the composite radices)
    while (n % p == 0) {
      if (pl.nst >= kMaxStages) fail(LRFG_ENOTSUP, "grid size %d has too many factors", N);
      pl.radix[pl.nst++] = p;
      n /= p;
    }
  }
  for (int p = 11; n > 1; p += 2) {
    while (n % p == 0) {
      if (p > kMaxGenericRadix) fail(LRFG_ENOTSUP, "grid size %d has a prime factor %d > %d", N, p, kMaxGenericRadix);
      if (pl.nst >= kMaxStages) fail(LRFG_ENOTSUP, "grid size %d has too many factors", N);
      pl.radix[pl.nst++] = p;
      n /= p;
    }
  }
  return pl;
}

const Twiddles& twiddles_for(lrfg_ctx* ctx, int N) {
  LRFG_CUDA(ensure_roots(ctx->device));
  auto it = ctx->twiddles.find(N);
  if (it != ctx->twiddles.end()) return it->second;
  std::vector<int4> h(N);
  for (int j = 0; j < N; ++j) h[j] = fixed_root(j, N);
  Twiddles t;
  t.N = N;
  LRFG_CUDA(cudaMalloc(&t.W, sizeof(int4) * N));
  // on the context's stream (ordered before its kernels, also when that stream is non-blocking)
  LRFG_CUDA(cudaMemcpyAsync(t.W, h.data(), sizeof(int4) * N, cudaMemcpyHostToDevice, ctx->stream));
  LRFG_CUDA(cudaStreamSynchronize(ctx->stream));
  return ctx->twiddles.emplace(N, t).first->second;
}

template <>
const int4* twiddle_table<double>(lrfg_ctx* ctx, int N) {
  return twiddles_for(ctx, N).W;
}

template <>
const float2* twiddle_table<float>(lrfg_ctx* ctx, int N) {
  Twiddles& t = const_cast<Twiddles&>(twiddles_for(ctx, N));
  if (!t.Wf) {
    std::vector<float2> h(N);
    const double two_pi = 6.283185307179586476925286766559;
    for (int j = 0; j < N; ++j) {
      double ang = two_pi * (double)j / (double)N;
      h[j] = make_float2((float)std::cos(ang), (float)-std::sin(ang));
    }
    LRFG_CUDA(cudaMalloc(&t.Wf, sizeof(float2) * N));
    LRFG_CUDA(cudaMemcpyAsync(t.Wf, h.data(), sizeof(float2) * N, cudaMemcpyHostToDevice, ctx->stream));
    LRFG_CUDA(cudaStreamSynchronize(ctx->stream));
  }
  return t.Wf;
}

// rows of a real-fibre tile that fit in shared memory: N twiddles and `fixed` further tables of N, `per` buffers of N
// for each row
static int tile_fibres(lrfg_ctx* ctx, int N, size_t elem, int fixed, int per) {
  size_t limit = 100 * 1024;
  if (N > 300) limit = (size_t)std::min(ctx->max_smem_optin, 200 * 1024);
  const long long row = (long long)N * (long long)elem;
  return (int)std::max(1LL, std::min(64LL, ((long long)limit - (1 + fixed) * row) / (per * row)));
}

// ----------------------------------------------------------------------------------------------------
// complex fibres
// ----------------------------------------------------------------------------------------------------
// the two frequencies (ka, kb) that are constant on fibre (o, i), in the order of their axes
template <typename R>
__device__ __forceinline__ void fibre_freqs(const FibreMul<R>& fm, long long o, long long i, int& ka, int& kb) {
  if (fm.axis == 1) {
    ka = freq_of((int)o, fm.N0);
    kb = (int)i;
  } else if (fm.d == 3) {
    const int i1 = (int)(i / fm.H);
    ka = freq_of(i1, fm.N1);
    kb = (int)(i - (long long)i1 * fm.H);
  } else {
    ka = (int)i;
    kb = 0;
  }
}

// frequency k_alpha of an element: kn along the fibre, (ka, kb) constant on it
template <typename R>
__device__ __forceinline__ int freq_alpha(const FibreMul<R>& fm, int kn, int ka, int kb) {
  return fm.alpha == fm.axis ? kn : (fm.alpha == (fm.axis == 0 ? 1 : 0) ? ka : kb);
}

// v * (2 pi i k) * scale, f = c2 k
template <typename V>
__device__ __forceinline__ V times_2pi_ik(V v, typename RealOf<V>::T f) {
  return mkc<V>(-v.y * f, v.x * f);
}

// mode 2 of FibreMul: the divergence term of element kn of a fibre accumulated into *dst
template <typename V>
__device__ __forceinline__ void acc_div_store(const FibreMul<typename RealOf<V>::T>& fm, V* dst, V x, int kn, int ka,
                                              int kb) {
  using R = typename RealOf<V>::T;
  V r = fm.alpha < 0 ? x : times_2pi_ik<V>(x, -fm.c2 * (R)freq_alpha(fm, kn, ka, kb));
  if (!fm.init) {
    const V o = *dst;
    r.x += o.x;
    r.y += o.y;
  }
  if (fm.precond) {
    const R s = fm.inv_kk[kn * kn + ka * ka + kb * kb];
    r.x *= s;
    r.y *= s;
  }
  *dst = r;
}

// index in a spectrum of length m of the frequency stored at index n of one of length N, -1 where it has none
__device__ __forceinline__ int same_freq(int n, int N, int m) {
  const int f = freq_of(n, N);
  return abs(f) > (m - 1) / 2 ? -1 : (f < 0 ? f + m : f);
}

// OP 0: plain transform; OP 1 and 2: the modes of FibreMul.  PAD: the input holds nin <= N frequencies of a fibre, the
// others are zero, or the output keeps nout <= N of them (the double grid of the exact integration)
template <int SIGN, typename V, int OP, bool PAD>
__global__ void __launch_bounds__(256, 3) fft_fibres_kernel(const V* in, V* out, long long outer, int N, long long inner,
                                                         int TF, FftPlan pl, const typename TwOf<V>::T* __restrict__ Wg,
                                                         FibreMul<typename RealOf<V>::T> fm, int nin,
                                                         int nout) {
  using R = typename RealOf<V>::T;
  extern __shared__ __align__(16) unsigned char smraw_fib[];
  V* sm = (V*)smraw_fib;
  auto* W = reinterpret_cast<typename TwOf<V>::T*>(sm);
  V* a = sm + 2 * N;
  V* b = a + (size_t)TF * N;
  const long long nfib = outer * inner;
  const long long g0 = (long long)blockIdx.x * TF;
  const int nf = (int)min((long long)TF, nfib - g0);
  const int total = nf * N;
  const bool across = inner >= TF;
  if (across) {
    // thread -> one fibre f of the tile and every step-th element of it: neighbouring threads take
    // neighbouring fibres (contiguous addresses); all index division happens once per thread
    const int step = blockDim.x / nf;
    const int f = threadIdx.x % nf, n0 = threadIdx.x / nf;
    const long long g = g0 + f;
    const long long o = g / inner, i = g - o * inner;
    const V* src = in + (size_t)o * (PAD ? nin : N) * (size_t)inner + (size_t)i;
    if (n0 < step)
      for (int n = n0; n < N; n += step) {
        const int m = PAD ? same_freq(n, N, nin) : n;
        if (m >= 0) cp_async<sizeof(V)>(a + (size_t)f * N + n, src + (size_t)m * inner);
        else a[(size_t)f * N + n] = mkc<V>(0, 0);
      }
  } else {
    for (int t = threadIdx.x; t < total; t += blockDim.x) {
      const int f = small_div(t, N, 1.0f / (float)N), n = t - f * N;
      const long long g = g0 + f;
      const long long o = g / inner, i = g - o * inner;
      const int m = PAD ? same_freq(n, N, nin) : n;
      if (m >= 0) cp_async<sizeof(V)>(a + t, in + ((size_t)o * (PAD ? nin : N) + m) * (size_t)inner + (size_t)i);
      else a[t] = mkc<V>(0, 0);
    }
  }
  for (int j = threadIdx.x; j < N; j += blockDim.x) W[j] = Wg[j];
  cp_async_wait_all();
  if constexpr (OP == 1) {
    // each thread scales the elements it copied itself (its own copies are complete after the wait)
    if (across) {
      const int step = blockDim.x / nf;
      const int f = threadIdx.x % nf, n0 = threadIdx.x / nf;
      const long long o = (g0 + f) / inner;
      int ka, kb;
      fibre_freqs(fm, o, g0 + f - o * inner, ka, kb);
      if (n0 < step)
        for (int n = n0; n < N; n += step) {
          V* p = a + (size_t)f * N + n;
          *p = times_2pi_ik<V>(*p, fm.c2 * (R)freq_alpha(fm, freq_of(n, N), ka, kb));
        }
    } else {
      for (int t = threadIdx.x; t < total; t += blockDim.x) {
        const int f = small_div(t, N, 1.0f / (float)N), n = t - f * N;
        const long long o = (g0 + f) / inner;
        int ka, kb;
        fibre_freqs(fm, o, g0 + f - o * inner, ka, kb);
        a[t] = times_2pi_ik<V>(a[t], fm.c2 * (R)freq_alpha(fm, freq_of(n, N), ka, kb));
      }
    }
  }
  __syncthreads();
  V* res = stockham_rows<SIGN>(a, b, nf, N, pl, W);
  if (across) {
    const int step = blockDim.x / nf;
    const int f = threadIdx.x % nf, n0 = threadIdx.x / nf;
    const long long g = g0 + f;
    const long long o = g / inner, i = g - o * inner;
    const int no = PAD ? nout : N;
    V* dst = out + (size_t)o * no * (size_t)inner + (size_t)i;
    const V* row = res + (size_t)f * N;
    if constexpr (OP == 2) {
      int ka, kb;
      fibre_freqs(fm, o, i, ka, kb);
      if (n0 < step)
        for (int n = n0; n < no; n += step)
          acc_div_store<V>(fm, dst + (size_t)n * inner, row[PAD ? same_freq(n, no, N) : n], freq_of(n, no), ka, kb);
    } else {
      if (n0 < step)
        for (int n = n0; n < no; n += step) dst[(size_t)n * inner] = row[PAD ? same_freq(n, no, N) : n];
    }
  } else {
    const int no = PAD ? nout : N;
    for (int t = threadIdx.x; t < nf * no; t += blockDim.x) {
      const int f = small_div(t, no, 1.0f / (float)no), n = t - f * no;
      const long long g = g0 + f;
      const long long o = g / inner, i = g - o * inner;
      V* dst = out + ((size_t)o * no + n) * (size_t)inner + (size_t)i;
      const V value = res[(size_t)f * N + (PAD ? same_freq(n, no, N) : n)];
      if constexpr (OP == 2) {
        int ka, kb;
        fibre_freqs(fm, o, i, ka, kb);
        acc_div_store<V>(fm, dst, value, freq_of(n, no), ka, kb);
      } else {
        *dst = value;
      }
    }
  }
}

// ----------------------------------------------------------------------------------------------------
// FP32 complex fibres of length N = P1 P2 in two register passes with one trip through shared memory.
// A block takes 32 consecutive fibres, lane = fibre, so every global access of a warp touches 32
// neighbouring inner indices.  The two Stockham stages of the header of fft_device.cuh, written out:
//  pass 1 (radix P1, L = 1; warp w = c < P2): x[c + P2 r], r < P1, loaded straight from global memory,
//         a P1-point DFT in registers, Z[c P1 + q] (q < P1) to shared memory;
//  pass 2 (radix P2, L = P1; f = w, w + P2, ... < P1): Z[r P1 + f] (r < P2) times w_N^{f r}, a P2-point
//         DFT, X[f + P1 q] (q < P2) stored straight to global memory.
// Against the staged kernel this saves the staging round trips through shared memory, one of its
// two buffers and the per-butterfly index arithmetic.  A block reads all of its fibres before it
// writes any, and fibres belong to one block, so in == out is allowed.  OP as in fft_fibres_kernel.
// ----------------------------------------------------------------------------------------------------
// three blocks per SM where their shared memory fits
template <int P1, int P2, int OP>
constexpr int fft2_min_blocks() {
  return P1 * P2 * 32 * 8 * 3 <= 200 * 1024 ? 3 : 2;
}

template <int SIGN, int P1, int P2, int OP>
__global__ void __launch_bounds__(32 * P2, fft2_min_blocks<P1, P2, OP>()) fft2_fibres_kernel(
    const float2* in, float2* out, long long outer, long long inner, const float2* __restrict__ Wg, FibreMul<float> fm) {
  static_assert(P1 % P2 == 0, "pass 2 takes P1 / P2 butterflies per warp");
  constexpr int N = P1 * P2;
  extern __shared__ __align__(16) unsigned char smraw_fib2[];
  float2* Z = (float2*)smraw_fib2;  // [N][32]
  float2* W = Z + N * 32;           // w_N^j, j < N
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const long long g = (long long)blockIdx.x * 32 + lane;
  const bool valid = g < outer * inner;
  long long o = 0, i = 0;
  if (valid) {
    o = g / inner;
    i = g - o * inner;
  }
  int ka = 0, kb = 0;
  if constexpr (OP != 0) fibre_freqs(fm, o, i, ka, kb);
  const size_t base = (size_t)o * N * (size_t)inner + (size_t)i;
  for (int j = threadIdx.x; j < N; j += blockDim.x) W[j] = Wg[j];

  float2 x[P1];
#pragma unroll
  for (int r = 0; r < P1; ++r) x[r] = valid ? in[base + (size_t)(w + P2 * r) * (size_t)inner] : make_float2(0.f, 0.f);
  if constexpr (OP == 1) {
    // k of the fibre's own axis varies along it: multiply before the transform; the others are constant on it and
    // the product commutes with the transform, so it is taken after pass 2 (fewer live registers)
    if (fm.alpha == fm.axis) {
#pragma unroll
      for (int r = 0; r < P1; ++r) x[r] = times_2pi_ik<float2>(x[r], fm.c2 * (float)freq_of(w + P2 * r, N));
    }
  }
  RegDFT<P1, SIGN, float2>::run(x);
#pragma unroll
  for (int q = 0; q < P1; ++q) Z[(w * P1 + q) * 32 + lane] = x[q];
  __syncthreads();

#pragma unroll
  for (int jb = 0; jb < P1 / P2; ++jb) {
    const int f = w + P2 * jb;
    float2 y[P2], prev[P2];
    if constexpr (OP == 2) {
      // the accumulator's old values, all requested before the transform so that their latencies overlap
#pragma unroll
      for (int q = 0; q < P2; ++q)
        prev[q] = valid && !fm.init ? out[base + (size_t)(f + P1 * q) * (size_t)inner] : make_float2(0.f, 0.f);
    }
#pragma unroll
    for (int r = 0; r < P2; ++r) {
      y[r] = Z[(r * P1 + f) * 32 + lane];
      if (r) y[r] = cmul(y[r], tw<SIGN>((const float2*)W, f * r));
    }
    RegDFT<P2, SIGN, float2>::run(y);
    if (valid) {
#pragma unroll
      for (int q = 0; q < P2; ++q) {
        const int n = f + P1 * q;
        float2* dst = out + base + (size_t)n * (size_t)inner;
        if constexpr (OP == 2) {
          const int kn = freq_of(n, N);
          float2 r = fm.alpha < 0 ? y[q] : times_2pi_ik<float2>(y[q], -fm.c2 * (float)freq_alpha(fm, kn, ka, kb));
          if (!fm.init) {
            r.x += prev[q].x;
            r.y += prev[q].y;
          }
          if (fm.precond) {
            // the correctly rounded reciprocal, the value the table holds, without its scattered gather
            const int kk = kn * kn + ka * ka + kb * kb;
            const float sc = kk ? __frcp_rn((float)kk) : 0.f;
            r.x *= sc;
            r.y *= sc;
          }
          *dst = r;
        } else if constexpr (OP == 1) {
          *dst = fm.alpha == fm.axis ? y[q] : times_2pi_ik<float2>(y[q], fm.c2 * (float)freq_alpha(fm, 0, ka, kb));
        } else {
          *dst = y[q];
        }
      }
    }
  }
}

// N = P1 P2 served by fft2_fibres_kernel (FP32), else 0
static int fft2_split(int N) {
  if (N == 243) return 27;
  if (N == 81) return 9;
  return 0;
}

template <int SIGN, int P1, int P2, int OP>
static void fft2_launch(lrfg_ctx* ctx, const float2* in, float2* out, long long outer, long long inner,
                        const FibreMul<float>& fm, double flops, double bytes) {
  constexpr int N = P1 * P2;
  const size_t smem = sizeof(float2) * (size_t)N * 33;
  const long long blocks = (outer * inner + 31) / 32;
  LRFG_REQUIRE(blocks < (1LL << 31), "too many fibres");
  const float2* W = twiddle_table<float>(ctx, N);
  LRFG_CUDA(raise_smem_limit((const void*)fft2_fibres_kernel<SIGN, P1, P2, OP>, smem));
  LRFG_LAUNCH(ctx, KC_FFT_FIBRES, flops, bytes,
              fft2_fibres_kernel<SIGN, P1, P2, OP><<<(unsigned)blocks, 32 * P2, smem, ctx->stream>>>(in, out, outer,
                                                                                                 inner, W, fm));
}

template <int SIGN, int OP>
static bool fft2_dispatch(lrfg_ctx* ctx, const float2* in, float2* out, long long outer, int N, long long inner,
                          const FibreMul<float>& fm, double flops, double bytes) {
  switch (fft2_split(N)) {
    case 27: fft2_launch<SIGN, 27, 9, OP>(ctx, in, out, outer, inner, fm, flops, bytes); return true;
    case 9: fft2_launch<SIGN, 9, 9, OP>(ctx, in, out, outer, inner, fm, flops, bytes); return true;
    default: return false;
  }
}

template <typename V, int SIGN, int OP>
static bool fft2_try(lrfg_ctx* ctx, const V* in, V* out, long long outer, int N, long long inner,
                     const FibreMul<typename RealOf<V>::T>& fm, double flops, double bytes) {
  if constexpr (sizeof(V) == sizeof(float2)) {
    return fft2_dispatch<SIGN, OP>(ctx, (const float2*)in, (float2*)out, outer, N, inner, fm, flops, bytes);
  } else {
    return false;
  }
}

// instructions of a radix-p butterfly in fixed point with its twiddles
static double butterfly_ops(int p) {
  switch (p) {
    case 3: return 150.0;
    case 5: return 400.0;
    case 7: return 750.0;
    case 9: return 800.0;
    default: return 20.0 * (double)(p - 1) * (p - 1) + 60.0 * p;
  }
}

// Cycles of one transform of tf rows in each of `blocks` blocks on the SM with the most of them: a pass takes the
// instructions of the warps on the busiest of the SM's four schedulers, or those of one warp at its latency where there
// are few, and a barrier; the conversions count as another pass.
double fft_cycles(lrfg_ctx* ctx, const FftPlan& pl, long long tf, long long blocks) {
  const long long nsm = ctx->num_sms > 0 ? ctx->num_sms : 152;
  const long long per_sm = (blocks + nsm - 1) / nsm;
  auto pass = [&](long long threads, double ops) {
    const long long warps = per_sm * ((threads + 31) / 32);
    return std::max((double)((warps + 3) / 4) * ops * 1.5, (double)(((threads + 255) / 256)) * ops * 3.0) + 200.0;
  };
  double c = pass(tf * pl.N, 120.0);
  for (int s = 0; s < pl.nst; ++s) c += pass(tf * (pl.N / pl.radix[s]), butterfly_ops(pl.radix[s]));
  return c;
}

// the context's earlier choice for a launch shape (tf = 0: none yet); the table is emptied when it has grown to 4096
static FftChoice& fft_choice(lrfg_ctx* ctx, int N, int kind, long long nrows, int extra) {
  auto& m = ctx->fft_choices;
  if (m.size() >= 4096) m.clear();
  return m[std::make_tuple(N, kind, nrows, extra)];
}

// Plan and tile for nrows rows, at most tf_max rows a tile: the cheapest by fft_cycles over the tiles and, for FP64 rows,
// over radix-9 passes or radix-3 ones (more instructions in shorter chains, for launches with few butterflies), the
// larger tile on a tie (fewer blocks restage fewer tables).  A 63 x 63 grid in 32-row tiles ran on one or two SMs: 46 us
// per fibre pass and 88 us per fused row pass under event timing (9 and 17 us with even tiles and fixed point).  From six
// full tiles per SM on the rounding up costs less than the shorter memory segments of a smaller tile, and tf_max stays.
// segments: long FP32 rows strided in memory, where a pass is bound by the accesses and not by its instructions.  A smaller tile
// then keeps whole 32-byte sectors (four rows, unless there are fewer than two for an SM), has to leave fewer rows to the busiest SM, all of whose blocks fit its shared
// memory, and is tried only where the largest gives an SM fewer than two blocks (down to half of it where it gives one): by
// the instructions alone 8000 rows of 625 points took 135 us in tiles of 1 (54 in tiles of 16), 1000 of 3125 points 75 us (62).
FftPlan choose_plan(lrfg_ctx* ctx, int N, bool fp64, long long nrows, int tf_max, int* tf, bool segments) {
  const long long nsm = ctx->num_sms > 0 ? ctx->num_sms : 152;
  FftPlan best = make_plan(N, fp64 ? plan_radix<double2>() : plan_radix<float2>());
  *tf = tf_max;
  const long long full = (nrows + tf_max - 1) / tf_max, full_rows = (full + nsm - 1) / nsm * tf_max;
  if (full >= (segments ? 2 : 6) * nsm) return best;
  FftChoice& known = fft_choice(ctx, N, segments ? 4 : (fp64 ? 1 : 0), nrows, tf_max);
  if (known.tf) {
    *tf = known.tf;
    return known.plan;
  }
  const FftPlan small = make_plan(N, 3);
  double cost = 0.0;
  for (int q = 0; q < (fp64 ? 2 : 1); ++q) {
    const FftPlan pl = q ? small : best;
    for (int t = tf_max; t >= 1; --t) {
      const long long blocks = (nrows + t - 1) / t, per_sm = (blocks + nsm - 1) / nsm;
      if (segments && t < tf_max &&
          ((nrows > 2 * nsm && t % 4) || per_sm * t >= full_rows || (full >= nsm && 2 * t < tf_max) ||
           (per_sm > 1 && per_sm * (2LL + 2 * t) * N * (long long)sizeof(float2) > ctx->max_smem_optin)))
        continue;
      const double c = fft_cycles(ctx, pl, t, blocks);
      if (cost == 0.0 || c < 0.97 * cost) {
        cost = c;
        best = pl;
        *tf = t;
      }
    }
  }
  known = {best, *tf, 0};
  return best;
}

// Plan and tile for the complex fibre FFT: whole 128-byte segments along the contiguous index (TF * sizeof(V) >=
// 128) and at most 72 KB of shared memory, so that three blocks share an SM and one block's transform
// overlaps the others' loads and stores; fewer fibres where that fills the SMs more evenly.
static FftPlan tile_complex(lrfg_ctx* ctx, int N, size_t elem, long long nfib, int* tf_out, size_t* smem_out) {
  const long long row = (long long)N * (long long)elem;
  long long limit = 72 * 1024;
  const long long tf_min = std::max<long long>(1, 128 / (long long)elem);
  if (2 * row + 2 * tf_min * row > limit) limit = std::min<long long>(ctx->max_smem_optin, 200 * 1024);
  long long tf = (limit - 2 * row) / (2 * row);
  tf = std::max<long long>(1, std::min<long long>(tf, 32));
  if (tf > tf_min) tf = (tf / tf_min) * tf_min;
  const bool fp64 = elem == sizeof(double2);
  const FftPlan pl = choose_plan(ctx, N, fp64, nfib, (int)tf, tf_out, !fp64 && limit > 72 * 1024);
  *smem_out = (size_t)(2 * row + 2 * *tf_out * row);
  return pl;
}

template <typename V>
void fft_fibres(lrfg_ctx* ctx, const V* in, V* out, long long outer, int N, long long inner, int sign) {
  using R = typename RealOf<V>::T;
  LRFG_REQUIRE(N >= 1 && (N % 2 == 1), "fft length must be odd (got %d)", N);
  LRFG_REQUIRE(outer >= 0 && inner >= 0, "negative batch");
  if (outer == 0 || inner == 0) return;
  const auto* W = twiddle_table<R>(ctx, N);
  size_t smem;
  int TF;
  long long nfib = outer * inner;
  const FftPlan pl = tile_complex(ctx, N, sizeof(V), nfib, &TF, &smem);
  long long blocks = (nfib + TF - 1) / TF;
  LRFG_REQUIRE(blocks < (1LL << 31), "too many fibres");
  const double flops = 5.0 * N * std::log2((double)N) * (double)nfib;   // radix-2-equivalent count
  const double bytes = 2.0 * sizeof(V) * (double)N * (double)nfib;
  const FibreMul<R> none{};
  if (sign < 0 ? fft2_try<V, -1, 0>(ctx, in, out, outer, N, inner, none, flops, bytes)
               : fft2_try<V, 1, 0>(ctx, in, out, outer, N, inner, none, flops, bytes))
    return;
  if (sign < 0) {
    LRFG_CUDA(raise_smem_limit((const void*)fft_fibres_kernel<-1, V, 0, false>, smem));
    LRFG_LAUNCH(ctx, KC_FFT_FIBRES, flops, bytes,
                fft_fibres_kernel<-1, V, 0, false><<<(unsigned)blocks, 256, smem, ctx->stream>>>(in, out, outer, N, inner, TF,
                                                                                         pl, W, none, N, N));
  } else {
    LRFG_CUDA(raise_smem_limit((const void*)fft_fibres_kernel<1, V, 0, false>, smem));
    LRFG_LAUNCH(ctx, KC_FFT_FIBRES, flops, bytes,
                fft_fibres_kernel<1, V, 0, false><<<(unsigned)blocks, 256, smem, ctx->stream>>>(in, out, outer, N, inner, TF,
                                                                                        pl, W, none, N, N));
  }
}
template void fft_fibres<double2>(lrfg_ctx*, const double2*, double2*, long long, int, long long, int);
template void fft_fibres<float2>(lrfg_ctx*, const float2*, float2*, long long, int, long long, int);

template <typename V>
void fft_fibres_mul(lrfg_ctx* ctx, const V* in, V* out, const FibreMul<typename RealOf<V>::T>& fm) {
  using R = typename RealOf<V>::T;
  LRFG_REQUIRE(fm.mode == 1 || fm.mode == 2, "multiplier mode %d", fm.mode);
  LRFG_REQUIRE(fm.d == 2 || fm.d == 3, "d = %d", fm.d);
  LRFG_REQUIRE(fm.axis == 0 || (fm.axis == 1 && fm.d == 3), "axis %d of a half spectrum with d = %d", fm.axis, fm.d);
  LRFG_REQUIRE(fm.alpha >= (fm.mode == 2 ? -1 : 0) && fm.alpha < fm.d, "component %d", fm.alpha);
  // the grid's length along the axis, and the transform's (the double grid's where fm.L is set)
  const int Ng = fm.axis == 0 ? fm.N0 : fm.N1;
  const int N = fm.L ? fm.L : Ng;
  const long long outer = fm.axis == 0 ? 1 : (fm.L0 ? fm.L0 : fm.N0);
  const long long inner = fm.axis == 0 ? (long long)(fm.d == 3 ? fm.N1 : 1) * fm.H : fm.H;
  LRFG_REQUIRE(N >= 1 && (N % 2 == 1), "fft length must be odd (got %d)", N);
  LRFG_REQUIRE(fm.mode == 1 || in != out, "the accumulator cannot hold the input");
  LRFG_REQUIRE(!(fm.mode == 2 && fm.precond) || fm.inv_kk, "reciprocal table missing");
  if (inner == 0) return;
  const auto* W = twiddle_table<R>(ctx, N);
  size_t smem;
  int TF;
  const FftPlan pl = tile_complex(ctx, N, sizeof(V), outer * inner, &TF, &smem);
  long long blocks = (outer * inner + TF - 1) / TF;
  LRFG_REQUIRE(blocks < (1LL << 31), "too many fibres");
  const double n_el = (double)N * (double)outer * (double)inner;
  const double flops = 5.0 * std::log2((double)N) * n_el + (fm.mode == 1 ? 2.0 : 4.0) * n_el;
  const double bytes = (fm.mode == 1 || fm.init ? 2.0 : 3.0) * sizeof(V) * n_el;
  if (N != Ng) {
    LRFG_REQUIRE((std::is_same<V, double2>::value) && N > Ng, "a padded transform is longer than its grid (FP64)");
    if constexpr (std::is_same<V, double2>::value) {
      if (fm.mode == 1) {
        LRFG_CUDA(raise_smem_limit((const void*)fft_fibres_kernel<1, V, 1, true>, smem));
        LRFG_LAUNCH(ctx, KC_FFT_FIBRES, flops, bytes,
                    fft_fibres_kernel<1, V, 1, true><<<(unsigned)blocks, 256, smem, ctx->stream>>>(
                        in, out, outer, N, inner, TF, pl, W, fm, Ng, N));
      } else {
        LRFG_CUDA(raise_smem_limit((const void*)fft_fibres_kernel<-1, V, 2, true>, smem));
        LRFG_LAUNCH(ctx, KC_FFT_FIBRES, flops, bytes,
                    fft_fibres_kernel<-1, V, 2, true><<<(unsigned)blocks, 256, smem, ctx->stream>>>(
                        in, out, outer, N, inner, TF, pl, W, fm, N, Ng));
      }
    }
    return;
  }
  if (fm.mode == 1 ? fft2_try<V, 1, 1>(ctx, in, out, outer, N, inner, fm, flops, bytes)
                   : fft2_try<V, -1, 2>(ctx, in, out, outer, N, inner, fm, flops, bytes))
    return;
  if (fm.mode == 1) {
    LRFG_CUDA(raise_smem_limit((const void*)fft_fibres_kernel<1, V, 1, false>, smem));
    LRFG_LAUNCH(ctx, KC_FFT_FIBRES, flops, bytes,
                fft_fibres_kernel<1, V, 1, false><<<(unsigned)blocks, 256, smem, ctx->stream>>>(in, out, outer, N, inner, TF, pl,
                                                                                        W, fm, N, N));
  } else {
    LRFG_CUDA(raise_smem_limit((const void*)fft_fibres_kernel<-1, V, 2, false>, smem));
    LRFG_LAUNCH(ctx, KC_FFT_FIBRES, flops, bytes,
                fft_fibres_kernel<-1, V, 2, false><<<(unsigned)blocks, 256, smem, ctx->stream>>>(in, out, outer, N, inner, TF, pl,
                                                                                         W, fm, N, N));
  }
}

// The axis-0 passes of both components of a d = 2 half spectrum (N, H), FP64 (OP as in fft_fibres_kernel): rows f and nf + f
// of a tile of nf fibres are the components 0 and 1 of fibre f.
template <int OP>
__global__ void __launch_bounds__(256, 3) fft_pair_2d_kernel(const double2* in, double2* out, int N, int H, int F, FftPlan pl,
                                                             const int4* __restrict__ Wg, FibreMul<double> fm) {
  extern __shared__ __align__(16) unsigned char smraw_2d[];
  double2* sm = (double2*)smraw_2d;
  int4* W = reinterpret_cast<int4*>(sm);
  double2* a = sm + N;
  double2* b = a + (size_t)2 * F * N;
  const int i0 = blockIdx.x * F, nf = min(F, H - i0);
  const size_t half = (size_t)N * H;
  for (int j = threadIdx.x; j < N; j += blockDim.x) W[j] = Wg[j];
  // neighbouring threads take neighbouring fibres
  const float inv_nf = 1.0f / (float)nf;
  for (int t = threadIdx.x; t < nf * N; t += blockDim.x) {
    const int n = small_div(t, nf, inv_nf), f = t - n * nf;
    const double2* src = in + (size_t)n * H + i0 + f;
    double2* p = a + (size_t)f * N + n;
    if constexpr (OP == 1) {
      const double2 v = *src;
      p[0] = times_2pi_ik<double2>(v, fm.c2 * (double)freq_of(n, N));
      p[(size_t)nf * N] = times_2pi_ik<double2>(v, fm.c2 * (double)(i0 + f));
    } else {
      p[0] = src[0];
      p[(size_t)nf * N] = src[half];
    }
  }
  __syncthreads();
  const double2* res = stockham_rows<OP == 1 ? 1 : -1>(a, b, 2 * nf, N, pl, W);
  for (int t = threadIdx.x; t < nf * N; t += blockDim.x) {
    const int n = small_div(t, nf, inv_nf), f = t - n * nf;
    double2* dst = out + (size_t)n * H + i0 + f;
    const double2 x0 = res[(size_t)f * N + n], x1 = res[(size_t)(nf + f) * N + n];
    if constexpr (OP == 1) {
      dst[0] = x0;
      dst[half] = x1;
    } else {
      const int k0 = freq_of(n, N), k1 = i0 + f;
      const double2 r0 = times_2pi_ik<double2>(x0, -fm.c2 * (double)k0), r1 = times_2pi_ik<double2>(x1, -fm.c2 * (double)k1);
      double2 r = make_double2(r0.x + r1.x, r0.y + r1.y);
      if (fm.precond) {
        const double s = fm.inv_kk[k0 * k0 + k1 * k1];
        r.x *= s;
        r.y *= s;
      }
      *dst = r;
    }
  }
}

bool fft_pair_2d_fits(lrfg_ctx* ctx, int N) {
  return sizeof(double2) * 5 * (size_t)N <= (size_t)std::min(ctx->max_smem_optin, 200 * 1024);
}

template <int OP>
static void fft_pair_2d(lrfg_ctx* ctx, const double2* in, double2* out, const FibreMul<double>& fm) {
  LRFG_REQUIRE(fm.d == 2 && fm.axis == 0 && fm.L == 0 && in != out, "both components of a d = 2 half spectrum expected");
  LRFG_REQUIRE(!(OP == 2 && fm.precond) || fm.inv_kk, "reciprocal table missing");
  const int N = fm.N0, H = fm.H;
  const auto* W = twiddle_table<double>(ctx, N);
  size_t smem;
  int TF;
  const FftPlan pl = tile_complex(ctx, N, sizeof(double2), 2LL * H, &TF, &smem);
  const int F = std::max(1, TF / 2);
  smem = sizeof(double2) * (size_t)N * (1 + 4 * F);
  const double n_el = (double)N * H;
  LRFG_CUDA(raise_smem_limit((const void*)fft_pair_2d_kernel<OP>, smem));
  LRFG_LAUNCH(ctx, KC_FFT_FIBRES, 2.0 * (5.0 * std::log2((double)N) + 2.0 * OP) * n_el, 3.0 * sizeof(double2) * n_el,
              fft_pair_2d_kernel<OP><<<(unsigned)((H + F - 1) / F), 256, smem, ctx->stream>>>(in, out, N, H, F, pl, W, fm));
}

void fft_grad_2d(lrfg_ctx* ctx, const double2* v, double2* w, const FibreMul<double>& fm) { fft_pair_2d<1>(ctx, v, w, fm); }
void fft_div_2d(lrfg_ctx* ctx, const double2* w, double2* out, const FibreMul<double>& fm) { fft_pair_2d<2>(ctx, w, out, fm); }

// Plain transforms between n frequencies and the L > n points of the double grid along the middle axis: inverse
// (outer, n, inner) -> (outer, L, inner) with zeros for the other frequencies, forward (outer, L, inner) -> (outer, n,
// inner) keeping n of them.
void fft_fibres_pad(lrfg_ctx* ctx, const double2* in, double2* out, long long outer, int n, int L, long long inner,
                    int sign) {
  LRFG_REQUIRE(L > n && L % 2 == 1 && n % 2 == 1 && in != out, "padded transform %d -> %d", n, L);
  if (outer == 0 || inner == 0) return;
  const auto* W = twiddle_table<double>(ctx, L);
  size_t smem;
  int TF;
  const FftPlan pl = tile_complex(ctx, L, sizeof(double2), outer * inner, &TF, &smem);
  const long long blocks = (outer * inner + TF - 1) / TF;
  LRFG_REQUIRE(blocks < (1LL << 31), "too many fibres");
  const double nfib = (double)outer * (double)inner;
  const double flops = 5.0 * L * std::log2((double)L) * nfib, bytes = sizeof(double2) * (double)(n + L) * nfib;
  const FibreMul<double> none{};
  if (sign > 0) {
    LRFG_CUDA(raise_smem_limit((const void*)fft_fibres_kernel<1, double2, 0, true>, smem));
    LRFG_LAUNCH(ctx, KC_FFT_FIBRES, flops, bytes,
                fft_fibres_kernel<1, double2, 0, true><<<(unsigned)blocks, 256, smem, ctx->stream>>>(
                    in, out, outer, L, inner, TF, pl, W, none, n, L));
  } else {
    LRFG_CUDA(raise_smem_limit((const void*)fft_fibres_kernel<-1, double2, 0, true>, smem));
    LRFG_LAUNCH(ctx, KC_FFT_FIBRES, flops, bytes,
                fft_fibres_kernel<-1, double2, 0, true><<<(unsigned)blocks, 256, smem, ctx->stream>>>(
                    in, out, outer, L, inner, TF, pl, W, none, L, n));
  }
}
template void fft_fibres_mul<double2>(lrfg_ctx*, const double2*, double2*, const FibreMul<double>&);
template void fft_fibres_mul<float2>(lrfg_ctx*, const float2*, float2*, const FibreMul<float>&);

// ----------------------------------------------------------------------------------------------------
// real fibres under a multiplier: row f holds fibre 2 f (real part) and fibre 2 f + 1 (imaginary part), so a fibre's partner
// does not depend on the tile (the FP32 transforms' rounding does depend on the partner)
// ----------------------------------------------------------------------------------------------------
__device__ __forceinline__ double2 multiplier(int kind, int k, double param) {
  if (kind == LRFG_MUL_DERIV) return make_double2(0.0, 6.283185307179586476925286766559 * (double)k);
  if (kind == LRFG_MUL_GAUSS) return make_double2(exp(-param * (double)k * (double)k), 0.0);
  return make_double2(1.0, 0.0);
}

// V = double2 (FP64 transforms) or float2 (FP32 transforms of FP64 data: the mixed-precision path); the fibres
// are read and written in FP64 either way.
template <typename V>
__global__ void __launch_bounds__(256) fibre_op_kernel(const double* in, double* out, long long outer,
                                                       int N, long long inner, int TF, FftPlan pl,
                                                       const typename TwOf<V>::T* __restrict__ Wg, int kind, double param,
                                                       double scale) {
  using R = typename RealOf<V>::T;
  extern __shared__ __align__(16) unsigned char smraw_op[];
  V* sm = (V*)smraw_op;
  auto* W = reinterpret_cast<typename TwOf<V>::T*>(sm);
  V* M = sm + N;
  V* a = sm + 2 * N;
  V* b = a + (size_t)TF * N;
  for (int j = threadIdx.x; j < N; j += blockDim.x) {
    W[j] = Wg[j];
    const double2 m = multiplier(kind, freq_of(j, N), param);
    M[j] = mkc<V>((R)m.x, (R)m.y);
  }
  const long long nfib = outer * inner;
  const long long g0 = (long long)blockIdx.x * (2LL * TF);
  const int nf = (int)min(2LL * TF, nfib - g0);   // real fibres in this tile
  const int rows = (nf + 1) / 2;
  for (int t = threadIdx.x; t < rows * N; t += blockDim.x) a[t] = mkc<V>((R)0, (R)0);
  __syncthreads();
  const int total = nf * N;
  const bool across = inner >= 2 * TF;
  for (int t = threadIdx.x; t < total; t += blockDim.x) {
    int f, n;
    if (across) { f = t % nf; n = t / nf; } else { f = t / N; n = t % N; }
    long long g = g0 + f;
    long long o = g / inner, i = g - o * inner;
    const R v = (R)in[((size_t)o * N + n) * (size_t)inner + (size_t)i];
    V* z = a + (size_t)(f >> 1) * N + n;
    if (f & 1) z->y = v; else z->x = v;
  }
  __syncthreads();
  V* res = stockham_rows<-1>(a, b, rows, N, pl, W);
  V* other = (res == a) ? b : a;
  for (int t = threadIdx.x; t < rows * N; t += blockDim.x) {
    int n = t % N;
    res[t] = cmul(res[t], M[n]);
  }
  __syncthreads();
  res = stockham_rows<1>(res, other, rows, N, pl, W);
  const double s = scale / (double)N;
  for (int t = threadIdx.x; t < total; t += blockDim.x) {
    int f, n;
    if (across) { f = t % nf; n = t / nf; } else { f = t / N; n = t % N; }
    long long g = g0 + f;
    long long o = g / inner, i = g - o * inner;
    const V v = res[(size_t)(f >> 1) * N + n];
    out[((size_t)o * N + n) * (size_t)inner + (size_t)i] = s * (double)((f & 1) ? v.y : v.x);
  }
}

template <typename V>
static void fibre_operator_t(lrfg_ctx* ctx, const double* in, double* out, long long outer, int N, long long inner,
                             int kind, double param, double scale) {
  const auto* W = twiddle_table<typename RealOf<V>::T>(ctx, N);
  const long long nfib = outer * inner;
  int TF;  // a row carries two real fibres
  const FftPlan pl = choose_plan(ctx, N, sizeof(V) == sizeof(double2), (nfib + 1) / 2, tile_fibres(ctx, N, sizeof(V), 1, 2),
                                 &TF);
  const size_t smem = (size_t)(2LL * N * sizeof(V) + (long long)TF * 2LL * N * sizeof(V));
  long long blocks = (nfib + 2LL * TF - 1) / (2LL * TF);
  LRFG_REQUIRE(blocks < (1LL << 31), "too many fibres");
  LRFG_CUDA(raise_smem_limit((const void*)fibre_op_kernel<V>, smem));
  // two complex transforms per pair of real fibres
  const double flops = 5.0 * N * std::log2((double)N) * (double)nfib;
  const double bytes = 2.0 * sizeof(double) * (double)N * (double)nfib;
  LRFG_LAUNCH(ctx, KC_FIBRE_OP, flops, bytes,
              fibre_op_kernel<V><<<(unsigned)blocks, 256, smem, ctx->stream>>>(in, out, outer, N, inner, TF, pl, W,
                                                                                kind, param, scale));
}

void fibre_operator(lrfg_ctx* ctx, const double* in, double* out, long long outer, int N, long long inner,
                    int kind, double param, double scale, bool fp32) {
  LRFG_REQUIRE(N >= 1 && (N % 2 == 1), "fibre length must be odd (got %d)", N);
  LRFG_REQUIRE(kind == LRFG_MUL_IDENTITY || kind == LRFG_MUL_DERIV || kind == LRFG_MUL_GAUSS,
               "unknown multiplier %d", kind);
  if (outer == 0 || inner == 0) return;
  if (fp32) fibre_operator_t<float2>(ctx, in, out, outer, N, inner, kind, param, scale);
  else fibre_operator_t<double2>(ctx, in, out, outer, N, inner, kind, param, scale);
}

// Many Gaussian multipliers of one input: the forward transform is shared, each term m gets its own
// multiply + inverse transform and is written to out + m * out_stride.  The nodes and scales travel as a kernel argument
// (two copies from host memory per call before).
constexpr int kMaxGaussTerms = 64;
constexpr int kMaxGaussHalf = 512;
struct GaussTerms {
  double t[kMaxGaussTerms], s[kMaxGaussTerms];
};

template <typename V>
__global__ void __launch_bounds__(256) fibre_gauss_multi_kernel(const double* __restrict__ in, double* out,
                                                                long long out_stride, long long outer, int N,
                                                                long long inner, int TF, FftPlan pl,
                                                                const typename TwOf<V>::T* __restrict__ Wg,
                                                                const __grid_constant__ GaussTerms terms, int nm,
                                                                int mper) {
  using R = typename RealOf<V>::T;
  extern __shared__ __align__(16) unsigned char smraw_gm[];
  V* sm = (V*)smraw_gm;
  auto* W = reinterpret_cast<typename TwOf<V>::T*>(sm);
  V* spec = sm + N;              // TF rows: the shared forward spectrum
  V* a = spec + (size_t)TF * N;  // TF rows
  V* b = a + (size_t)TF * N;     // TF rows
  R* mult = (R*)(b + (size_t)TF * N);  // exp(-t_m k^2), k = 0..(N-1)/2 < kMaxGaussHalf: an FP64 exponential takes tens of
                                       // operations
  for (int j = threadIdx.x; j < N; j += blockDim.x) W[j] = Wg[j];
  const long long nfib = outer * inner;
  const long long g0 = (long long)blockIdx.x * (2LL * TF);
  const int nf = (int)min(2LL * TF, nfib - g0);
  const int rows = (nf + 1) / 2;
  for (int t = threadIdx.x; t < rows * N; t += blockDim.x) a[t] = mkc<V>((R)0, (R)0);
  __syncthreads();
  const int total = nf * N;
  const bool across = inner >= 2 * TF;
  for (int t = threadIdx.x; t < total; t += blockDim.x) {
    int f, n;
    if (across) { f = t % nf; n = t / nf; } else { f = t / N; n = t % N; }
    long long g = g0 + f;
    long long o = g / inner, i = g - o * inner;
    const R v = (R)in[((size_t)o * N + n) * (size_t)inner + (size_t)i];
    V* z = a + (size_t)(f >> 1) * N + n;
    if (f & 1) z->y = v; else z->x = v;
  }
  __syncthreads();
  V* res = stockham_rows<-1>(a, b, rows, N, pl, W);
  for (int t = threadIdx.x; t < rows * N; t += blockDim.x) spec[t] = res[t];
  __syncthreads();
  const int m_end = min(nm, (int)(blockIdx.y + 1) * mper);
  for (int m = blockIdx.y * mper; m < m_end; ++m) {
    const double t_m = terms.t[m];
    const int half = (N - 1) / 2;
    if (half < kMaxGaussHalf) {
      for (int k = threadIdx.x; k <= half; k += blockDim.x) mult[k] = (R)exp(-t_m * (double)k * (double)k);
      __syncthreads();
      for (int t = threadIdx.x; t < rows * N; t += blockDim.x) a[t] = cscale(spec[t], mult[abs(freq_of(t % N, N))]);
    } else {
      for (int t = threadIdx.x; t < rows * N; t += blockDim.x) {
        const int k = freq_of(t % N, N);
        a[t] = cscale(spec[t], (R)exp(-t_m * (double)k * (double)k));
      }
    }
    __syncthreads();
    V* r2 = stockham_rows<1>(a, b, rows, N, pl, W);
    const double s = terms.s[m] / (double)N;
    double* o_m = out + (size_t)m * (size_t)out_stride;
    for (int t = threadIdx.x; t < total; t += blockDim.x) {
      int f, n;
      if (across) { f = t % nf; n = t / nf; } else { f = t / N; n = t % N; }
      long long g = g0 + f;
      long long o = g / inner, i = g - o * inner;
      const V v = r2[(size_t)(f >> 1) * N + n];
      o_m[((size_t)o * N + n) * (size_t)inner + (size_t)i] = s * (double)((f & 1) ? v.y : v.x);
    }
    __syncthreads();
  }
}

template <typename V>
static void fibre_gauss_multi_t(lrfg_ctx* ctx, const double* in, double* out, long long out_stride, long long outer,
                                int N, long long inner, const double* t, const double* scale, int nm) {
  const auto* Wt = twiddle_table<typename RealOf<V>::T>(ctx, N);
  // few fibres (low-rank carriages): small tiles, and the terms split over grid.y (each block redoes the shared forward
  // transform of its tile), so that the launch covers the SMs: the cheapest of the splits by the inverse transforms a
  // block runs plus its forward one
  const int nsm = ctx->num_sms > 0 ? ctx->num_sms : 152;
  const long long nfib = outer * inner, nrows = (nfib + 1) / 2;
  const long long per = 3LL * N * (long long)sizeof(V);
  const int tf_max = tile_fibres(ctx, N, sizeof(V), 0, 3);
  int tf = 1, mper = nm;
  FftPlan pl{};
  double cost = 0.0;
  FftChoice& known = fft_choice(ctx, N, sizeof(V) == sizeof(double2) ? 3 : 2, nrows, nm);
  if (known.tf) {
    pl = known.plan;
    tf = known.tf;
    mper = known.mper;
  }
  for (int q = 0; !known.tf && q < (sizeof(V) == sizeof(double2) ? 2 : 1); ++q) {
    const FftPlan cand = make_plan(N, q ? 3 : plan_radix<V>());
    for (int t = tf_max; t >= 1; --t) {
      const long long bx = (nrows + t - 1) / t;
      if (t < tf_max && bx > 8LL * nsm) break;
      for (int chunks = 1; chunks <= nm; ++chunks) {
        const int mp = (nm + chunks - 1) / chunks, mg = (nm + mp - 1) / mp;
        if (chunks > 1 && bx * mg > 8LL * nsm) break;
        const double c = fft_cycles(ctx, cand, t, bx * mg) * (1 + mp);
        if (cost == 0.0 || c < 0.97 * cost) {
          cost = c;
          pl = cand;
          tf = t;
          mper = mp;
        }
      }
    }
  }
  known = {pl, tf, mper};
  const int half = (N - 1) / 2;
  size_t smem = (size_t)(N * sizeof(V) + tf * per) + (half < kMaxGaussHalf ? sizeof(V) / 2 * (half + 1) : 0);
  GaussTerms terms{};
  for (int m = 0; m < nm; ++m) {
    terms.t[m] = t[m];
    terms.s[m] = scale[m];
  }
  long long blocks = (nrows + tf - 1) / tf;
  LRFG_REQUIRE(blocks < (1LL << 31), "too many fibres");
  LRFG_CUDA(raise_smem_limit((const void*)fibre_gauss_multi_kernel<V>, smem));
  // one forward and nm inverse complex transforms per pair of real fibres (algorithmic count)
  const double flops = 2.5 * N * std::log2((double)N) * (double)nfib * (1.0 + nm);
  const double bytes = sizeof(double) * (double)N * (double)nfib * (1.0 + nm);
  const int mgrid = (nm + mper - 1) / mper;
  LRFG_LAUNCH(ctx, KC_GAUSS_MULTI, flops, bytes,
              fibre_gauss_multi_kernel<V><<<dim3((unsigned)blocks, (unsigned)mgrid), 256, smem, ctx->stream>>>(
                  in, out, out_stride, outer, N, inner, (int)tf, pl, Wt, terms, nm, mper));
}

void fibre_gauss_multi(lrfg_ctx* ctx, const double* in, double* out, long long out_stride, long long outer,
                       int N, long long inner, const double* t, const double* scale, int nm, bool fp32) {
  LRFG_REQUIRE(N >= 1 && (N % 2 == 1), "fibre length must be odd (got %d)", N);
  if (outer == 0 || inner == 0 || nm == 0) return;
  for (int m = 0; m < nm; m += kMaxGaussTerms) {
    const int q = std::min(kMaxGaussTerms, nm - m);
    double* o = out + (size_t)m * (size_t)out_stride;
    if (fp32) fibre_gauss_multi_t<float2>(ctx, in, o, out_stride, outer, N, inner, t + m, scale + m, q);
    else fibre_gauss_multi_t<double2>(ctx, in, o, out_stride, outer, N, inner, t + m, scale + m, q);
  }
}


// ------------------------------------------------------------------------------------------------
// Ga mode maps (Sec. 2.2.3) on real fibres: forward transform on n_in points, a spectral map to n_out
// points, inverse transform; the maps are exact in exact arithmetic (zero padding, truncation, periodic
// extension with the cell sinc), the transforms the library's fibre FFTs.
// ------------------------------------------------------------------------------------------------
__global__ void real_to_complex_kernel(const double* __restrict__ in, double2* __restrict__ out, long long n) {
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < n; t += (long long)gridDim.x * blockDim.x)
    out[t] = make_double2(in[t], 0.0);
}

__global__ void complex_to_real_kernel(const double2* __restrict__ in, double* __restrict__ out, long long n) {
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < n; t += (long long)gridDim.x * blockDim.x)
    out[t] = in[t].x;
}

__device__ __forceinline__ int freq_rep(int i, int n) { return i <= (n - 1) / 2 ? i : i - n; }

// out[o][m][i] = weight(m) * in[o][src(m)][i] over (outer, n_out, inner)
__global__ void ga_spectral_map_kernel(const double2* __restrict__ in, double2* __restrict__ out, long long outer,
                                       int n_in, long long inner, int n_out, int mode, int n_grid) {
  const long long total = outer * n_out * inner;
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < total; t += (long long)gridDim.x * blockDim.x) {
    const long long i = t % inner;
    const long long q = t / inner;
    const int m = (int)(q % n_out);
    const long long o = q / n_out;
    const int f = freq_rep(m, n_out);
    int src = -1;
    double wgt = 0.0;
    if (mode == GA_UP) {  // zero padding, F_N = Phi_N / N
      if (abs(f) <= (n_in - 1) / 2) { src = f < 0 ? f + n_in : f; wgt = 1.0 / n_in; }
    } else if (mode == GA_DOWN) {  // the frequencies of the small grid, F_M = Phi_M / M
      src = f < 0 ? f + n_in : f;
      wgt = 1.0 / n_in;
    } else {  // periodic extension times the cell sinc of the pixel grid n_grid, and M^-1
      src = ((f % n_in) + n_in) % n_in;
      const double x = 3.141592653589793238462643383279502884 * (double)f;
      const double s = f == 0 ? 1.0 / n_grid : sin(x / (double)n_grid) / x;
      wgt = s / n_out;
    }
    double2 v = make_double2(0.0, 0.0);
    if (src >= 0) {
      const double2 u = in[(o * n_in + src) * inner + i];
      v = make_double2(wgt * u.x, wgt * u.y);
    }
    out[t] = v;
  }
}

void ga_resample(lrfg_ctx* ctx, const double* in, double* out, long long outer, int n_in, long long inner, int n_out,
                 int mode) {
  const long long nin = outer * n_in * inner, nout = outer * n_out * inner;
  if (nin == 0 || nout == 0) return;
  const unsigned gin = (unsigned)std::min<long long>((nin + 255) / 256, 8LL * ctx->num_sms);
  const unsigned gout = (unsigned)std::min<long long>((nout + 255) / 256, 8LL * ctx->num_sms);
  DBuf<double2> a(ctx->pool, (size_t)nin), b(ctx->pool, (size_t)nout);
  LRFG_LAUNCH(ctx, KC_TT_MISC, 0.0, 24.0 * nin, real_to_complex_kernel<<<gin, 256, 0, ctx->stream>>>(in, a.get(), nin));
  fft_fibres<double2>(ctx, a.get(), a.get(), outer, n_in, inner, -1);
  LRFG_LAUNCH(ctx, KC_TT_MISC, 2.0 * nout, 32.0 * nout,
              ga_spectral_map_kernel<<<gout, 256, 0, ctx->stream>>>(a.get(), b.get(), outer, n_in, inner, n_out, mode,
                                                                    mode == GA_EXTEND ? n_in : 0));
  fft_fibres<double2>(ctx, b.get(), b.get(), outer, n_out, inner, 1);
  LRFG_LAUNCH(ctx, KC_TT_MISC, 0.0, 24.0 * nout,
              complex_to_real_kernel<<<gout, 256, 0, ctx->stream>>>(b.get(), out, nout));
}

}  // namespace lrfg
