// Dense FP64 building blocks for the rank truncation and the solvers: batched GEMM (Gram matrices and
// core contractions) and reductions.
#include <algorithm>
#include <cmath>
#include <type_traits>

#include "ops.cuh"

namespace lrfg {

// ------------------------------------------------------------------------------------------------
// GEMM, FP64.  On this part the FP64 pipe (2 FMA/clk/SM) is the bottleneck of every product here, so
// the kernel is built to waste none of it: a block owns a 64 x 64 (small products: 32 x 32) output block
// (clipped to the active sizes, which may be read from the device), each of its 256 threads owns up to 16
// (4) outputs of that block exactly (no padded tile rows or columns are computed), operands are staged
// through shared memory in k-steps of 32, and long K is split across blocks (see gemm_impl; split-K: each
// split writes its partial block to a workspace; the last split of a tile to arrive, found by an arrival
// counter, sums the partials in split order, so every product, and with it every solve, is bitwise
// reproducible whatever else runs on the GPU, and no second launch is needed).  With many splits the sum is
// two-level: the splits form groups of about sqrt(splits); the last split of each group to arrive sums its
// group's partials in order into a group partial, and the last group sums the group partials in order — the
// reduction then runs on as many blocks as there are groups instead of on one.  An output costs two
// shared-memory reads per FMA, far below the shared-memory bandwidth at the FP64 rate.
// ------------------------------------------------------------------------------------------------
constexpr int GK = 32;  // k-step

// pk[j] = (row << 16) | column of output j within the block
template <int NR, int TILE, typename T>
__device__ __forceinline__ void gemm_fma_rows(T* acc, const T (*As)[TILE + 1], const T (*Bs)[TILE + 1],
                                              const int* pk, int kk_end) {
  for (int kk = 0; kk < kk_end; ++kk) {
#pragma unroll
    for (int j = 0; j < NR; ++j) acc[j] = fma(As[kk][pk[j] >> 16], Bs[kk][pk[j] & 0xffff], acc[j]);
  }
}

// dynM / dynN (optional, per batch item): the product is computed only for rows < dynM[b] * mulM and
// columns < dynN[b] * mulN (data-dependent active sizes, e.g. numerical ranks); the rest of C is not
// written.  With splits > 1 the partial sums go to part[((split * batches + item) * M + row) * N + column]
// (M, N the static sizes).  TILE = 64 (16 outputs per thread), 32 (4 per thread, for small products:
// four times the blocks, so that a product of a few tiles still spreads over the SMs) or 16 (one per thread,
// for products of one or a few 32-tiles with a short K, see gemm_impl).
// T = double (the FP64 products) or float (the FP32 sketch products of the mixed-precision path).
// SYM: the product is symmetric (a Gram matrix, or F R F^T with a symmetric R); only the tiles and outputs on and below
// the diagonal are computed, each written to both places: half the FP64 work of a product that is bound by it.
template <bool TA, bool TB, int TILE, typename T, bool SYM>
__global__ void __launch_bounds__(256) dgemm_kernel(int M, int N, int K, double alpha_d, const T* __restrict__ A,
                                                    int lda, long long sA, const T* __restrict__ B, int ldb,
                                                    long long sB, double beta_d, T* C, int ldc, long long sC,
                                                    int splits, int kchunk, const int* __restrict__ dynM, int mulM,
                                                    const int* __restrict__ dynN, int mulN, double* work,
                                                    T* __restrict__ part, unsigned int* __restrict__ cnt,
                                                    int gsize) {
  constexpr int NMAX = TILE * TILE / 256;
  const T alpha = (T)alpha_d, beta = (T)beta_d;
  __shared__ T As[GK][TILE + 1];
  __shared__ T Bs[GK][TILE + 1];
  const int batch = blockIdx.z;
  const int bm = blockIdx.y / splits, split = blockIdx.y - (blockIdx.y / splits) * splits;
  const int bn = blockIdx.x;
  A += (size_t)batch * sA;
  B += (size_t)batch * sB;
  C += (size_t)batch * sC;
  const int Ms = M, Ns = N;
  if (dynM) M = min(M, dynM[batch] * mulM);
  if (dynN) N = min(N, dynN[batch] * mulN);
  if (work && bm == 0 && bn == 0 && split == 0 && threadIdx.x == 0)
    add_work(work, (SYM ? 1.0 * M * (M + 1.0) : 2.0 * M * N) * (double)K, (double)sizeof(T) * ((double)M * K + (double)K * N + (double)M * N));
  const int m0 = bm * TILE, n0 = bn * TILE;
  const int Mb = min(TILE, M - m0), Nb = min(TILE, N - n0);
  if (Mb <= 0 || Nb <= 0) return;
  if (SYM && bn > bm) return;
  const bool tri = SYM && bn == bm;
  const int kbeg = split * kchunk, kend = min(K, kbeg + kchunk);
  // this thread's outputs o = t + 256 j < Mb Nb, as (row, column) within the block
  const int tot = tri ? Mb * (Mb + 1) / 2 : Mb * Nb;
  const int nact = tot > (int)threadIdx.x ? min(NMAX, (tot - (int)threadIdx.x + 255) / 256) : 0;
  int pk[NMAX];
  T acc[NMAX];
#pragma unroll
  for (int j = 0; j < NMAX; ++j) {
    const int o = threadIdx.x + 256 * j;
    int m, c0;  // row and the index of its first output
    if (tri) {
      m = (int)((sqrtf(8.0f * (float)o + 1.0f) - 1.0f) * 0.5f);
      while (m * (m + 1) / 2 > o) --m;
      while ((m + 1) * (m + 2) / 2 <= o) ++m;
      c0 = m * (m + 1) / 2;
    } else {
      m = o / Nb;
      c0 = m * Nb;
    }
    pk[j] = j < nact ? (m << 16) | (o - c0) : 0;
    acc[j] = (T)0;
  }
  // the next k-step's operands are on their way to registers while this one's are multiplied (135 x 135 x 18225 Gram product
  // 404 -> 334 us, the small products of an application 5-15% shorter).  The 64 x 64 FP64 kernels take 229-240 registers with
  // them in four of their six forms, one block an SM; the 32 x 32 ones at most 112, two or more.
  constexpr int NL = TILE * GK / 256;
  T ra[NL], rb[NL];
  auto fetch = [&](int k0) {
    const int kc = kend - k0;
#pragma unroll
    for (int u = 0; u < NL; ++u) {
      const int e = threadIdx.x + 256 * u;
      const int mm = TA ? e % TILE : e / GK, ka = TA ? e / TILE : e % GK;
      const int nn = TB ? e / GK : e % TILE, kb = TB ? e % GK : e / TILE;
      ra[u] = (mm < Mb && ka < kc) ? (TA ? A[(size_t)(k0 + ka) * lda + m0 + mm] : A[(size_t)(m0 + mm) * lda + k0 + ka]) : (T)0;
      rb[u] = (nn < Nb && kb < kc) ? (TB ? B[(size_t)(n0 + nn) * ldb + k0 + kb] : B[(size_t)(k0 + kb) * ldb + n0 + nn]) : (T)0;
    }
  };
  if (kbeg < kend) fetch(kbeg);
  for (int k0 = kbeg; k0 < kend; k0 += GK) {
    const int kc = min(GK, kend - k0);
#pragma unroll
    for (int u = 0; u < NL; ++u) {
      const int e = threadIdx.x + 256 * u;
      As[TA ? e / TILE : e % GK][TA ? e % TILE : e / GK] = ra[u];
      Bs[TB ? e % GK : e / TILE][TB ? e / GK : e % TILE] = rb[u];
    }
    __syncthreads();
    if (k0 + GK < kend) fetch(k0 + GK);
    if constexpr (NMAX == 16) {
      switch (nact) {
        case 16: gemm_fma_rows<16, TILE>(acc, As, Bs, pk, kc); break;
        case 15: gemm_fma_rows<15, TILE>(acc, As, Bs, pk, kc); break;
        case 14: gemm_fma_rows<14, TILE>(acc, As, Bs, pk, kc); break;
        case 13: gemm_fma_rows<13, TILE>(acc, As, Bs, pk, kc); break;
        case 12: gemm_fma_rows<12, TILE>(acc, As, Bs, pk, kc); break;
        case 11: gemm_fma_rows<11, TILE>(acc, As, Bs, pk, kc); break;
        case 10: gemm_fma_rows<10, TILE>(acc, As, Bs, pk, kc); break;
        case 9: gemm_fma_rows<9, TILE>(acc, As, Bs, pk, kc); break;
        case 8: gemm_fma_rows<8, TILE>(acc, As, Bs, pk, kc); break;
        case 7: gemm_fma_rows<7, TILE>(acc, As, Bs, pk, kc); break;
        case 6: gemm_fma_rows<6, TILE>(acc, As, Bs, pk, kc); break;
        case 5: gemm_fma_rows<5, TILE>(acc, As, Bs, pk, kc); break;
        case 4: gemm_fma_rows<4, TILE>(acc, As, Bs, pk, kc); break;
        case 3: gemm_fma_rows<3, TILE>(acc, As, Bs, pk, kc); break;
        case 2: gemm_fma_rows<2, TILE>(acc, As, Bs, pk, kc); break;
        case 1: gemm_fma_rows<1, TILE>(acc, As, Bs, pk, kc); break;
        default: break;
      }
    } else if constexpr (NMAX == 4) {
      switch (nact) {
        case 4: gemm_fma_rows<4, TILE>(acc, As, Bs, pk, kc); break;
        case 3: gemm_fma_rows<3, TILE>(acc, As, Bs, pk, kc); break;
        case 2: gemm_fma_rows<2, TILE>(acc, As, Bs, pk, kc); break;
        case 1: gemm_fma_rows<1, TILE>(acc, As, Bs, pk, kc); break;
        default: break;
      }
    } else {
      if (nact == 1) gemm_fma_rows<1, TILE>(acc, As, Bs, pk, kc);
    }
    __syncthreads();
  }
  if (splits > 1) {
    const size_t pstride = (size_t)gridDim.z * Ms * Ns;  // between the splits of one output
    T* P = part + (size_t)batch * Ms * Ns;
#pragma unroll
    for (int j = 0; j < NMAX; ++j) {
      if (j >= nact) break;
      P[split * pstride + (size_t)(m0 + (pk[j] >> 16)) * Ns + n0 + (pk[j] & 0xffff)] = acc[j];
    }
    __shared__ unsigned int s_last;
    const size_t tile_id = ((size_t)batch * gridDim.y / splits + bm) * gridDim.x + bn;
    unsigned int* c = cnt + tile_id;
    // the partials the tile's last block sums: every split's (one level), or every group's (two levels: the
    // group partials sit after the splits' in the workspace)
    int nsum = splits;
    const T* S = P;
    if (gsize < splits) {
      const int ngroups = (splits + gsize - 1) / gsize;
      const int g = split / gsize, g0 = g * gsize, gn = min(gsize, splits - g0);
      unsigned int* cg = cnt + kSplitKCounters + tile_id * kSplitKGroups + g;
      __threadfence();
      __syncthreads();
      if (threadIdx.x == 0) {
        const unsigned int prev = atomicAdd(cg, 1u);
        s_last = (prev == (unsigned int)gn - 1u) ? 1u : 0u;
      }
      __syncthreads();
      if (!s_last) return;
      __threadfence();
      // the group's last split: its partials in split order into group partial g
#pragma unroll
      for (int j = 0; j < NMAX; ++j) {
        if (j >= nact) break;
        const size_t off = (size_t)(m0 + (pk[j] >> 16)) * Ns + n0 + (pk[j] & 0xffff);
        T v = (T)0;
        for (int s = g0; s < g0 + gn; ++s) v += __ldcg(P + s * pstride + off);
        P[(size_t)(splits + g) * pstride + off] = v;
      }
      if (threadIdx.x == 0) *cg = 0u;
      nsum = ngroups;
      S = P + (size_t)splits * pstride;
    }
    // the last (split or group) of this tile to arrive sums the partials in order
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) {
      const unsigned int prev = atomicAdd(c, 1u);
      s_last = (prev == (unsigned int)nsum - 1u) ? 1u : 0u;
    }
    __syncthreads();
    if (!s_last) return;
    __threadfence();
#pragma unroll
    for (int j = 0; j < NMAX; ++j) {
      if (j >= nact) break;
      const size_t off = (size_t)(m0 + (pk[j] >> 16)) * Ns + n0 + (pk[j] & 0xffff);
      T v = (T)0;
      for (int s = 0; s < nsum; ++s) v += __ldcg(S + s * pstride + off);
      T* cp = C + (size_t)(m0 + (pk[j] >> 16)) * ldc + n0 + (pk[j] & 0xffff);
      v = (beta_d == 0.0) ? alpha * v : alpha * v + beta * (*cp);
      *cp = v;
      if (SYM) C[(size_t)(n0 + (pk[j] & 0xffff)) * ldc + m0 + (pk[j] >> 16)] = v;
    }
    if (threadIdx.x == 0) *c = 0u;  // ready for the next product
    return;
  }
#pragma unroll
  for (int j = 0; j < NMAX; ++j) {
    if (j >= nact) break;
    T* c = C + (size_t)(m0 + (pk[j] >> 16)) * ldc + n0 + (pk[j] & 0xffff);
    const T v = (beta_d == 0.0) ? alpha * acc[j] : alpha * acc[j] + beta * (*c);
    *c = v;
    if (SYM) C[(size_t)(n0 + (pk[j] & 0xffff)) * ldc + m0 + (pk[j] >> 16)] = v;
  }
}

template <int TILE, typename T>
static void launch_dgemm(lrfg_ctx* ctx, int transA, int transB, dim3 grid, double flops, double bytes, int M, int N,
                         int K, double alpha, const T* A, int lda, long long sA, const T* B, int ldb,
                         long long sB, double beta, T* C, int ldc, long long sC, int splits, int kchunk,
                         const int* dynM, int mulM, const int* dynN, int mulN, double* work, T* part,
                         int gsize = 1 << 30, bool sym = false) {
  auto launch = [&](auto kernel) {
    LRFG_LAUNCH_KC(ctx, (std::is_same<T, float>::value ? KC_GEMM32 : KC_GEMM), flops, bytes,
                   kernel<<<grid, 256, 0, ctx->stream>>>(M, N, K, alpha, A, lda, sA, B, ldb, sB, beta, C, ldc, sC, splits,
                                                         kchunk, dynM, mulM, dynN, mulN, work, part, ctx->splitk_cnt,
                                                         gsize));
  };
  if constexpr (std::is_same<T, double>::value) {
    if (sym) {
      if (transA && !transB) launch(dgemm_kernel<true, false, TILE, T, true>);
      else launch(dgemm_kernel<false, true, TILE, T, true>);
      return;
    }
  }
  if (!transA && !transB) launch(dgemm_kernel<false, false, TILE, T, false>);
  else if (transA && !transB) launch(dgemm_kernel<true, false, TILE, T, false>);
  else if (!transA && transB) launch(dgemm_kernel<false, true, TILE, T, false>);
  else launch(dgemm_kernel<true, true, TILE, T, false>);
}

__global__ void scale_matrix_kernel(double* C, int M, int N, int ldc, long long sC, int batch, double beta) {
  long long total = (long long)M * N * batch;
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < total; t += (long long)gridDim.x * blockDim.x) {
    long long b = t / ((long long)M * N);
    long long rem = t - b * M * N;
    int i = (int)(rem / N), j = (int)(rem % N);
    double* c = C + (size_t)b * sC + (size_t)i * ldc + j;
    *c = (beta == 0.0) ? 0.0 : beta * (*c);
  }
}

void gemm(lrfg_ctx* ctx, int transA, int transB, int M, int N, int K, double alpha, const double* A, int lda,
          long long sA, const double* B, int ldb, long long sB, double beta, double* C, int ldc, long long sC,
          int batch) {
  gemm_dyn(ctx, transA, transB, M, N, K, alpha, A, lda, sA, B, ldb, sB, beta, C, ldc, sC, batch, nullptr, 1,
           nullptr, 1);
}

template <typename T>
static void gemm_impl(lrfg_ctx* ctx, int transA, int transB, int M, int N, int K, double alpha, const T* A, int lda,
                      long long sA, const T* B, int ldb, long long sB, double beta, T* C, int ldc, long long sC,
                      int batch, const int* dynM, int mulM, const int* dynN, int mulN, bool sym = false, bool once = false) {
  if (M <= 0 || N <= 0 || batch <= 0) return;
  LRFG_REQUIRE(!sym || (M == N && transA != transB && beta == 0.0), "not a symmetric product");
  if (K <= 0) {
    LRFG_REQUIRE((std::is_same<T, double>::value), "FP32 product with an empty inner dimension");
    LRFG_LAUNCH(ctx, KC_GEMM, (double)M * N * batch, 2.0 * sizeof(double) * M * N * batch,
                scale_matrix_kernel<<<std::min(1024LL, ((long long)M * N * batch + 255) / 256), 256, 0, ctx->stream>>>(
                    (double*)C, M, N, ldc, sC, batch, beta));
    return;
  }
  LRFG_REQUIRE(batch < 65536, "gemm batch too large");
  const int nsm = ctx->num_sms > 0 ? ctx->num_sms : 152;
  // blocks expected to be active: the static count, or for data-dependent sizes a quarter of it (the
  // numerical ranks are typically well below their bounds), at least one per item
  auto active_tiles = [&](int tile) {
    const long long tm = (M + tile - 1) / tile, tn = (N + tile - 1) / tile;
    long long a = (sym ? tm * (tm + 1) / 2 : tm * tn) * batch;
    if (dynM || dynN) a = std::max<long long>(batch, a / 4);
    return a;
  };
  // 32 x 32 tiles for thin products (one side <= 32: the 64-row staging would be mostly padding), when
  // 64 x 64 ones would leave most SMs idle, or when they fill the SMs more evenly: the FP64 pipe is shared by
  // the blocks of an SM, so a product takes as long as its busiest SM, ceil(blocks / SMs) blocks (static
  // sizes only: with data-dependent sizes the active tiles are not known here, and the split count is what
  // spreads those products)
  auto fill = [&](long long blocks) { return (double)blocks / (double)(((blocks + nsm - 1) / nsm) * nsm); };
  const bool dyn = dynM || dynN;
  // (data-dependent sizes are judged by their static bounds: the tile's evenness costs little where they are far below)
  auto tiles_of = [&](int tile) {
    const long long tm = (M + tile - 1) / tile, tn = (N + tile - 1) / tile;
    return (sym ? tm * (tm + 1) / 2 : tm * tn) * batch;
  };
  int tile = ((!dyn && (std::min(M, N) <= 32 || active_tiles(64) < nsm)) ||
              fill(tiles_of(32)) > fill(tiles_of(64)) + 0.05)
                 ? 32
                 : 64;
  // 16 x 16 tiles when even the largest split of the 32-tiles leaves most SMs idle: one k-step of a 32-tile
  // block is 32 K FMAs, 8 us of one SM's FP64 pipe, so a product of a few 32-tiles whose K is too short to
  // split further runs on a few SMs for that long; 16-tiles give four times the blocks at a quarter of the work
  if (tile == 32 && active_tiles(32) * std::max(1, K / GK) < nsm) tile = 16;
  const long long active = active_tiles(tile);
  // Split long K so that the busiest SM has the fewest k-steps: a block of c k-steps, active * ceil(steps / c) blocks, and
  // a round of blocks costs c steps plus about one for its first loads and its partial sums.  At most four blocks per SM; in a
  // context whose pool has a budget two, the tiles above the diagonal of a symmetric product counted as well (the partial
  // sums have the space of all of them), and no split of less than a whole k-step.
  // once: a product no lockstep batch repeats, so that its order of summation is free (a solve alone and in lockstep takes the
  // same steps to 1e-9 only where both split alike).  Several blocks an SM, side by side or in turn, even out to the average
  // tile, `filled` of its outputs, and a lone block's first loads and last sums are covered by nothing (about a third of a
  // step each).  Limited to one / two / four blocks an SM, a compression of 135^3 values, whose 135 x 135 x 18225 Gram product is a
  // third padding, takes 4.09 / 3.63 / 3.49 ms, the lockstep tensor at 81^3 28.4 / 27.2 / 27.1 ms, the other roundings the same
  // within 1%.
  const int steps = (K + GK - 1) / GK;
  const double filled = dyn || !once ? 1.0 : (sym ? 0.5 * M * (M + 1.0) : (double)M * N) * batch / ((double)tiles_of(tile) * tile * tile);
  int per = steps;
  if (active < 2LL * nsm) {
    double best = 0.0;
    const bool tight = ctx->pool->budget() != 0;
    const long long most = (tight ? 2LL : 4LL) * nsm;
    const long long all = (long long)((M + tile - 1) / tile) * ((N + tile - 1) / tile) * batch;
    const long long stored = tight ? std::max(active, dyn ? all / 4 : all) : active;
    for (int c = (int)std::max(1LL, std::min<long long>(steps, stored * steps / most)); c <= steps; ++c) {
      const int parts = (steps + c - 1) / c;
      const long long blocks = active * parts;
      if (tight && (stored * parts > most || parts > std::max(1, K / GK))) continue;
      const double q = (double)((blocks + nsm - 1) / nsm);
      const double cost = (filled * q + (1.0 - filled)) * c + (q < 2.0 && once ? 0.35 * c : 0.0) + q;
      if (best == 0.0 || cost < best) {
        best = cost;
        per = c;
      }
      if (blocks <= nsm) break;  // longer blocks only add steps from here on
    }
  }
  const int kchunk = per * GK;
  int splits = (steps + per - 1) / per;
  const int bmn = (M + tile - 1) / tile, bnn = (N + tile - 1) / tile;
  LRFG_REQUIRE((long long)bmn * splits < 65536, "gemm too many row blocks x splits");
  if (splits > 1)
    LRFG_REQUIRE((long long)bmn * bnn * batch <= kSplitKCounters, "split-K product with too many output tiles");
  // two-level reduction of the partials from 9 splits on: groups of ceil(sqrt(splits))
  int gsize = 1 << 30, ngroups = 0;
  if (splits > 8) {
    gsize = (int)std::ceil(std::sqrt((double)splits));
    ngroups = (splits + gsize - 1) / gsize;
    LRFG_REQUIRE(ngroups <= kSplitKGroups, "split-K product with too many groups (%d)", ngroups);
  }
  DBuf<T> part;
  if (splits > 1) part = DBuf<T>(ctx->pool, (size_t)(splits + ngroups) * M * N * batch);
  // products with data-dependent sizes count their work on the device
  double* work = (dynM || dynN) ? work_counter(ctx, KC_GEMM) : nullptr;
  const double flops = work ? 0.0 : (sym ? 1.0 * M * (M + 1.0) : 2.0 * M * N) * (double)K * batch;
  const double bytes = work ? 0.0 : sizeof(T) * ((double)M * K + (double)K * N + (double)M * N) * batch;
  dim3 grid(bnn, bmn * splits, batch);
  if (tile == 16)
    launch_dgemm<16, T>(ctx, transA, transB, grid, flops, bytes, M, N, K, alpha, A, lda, sA, B, ldb, sB, beta, C, ldc,
                     sC, splits, kchunk, dynM, mulM, dynN, mulN, work, part.get(), gsize, sym);
  else if (tile == 32)
    launch_dgemm<32, T>(ctx, transA, transB, grid, flops, bytes, M, N, K, alpha, A, lda, sA, B, ldb, sB, beta, C, ldc,
                     sC, splits, kchunk, dynM, mulM, dynN, mulN, work, part.get(), gsize, sym);
  else
    launch_dgemm<64, T>(ctx, transA, transB, grid, flops, bytes, M, N, K, alpha, A, lda, sA, B, ldb, sB, beta, C, ldc,
                     sC, splits, kchunk, dynM, mulM, dynN, mulN, work, part.get(), gsize, sym);
}

void gemm_dyn(lrfg_ctx* ctx, int transA, int transB, int M, int N, int K, double alpha, const double* A, int lda,
              long long sA, const double* B, int ldb, long long sB, double beta, double* C, int ldc, long long sC,
              int batch, const int* dynM, int mulM, const int* dynN, int mulN) {
  gemm_impl<double>(ctx, transA, transB, M, N, K, alpha, A, lda, sA, B, ldb, sB, beta, C, ldc, sC, batch, dynM, mulM,
                    dynN, mulN);
}

void gemm_sym(lrfg_ctx* ctx, int trans, int M, int K, const double* A, int lda, long long sA, const double* B, int ldb,
              long long sB, double* C, int ldc, long long sC, int batch, const int* dyn, bool once) {
  gemm_impl<double>(ctx, trans, !trans, M, M, K, 1.0, A, lda, sA, B, ldb, sB, 0.0, C, ldc, sC, batch, dyn, 1, dyn, 1, true, once);
}

void gemm_f32(lrfg_ctx* ctx, int transA, int transB, int M, int N, int K, double alpha, const float* A, int lda,
              long long sA, const float* B, int ldb, long long sB, double beta, float* C, int ldc, long long sC,
              int batch) {
  gemm_impl<float>(ctx, transA, transB, M, N, K, alpha, A, lda, sA, B, ldb, sB, beta, C, ldc, sC, batch, nullptr, 1,
                   nullptr, 1);
}

// The same product in one pass over K (no split-K): it needs no partial-sum workspace, so it takes nothing
// from the context's pool.  For callers that must not allocate.
void gemm_nosplit(lrfg_ctx* ctx, int transA, int transB, int M, int N, int K, double alpha, const double* A, int lda,
                  long long sA, const double* B, int ldb, long long sB, double beta, double* C, int ldc, long long sC,
                  int batch) {
  if (M <= 0 || N <= 0 || batch <= 0) return;
  if (K <= 0) {
    LRFG_LAUNCH(ctx, KC_GEMM, (double)M * N * batch, 2.0 * sizeof(double) * M * N * batch,
                scale_matrix_kernel<<<std::min(1024LL, ((long long)M * N * batch + 255) / 256), 256, 0, ctx->stream>>>(
                    C, M, N, ldc, sC, batch, beta));
    return;
  }
  LRFG_REQUIRE(batch < 65536, "gemm batch too large");
  const int nsm = ctx->num_sms > 0 ? ctx->num_sms : 152;
  const long long tiles64 = (long long)((M + 63) / 64) * ((N + 63) / 64) * batch;
  const int tile = tiles64 < nsm ? 32 : 64;
  const int bmn = (M + tile - 1) / tile, bnn = (N + tile - 1) / tile;
  LRFG_REQUIRE(bmn < 65536, "gemm too many row blocks");
  const int kchunk = ((K + GK - 1) / GK) * GK;
  const double flops = 2.0 * M * N * (double)K * batch;
  const double bytes = sizeof(double) * ((double)M * K + (double)K * N + (double)M * N) * batch;
  dim3 grid(bnn, bmn, batch);
  if (tile == 32)
    launch_dgemm<32, double>(ctx, transA, transB, grid, flops, bytes, M, N, K, alpha, A, lda, sA, B, ldb, sB, beta, C,
                             ldc, sC, 1, kchunk, nullptr, 1, nullptr, 1, nullptr, nullptr);
  else
    launch_dgemm<64, double>(ctx, transA, transB, grid, flops, bytes, M, N, K, alpha, A, lda, sA, B, ldb, sB, beta, C,
                             ldc, sC, 1, kchunk, nullptr, 1, nullptr, 1, nullptr, nullptr);
}

// ------------------------------------------------------------------------------------------------
// elementwise and reductions
// ------------------------------------------------------------------------------------------------
__global__ void fill_kernel(double* x, double v, long long n) {
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < n; t += (long long)gridDim.x * blockDim.x)
    x[t] = v;
}

__global__ void axpby_kernel(long long n, double a, const double* __restrict__ x, double b, double* y) {
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < n; t += (long long)gridDim.x * blockDim.x)
    y[t] = (b == 0.0) ? a * x[t] : a * x[t] + b * y[t];
}

static unsigned grid_for(lrfg_ctx* ctx, long long n) {
  long long g = (n + 255) / 256;
  long long cap = 8LL * (ctx->num_sms > 0 ? ctx->num_sms : 152);
  return (unsigned)std::max(1LL, std::min(g, cap));
}

void fill(lrfg_ctx* ctx, double* x, double v, long long n) {
  if (n <= 0) return;
  LRFG_LAUNCH(ctx, KC_TT_MISC, 0, sizeof(double) * (double)n,
              fill_kernel<<<grid_for(ctx, n), 256, 0, ctx->stream>>>(x, v, n));
}

void axpby(lrfg_ctx* ctx, long long n, double alpha, const double* x, double beta, double* y) {
  if (n <= 0) return;
  LRFG_LAUNCH(ctx, KC_TT_MISC, 3.0 * n, 3.0 * sizeof(double) * n,
              axpby_kernel<<<grid_for(ctx, n), 256, 0, ctx->stream>>>(n, alpha, x, beta, y));
}

// two-stage deterministic dot: fixed grid of partial sums, then one block sums them in order
constexpr int kDotBlocks = 304;

__global__ void __launch_bounds__(256) dot_partial_kernel(const double* __restrict__ x, const double* __restrict__ y,
                                                          long long n, double* partial) {
  __shared__ double red[8];
  double s = 0.0;
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < n; t += (long long)gridDim.x * blockDim.x)
    s = fma(x[t], y[t], s);
  for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(0xffffffff, s, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    double v = 0.0;
    for (int i = 0; i < 8; ++i) v += red[i];
    partial[blockIdx.x] = v;
  }
}

__global__ void sum_partials_kernel(const double* __restrict__ partial, int n, double* out) {
  __shared__ double red[8];
  double s = 0.0;
  for (int t = threadIdx.x; t < n; t += blockDim.x) s += partial[t];
  for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(0xffffffff, s, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    double v = 0.0;
    for (int i = 0; i < 8; ++i) v += red[i];
    *out = v;
  }
}

void dot_device(lrfg_ctx* ctx, const double* x, const double* y, long long n, double* out) {
  DBuf<double> partial(ctx->pool, kDotBlocks);
  LRFG_LAUNCH(ctx, KC_REDUCE, 2.0 * n, 2.0 * sizeof(double) * n,
              dot_partial_kernel<<<kDotBlocks, 256, 0, ctx->stream>>>(x, y, n, partial.get()));
  LRFG_LAUNCH(ctx, KC_REDUCE, kDotBlocks, kDotBlocks * sizeof(double),
              sum_partials_kernel<<<1, 256, 0, ctx->stream>>>(partial.get(), kDotBlocks, out));
}

double dot_host(lrfg_ctx* ctx, const double* x, const double* y, long long n) {
  DBuf<double> d(ctx->pool, 1);
  dot_device(ctx, x, y, n, d.get());
  double h = 0.0;
  LRFG_CUDA(cudaMemcpyAsync(&h, d.get(), sizeof(double), cudaMemcpyDeviceToHost, ctx->stream));
  LRFG_CUDA(cudaStreamSynchronize(ctx->stream));
  return h;
}

__global__ void to_f32_kernel(const double* __restrict__ in, float* __restrict__ out, long long n) {
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < n; t += (long long)gridDim.x * blockDim.x)
    out[t] = (float)in[t];
}

__global__ void to_f64_kernel(const float* __restrict__ in, double* __restrict__ out, long long n) {
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < n; t += (long long)gridDim.x * blockDim.x)
    out[t] = (double)in[t];
}

void to_f32(lrfg_ctx* ctx, const double* in, float* out, long long n) {
  if (n <= 0) return;
  LRFG_LAUNCH(ctx, KC_TT_MISC, 0.0, 12.0 * n, to_f32_kernel<<<grid_for(ctx, n), 256, 0, ctx->stream>>>(in, out, n));
}

void to_f64(lrfg_ctx* ctx, const float* in, double* out, long long n) {
  if (n <= 0) return;
  LRFG_LAUNCH(ctx, KC_TT_MISC, 0.0, 12.0 * n, to_f64_kernel<<<grid_for(ctx, n), 256, 0, ctx->stream>>>(in, out, n));
}

}  // namespace lrfg
