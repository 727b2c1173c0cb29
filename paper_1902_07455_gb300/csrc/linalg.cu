// Dense FP64 building blocks for the rank truncation and the solvers: batched GEMM (Gram matrices and
// core contractions), a cyclic Jacobi eigensolver and reductions.
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
// Symmetric eigensolver by cyclic two-sided Jacobi rotations with the round-robin (circle) ordering, so that each round applies
// m'/2 disjoint rotations in parallel (Golub & Van Loan, "Matrix Computations", 4th ed., Sec. 8.5: the 2 x 2 symmetric Schur
// step and parallel orderings).  One block per matrix, working matrices in shared memory when they fit, else in a global
// scratch slice.  Its errors on small eigenvalues are a tenth of eps64 ||A||, the level of the rounding of a Gram matrix
// itself, where the tridiagonal solver's are eps64 ||A||: compressions that reach that level take it (see tt_compress).
// 46 ms for one matrix of 135 rows, against 1.45 ms for ten eigenpairs by the tridiagonal solver.
// syevj_floor is launched behind the tridiagonal solver and reads its eigenvalues on the device: the host, which has the
// compression's other launches to queue meanwhile, does not wait for them (80 us of a 3.5 ms compression).
// ------------------------------------------------------------------------------------------------
constexpr int kJacobiMaxSweeps = 30;
constexpr int kJacobiThreads = 512;

__device__ __forceinline__ void rr_pair(int round, int i, int mp, int* p, int* q) {
  // circle method: player mp-1 fixed, the others rotate
  const int n1 = mp - 1;
  if (i == 0) { *p = round % n1; *q = n1; return; }
  *p = (round + i) % n1;
  *q = (round - i + n1) % n1;
}

__device__ __forceinline__ double block_total(double v, double* red) {
  for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffff, v, o);
  __syncthreads();
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  double s = 0;
  for (int i = 0; i < (int)(blockDim.x >> 5); ++i) s += red[i];
  return s;
}

// power of two that brings the largest entry (bits of its upper word, over the block) near 1; red: 32 ints
__device__ double pow2_near_one(int hi_abs, int* red) {
  const int m = __reduce_max_sync(0xffffffff, hi_abs);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
  __syncthreads();
  int b = 0;
  for (int q = 0; q < (int)(blockDim.x >> 5); ++q) b = max(b, red[q]);
  const int ex = b >> 20;
  return ex == 0 || ex == 0x7ff ? 1.0 : __hiloint2double(min(2046, max(1, 2046 - ex)) << 20, 0);
}

// whether k eigenvalues w of a Gram matrix reach down to its rounding
__device__ __forceinline__ bool at_floor(const double* w, int k) { return w[k - 1] < 64.0 * 2.220446049250313e-16 * w[0]; }

// combinations of the columns or rows of C that judge what the known vectors leave of it
constexpr int kImages = 4;

// k > 0: only where the first k of the eigenvalues w, known already, reach the floor, and the k vectors known (in Vout) leave more
// than 1e-13 of C (m x n, or of_rows 0: n x m, whose Gram matrix is given): of four combinations of its columns (rows)
// with random signs
__global__ void __launch_bounds__(kJacobiThreads) jacobi_kernel(const double* __restrict__ Ag, double* w,
                                                               double* Vout, int m, double* scratch, int use_smem,
                                                               double eps, int k, const double* __restrict__ C, int n,
                                                               int of_rows) {
  extern __shared__ __align__(16) unsigned char smraw[];
  const int mp = m + (m & 1);
  const int npair = mp / 2;
  double* cs = (double*)smraw;                         // 2 npair (c, s)
  int* pq = (int*)(cs + 2 * npair);                    // 2 npair
  double* red = (double*)(pq + 2 * npair);             // 32 partial sums
  int* rank = (int*)(red + 32);                        // m (+1) ints
  double* A;
  double* V;
  if (use_smem == 2) {         // A and V in shared memory
    A = (double*)(rank + m + (m & 1));
    V = A + (size_t)m * m;
  } else if (use_smem == 1) {  // A in shared memory, V in a global scratch slice
    A = (double*)(rank + m + (m & 1));
    V = scratch + (size_t)blockIdx.x * m * m;
  } else {
    A = scratch + (size_t)blockIdx.x * 2 * m * m;
    V = A + (size_t)m * m;
  }
  if (k > 0) {
    if (!at_floor(w, k)) return;
    double *Y = A, *T = A + m * kImages;  // m x 4, k x 4
    const int lane = threadIdx.x & 31, part = of_rows ? lane : 0, step = of_rows ? 32 : 1;
    for (int i = of_rows ? threadIdx.x >> 5 : threadIdx.x; i < m; i += of_rows ? blockDim.x >> 5 : blockDim.x) {
      double y[kImages] = {0.0, 0.0, 0.0, 0.0};
      for (int j = part; j < n; j += step) {
        const double v = of_rows ? C[(size_t)i * n + j] : C[(size_t)j * m + i];
        const unsigned h = ((unsigned)j + 1u) * 2654435761u, bits = (h ^ (h >> 15)) * 2246822519u;
#pragma unroll
        for (int l = 0; l < kImages; ++l) y[l] += (bits >> (28 + l) & 1u) ? v : -v;
      }
#pragma unroll
      for (int l = 0; l < kImages; ++l) {
        if (of_rows)
          for (int o = 16; o; o >>= 1) y[l] += __shfl_xor_sync(0xffffffff, y[l], o);
        if (part == 0) Y[i * kImages + l] = y[l];
      }
    }
    __syncthreads();
    for (int q = threadIdx.x; q < k * kImages; q += blockDim.x) {
      const int t = q % k, l = q / k;
      double s = 0.0;
      for (int i = 0; i < m; ++i) s = fma(Vout[(size_t)i * m + t], Y[i * kImages + l], s);
      T[q] = s;
    }
    __syncthreads();
    double all = 0.0, left = 0.0;
    for (int q = threadIdx.x; q < m * kImages; q += blockDim.x) {
      const int i = q / kImages, l = q % kImages;
      double r = Y[q];
      all = fma(r, r, all);
      for (int t = 0; t < k; ++t) r = fma(-Vout[(size_t)i * m + t], T[l * k + t], r);
      left = fma(r, r, left);
    }
    all = block_total(all, red);
    left = block_total(left, red);
    if (left <= 1e-26 * all) return;
    __syncthreads();
  }
  const double* Ain = Ag + (size_t)blockIdx.x * m * m;
  // scaled by a power of two to entries near 1, so that the squares stay in range
  int top = 0;
  for (int t = threadIdx.x; t < m * m; t += blockDim.x) {
    A[t] = Ain[t];
    V[t] = ((t / m) == (t % m)) ? 1.0 : 0.0;
    top = max(top, __double2hiint(A[t]) & 0x7fffffff);
  }
  const double scale = pow2_near_one(top, (int*)red);
  double loc = 0.0;
  for (int t = threadIdx.x; t < m * m; t += blockDim.x) {
    A[t] *= scale;
    loc += A[t] * A[t];
  }
  const double fro2 = block_total(loc, red);
  const double tol2 = 16.0 * eps * eps * fro2;
  double prev_off = fro2;
  if (m > 1 && fro2 > 0.0) {
    for (int sweep = 0; sweep < kJacobiMaxSweeps; ++sweep) {
      for (int round = 0; round < mp - 1; ++round) {
        for (int i = threadIdx.x; i < npair; i += blockDim.x) {
          int p, q;
          rr_pair(round, i, mp, &p, &q);
          if (p > q) { int t = p; p = q; q = t; }
          double c = 1, s = 0;
          if (q < m) {
            double apq = A[(size_t)p * m + q];
            double app = A[(size_t)p * m + p], aqq = A[(size_t)q * m + q];
            if (apq != 0.0 && fabs(apq) > 0.01 * eps * sqrt(fabs(app * aqq))) {
              double tau = (aqq - app) / (2.0 * apq);
              double t = (tau >= 0.0 ? 1.0 : -1.0) / (fabs(tau) + sqrt(1.0 + tau * tau));
              c = 1.0 / sqrt(1.0 + t * t);
              s = t * c;
            }
          } else {
            q = -1;
          }
          cs[2 * i] = c;
          cs[2 * i + 1] = s;
          pq[2 * i] = p;
          pq[2 * i + 1] = (s == 0.0) ? -1 : q;
        }
        __syncthreads();
        // rows: A <- J^T A
        for (int t = threadIdx.x; t < npair * m; t += blockDim.x) {
          int i = t / m, j = t - (t / m) * m;
          int q = pq[2 * i + 1];
          if (q < 0) continue;
          int p = pq[2 * i];
          double c = cs[2 * i], s = cs[2 * i + 1];
          double ap = A[(size_t)p * m + j], aq = A[(size_t)q * m + j];
          A[(size_t)p * m + j] = c * ap - s * aq;
          A[(size_t)q * m + j] = s * ap + c * aq;
        }
        __syncthreads();
        // columns: A <- A J, V <- V J
        for (int t = threadIdx.x; t < npair * m; t += blockDim.x) {
          int i = t / m, j = t - (t / m) * m;
          int q = pq[2 * i + 1];
          if (q < 0) continue;
          int p = pq[2 * i];
          double c = cs[2 * i], s = cs[2 * i + 1];
          double ap = A[(size_t)j * m + p], aq = A[(size_t)j * m + q];
          A[(size_t)j * m + p] = c * ap - s * aq;
          A[(size_t)j * m + q] = s * ap + c * aq;
          double vp = V[(size_t)j * m + p], vq = V[(size_t)j * m + q];
          V[(size_t)j * m + p] = c * vp - s * vq;
          V[(size_t)j * m + q] = s * vp + c * vq;
        }
        __syncthreads();
      }
      double off = 0;
      for (int t = threadIdx.x; t < m * m; t += blockDim.x) {
        int i = t / m, j = t - (t / m) * m;
        if (i != j) off += A[t] * A[t];
      }
      off = block_total(off, red);
      // converged, or rounding has stopped the decrease (off-diagonal mass at the precision floor)
      if (off <= tol2 || (off > 0.25 * prev_off && off <= 4096.0 * eps * eps * fro2)) break;
      prev_off = off;
    }
  }
  // sort descending: rank[j] = position of eigenvalue j (ties by index)
  for (int j = threadIdx.x; j < m; j += blockDim.x) {
    double lj = A[(size_t)j * m + j];
    int pos = 0;
    for (int i = 0; i < m; ++i) {
      double li = A[(size_t)i * m + i];
      if (li > lj || (li == lj && i < j)) ++pos;
    }
    rank[j] = pos;
  }
  __syncthreads();
  double* wb = w + (size_t)blockIdx.x * m;
  double* Vb = Vout + (size_t)blockIdx.x * m * m;
  for (int j = threadIdx.x; j < m; j += blockDim.x) wb[rank[j]] = A[(size_t)j * m + j] / scale;
  for (int t = threadIdx.x; t < m * m; t += blockDim.x) {
    int i = t / m, j = t - (t / m) * m;
    Vb[(size_t)i * m + rank[j]] = V[t];
  }
}

static void jacobi_launch(lrfg_ctx* ctx, const double* A, double* w, double* V, int m, int batch, int k,
                          const double* C, int n, bool of_rows) {
  const int npair = (m + 1) / 2;
  size_t head = sizeof(double) * 2 * npair + sizeof(int) * 2 * npair + sizeof(double) * 32 + sizeof(int) * (m + (m & 1));
  head = (head + 15) / 16 * 16;
  const size_t limit = (size_t)std::min(ctx->max_smem_optin, 220 * 1024);
  const size_t one = head + sizeof(double) * (size_t)m * std::max(m, 2 * kImages), two = one + sizeof(double) * (size_t)m * m;
  const int use_smem = two <= limit ? 2 : (one <= limit ? 1 : 0);
  const size_t smem = use_smem == 2 ? two : (use_smem == 1 ? one : head);
  DBuf<double> scratch;
  if (use_smem < 2) scratch = DBuf<double>(ctx->pool, (size_t)(2 - use_smem) * m * m * batch);
  LRFG_CUDA(raise_smem_limit((const void*)jacobi_kernel, smem));
  // one sweep of the two-sided cyclic Jacobi costs about 9 m^3 flops (rows, columns and V)
  LRFG_LAUNCH(ctx, KC_EIGEN, k > 0 ? 0.0 : 9.0 * (double)m * m * m * batch, k > 0 ? 0.0 : 3.0 * sizeof(double) * (double)m * m * batch,
              jacobi_kernel<<<batch, kJacobiThreads, smem, ctx->stream>>>(A, w, V, m, scratch.get(), use_smem,
                                                                         2.220446049250313e-16, k, C, n, of_rows));
}

void syevj(lrfg_ctx* ctx, const double* A, double* w, double* V, int m, int batch) {
  if (m <= 0 || batch <= 0) return;
  jacobi_launch(ctx, A, w, V, m, batch, 0, nullptr, 0, false);
}

void syevj_floor(lrfg_ctx* ctx, const double* G, double* w, double* V, int m, int k, const double* C, int n, bool of_rows) {
  jacobi_launch(ctx, G, w, V, m, 1, k, C, n, of_rows);
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
