// Batched tensor-train operations for solving several right-hand sides of one problem in lockstep: nb tensor
// trains of identical shape and ranks stored item after item (TTBatch), every launch covering all items.
// These are the block sum of Sec. 3.1 (the TT sum in block form), the inner products of Sec. 3.3 and the
// exponential-sum preconditioner of Sec. 2.3 in its low-rank form, each the batched counterpart of tt.cu's.
#include <algorithm>
#include <cmath>

#include "ops.cuh"

namespace lrfg {

void ttb_dot_device(lrfg_ctx* ctx, const TTBatchView& x, const TTBatchView& y, double* out_dev) {
  LRFG_REQUIRE(x.d == y.d && x.nb == y.nb, "batched dot of unlike batches");
  const int nb = x.nb;
  DBuf<double> W;
  for (int j = 0; j < x.d; ++j) {
    const int a = x.r[j], b = x.r[j + 1], c = y.r[j], e = y.r[j + 1], n = x.N[j];
    LRFG_REQUIRE(n == y.N[j], "dot of TTs on different grids");
    // V_i (c x (n b)) = W_i^T (c x a) x_i,j (a x (n b));  W'_i (b x e) = V_i^T y_i,j over (c n); W_i = 1 at the first
    // carriage
    DBuf<double> Vb;
    const double* V = x.core[0];
    if (j > 0) {
      Vb = DBuf<double>(ctx->pool, (size_t)c * n * b * nb);
      V = Vb.get();
      gemm(ctx, 1, 0, c, n * b, a, 1.0, W.get(), c, (long long)a * c, x.core[j], n * b, (long long)x.elems(j), 0.0,
           Vb.get(), n * b, (long long)c * n * b, nb);
    }
    double* dst = (j == x.d - 1) ? out_dev : nullptr;
    DBuf<double> Wn;
    if (!dst) { Wn = DBuf<double>(ctx->pool, (size_t)b * e * nb); dst = Wn.get(); }
    gemm(ctx, 1, 0, b, e, c * n, 1.0, V, b, (long long)c * n * b, y.core[j], e, (long long)y.elems(j), 0.0,
         dst, e, (long long)b * e, nb);
    if (j != x.d - 1) W = std::move(Wn);
  }
}

void ttb_precond(lrfg_ctx* ctx, const TTBatchView& x, const std::vector<double>& ts, const std::vector<double>& w,
                 int rmax, TTBatch& out, double tol, const TTView* omega, bool fp32, bool final) {
  const int d = x.d, nb = x.nb;
  const int R = (int)ts.size();
  std::vector<double> ones(R, 1.0);
  int rk[4];
  for (int j = 0; j <= d; ++j) rk[j] = (j == 0 || j == d) ? 1 : R * x.r[j];
  // the blocks G_m x_j of items b0 .. b0 + g - 1 in one launch: [m][item] (a x N x b each)
  auto blocks = [&](int j, int b0, int g) {
    const size_t e = x.elems(j);
    DBuf<double> t(ctx->pool, e * g * R);
    fibre_gauss_multi(ctx, x.core[j] + b0 * e, t.get(), (long long)(e * g), (long long)x.r[j] * g, x.N[j], x.r[j + 1],
                      ts.data(), (j == 0) ? w.data() : ones.data(), R, fp32);
    return t;
  };
  if (omega) {
    // the blocks enter the sketch contractions as they are (never embedded in the block-diagonal carriage)
    SketchSource z;
    z.kind = SketchSource::BLOCKS;
    z.d = d;
    z.nb = nb;
    z.nblocks = R;
    DBuf<double> terms[3];
    for (int j = 0; j < d; ++j) {
      z.N[j] = x.N[j];
      terms[j] = blocks(j, 0, nb);
      z.blocks[j] = terms[j].get();
      z.bstride[j] = (long long)(x.elems(j) * nb);
    }
    for (int j = 0; j <= d; ++j) {
      z.s[j] = rk[j];
      z.ry[j] = x.r[j];
    }
    tt_round_sketch(ctx, z, *omega, rmax, out, tol, fp32, final);
    return;
  }
  // deterministic rounding: the carriages are block rows (first), block diagonal (middle) and block columns (last) over
  // m.  The items of a batch are rounded together (their eigenproblems and factors run on an SM each), in groups whose
  // block-diagonal carriages stay below 1 GB; with a pool budget, or where the device has no room for a group, one at a time,
  // with one carriage's blocks at a time: the least memory the product takes.
  long long item_elems = 0;
  for (int j = 0; j < d; ++j) item_elems += (long long)rk[j] * x.N[j] * rk[j + 1];
  int group = ctx->pool->budget() ? 1 : (int)std::max(1LL, std::min<long long>(nb, (1LL << 27) / item_elems));
  auto round_items = [&](int b0, int g, TTBatch& part) {
    TTBatch big;
    ttb_alloc(ctx, big, d, x.N, rk, g);
    for (int j = 0; j < d; ++j) {
      const DBuf<double> t = blocks(j, b0, g);
      stack_blocks(ctx, t.get(), (long long)(x.elems(j) * g), x.r[j], x.N[j], x.r[j + 1], R,
                   j == 0 ? 0 : (j == d - 1 ? 2 : 1), g, big.core[j].get());
    }
    tt_round_batch(ctx, batch_view(big), rmax, part, tol);
  };
  std::vector<TTBatch> parts;
  for (int b0 = 0; b0 < nb;) {
    const int g = std::min(group, nb - b0);
    TTBatch part;
    try {
      round_items(b0, g, part);
    } catch (const Error& err) {
      if (err.status != LRFG_ENOMEM || g == 1) throw;
      group = 1;
      continue;
    }
    if (g == nb) {
      out = std::move(part);
      return;
    }
    parts.push_back(std::move(part));
    b0 += g;
  }
  LRFG_REQUIRE(tol == 0.0, "tolerance truncation of a batch in groups");
  ttb_alloc(ctx, out, d, x.N, parts[0].r, nb);
  int at = 0;
  for (TTBatch& q : parts) {
    for (int j = 0; j < d; ++j)
      LRFG_CUDA(cudaMemcpyAsync(out.core[j].get() + (size_t)at * out.elems(j), q.core[j].get(),
                                sizeof(double) * q.elems(j) * q.nb, cudaMemcpyDeviceToDevice, ctx->stream));
    at += q.nb;
  }
}

TTView item_view_of(const TTBatchView& x, int b) {
  TTView v{};
  v.d = x.d;
  for (int j = 0; j < 3; ++j) v.N[j] = x.N[j];
  for (int j = 0; j < 4; ++j) v.r[j] = x.r[j];
  for (int j = 0; j < x.d; ++j) v.core[j] = x.core[j] + (size_t)b * x.elems(j);
  return v;
}

}  // namespace lrfg
