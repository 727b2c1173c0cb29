"""Block sums in one launch: alpha x + beta y of trains of unequal ranks against the sum of their values, and the operator's
preconditioner with the items of a batch rounded together against item by item (a pool budget rounds them one at a
time)."""
import numpy as np
import pytest
import torch

import paper_1902_07455_gb300 as lrfg
from synthetic import lognormal_grf, random_tt

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape,rx,ry", [((9, 5), [1], [4]), ((63, 45), [7], [3]), ((9, 15, 7), [1, 1], [1, 1]),
                                         ((45, 27, 63), [3, 5], [6, 2])])
def test_add(ctx, shape, rx, ry):
    x, y = (lrfg.TTensor.from_numpy(random_tt(shape, r, seed=s)) for s, r in ((1, rx), (2, ry)))
    got = ctx.tt_add(0.75, x, -2.5, y)
    assert got.ranks == [1] + [a + b for a, b in zip(rx, ry)] + [1]
    ref = 0.75 * ctx.tt_expand(x) - 2.5 * ctx.tt_expand(y)
    assert float((ctx.tt_expand(got) - ref).abs().max()) <= 1e-13 * float(ref.abs().max()) * 16


@pytest.mark.parametrize("d,N", [(2, 45), (3, 27)])
def test_batched_precond_under_budget(ctx, d, N):
    a = ctx.tt_compress(torch.as_tensor(lognormal_grf(d, N, seed=3), device="cuda"), 4)
    kw = dict(rank=5, tol=1e-12, maxit=2, stop_on_increase=False)
    free = ctx.problem(a, lrfg.TT, **kw).aeff_tensor()
    small = lrfg.Context(0, budget=1 << 30)
    try:
        tight = small.problem(lrfg.TTensor([c.clone() for c in a.cores]), lrfg.TT, **kw).aeff_tensor()
    finally:
        small.close()
    assert np.abs(free - tight).max() <= 1e-9 * np.abs(free).max()
