"""Calls that a context with a pool budget of this size has always had room for: a work space that grows past it turns them
into LRFG_ENOMEM.  The results are compared with those of a context without a budget, to the truncation's 1e-7."""
import pytest
import torch

import paper_1902_07455_gb300 as lrfg
from synthetic import lognormal_grf, random_tt

pytestmark = pytest.mark.gpu


def _check(ctx, budget, call):
    small = lrfg.Context(0, budget=budget)
    try:
        got = small.tt_expand(call(small)).clone()
    finally:
        small.close()
    ref = ctx.tt_expand(call(ctx))
    assert float((got - ref).norm()) <= 1e-7 * float(ref.norm())


@pytest.mark.parametrize("shape,ranks,eps,rmax,budget", [((729, 729), [20], 1e-3, 20, 34_500_000),
                                                         ((81, 81, 81), [8, 8], 1e-2, 8, 44_500_000)])
def test_precond(ctx, shape, ranks, eps, rmax, budget):
    x = random_tt(shape, ranks, seed=1)
    _check(ctx, budget, lambda c: c.tt_precond(lrfg.TTensor.from_numpy(x), eps, rmax))
