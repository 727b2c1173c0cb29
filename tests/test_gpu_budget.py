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


def test_compress(ctx):
    a = torch.as_tensor(lognormal_grf(3, 81, seed=5), device="cuda")
    _check(ctx, 10_900_000, lambda c: c.tt_compress(a, 10))


def test_solve(ctx):
    cores = ctx.tt_compress(torch.as_tensor(lognormal_grf(3, 27, seed=5), device="cuda"), 4).cores

    def solve(c):
        P = c.problem(lrfg.TTensor([x.clone() for x in cores]), lrfg.TT, rank=5, tol=1e-12, maxit=2, stop_on_increase=False)
        return P.solve([1.0, 0.0, 0.0], want_field=False)[0].Aeff

    small = lrfg.Context(0, budget=2_530_000)
    try:
        got = solve(small)
    finally:
        small.close()
    assert abs(got - solve(ctx)) <= 1e-9 * got
