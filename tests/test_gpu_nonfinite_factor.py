"""Data that a Gram factor cannot hold stay visible: a NaN, or entries whose squares overflow, make a truncation NaN as a whole at
every kernel of the pivoted Cholesky (registers up to 32, 64 and 96 rows, above them shared memory), not the zero tensor of a
factor of rank 0; with the deterministic rounding and the randomised one."""
import pytest
import torch

import paper_1902_07455_gb300 as lrfg
from synthetic import random_tt

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("r", [4, 40, 80, 100, 130])
@pytest.mark.parametrize("j", [0, 1, 2])
@pytest.mark.parametrize("value", [float("nan"), 1e200])
def test_round(ctx, r, j, value):
    x = lrfg.TTensor.from_numpy(random_tt((135, 9, 135), [r, r], seed=r))
    x.cores[j].view(-1)[7] = value
    assert bool(torch.isnan(ctx.tt_expand(ctx.tt_round(x, 5))).all())


@pytest.mark.parametrize("value", [float("nan"), 1e200])
def test_round_2d(ctx, value):
    for r in (30, 110):
        x = lrfg.TTensor.from_numpy(random_tt((135, 135), [r], seed=r))
        x.cores[1].view(-1)[3] = value
        assert bool(torch.isnan(ctx.tt_expand(ctx.tt_round(x, 5))).all())
