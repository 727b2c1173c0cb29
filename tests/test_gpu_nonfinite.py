"""A NaN stays one: truncations and eigenpairs of data with a NaN are NaN as a whole, not the zeros or unit vectors of a
factor of rank 0 (the register Cholesky of up to 32, 64 and 96 rows, the eigensolver's register and shared-memory
tridiagonalisations)."""
import pytest
import torch

import paper_1902_07455_gb300 as lrfg
from synthetic import random_tt

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("r", [4, 40, 80])
@pytest.mark.parametrize("j", [0, 1, 2])
def test_round(ctx, r, j):
    x = lrfg.TTensor.from_numpy(random_tt((81, 45, 81), [r, r], seed=r))
    x.cores[j].view(-1)[7] = float("nan")
    assert bool(torch.isnan(ctx.tt_expand(ctx.tt_round(x, 5))).all())


@pytest.mark.parametrize("n", [2, 30, 60, 90, 135])
def test_eig(ctx, n):
    A = torch.eye(n, dtype=torch.float64, device="cuda").repeat(2, 1, 1)
    A[0, n // 2, n - 1] = A[0, n - 1, n // 2] = float("nan")
    w, V = ctx.sym_eig(A, min(n, 5))
    assert bool(torch.isnan(w[0]).all()) and bool(torch.isnan(V[0]).all())
    assert float((w[1] - 1.0).abs().max()) <= 1e-13
