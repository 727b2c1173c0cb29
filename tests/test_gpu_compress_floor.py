"""Compressions whose rank or tolerance reaches the rounding of the Gram matrices: their error stays at the resolution of that
rounding, sqrt(eps) / 1.5 = 1e-8 of the values' norm (a larger share of eps ||G|| in the small eigenpairs goes straight into
it), and data of a low rank come back to rounding whatever rank is asked for."""
import numpy as np
import pytest
import torch

from synthetic import lognormal_grf

pytestmark = pytest.mark.gpu


def _err(ctx, a, rmax, tol=0.0):
    y = ctx.tt_compress(a, rmax, tol)
    return float((ctx.tt_expand(y) - a).norm() / a.norm()), y


@pytest.mark.parametrize("d,N,rmax,tol", [(2, 45, 22, 0.0), (2, 135, 67, 0.0), (3, 45, 33, 0.0), (3, 81, 40, 0.0),
                                          (2, 45, 45, 1e-9), (2, 135, 135, 1e-9), (3, 27, 27, 1e-9), (3, 45, 45, 1e-9),
                                          (3, 81, 81, 1e-9)])
def test_floor(ctx, d, N, rmax, tol):
    a = torch.as_tensor(lognormal_grf(d, N, ell=0.2, seed=3), device="cuda")
    assert _err(ctx, a, rmax, tol)[0] <= 1e-8


@pytest.mark.parametrize("scale", [1.0, 1e100, 1e-100])
@pytest.mark.parametrize("shape", [(135, 45), (27, 81, 9)])
def test_low_rank(ctx, shape, scale):
    rng = np.random.default_rng(len(shape))
    a = 0.0
    for _ in range(3):
        t = scale
        for n in shape:
            t = np.multiply.outer(t, rng.standard_normal(n))
        a = a + t
    a = torch.as_tensor(np.ascontiguousarray(a), device="cuda")
    for rmax in (3, 7, 9):
        e, y = _err(ctx, a, rmax)
        assert e <= 1e-13 and y.ranks[1:-1] == [rmax] * (len(shape) - 1)


def test_large_and_small_values(ctx):
    """the same at the ends of the range the Gram matrix has"""
    a = torch.as_tensor(lognormal_grf(2, 45, ell=0.2, seed=3), device="cuda")
    for scale in (2.0 ** 400, 2.0 ** -400):
        assert abs(_err(ctx, a * scale, 22)[0] - _err(ctx, a, 22)[0]) <= 1e-10
