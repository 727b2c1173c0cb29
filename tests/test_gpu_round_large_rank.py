"""Rounding at bonds of stored rank above 3072, where the balancing's scales exceed 48 KB of shared memory (products with
the exponential sum reach it: 11 terms of rank 300), against the truncated SVD of the values.  The stored rank is far above
the numerical one (at most 9), so the Gram-SVD's 1e-8 of the largest singular value is what the rounding may lose."""
import numpy as np
import pytest
import torch

import paper_1902_07455_gb300 as lrfg

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("b", [3072, 3073, 3300])
@pytest.mark.parametrize("d", [2, 3])
def test_round(ctx, b, d):
    rng = np.random.default_rng(b)
    # the last bond of rank b (d = 3: behind one of rank 2)
    cores = [rng.standard_normal((1, 9, 2)), rng.standard_normal((2, 3, b))] if d == 3 else [rng.standard_normal((1, 9, b))]
    cores.append(rng.standard_normal((b, 7, 1)) / np.sqrt(b))
    x = lrfg.TTensor.from_numpy(cores)
    full = np.einsum("aib,bjc->aijc", cores[0], cores[1])[0, ..., 0] if d == 2 else \
        np.einsum("aib,bjc,ckd->ijk", *cores)
    lossless = ctx.tt_expand(ctx.tt_round(x, 9)).cpu().numpy()
    assert np.linalg.norm(lossless - full) <= 1e-8 * np.linalg.norm(full)
    if d == 2:
        u, s, vt = np.linalg.svd(full)
        ref = (u[:, :3] * s[:3]) @ vt[:3]
        got = ctx.tt_expand(ctx.tt_round(x, 3)).cpu().numpy()
        assert np.linalg.norm(got - ref) <= 1e-7 * np.linalg.norm(ref)
