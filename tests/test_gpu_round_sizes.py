"""TT rounding at the bond ranks where the pivoted Cholesky factor changes kernels (registers up to 32, 64 and 96 rows,
shared memory above) and where the symmetric products change tiles: a train of rank b stored with a redundant rank must
come back exactly when nothing is cut.  The Gram-SVD keeps directions above sqrt(eps) = 1e-8 of the largest, which covers
what the rounding may lose here; the left carriages are orthonormal to 1e-8 as elsewhere."""
import numpy as np
import pytest
import torch

import paper_1902_07455_gb300 as lrfg

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("b", [1, 2, 31, 32, 33, 63, 64, 65, 96, 97, 130])
@pytest.mark.parametrize("d", [2, 3])
def test_lossless(ctx, b, d):
    rng = np.random.default_rng(b)
    n = 135
    shape, ranks = (n,) * d, [1] + [b] * (d - 1) + [1]
    cores = [rng.standard_normal((ranks[j], n if j != 1 or d == 2 else 9, ranks[j + 1])) for j in range(d)]
    r = max(1, b // 2)
    # bond 1 of rank r, stored with b columns
    cores[0] = (cores[0][0, :, :r] @ rng.standard_normal((r, b)))[None]
    x = lrfg.TTensor.from_numpy(cores)
    y = ctx.tt_round(x, b)
    X, Y = ctx.tt_expand(x), ctx.tt_expand(y)
    assert float((X - Y).norm() / X.norm()) <= 1e-8
    q = y.cores[0][0, :, :r].cpu().numpy()
    assert np.abs(q.T @ q - np.eye(r)).max() <= 1e-8
    assert shape[0] == y.shape[0]
