"""The FP64 full-format operator in d = 2 (both components in each launch) against FFTs of the whole grid: the smallest grids,
axes much longer than the other, prime factors 3 to 31, an axis whose fibres of both components exceed shared memory (the
components run one by one), with and without an anisotropic part.  Tolerance 1e-12 of the largest value, as for FP64 results
of the operator elsewhere."""
import math

import numpy as np
import pytest
import torch

import paper_1902_07455_gb300 as lrfg

pytestmark = pytest.mark.gpu


def _apply(a, v, B):
    ks = np.meshgrid(*[np.fft.fftfreq(n, 1.0 / n) for n in a.shape], indexing="ij")
    vh, out = np.fft.fftn(v), 0.0
    for k in ks:
        out = out - 2j * math.pi * k * np.fft.fftn(a * np.fft.ifftn(2j * math.pi * k * vh))
    if B is not None:
        out = out + 4 * math.pi ** 2 * sum(B[i][j] * ks[i] * ks[j] for i in range(2) for j in range(2)) * vh
    kk = ks[0] ** 2 + ks[1] ** 2
    return np.fft.ifftn(np.where(kk > 0, out / np.where(kk > 0, kk, 1.0), 0.0)).real


@pytest.mark.parametrize("shape", [(3, 3), (5, 3), (3, 31), (31, 33), (63, 105), (243, 27), (27, 343), (729, 9), (2187, 5),
                                   (2625, 3)])
@pytest.mark.parametrize("aniso", [False, True])
def test_apply(ctx, shape, aniso):
    rng = np.random.default_rng(sum(shape))
    a = np.exp(rng.standard_normal(shape))
    v = rng.standard_normal(shape)
    v -= v.mean()
    B = np.array([[2.0, 0.5], [0.5, 1.0]]) if aniso else None
    P = ctx.problem(torch.as_tensor(a, device="cuda"), lrfg.FULL, B=B)
    got = P.apply(ctx.field_from_full(torch.as_tensor(v, device="cuda"))).full(device=True).cpu().numpy()
    ref = _apply(a, v, B)
    assert np.abs(got - ref).max() <= 1e-12 * np.abs(ref).max()
