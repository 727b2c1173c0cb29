"""Rows of one FP64 butterfly (3 to 9 points) around the rows a block holds, under transforms and multipliers, against NumPy's
transforms: rounding of at most nine terms, 2^-50 of a row's norm."""
import numpy as np
import pytest
import torch

import paper_1902_07455_gb300 as lrfg

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", [3, 5, 7, 9])
@pytest.mark.parametrize("outer,inner", [(1, 1), (2, 31), (1, 65), (7, 1000)])
def test_fp64(ctx, N, outer, inner):
    rng = np.random.default_rng(N * inner)
    z = rng.standard_normal((outer, N, inner)) + 1j * rng.standard_normal((outer, N, inner))
    norm = np.sqrt(N) * np.linalg.norm(z, axis=1, keepdims=True)
    for sign, ref in ((-1, np.fft.fft(z, axis=1)), (1, N * np.fft.ifft(z, axis=1))):
        got = ctx.fft_fibres(torch.as_tensor(z, device="cuda"), sign).cpu().numpy()
        assert (np.abs(got - ref) <= 2.0 ** -50 * norm).all()
    k = np.fft.fftfreq(N, 1.0 / N)[None, :, None]
    ref = np.fft.ifft(2j * np.pi * k * np.fft.fft(z.real, axis=1), axis=1).real
    got = ctx.fibre_operator(torch.as_tensor(np.ascontiguousarray(z.real), device="cuda"), lrfg.MUL_DERIV).cpu().numpy()
    assert (np.abs(got - ref) <= 2.0 ** -50 * 2 * np.pi * N * norm).all()
