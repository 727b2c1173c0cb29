"""FP32 rows strided in memory where their tiles change (one row an SM, four rows and more, the largest tile), against NumPy's
FP64 transforms: 1e-6 of the largest value."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,outer,inner", [(625, 50, 20), (625, 1, 4900), (1701, 1, 700), (2187, 3, 3), (2401, 20, 20),
                                           (3125, 20, 20), (343, 1, 8000)])
def test_transform(ctx, N, outer, inner):
    rng = np.random.default_rng(N)
    z = (rng.standard_normal((outer, N, inner)) + 1j * rng.standard_normal((outer, N, inner))).astype(np.complex64)
    ref = np.fft.fft(z.astype(np.complex128), axis=1)
    got = ctx.fft_fibres(torch.as_tensor(z, device="cuda"), -1).cpu().numpy()
    assert np.abs(got - ref).max() <= 1e-6 * np.abs(ref).max()
