"""Transform tiles chosen by the number of fibres: FP64 and FP32 fibre FFTs at the fibre counts where the tile changes
(one fibre, one short of and past a fibre per SM, the switch to the largest tile), against torch.fft in FP64.  Tolerances
as for the fibre tests: 1e-12 N max|x| in FP64, 4 u_32 log2(N) sqrt(N) max|x| in FP32."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", [7, 63, 105, 135, 243])
@pytest.mark.parametrize("dtype", [torch.complex128, torch.complex64])
def test_fibre_counts(ctx, N, dtype):
    nsm = torch.cuda.get_device_properties(0).multi_processor_count
    for nfib in (1, 2, nsm - 1, nsm + 1, 3 * nsm + 7, 48 * nsm - 1, 48 * nsm + 1):
        for outer, inner in ((1, nfib), (nfib, 1)):
            g = torch.Generator(device="cuda").manual_seed(nfib)
            x = torch.randn((outer, N, inner, 2), generator=g, device="cuda", dtype=torch.float64)
            x = torch.view_as_complex(x).to(dtype)
            ref = torch.fft.fft(x.to(torch.complex128), dim=1)
            got = ctx.fft_fibres(x, -1)
            big = float(x.abs().max())
            tol = 1e-12 * N * big if dtype == torch.complex128 else 4 * 2.0 ** -24 * np.log2(N + 1) * np.sqrt(N) * big
            assert float((got - ref).abs().max()) <= tol, (outer, inner)
