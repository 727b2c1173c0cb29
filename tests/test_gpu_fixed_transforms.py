"""The fixed-point transforms of FP64 rows against the sum of their definition in extended precision: every butterfly and the
order of passes that a length takes, rows of very different size side by side, single entries, zero and subnormal rows,
and rows that are not finite beside rows that are.  Tolerance: a row's rounding is half a unit of 2^-53 at its input and
output and about a unit of the row's sum times 2^-61 per pass, taken as (1 + passes) 2^-52 of its 2-norm."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def _dft(x, sign):
    N = x.shape[1]
    j = np.outer(np.arange(N), np.arange(N)) % N
    ang = np.longdouble("6.283185307179586476925286766559005768") * np.arange(N, dtype=np.longdouble) / N
    c, s = np.cos(ang)[j], sign * np.sin(ang)[j]
    re, im = x.real.astype(np.longdouble), x.imag.astype(np.longdouble)
    return re @ c - im @ s, re @ s + im @ c


def _run(ctx, x, sign):
    y = ctx.fft_fibres(torch.as_tensor(x[:, :, None].copy(), device="cuda"), sign)
    return y.cpu().numpy()[:, :, 0]


@pytest.mark.parametrize("N", [3, 5, 7, 9, 11, 15, 31, 35, 99, 121, 243, 403, 729, 1215])
@pytest.mark.parametrize("sign", [-1, 1])
def test_rows(ctx, N, sign):
    rng = np.random.default_rng(N)
    x = rng.standard_normal((11, N)) + 1j * rng.standard_normal((11, N))
    x[1] = np.exp(3 * rng.standard_normal(N))          # all of one sign, far from its mean
    x[2] *= 1e-200
    x[3] *= 1e290
    x[4] = 0.0
    x[5] = 0.0
    x[5, N // 2] = 1.0 + 2.0j                          # one entry carries the row
    x[6] *= 10.0 ** rng.uniform(-30, 0, N)
    x[7] = 1.0
    x[8] = x[8].real
    x[9] *= 1e-310                                     # subnormal
    got = _run(ctx, x, sign)
    re, im = _dft(x, sign)
    passes = len([1 for p in (3, 5, 7, 11, 13, 31) for _ in range(12) if N % p == 0 and N % p ** (_ + 1) == 0])
    for r in range(11):
        e2 = (((got[r].real - re[r]) / np.longdouble(1)) ** 2 + (got[r].imag - im[r]) ** 2).sum()
        n2 = (re[r] ** 2 + im[r] ** 2).sum()
        assert np.sqrt(e2) <= (1 + passes) * 2.0 ** -52 * np.sqrt(n2) + N * 2.0 ** -1074, (r, np.sqrt(e2 / n2))


@pytest.mark.parametrize("N,rows", [(27, 1), (27, 5), (105, 40), (729, 3)])
def test_not_finite(ctx, N, rows):
    rng = np.random.default_rng(N + rows)
    x = rng.standard_normal((rows + 3, N)) + 1j * rng.standard_normal((rows + 3, N))
    clean = _run(ctx, x, -1)
    x[0, 1] = np.nan
    x[1, 2] = 1j * np.inf
    x[rows + 2, 0] = -np.inf
    got = _run(ctx, x, -1)
    for r in (0, 1, rows + 2):
        assert np.isnan(got[r].real).all() and np.isnan(got[r].imag).all()
    assert np.array_equal(got[2:rows + 2], clean[2:rows + 2])
