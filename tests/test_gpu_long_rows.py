"""The longest FP64 transforms a block's shared memory takes, 64 bytes a point up to 227 KB: every entry that runs them at the
lengths of prime factors up to 31 from 3553 on.  Tolerances: 1e-12 of the largest value for transforms and the operator, 1e-7 for
the truncated preconditioner, as for shorter ones elsewhere."""
import numpy as np
import pytest
import torch

import paper_1902_07455_gb300 as lrfg
from oracle import lowrank as lr
from synthetic import random_tt

pytestmark = pytest.mark.gpu

LENGTHS = [3553, 3575, 3591, 3625, 3627]


@pytest.mark.parametrize("N", LENGTHS)
def test_fibres(ctx, N):
    rng = np.random.default_rng(N)
    z = rng.standard_normal((2, N, 1)) + 1j * rng.standard_normal((2, N, 1))
    for sign, f in ((-1, np.fft.fft), (1, lambda v, axis: N * np.fft.ifft(v, axis=axis))):
        ref = f(z, axis=1)
        got = ctx.fft_fibres(torch.as_tensor(z, device="cuda"), sign).cpu().numpy()
        assert np.abs(got - ref).max() <= 1e-12 * np.abs(ref).max()
    x = rng.standard_normal((1, N, 3))
    ref = np.fft.ifft(2j * np.pi * np.fft.fftfreq(N, 1.0 / N)[None, :, None] * np.fft.fft(x, axis=1), axis=1).real
    got = ctx.fibre_operator(torch.as_tensor(x, device="cuda"), lrfg.MUL_DERIV).cpu().numpy()
    assert np.abs(got - ref).max() <= 1e-12 * np.abs(ref).max()


@pytest.mark.parametrize("N", LENGTHS)
def test_precond(ctx, N):
    shape, rmax, eps = (N, 3), 3, 1e-3
    x = random_tt(shape, [2], seed=5)
    op = lr.LowRankGaNi(lr.tt_from_separable([[np.ones(n) for n in shape]]), shape, fmt="tt", rank=rmax, pinv_eps=eps)
    ref = np.real(lr.tt_full(lr.tt_idft(op.T(lr.tt_hadamard(op.Pinv, lr.tt_dft(x))))))
    got = ctx.tt_expand(ctx.tt_precond(lrfg.TTensor.from_numpy(x), eps, rmax)).cpu().numpy()
    assert np.linalg.norm(got - ref) <= 1e-7 * np.linalg.norm(ref)


@pytest.mark.parametrize("shape", [(3, 3627), (3627, 3), (3, 3, 3625)])
def test_operator(ctx, shape):
    rng = np.random.default_rng(len(shape))
    a, v = np.exp(rng.standard_normal(shape)), rng.standard_normal(shape)
    v -= v.mean()
    ks = np.meshgrid(*[np.fft.fftfreq(n, 1.0 / n) for n in shape], indexing="ij")
    vh = np.fft.fftn(v)
    out = sum(-2j * np.pi * k * np.fft.fftn(a * np.fft.ifftn(2j * np.pi * k * vh)) for k in ks)
    kk = sum(k ** 2 for k in ks)
    ref = np.fft.ifftn(np.where(kk > 0, out / np.where(kk > 0, kk, 1.0), 0.0)).real
    P = ctx.problem(torch.as_tensor(a, device="cuda"), lrfg.FULL)
    got = P.apply(ctx.field_from_full(torch.as_tensor(v, device="cuda"))).full(device=True).cpu().numpy()
    assert np.abs(got - ref).max() <= 1e-12 * np.abs(ref).max()
