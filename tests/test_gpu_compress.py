"""TT compression of grid values (App. A.3.3) where only the kept eigenpairs of each unfolding's Gram matrix are
decomposed: fixed ranks up to the full one and tolerances, against NumPy's TT-SVD.  A Gram matrix determines singular
vectors to eps (sigma_1 / sigma_k)^2 and drops content below sqrt(eps) sigma_1: 1e-8 of the tensor's norm covers both for
the kept values here (sigma_k >= 1e-4 sigma_1), and the rounding noise where every value is kept."""
import numpy as np
import pytest

from oracle import lowrank as lr
from synthetic import lognormal_grf, random_field

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def rel(a, b):
    return np.linalg.norm(a - b) / np.linalg.norm(b)


@pytest.mark.parametrize("shape,rmax", [((9, 7), 7), ((63, 243), 10), ((405, 49), 8), ((9, 15, 7), 1), ((15, 9, 21), 60),
                                        ((27, 175, 45), 6), ((175, 27, 35), 10)])
def test_fixed_rank(ctx, shape, rmax):
    A = random_field(shape, seed=4) if min(shape) < 20 else lognormal_grf(len(shape), max(shape), seed=3)[tuple(slice(0, n) for n in shape)]
    A = np.ascontiguousarray(A)
    ref = lr.tt_full(lr.tt_svd(A, rmax=rmax))
    got = ctx.tt_expand(ctx.tt_compress(torch.as_tensor(A, device="cuda"), rmax)).cpu().numpy()
    assert rel(got, ref) <= 1e-8


@pytest.mark.parametrize("shape,tol", [((63, 81), 1e-3), ((45, 27, 63), 1e-2)])
def test_tolerance_ranks(ctx, shape, tol):
    """The smallest ranks whose dropped tail is within tol / sqrt(d - 1) of the unfolding's norm, with every eigenvalue
    summed: the ranks NumPy's singular values give."""
    A = np.ascontiguousarray(lognormal_grf(len(shape), max(shape), seed=6)[tuple(slice(0, n) for n in shape)])
    got = ctx.tt_compress(torch.as_tensor(A, device="cuda"), 40, tol)
    s = np.linalg.svd(A.reshape(shape[0], -1), compute_uv=False)
    tail = np.sqrt(np.cumsum(s[::-1] ** 2)[::-1])
    k = int(np.argmax(np.append(tail, 0.0) <= tol / np.sqrt(len(shape) - 1) * tail[0]))
    assert got.ranks[1] == k
    assert rel(ctx.tt_expand(got).cpu().numpy(), A) <= tol
