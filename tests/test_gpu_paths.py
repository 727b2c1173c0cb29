"""The full-format operator through the passes its components share against the component-by-component passes (taken when a
pool budget has no room for the shared ones' work space), FP64 to 1e-12 and FP32 to the operator's 1e-5."""
import pytest
import torch

import paper_1902_07455_gb300 as lrfg
from synthetic import lognormal_grf

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(3, 3, 3), (27, 45, 63), (81, 9, 243), (35, 105, 11)])
@pytest.mark.parametrize("prec,tol", [(lrfg.FP64, 1e-12), (lrfg.MIXED, 1e-5)])
def test_shared_passes(ctx, shape, prec, tol):
    a = torch.as_tensor(lognormal_grf(3, max(shape) | 1, seed=5)[tuple(slice(0, n) for n in shape)].copy(), device="cuda")
    g = torch.Generator(device="cuda").manual_seed(3)
    v = torch.randn(shape, generator=g, device="cuda", dtype=torch.float64)
    ref = ctx.problem(a, lrfg.FULL, prec=prec).apply(ctx.field_from_full(v)).full(device=True)
    # the smallest budget the application runs in: grown until it no longer fails
    budget, got = 1 << 16, None
    while got is None:
        small = lrfg.Context(0, budget=budget)
        try:
            got = small.problem(a, lrfg.FULL, prec=prec).apply(small.field_from_full(v)).full(device=True).clone()
        except lrfg.LrfgError:
            budget += budget // 8
        finally:
            small.close()
    assert float((got - ref).norm() / ref.norm()) <= tol
