"""The work space of the full-format operator under a pool budget: which passes a problem takes is decided once, from its grid, the
budget and the blocks in use, so blocks the pool still caches from earlier work change no bit of an application; where
other blocks have taken the memory by then, the components run one by one, as in a context whose budget never had it, and
go on so."""
import gc

import pytest
import torch

import paper_1902_07455_gb300 as lrfg
from synthetic import lognormal_grf

pytestmark = pytest.mark.gpu

N = 27
SHAPES = [(N, N, N), (N, N)]


def _block(shape):  # a half spectrum's block in the pool
    half, b = 16 * (shape[-1] + 1) // 2, 256
    for n in shape[:-1]:
        half *= n
    while b < half:
        b *= 2
    return b


def _data(shape):
    a = torch.as_tensor(lognormal_grf(len(shape), N, seed=5), device="cuda")
    g = torch.Generator(device="cuda").manual_seed(3)
    return a, torch.randn(shape, generator=g, device="cuda", dtype=torch.float64)


def _apply(c, P, v):
    return P.apply(c.field_from_full(v)).full(device=True).clone()


@pytest.fixture
def setup(request):
    a, v = _data(request.param)
    block = _block(request.param)
    c = lrfg.Context(0)
    P = c.problem(a, lrfg.FULL)
    base = c.pool_bytes()[0]
    shared = _apply(c, P, v)
    del P
    c.close()
    c = lrfg.Context(0, budget=base + 4 * block)
    single = _apply(c, c.problem(a, lrfg.FULL), v)
    c.close()
    assert not torch.equal(shared, single)
    assert float((shared - single).norm() / single.norm()) <= 1e-12
    return a, v, block, base + 7 * block, shared, single


@pytest.mark.parametrize("setup", SHAPES, indirect=True)
def test_cached_blocks(setup):
    a, v, block, budget, shared, _ = setup
    c = lrfg.Context(0, budget=budget)
    other = torch.zeros((27,) * (a.dim() - 1) + (105,), dtype=torch.float64, device="cuda")  # blocks of another size
    f = c.field_from_full(other)
    del f
    gc.collect()
    assert c.pool_bytes()[1] >= 4 * block
    P = c.problem(a, lrfg.FULL)
    assert torch.equal(_apply(c, P, v), shared)
    del P
    c.close()


@pytest.mark.parametrize("setup", SHAPES, indirect=True)
def test_memory_gone(setup):
    a, v, block, budget, shared, single = setup
    c = lrfg.Context(0, budget=budget)
    P = c.problem(a, lrfg.FULL)
    held = []
    while budget - c.pool_bytes()[0] >= 4 * block:  # in, out and work space are four, an export needs three
        held.append(c.field_from_full(v))
    assert torch.equal(_apply(c, P, v), single)
    held.clear()
    gc.collect()
    assert torch.equal(_apply(c, P, v), single)
    del P
    P = c.problem(a, lrfg.FULL)
    assert torch.equal(_apply(c, P, v), shared)
    del P
    c.close()
