"""Device memory that a network holds between calls, counted through the
allocator hooks."""
import numpy as np
import pytest

from paper_2506_13072_gb300 import workloads as W

from gpu_common import fvlb

pytestmark = pytest.mark.gpu

KEPT = 262144               # samples whose memory a network may keep


@pytest.mark.parametrize("lattice", [W.D2Q9, W.D3Q19])
def test_large_inference_gives_its_memory_back(lattice):
    import torch

    F = fvlb()
    live = {}

    def alloc(n, ctx):
        p = torch.cuda.caching_allocator_alloc(int(n))
        live[p] = int(n)
        return p

    def free(p, ctx):
        live.pop(p)
        torch.cuda.caching_allocator_delete(p)

    hooks, others = (F.ALLOC_FN(alloc), F.FREE_FN(free)), F._alloc_refs
    F.check(F.lib.fvlb_set_allocator(*hooks, None))
    try:
        net = F.Mlp(lattice, capacity=64, seed=2)
    finally:                # the hooks are captured by the network
        F.check(F.lib.fvlb_set_allocator(*others, None))
    rng = np.random.default_rng(5)
    x = rng.standard_normal((KEPT + 70001, net.IN)).astype(np.float32)
    base = sum(live.values())
    y = net.infer(x)
    assert sum(live.values()) == base
    sample = 4 * (net.IN + net.OUT)
    net.grad(x[:1000], y[:1000])
    assert sum(live.values()) <= base + 1000 * sample + 256
    again = net.infer(x)    # with a smaller buffer kept
    assert np.array_equal(y, again)
    small = net.infer(x[:KEPT])
    assert np.array_equal(small, y[:KEPT])
    assert sum(live.values()) <= base + KEPT * sample + 256
    net.close()
    assert not live
