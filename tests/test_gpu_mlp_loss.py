"""The loss of a gradient call beside residuals of very different size."""
import numpy as np
import pytest

from paper_2506_13072_gb300 import workloads as W

from gpu_common import fvlb

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lattice", [W.D2Q9, W.D3Q19])
@pytest.mark.parametrize("n", [262144, 100003])
def test_loss_keeps_small_residuals(lattice, n):
    """A network of zeros gives 0, so the residuals are the targets: 1 for the
    first 14592 pairs (a tile of 32 for each of 456 blocks), 2^-12 (its square
    2^-24) for all others.
    Each product is exact; a pair's squares add up exactly, and so does any
    sum of them in FP64 (below 2^18 with 24 fractional bits), while an FP32
    sum drops 2^-24 beside 1.  Bound: the roundings of the one product with
    1 / (n OUT)."""
    F = fvlb()
    net = F.Mlp(lattice, capacity=64, seed=1)
    net.set_params(np.zeros_like(net.params()))
    x = np.ones((n, net.IN), np.float32)
    y = np.full((n, net.OUT), 2.0 ** -12, np.float32)
    y[:14592] = 1.0
    loss, _ = net.grad(x, y)
    ref = float((y.astype(np.float64) ** 2).mean())
    net.close()
    assert abs(loss - ref) <= 4 * 2.0 ** -53 * ref
