"""A batch's update is the one of fvlb_step: where the arithmetic is FP32, its
order is fixed, so every instance of a batch has the bits of the same grid run
alone, periodic or walled, whatever the tile shape."""
import numpy as np
import pytest

from gpu_common import fvlb
from paper_2506_13072_gb300 import workloads as W

pytestmark = pytest.mark.gpu

# nx x ny, walls: one row and column, row starts off the 16-byte grid, rows
# that end inside a tile, several tiles and chunks; both fills of the 16-bit
# forms (pairs of nodes where nx is even, single nodes otherwise)
GRIDS = [((1, 1), 0), ((5, 3), 0), ((31, 2), 0), ((32, 32), 0), ((33, 40), 0), ((131, 70), 0),
         ((258, 33), 0), ((33, 40), 0b10), ((131, 70), 0b10), ((40, 9), 0b01)]


@pytest.mark.parametrize("tma", ["1", "0"])
@pytest.mark.parametrize("prec", [1, 2, 3])
def test_batch_has_the_bits_of_single_grids(prec, tma, monkeypatch):
    monkeypatch.setenv("FVLB_STAGE_TMA", tma)
    F = fvlb()
    probs = []
    for i, (shape, walls) in enumerate(GRIDS):
        pr = W.Problem("r", W.D2Q9, *shape, 1, 0.7 + 0.02 * i, 0.15, 11.0, W.FORCE_CONST,
                       (1e-5, -2e-5, 0.0), walls=walls)
        pr.u0, pr.p0, pr.A0 = W.random_smooth(pr.lattice, pr.shape, seed=i)
        probs.append(pr)
    steps = 41      # the first step, 18 of the tuner over its shapes, graph replays
    bt = F.Batch(probs, precision=prec)
    for i, pr in enumerate(probs):
        bt.init_fields(i, pr.u0, pr.p0, pr.A0)
    bt.step(steps)
    for i, pr in enumerate(probs):
        s = F.Simulation.from_problem(pr, precision=prec)
        s.init_fields(pr.u0, pr.p0, pr.A0)
        s.step(steps)
        for which in (F.FVLB_FIELD_U, F.FVLB_FIELD_P, F.FVLB_FIELD_A):
            assert np.array_equal(np.ravel(bt.fields(i, which)), np.ravel(s.fields(which))), \
                (pr.nx, pr.ny, pr.walls, which)
        s.close()
    bt.close()
