"""The fused step at the edges of its tiles and launch rules: row starts off
the 16-byte grid (padded stage), rows that end inside a tile, one-plane and
ragged chunks, and grids on both sides of the choice between the one-warp and
the wide tile.  Checked against the split kernels (one thread per node, no
staging), and with bulk tensor copies against plain copies bit for bit."""
import numpy as np
import pytest

from gpu_common import gpu_sim, rel_l2
from paper_2506_13072_gb300 import workloads as W

pytestmark = pytest.mark.gpu

FP64, FP32, FP16, BF16 = 0, 1, 2, 3

SHAPES_2D = [(5, 3), (31, 2), (33, 40), (127, 9), (129, 65), (131, 700), (258, 333), (1030, 257)]
SHAPES_3D = [(3, 2, 2), (31, 3, 5), (33, 7, 4), (65, 5, 33), (66, 30, 40), (100, 41, 37), (127, 64, 20)]


def _problem(shape, walls):
    if len(shape) == 2:
        pr = W.Problem("r", W.D2Q9, *shape, 1, 0.7, 0.15, 11.0, W.FORCE_CONST, (1e-5, -2e-5, 0.0),
                       walls=walls)
    else:
        pr = W.Problem("r3", W.D3Q19, *shape, 0.75, 0.1, 13.0, W.FORCE_CONST, (1e-5, 2e-5, -1e-5),
                       walls=walls)
    pr.u0, pr.p0, pr.A0 = W.random_smooth(pr.lattice, pr.shape, seed=sum(shape) + walls)
    return pr


# fused and split differ by roundings only: per step about eps (FP64 2e-16,
# FP32 1.2e-7, 16-bit storage half an ulp 2.4e-4 / 2e-3 of the largest stored
# value) times a few operations; p is of size 0.1 |u| in these units
TOL = {FP64: 1e-12, FP32: 1e-5, FP16: 2e-3, BF16: 1.6e-2}


@pytest.mark.parametrize("prec", [FP64, FP32, FP16, BF16])
@pytest.mark.parametrize("shape,walls", [(s, w) for s in SHAPES_2D for w in (0, 0b10, 0b01)]
                         + [(s, w) for s in SHAPES_3D for w in (0, 0b110, 0b001)])
def test_tile_edges_against_split(shape, walls, prec):
    pr = _problem(shape, walls)
    got = []
    for kernel in (0, 1):
        s = gpu_sim(pr, prec, kernel)
        s.step(7)
        got.append((s.u(), s.A(), s.p()))
        s.close()
    (u, A, p), (ur, Ar, prf) = got
    assert rel_l2(u, ur, 1e-30) <= TOL[prec]
    assert rel_l2(A, Ar, 1e-30) <= TOL[prec]
    assert np.linalg.norm(p - prf) <= TOL[prec] * max(np.linalg.norm(prf), 0.1 * np.linalg.norm(ur))


@pytest.mark.parametrize("prec", [FP64, FP32, FP16, BF16])
@pytest.mark.parametrize("shape,walls", [((33, 40), 0), ((131, 300), 0b10), ((37, 5), 0b01),
                                         ((66, 30, 40), 0), ((35, 9, 6), 0b011), ((101, 4, 3), 0b100)])
def test_padded_stage_bitwise(prec, shape, walls, monkeypatch):
    pr = _problem(shape, walls)
    out = []
    for flag in ("1", "0"):
        monkeypatch.setenv("FVLB_STAGE_TMA", flag)
        s = gpu_sim(pr, prec)
        s.step(9)
        out.append(np.concatenate([s.u().ravel(), s.A().ravel(), s.p().ravel()]))
        s.close()
    assert np.array_equal(out[0], out[1])


@pytest.mark.parametrize("prec", [FP64, FP32, FP16])
@pytest.mark.parametrize("shape", [(64, 40), (40, 9, 6)])
def test_steps_in_a_captured_graph(shape, prec):
    """Consecutive launches overlap their starts and ends; replayed from a
    captured graph (two steps, so the buffers return to their places) they
    give the same fields as launched directly."""
    import torch

    pr = _problem(shape, 0b10)
    out = []
    for captured in (False, True):
        st = torch.cuda.Stream()
        s = gpu_sim(pr, prec)
        s.synchronize()
        s.set_stream(st)
        s.step(2)
        st.synchronize()
        if captured:
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g, stream=st):
                s.step(2)
            with torch.cuda.stream(st):
                for _ in range(4):
                    g.replay()
            st.synchronize()
        else:
            s.step(8)
        out.append(np.concatenate([s.u().ravel(), s.A().ravel(), s.p().ravel()]))
        s.close()
    assert np.array_equal(out[0], out[1])


@pytest.mark.parametrize("shape,walls", [((131, 300), 0b10), ((33, 40), 0), ((33, 7, 4), 0),
                                         ((66, 30, 40), 0b110), ((100, 41, 37), 0), ((64, 3, 70), 0b001)])
def test_closure_tile_edges(shape, walls):
    """The learned closure's tile (fill threads with two ring slots in 3D, counts
    added up per tile): with no network value accepted it is the plain step,
    and every node update is counted once."""
    from paper_2506_13072_gb300 import fvlb as F
    pr = _problem(shape, walls)
    net = F.Mlp(pr.lattice, seed=3)
    out = []
    for tol in (None, 1e-12):
        s = gpu_sim(pr, FP32)
        if tol is not None:
            s.set_closure(net, tol=tol)
        s.step(7)
        out.append((s.u(), s.A()))
        if tol is not None:
            st = s.closure_stats()
            assert st["fallback"] == 7 * pr.sites and st["network"] == 0
        s.close()
    net.close()
    assert rel_l2(out[1][0], out[0][0], 1e-30) <= TOL[FP32]
    assert rel_l2(out[1][1], out[0][1], 1e-30) <= TOL[FP32]
