"""Contact grid of a wall box with more cells than the grid may have: the cells
that hold nodes stay few to a node, whatever the box's shape.  A box with a distant
top, or side, wall against the close-fitting one: the same bits through rebuilds
of the lists, and rebuilds about as fast."""
import numpy as np
import pytest
import torch

from paper_2108_07212_gb300 import binding as B
from paper_2108_07212_gb300 import inputs as I

pytestmark = pytest.mark.gpu

# wall box over the close-fitting one: a column under a distant top, a bed
# beside a distant side wall, far both ways, and walls at no distance to speak of
SHAPES = [(1, 1e5), (1, 30), (1e5, 1), (1e4, 1e4), (3, 3)]


def _workload(nx, fx=1.0, fy=1.0, spread=1.0):
    """Grains in nx columns, at rest on one another, in a box fx by fy times as
    large; spread: rows as many times as far apart (and the box as high)."""
    R, rows = 1e-3, -(-48 // nx)
    w = I.settling(n_grains=48, h_ratio=11, seed=3)
    gap = 2.06 * 1.5 * R
    for g in range(48):
        w.grain_geom[g, :2] = gap * (g % nx + 0.5), gap * spread * (g // nx + 0.5)
    w.params["wall_lo"] = (0.0, 0.0)
    w.params["wall_hi"] = (gap * nx * fx, gap * rows * spread * fy)
    return w


def _rebuild_time(S):
    t = []
    for _ in range(9):
        S.clear_status()                     # the next evaluation rebuilds the lists
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        S.eval_forces()
        b.record()
        torch.cuda.synchronize()
        t.append(a.elapsed_time(b))
    return min(t)


@pytest.mark.parametrize("prec", [B.PD_FP64, B.PD_FP32_SPLIT])
@pytest.mark.parametrize("nx", [2, 12])
@pytest.mark.parametrize("shape", SHAPES)
def test_wide_boxes_rebuild_the_same_lists_as_fast(prec, nx, shape):
    # the FP32 split keeps positions relative to the box, so its bits and its cells follow the box's size
    if prec == B.PD_FP32_SPLIT and max(shape) > 100:
        pytest.skip("FP32 split: box sizes that leave its positions their precision")
    out, times = [], []
    for f in ((1, 1), shape):
        S = B.Simulation(_workload(nx, *f), precision=prec, device="cuda:0")
        S.set_path(2, 4, 128)
        S.set("VEL", 20.0 * np.random.default_rng(4).uniform(-1, 1, size=(48, 2))[S.get("GRAIN")])
        S.step(40)
        rc, st = S.status()
        assert rc == 0 and st[B.STATUS_REBUILDS] >= 3
        out.append((S.get("DISP"), S.get("VEL")))
        times.append(_rebuild_time(S))
        S.close()
    if prec == B.PD_FP64:
        for a, b in zip(*out):
            assert np.array_equal(a, b)
    assert times[1] <= 1.5 * times[0], times


@pytest.mark.parametrize("nx", [2, 12])
def test_grains_far_apart_rebuild_as_fast(nx):
    """More cells between the grains than the grid may have."""
    times = []
    for spread in (1, 300):
        S = B.Simulation(_workload(nx, spread=spread), precision=B.PD_FP64, device="cuda:0")
        times.append(_rebuild_time(S))
        S.close()
    assert times[1] <= 1.5 * times[0], times
