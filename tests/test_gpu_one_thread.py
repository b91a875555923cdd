"""One thread per node where it runs without bond tiles, and where FP64 begins to
use them: contexts whose bonds have no stencil (horizons other than 3 h) or reach
too far, and FP64 contexts of fewer nodes than one tile for each block that fits
the chip.  Forces and breaking against the oracle, the same bits on every form of
the step, and no step left to a few blocks."""
import numpy as np
import pytest
import torch

from oracle import oracle as O
from paper_2108_07212_gb300 import binding as B
from paper_2108_07212_gb300 import inputs as I

pytestmark = pytest.mark.gpu

# the per-step force tolerances of the two paths (of the largest nodal force)
TOL = {B.PD_FP64: 1e-12, B.PD_FP32_SPLIT: 1e-5}
PATHS = [(0, 1, 128), (2, 1, 128), (1, 1, 128), (1, 1, 256), (3, 1, 128), (3, 1, 256)]


def _grains(n, ratio=3.0, h_ratio=15):
    """Grains of every shape, about 412 nodes each (h_ratio 32: 1900)."""
    s = (n / 50) ** 0.5
    w = I.settling(n_grains=n, h_ratio=h_ratio, box=(20e-3 * s + 3e-3, 30e-3 * s + 3e-3), seed=3)
    w.params["horizon_ratio"] = ratio
    return w


def _edge():
    """Grains for one tile of 256 nodes for each of two blocks an SM, and half a tile less and more."""
    return round(2 * 256 * torch.cuda.get_device_properties(0).multi_processor_count / 412)


CASES = {
    "hor2": lambda: _grains(9, 2.0),                                       # 12 bonds, no stencil
    "hor4": lambda: _grains(9, 4.0),                                       # 48 bonds, no stencil
    "reach": lambda: I.two_disks(h_ratio=37, k_bulk=1e5, dt=1e-8),         # rows past the carried slots
    "few": lambda: I.two_disks(h_ratio=4, k_bulk=5e5),                     # fewer nodes than a block
    "below": lambda: _grains(int(0.9 * _edge())),                          # the last FP64 sizes without tiles
    "above": lambda: _grains(int(1.15 * _edge())),                         # the first with
    "wide": lambda: _grains(int(1.15 * _edge() * 412 / 1900), 3.0, 32),    # with, two rows of 63 nodes
}


def _state(X, seed, amp):
    rng = np.random.default_rng(seed)
    u = amp * 1e-3 * np.stack([np.sin(900 * X[:, 1] + 1), np.sin(700 * X[:, 0])], 1)
    return u, rng.normal(scale=0.2, size=X.shape)


@pytest.mark.parametrize("prec", [B.PD_FP64, B.PD_FP32_SPLIT])
@pytest.mark.parametrize("kind", list(CASES))
def test_forces_with_one_sided_breaks_match_the_oracle(prec, kind):
    w = CASES[kind]()
    P = O.OracleProblem.from_workload(w)
    S = B.Simulation(w, precision=prec, store_parts=True, device="cuda:0")
    u, v = _state(P.X, 5, 0.01)
    br = np.zeros(S.n_bonds, np.uint8)
    br[::17] = 1
    P.u[:], P.v[:] = u, v
    P.broken[: S.n_bonds] = br
    Fo, _ = P.forces()
    for path in [(0, 1, 128), (2, 1, 128)]:
        S.set_path(*path)
        S.set("DISP", u)
        S.set("VEL", v)
        S.set("BROKEN", br)
        S.eval_forces()
        err = np.abs(S.get("FORCE") - Fo).max() / np.abs(Fo).max()
        assert err <= TOL[prec], (path, err)
        assert np.array_equal(S.get("BROKEN"), P.broken[: S.n_bonds])


@pytest.mark.parametrize("prec", [B.PD_FP64, B.PD_FP32_SPLIT])
@pytest.mark.parametrize("kind", list(CASES))
def test_every_form_of_the_step_gives_the_same_bits(prec, kind):
    """Steps in which the strain passes the critical stretch in places."""
    w = CASES[kind]()
    w.params["Gc"] = 1e-4 * w.params["Gc"]
    runs = []
    for path in PATHS:
        S = B.Simulation(w, precision=prec, device="cuda:0")
        S.set_path(*path)
        u, v = _state(S.get("X"), 6, 0.02)
        S.set("DISP", u)
        S.set("VEL", v)
        S.step(12)
        runs.append((S.get("BROKEN"), S.get("DISP"), S.get("VEL")))
        S.close()
    assert 0 < runs[0][0].sum() < runs[0][0].size
    for path, got in zip(PATHS, runs):
        for a, b in zip(got, runs[0]):
            assert np.array_equal(a, b), path


@pytest.mark.parametrize("kind,most", [("hor4", 2.5), ("hor3", 2.0)])
def test_one_thread_per_node_is_spread_over_the_chip(kind, most):
    """FP64, 20600 nodes, kernel graph: one thread per node against four.  The four
    need about three quarters of the time; runs of 1024 nodes a block, which left
    most of the chip without work, took 3.3 (3 h) and 5.3 (4 h) times as long."""
    S = B.Simulation(_grains(50, 4.0 if kind == "hor4" else 3.0), precision=B.PD_FP64, device="cuda:0")
    best = {}
    for lanes in (1, 4):
        S.set_path(0, lanes, 128)
        S.step(8)
        t = []
        for _ in range(7):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            S.step(16)
            b.record()
            torch.cuda.synchronize()
            t.append(a.elapsed_time(b))
        best[lanes] = min(t)
    assert best[1] <= most * best[4], best
