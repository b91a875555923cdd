"""Bond tiles (one thread per node: each stencil bond evaluated once and handed
to its other node through shared memory): forces and breaking against the
oracle and against the several-threads-per-node loops, where tiles can go
wrong -- runs shorter than a tile, rows at and past the reach of the carried
slots, bonds broken in one direction only, bonds that break during the step."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2108_07212_gb300 import binding as B
from paper_2108_07212_gb300 import inputs as I

pytestmark = pytest.mark.gpu

# the per-step force tolerances of the two paths (of the largest nodal force)
TOL = {B.PD_FP64: 1e-12, B.PD_FP32_SPLIT: 1e-5}
PATHS = [(1, 1, 128), (1, 1, 256), (0, 1, 128), (3, 1, 256)]


def _workload(kind):
    if kind == "small":                       # 386 nodes: shorter than two tiles
        return I.two_disks(h_ratio=8, k_bulk=5e5)
    if kind in ("reach128", "beyond"):        # rows of 63 nodes (two rows: 128 places) and of 67
        return I.two_disks(h_ratio=32 if kind == "reach128" else 34, k_bulk=1e5, dt=1e-8)
    return I.settling(n_grains=40, h_ratio=9, box=(20e-3, 30e-3), seed=3)   # every shape, gapped rows


def _state(P, seed, amp):
    rng = np.random.default_rng(seed)
    u = amp * 1e-3 * np.stack([np.sin(900 * P.X[:, 1] + 1), np.sin(700 * P.X[:, 0])], 1)
    return u, rng.normal(scale=0.2, size=P.X.shape)


def _push(S, u, v, broken):
    S.set("DISP", u)
    S.set("VEL", v)
    S.set("BROKEN", broken)


@pytest.mark.parametrize("prec", [B.PD_FP64, B.PD_FP32_SPLIT])
@pytest.mark.parametrize("kind", ["small", "reach128", "beyond", "shapes"])
@pytest.mark.parametrize("broken", ["none", "one_sided"])
def test_tile_forces_match_the_oracle(prec, kind, broken):
    """Forces of a strained state; one_sided: every 17th directed bond is broken
    (its other direction mostly is not), so slots hold markers."""
    w = _workload(kind)
    P = O.OracleProblem.from_workload(w)
    S = B.Simulation(w, precision=prec, store_parts=True, device="cuda:0")
    u, v = _state(P, 5, 0.01)
    br = np.zeros(S.n_bonds, np.uint8)
    if broken == "one_sided":
        br[::17] = 1
    P.u[:], P.v[:] = u, v
    P.broken[: S.n_bonds] = br
    Fo, _ = P.forces()
    for path in [(0, 1, 128), (2, 1, 128), (0, 4, 128)]:
        S.set_path(*path)
        _push(S, u, v, br)
        S.eval_forces()
        err = np.abs(S.get("FORCE") - Fo).max() / np.abs(Fo).max()
        assert err <= TOL[prec], (path, err)
        assert np.array_equal(S.get("BROKEN"), P.broken[: S.n_bonds])


@pytest.mark.parametrize("prec", [B.PD_FP64, B.PD_FP32_SPLIT])
@pytest.mark.parametrize("kind", ["small", "reach128", "beyond", "shapes"])
def test_tile_steps_do_not_depend_on_where_tiles_begin(prec, kind):
    """Twenty steps in which the strain passes the critical stretch in places.
    A node adds its bonds in one order wherever its tile begins, so every block
    size, the fused and the split force phase, and the persistent kernel and the
    kernel graph give the same bits.  Another number of threads per node sums in
    another order: the same bonds break, and FP64 states agree to 1e-10 (in the
    FP32 split that rounding can move a break by one step)."""
    w = _workload(kind)
    P = O.OracleProblem.from_workload(w)
    w.params["Gc"] = 1e-4 * w.params["Gc"]          # critical stretch / 100: below the strain's peaks
    u, v = _state(P, 6, 0.02)
    runs = []
    for path in [(0, 4, 128)] + PATHS:
        S = B.Simulation(w, precision=prec, device="cuda:0")
        S.set_path(*path)
        _push(S, u, v, np.zeros(S.n_bonds, np.uint8))
        S.step(20)
        runs.append((S.get("BROKEN"), S.get("DISP"), S.get("VEL")))
    lanes, tiles = runs[0], runs[1:]
    assert 0 < lanes[0].sum() < lanes[0].size
    for path, got in zip(PATHS, tiles):
        assert np.array_equal(got[0], lanes[0]), path
        for a, b in zip(got, tiles[0]):
            assert np.array_equal(a, b), path
        if prec == B.PD_FP64:
            for a, b in zip(got[1:], lanes[1:]):
                assert np.linalg.norm(a - b) <= 1e-10 * np.linalg.norm(b), path
