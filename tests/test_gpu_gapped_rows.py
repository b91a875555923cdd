"""Nodes at the edge of a hole, whose lattice rows have a gap, in bond tiles:
forces and breaking against the oracle and the several-threads-per-node loops,
for holes cut at several lattice spacings."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2108_07212_gb300 import binding as B
from paper_2108_07212_gb300 import inputs as I

pytestmark = pytest.mark.gpu

# the per-step force tolerances of the two paths (of the largest nodal force)
TOL = {B.PD_FP64: 1e-12, B.PD_FP32_SPLIT: 1e-5}


def _workload(h_ratio):
    return I.settling(n_grains=6, h_ratio=h_ratio, box=(12e-3, 14e-3), seed=5, mix=("annulus", "plus"))


@pytest.mark.parametrize("prec", [B.PD_FP64, B.PD_FP32_SPLIT])
@pytest.mark.parametrize("h_ratio", [7, 15, 20, 31])
def test_forces_at_a_hole_match_the_oracle(prec, h_ratio):
    w = _workload(h_ratio)
    P = O.OracleProblem.from_workload(w)
    S = B.Simulation(w, precision=prec, store_parts=True, device="cuda:0")
    u = 1e-5 * np.stack([np.sin(900 * P.X[:, 1] + 1), np.sin(700 * P.X[:, 0])], 1)
    v = np.random.default_rng(8).normal(scale=0.2, size=P.X.shape)
    for br in (np.zeros(S.n_bonds, np.uint8), (np.arange(S.n_bonds) % 13 == 0).astype(np.uint8)):
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


@pytest.mark.parametrize("h_ratio", [15, 20])
def test_bonds_at_a_hole_break_alike_on_every_path(h_ratio):
    """FP64, twenty steps past the critical stretch in places."""
    w = _workload(h_ratio)
    X = O.OracleProblem.from_workload(w).X
    w.params["Gc"] = 1e-4 * w.params["Gc"]
    u = 2e-5 * np.stack([np.sin(900 * X[:, 1] + 1), np.sin(700 * X[:, 0])], 1)
    runs = []
    for path in [(0, 4, 128), (0, 1, 128), (1, 1, 128), (1, 1, 256), (3, 1, 256)]:
        S = B.Simulation(w, precision=B.PD_FP64, device="cuda:0")
        S.set_path(*path)
        S.set("DISP", u)
        S.step(20)
        runs.append((S.get("BROKEN"), S.get("DISP"), S.get("VEL")))
    assert 0 < runs[0][0].sum() < runs[0][0].size
    for got in runs[1:]:
        assert np.array_equal(got[0], runs[0][0])
        for a, b, first in zip(got, runs[1], runs[0]):
            assert np.array_equal(a, b)
            assert np.linalg.norm(a.astype(float) - first) <= 1e-10 * np.linalg.norm(first)
