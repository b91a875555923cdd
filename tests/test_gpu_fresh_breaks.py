"""Contacts of bonds that broke after the candidate lists were built.

The lists leave out pairs with an intact bond; a bond that breaks later brings
its pair back from the broken bits, without a rebuild.  A lattice pressed
together below the contact radius makes such pairs exert self-contact forces at
once: against the oracle, for bonds broken between the steps and in the step,
on every form of the force phase.  In the step some stretches lie so close to
the critical one that the FP32 split decides them in FP64, also at the edge of a
grain, where a node lacks neighbours.  And the order of a node's contacts does
not depend on when its list was built."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2108_07212_gb300 import binding as B
from paper_2108_07212_gb300 import inputs as I

pytestmark = pytest.mark.gpu

# the per-step force tolerances of the two paths (of the largest nodal acceleration)
TOL = {B.PD_FP64: 1e-12, B.PD_FP32_SPLIT: 1e-5}
PATHS = [(0, 1, 128), (2, 1, 128), (1, 1, 128), (3, 1, 256), (0, 4, 128), (2, 2, 128), (1, 4, 128), (3, 8, 128)]
H = 1e-3 / 8


def _pressed(press, Gc=None, ratio=3.0):
    """Two disks, every lattice pressed by `press` about its centre (0.95 h is the
    contact radius): workload, oracle, displacement, velocity."""
    w = I.two_disks(h_ratio=8, k_bulk=5e5, dt=2e-8, horizon_ratio=ratio, gap=0.4e-3, floor_gap=0.3e-3)
    if Gc:
        w.params["Gc"] = Gc
    P = O.OracleProblem.from_workload(w)
    u = -press * (P.X - w.grain_geom[P.grain, :2])
    v = np.random.default_rng(2).normal(scale=0.2, size=P.X.shape)
    return w, P, u, v


def _some_bonds(P, seed, share):
    """The directed bonds of a random share of the undirected ones, both directions."""
    src = np.repeat(np.arange(P.N), np.diff(P.row_ptr))
    lo, hi = np.minimum(src, P.col).astype(np.int64), np.maximum(src, P.col).astype(np.int64)
    _, pair = np.unique(lo * P.N + hi, return_inverse=True)
    return (np.random.default_rng(seed).random(pair.max() + 1) < share)[pair].astype(np.uint8)


def _wave(P):
    """A wave of 0.025 h that changes stretches by 1.7 % and moves no node past the
    rebuild trigger of 0.045 R_c."""
    return 0.025 * H * np.stack([np.sin(0.7 / H * P.X[:, 0]), np.sin(0.7 / H * P.X[:, 1])], 1)


def _rebuilds(S):
    return int(S.status()[1][B.STATUS_REBUILDS])


@pytest.mark.parametrize("prec", [B.PD_FP64, B.PD_FP32_SPLIT])
@pytest.mark.parametrize("ratio", [3.0, 4.0])           # 24 and up to 48 bonds a node
@pytest.mark.parametrize("when", ["between", "during"])
def test_contacts_of_fresh_breaks_match_the_oracle(prec, ratio, when):
    if when == "between":
        w, P, u, v = _pressed(0.08, ratio=ratio)
        u1, br = u, _some_bonds(P, 3, 0.3)
    else:
        # critical stretch 0.08, lattice at 0.07: the wave takes some bonds past it
        w, P, u, v = _pressed(0.07, ratio=ratio)
        _, s0 = O.bond_constants(w.params["E"], w.params["nu"], w.params["Gc"], ratio * H)
        w, P, u, v = _pressed(0.07, Gc=w.params["Gc"] * (0.08 / s0) ** 2, ratio=ratio)
        u1, br = u + _wave(P), np.zeros(len(P.col), np.uint8)
    P.u[:], P.v[:] = u1, v
    P.broken[: len(br)] = br
    P.a[:] = 0.0
    _, parts = P.run(1, want_parts=True)
    broken = P.broken[: len(br)]
    assert np.abs(parts[1]).max() > 0.05 * np.abs(parts[0]).max()      # self-contact counts
    assert when == "between" or 0.05 < broken.mean() < 0.95
    for path in PATHS:
        S = B.Simulation(w, precision=prec, device="cuda:0")
        S.set_path(*path)
        S.set("DISP", u)
        S.eval_forces()                                  # lists without the bonded pairs
        assert not S.get("BROKEN").any()
        n = _rebuilds(S)
        S.set("DISP", u1)
        S.set("VEL", v)
        S.set("ACC", np.zeros_like(v))
        S.set("BROKEN", br)
        S.step(1)
        assert _rebuilds(S) == n, path
        assert np.array_equal(S.get("BROKEN"), broken), path
        err = np.abs(S.get("ACC") - P.a).max() / np.abs(P.a).max()
        assert err <= TOL[prec], (path, err)


@pytest.mark.parametrize("prec", [B.PD_FP64, B.PD_FP32_SPLIT])
@pytest.mark.parametrize("path", PATHS)
def test_order_of_contacts_does_not_depend_on_the_last_rebuild(prec, path):
    """Half of the broken bonds are in the lists, half came after them; with the
    lists rebuilt all are in: the same bits."""
    w, P, u, v = _pressed(0.08)
    br = _some_bonds(P, 3, 0.4)
    listed = br * _some_bonds(P, 4, 0.5)
    assert 0 < listed.sum() < br.sum()
    runs = []
    for rebuild in (False, True):
        S = B.Simulation(w, precision=prec, device="cuda:0")
        S.set_path(*path)
        S.set("DISP", u)
        S.set("BROKEN", listed)
        S.eval_forces()
        S.set("VEL", v)
        S.set("ACC", np.zeros_like(v))
        S.set("BROKEN", br)
        if rebuild:
            S.clear_status()
        n = _rebuilds(S)
        S.step(1)
        assert _rebuilds(S) == n + rebuild
        runs.append((S.get("ACC"), S.get("VEL"), S.get("BROKEN")))
    for a, b in zip(*runs):
        assert np.array_equal(a, b)
