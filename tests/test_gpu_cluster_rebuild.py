"""Candidate lists of the kernel graph: up to 65536 nodes one thread-block
cluster rebuilds them, beyond that six kernels behind a conditional node.  Both
against the six kernels launched every step (mode 6): the same lists in the same
order, so the same bits, through several rebuilds with fewer nodes than the
cluster has threads, with several rounds of them, and on each side of the limit."""
import numpy as np
import pytest

from paper_2108_07212_gb300 import binding as B
from paper_2108_07212_gb300 import inputs as I

pytestmark = pytest.mark.gpu

LIMIT = 1 << 16
H = {"grains": 9, "below": 29, "above": 31}


def _workload(kind):
    if kind == "pair":
        return I.two_disks(h_ratio=8, k_bulk=5e5)
    return I.settling(n_grains=40, h_ratio=H[kind], box=(20e-3, 30e-3), seed=3)


@pytest.mark.parametrize("prec", [B.PD_FP64, B.PD_FP32_SPLIT])
@pytest.mark.parametrize("kind", ["pair", "grains", "below", "above"])
def test_cluster_rebuild_gives_the_same_lists(prec, kind):
    w = _workload(kind)
    runs = []
    for mode in (2, 6, 0, 4):
        S = B.Simulation(w, precision=prec, device="cuda:0")
        assert (S.N <= LIMIT) == (kind != "above"), S.N
        S.set_path(mode, 4, 128)
        v = np.random.default_rng(4).normal(scale=0.2, size=(S.N, 2))
        if kind != "pair":
            v[:, 1] -= 20.0                  # 24 um in 24 steps: 0.45 of the skin is 1.5 to 5 um
        S.set("VEL", v)
        S.step(24)
        rebuilds = int(S.status()[1][B.STATUS_REBUILDS])
        runs.append((S.get("DISP"), S.get("VEL"), S.get("BROKEN"), rebuilds))
    assert runs[0][3] >= (1 if kind == "pair" else 3)
    for r in runs[1:]:
        for a, b in zip(r, runs[0]):
            assert np.array_equal(a, b)
