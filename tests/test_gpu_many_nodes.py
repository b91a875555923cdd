"""The update pass of more than 2^20 nodes, FP32 split: the same bits as the fused
force phase, which has no such pass."""
import numpy as np
import pytest

from paper_2108_07212_gb300 import binding as B
from paper_2108_07212_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def test_update_pass_of_many_nodes_gives_the_bits_of_the_fused_phase():
    n = 1060
    w = I.compaction(n, width=40e-3 * (n / 500) ** 0.5 + 3e-3, h_ratio=23, seed=3)
    runs = []
    for mode in (0, 2):
        S = B.Simulation(w, precision=B.PD_FP32_SPLIT, device="cuda:0")
        assert S.N > 1 << 20
        S.set_path(mode, 1, 128)
        v = np.random.default_rng(4).normal(scale=3.0, size=(w.n_grains, 2))[S.get("GRAIN")]
        S.set("VEL", v)
        S.step(6)
        runs.append((S.get("DISP"), S.get("VEL"), S.get("ACC")))
        S.close()
    for a, b in zip(*runs):
        assert np.array_equal(a, b)
