"""Tile sizes of the network kernels: batches at the edges of 32, 64 and 128
samples a tile and of one and several tiles a block give the loss, gradient and
outputs of the reference, in rows and blocks that a wrong edge would leave out
or count twice."""
import numpy as np
import pytest

from oracle import mlp_oracle as M
from paper_2108_07212_gb300 import binding as B

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

# the element-wise tolerance of the BF16 network against the reference with the
# same rounding: four BF16 units of the output scale
TOL = 2.0 ** -6


def _worst(a, b):
    return float((np.abs(a - b) / np.maximum(TOL * (np.abs(b).max() + np.abs(b)), 1e-300)).max())


# 152 blocks of 32, 64 and 128 samples: 4864, 9728, 19456 (and one beyond each)
@pytest.mark.parametrize("n", [1, 31, 33, 127, 129, 4864, 4865, 9729, 19457, 20001])
def test_every_sample_counts_once(n):
    rng = np.random.default_rng(n)
    params = M.init_params(5)
    x = rng.normal(size=(n, 32)).astype(np.float32)
    t = (0.3 * np.tanh(x[:, ::-1])).astype(np.float32)
    net = B.MLP(max_batch=20001, params=params)
    xd = torch.from_numpy(x).cuda()
    y = net.forward(xd).cpu().numpy()
    y_ref, _ = M.forward(params.astype(np.float64), x, bf16=True)
    assert _worst(y, y_ref) <= 1.0
    loss, g = net.loss_grad(xd, torch.from_numpy(t).cuda())
    loss_ref, g_ref = M.loss_grad(params.astype(np.float64), x, t, bf16=True)
    assert loss == pytest.approx(loss_ref, rel=2e-3)
    off = 0
    for name, shape in M.SIZES:
        k = int(np.prod(shape))
        assert _worst(g[off:off + k], g_ref[off:off + k]) <= 1.0, name
        off += k
    # rows that start off a 16-byte boundary give the same bits
    buf = torch.zeros(n * 32 + 1, device="cuda")
    buf[1:] = xd.reshape(-1)
    assert np.array_equal(net.forward(buf[1:].view(n, 32)).cpu().numpy(), y)
