"""The loss of a batch whose partial sums are read back in several pieces (GPU).

Blocks of up to 128 rows, 1024 sums at a time: 131072 rows fill one piece.  FP32 products of a
few terms summed in FP64: 1e-5, as for every loss.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import mlp as omlp  # noqa: E402
from paper_0707_0159_gb300 import dmrg2d  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B", [131072, 131073, 300001])
def test_loss(B):
    H = 5
    net = dmrg2d.MLP(hidden=H, seed=3)
    rng = np.random.default_rng(B)
    p = net.get_params().astype(np.float64)
    X = rng.normal(size=(B, 4)).astype(np.float32)
    w, T = (rng.normal(size=B).astype(np.float32) for _ in range(2))
    g = torch.empty(net.n_params, dtype=torch.float32, device="cuda")
    loss = net.loss_grad(*(torch.from_numpy(a).cuda() for a in (X, w, T)), g)
    ref = omlp.loss(p, H, *(a.astype(np.float64) for a in (X, w, T)))
    assert abs(loss - ref) <= 1e-5 * abs(ref)
