"""The network's loss and gradient at the edges of their cuts, against the FP64 oracle (GPU).

Products run in 128 x 64 tiles with K chunks of 16 (16-byte loads when hidden % 4 == 0), the
batch is cut into at most 152 blocks of 16 to 128 rows.  Gradient sums of B FP32 terms of
relative rounding 2^-24 each, a few operations deep: 1e-4 covers them with a wide margin.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import mlp as omlp  # noqa: E402
from paper_0707_0159_gb300 import dmrg2d  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H,B", [(1, 1), (33, 15), (64, 129), (130, 2433), (256, 8192), (20, 20000)])
def test_loss_and_gradient(H, B):
    net = dmrg2d.MLP(hidden=H, seed=3)
    rng = np.random.default_rng(H + B)
    net.set_params((0.3 * rng.standard_normal(net.n_params)).astype(np.float32))
    p = net.get_params().astype(np.float64)
    X = rng.normal(size=(B, 4)).astype(np.float32)
    w, T = (rng.normal(size=B).astype(np.float32) for _ in range(2))
    Xt, wt, Tt = (torch.from_numpy(a).cuda() for a in (X, w, T))
    g = torch.empty(net.n_params, dtype=torch.float32, device="cuda")
    loss = net.loss_grad(Xt, wt, Tt, g)
    X, w, T = (a.astype(np.float64) for a in (X, w, T))
    g_ref = omlp.grad(p, H, X, w, T)
    assert abs(loss - omlp.loss(p, H, X, w, T)) <= 1e-5 * abs(loss)
    assert np.linalg.norm(g.cpu().numpy() - g_ref) <= 1e-4 * np.linalg.norm(g_ref)
    # a smaller batch afterwards uses the same scratch
    n = (B + 1) // 2
    loss = net.loss_grad(Xt[:n], wt[:n], Tt[:n], g)
    g_ref = omlp.grad(p, H, X[:n], w[:n], T[:n])
    assert np.linalg.norm(g.cpu().numpy() - g_ref) <= 1e-4 * np.linalg.norm(g_ref)
