"""The small eigensolve where its minors meet zeros, splits and extreme scales (GPU).

Eigenvalues by Sturm counts on minors scaled to the norm of T: backward stable, so within a
few 1e-15 of the norm of numpy's; the eigenvector's residual within 1e-13 of the norm.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_0707_0159_gb300 import dmrg2d  # noqa: E402

pytestmark = pytest.mark.gpu

RNG = np.random.default_rng(1)
CASES = {
    "one": ([3.0], [0.0]),
    "zero_diagonal": (np.zeros(9), np.ones(9)),
    "split": ([1.0, -2.0, 5.0, -2.5, 7.0], [0.0, 1e-3, 0.0, 1e-200, 0.0]),
    "graded": (10.0 ** np.arange(0, -24, -1.5), 0.1 * 10.0 ** np.arange(0, -24, -1.5)),
    "huge": (1e120 * RNG.normal(size=40), 1e120 * RNG.normal(size=40)),
    "tiny": (1e-120 * RNG.normal(size=40), 1e-120 * RNG.normal(size=40)),
    "longest": (RNG.normal(size=512), RNG.normal(size=512)),
    "equal": (np.full(100, 2.0), np.full(100, -1.0)),
}


@pytest.mark.parametrize("name", sorted(CASES))
def test_tridiag_lowest(name):
    a, b = (np.array(v, dtype=np.float64) for v in CASES[name])
    th, s, _, status = dmrg2d.tridiag_lowest(torch.from_numpy(a).cuda(), torch.from_numpy(b).cuda())
    T = np.diag(a) + np.diag(b[:-1], 1) + np.diag(b[:-1], -1)
    norm = np.abs(T).sum(1).max()
    s = s.cpu().numpy()
    assert status == 0
    assert abs(th - np.linalg.eigvalsh(T / norm)[0] * norm) <= 1e-14 * norm
    assert abs(np.linalg.norm(s) - 1.0) <= 1e-13
    assert np.linalg.norm(T @ s - th * s) <= 1e-13 * norm
