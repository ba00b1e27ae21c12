"""Every dense CUDA-core kernel at ragged sizes against the oracle (GPU).

test_simt_choice.py names the branch that each of these superblocks takes on 152 SMs and
checks it on the host; here its H·v runs.  FP64 bound of every FP64 test; FP32 as there.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle.superblock import Superblock  # noqa: E402
from paper_0707_0159_gb300 import dmrg2d, synth  # noqa: E402

from test_simt_choice import CASES  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("offset", [0, 1])
@pytest.mark.parametrize("prec,kind,legs,m1,m4,branch", CASES)
def test_branch(prec, kind, legs, m1, m4, branch, offset):
    make = synth.heisenberg_block if kind == "heisenberg" else synth.hubbard_block
    mdl, left, right = synth.model(kind, legs), make(m1, legs, 3), make(m4, legs, 4)
    sb = Superblock(mdl, left, right)
    v = synth.start_vector(sb.n_vec, 9)
    dt = torch.float64 if prec == "fp64" else torch.float32
    x = torch.zeros(sb.n_vec + offset, dtype=dt, device="cuda")
    x[offset:] = torch.from_numpy(v).to("cuda", dt)
    y = torch.full_like(x, 7.0)
    dmrg2d.apply_H(dmrg2d.build_ops(mdl, left, right), x[offset:], y[offset:], prec)
    ref = sb.apply(v)
    got = y[offset:].double().cpu().numpy()
    tol = 1e-12 if prec == "fp64" else 1e-5
    assert np.linalg.norm(got - ref) <= tol * np.linalg.norm(ref)
    assert np.abs(got - ref).max() <= 10 * tol * np.abs(ref).max()
    if offset:
        assert y[0].item() == 7.0
