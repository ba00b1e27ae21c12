"""The fused Lanczos step against the step of separate kernels (GPU).

dmrg2d_lanczos_ground runs a step's vector work in one cooperative kernel when the vector
fits in the SMs' shared memory; dmrg2d_lanczos_ground_noalloc runs it as separate kernels.
Same recurrence in FP64, other summation orders: over 20 steps from one start vector the
energies agree to 1e-12 and the vectors to 1e-9.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle.solvers import lanczos_ground as oracle_lanczos  # noqa: E402
from oracle.superblock import Superblock  # noqa: E402
from paper_0707_0159_gb300 import dmrg2d, synth  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("legs,m1,m4,k", [(1, 1, 1, 2), (1, 3, 5, 20), (2, 11, 13, 20),
                                          (2, 64, 64, 20), (2, 70, 65, 2)])
def test_fused_step_matches_separate_kernels(legs, m1, m4, k):
    mdl = synth.model("heisenberg", legs)
    ops = dmrg2d.build_ops(mdl, synth.heisenberg_block(m1, legs, 1),
                           synth.heisenberg_block(m4, legs, 2))
    x0 = torch.from_numpy(synth.start_vector(ops.info["n_vec"], 3)).cuda()
    opts = dict(max_iter=k, krylov_dim=k, fixed_steps=1)
    a, b = x0.clone(), x0.clone()
    ea, _, ca = dmrg2d.lanczos_ground(ops, a, **opts)
    eb, _, cb = dmrg2d.lanczos_ground_noalloc(ops, b, **opts)
    assert ca == cb == 0
    assert abs(ea - eb) <= 1e-12 * abs(eb)
    assert torch.linalg.norm(a - b) <= 1e-9


@pytest.mark.parametrize("thick_keep", [0, 4])
def test_fused_step_with_restarts(thick_keep):
    mdl = synth.model("heisenberg", 2)
    left, right = synth.heisenberg_block(12, 2, 1), synth.heisenberg_block(10, 2, 2)
    ops, sb = dmrg2d.build_ops(mdl, left, right), Superblock(mdl, left, right)
    v = synth.start_vector(sb.n_vec, 4)
    x = torch.from_numpy(v).cuda()
    e, st, code = dmrg2d.lanczos_ground(ops, x, max_iter=400, krylov_dim=14, tol=1e-10,
                                        thick_keep=thick_keep)
    e_ref, _, _ = oracle_lanczos(sb.apply, v, max_iter=300, tol=1e-12)
    assert code == 0 and abs(e - e_ref) <= 1e-10 * abs(e_ref)
    xr = x.cpu().numpy()
    assert np.linalg.norm(sb.apply(xr) - e * xr) <= 1e-8 * abs(e)


def test_vector_too_long_for_shared_memory():
    """n = 846400 > 152 x 5120: the separate kernels."""
    mdl = synth.model("heisenberg", 2)
    left, right = synth.heisenberg_block(230, 2, 1), synth.heisenberg_block(230, 2, 2)
    ops, sb = dmrg2d.build_ops(mdl, left, right), Superblock(mdl, left, right)
    v = synth.start_vector(sb.n_vec, 4)
    x = torch.from_numpy(v).cuda()
    e, _, code = dmrg2d.lanczos_ground(ops, x, max_iter=4, krylov_dim=4, fixed_steps=1)
    xr = x.cpu().numpy()
    assert code == 0 and abs(xr @ sb.apply(xr) - e) <= 1e-11 * abs(e)
