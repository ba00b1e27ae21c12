"""The mixed solver's counters: every low-precision H·v that ran, and steps that counted (GPU)."""
import numpy as np  # noqa: F401
import pytest

torch = pytest.importorskip("torch")

from paper_0707_0159_gb300 import dmrg2d, synth  # noqa: E402

pytestmark = pytest.mark.gpu

MIXED = dict(precision="tf32", refine=1, refine_precision="fp64x", krylov_dim=20, outer_max=8)


@pytest.fixture(scope="module")
def ops():
    mdl = synth.model("hubbard", 2, t=1.0, U=8.0)
    return dmrg2d.build_ops(mdl, synth.hubbard_block(32, 2, 5), synth.hubbard_block(32, 2, 6))


def solve(ops, **opts):
    x = torch.from_numpy(synth.start_vector(ops.info["n_vec"], 3)).cuda()
    return dmrg2d.lanczos_ground(ops, x, **{**MIXED, **opts})


def test_step_queued_ahead_is_counted(ops):
    """On a superblock this small the next CG step is queued before the last one's result is
    read: a correction solve that stops by itself has run one H·v more than it took steps."""
    _, st, code = solve(ops, inner_iter=500, tol=1e-9)
    assert code == 0 and st["outer"] >= 1
    assert st["n_hv_low"] == st["iters"] + st["outer"]


def test_correction_solve_cut_short(ops):
    """Stopped by inner_iter there is no such step."""
    _, st, _ = solve(ops, inner_iter=3, tol=1e-12, outer_max=2)
    assert st["outer"] == 2 and st["n_hv_low"] == st["iters"] == 3 + 2 * 3


def test_no_inner_steps(ops):
    """inner_iter = 0: one Lanczos step for the start vector, no CG step, nothing counted for it."""
    solve(ops, inner_iter=30, tol=1e-6)  # leaves other numbers behind
    _, st, code = solve(ops, inner_iter=0, tol=1e-12)
    assert code == -5
    assert st["n_hv_low"] == 1 and st["iters"] == 1


def test_no_step_queued_ahead_on_long_vectors():
    """n = 18.9e6: no H·v is run after the step that met the stopping test."""
    mdl = synth.model("hubbard", 3, t=1.0, U=8.0)
    long_ops = dmrg2d.build_ops(mdl, synth.hubbard_block(64, 3, 5), synth.hubbard_block(72, 3, 6))
    assert long_ops.info["n_vec"] >= 1 << 23
    _, st, code = solve(long_ops, inner_iter=500, tol=1e-5)
    assert code == 0 and st["outer"] >= 1
    assert st["n_hv_low"] == st["iters"]
