"""Segment kernels: the V tile of pass 2 in one 3-D box, or in 2-D boxes that stop at the
matrix's end, and operator rows in boxes of 128, 64 and 32 (GPU).

Sector extents put N at the edges of the boxes (one state, 31 .. 33, 95 .. 97, 127 .. 130 and
257 states) and the row counts of the matrices off the 64 rows of a box; the last matrix of
the packed vector is the one that takes 2-D boxes.  FP64 H v is the reference; bounds as for
every tile configuration.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_0707_0159_gb300 import dmrg2d, synth  # noqa: E402

pytestmark = pytest.mark.gpu


def spin_block(sizes, n_legs, seed, base=4):
    lab = synth.labels_from_sectors((base,), [(q,) for q in range(len(sizes))], sizes)
    return synth.heisenberg_block(sum(sizes), n_legs, seed, lab)


@pytest.mark.parametrize("left,right", [([1, 31, 33], [32, 64, 5]),
                                        ([95, 97, 3], [96, 127, 1]),
                                        ([129, 64], [257, 130]),
                                        ([8], [1]),
                                        ([40, 40, 40], [7, 65, 9])])
@pytest.mark.parametrize("prec,tol", [(dmrg2d.TF32, 1e-3), (dmrg2d.BF16, 6e-3),
                                      (dmrg2d.BF16X3, 1e-4)])
def test_segment_kernels(left, right, prec, tol):
    mdl = synth.model(synth.HEISENBERG, 2)
    target = (2 * 4 + len(left) // 2 + len(right) // 2 + 2,)
    ops = dmrg2d.build_ops(mdl, spin_block(left, 2, 5), spin_block(right, 2, 6), target=target)
    rng = np.random.default_rng(9)
    n = ops.info["n_vec"]
    # H times a random vector: zero on the layout's padding
    v0 = torch.from_numpy(rng.standard_normal(n)).cuda()
    y0 = torch.empty_like(v0)
    dmrg2d.apply_H(ops, v0, y0, dmrg2d.FP64)
    v = dmrg2d.convert_input(y0, prec)
    ref = torch.empty_like(y0)
    dmrg2d.apply_H(ops, y0, ref, dmrg2d.FP64)
    if prec != dmrg2d.BF16X3:
        dmrg2d.set_tile_config(ops, prec, 22)
    got = torch.full((n,), 7.0, dtype=torch.float32, device="cuda")
    dmrg2d.apply_H(ops, v, got, prec)
    assert torch.all(got.double()[ref == 0.0] == 0.0)
    assert float((got.double() - ref).norm()) <= tol * float(ref.norm())
