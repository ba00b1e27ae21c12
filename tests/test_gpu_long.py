"""The two-pass CUDA-core H·v at the edges of its items, against the oracle (GPU).

An item is up to 64 indices of one segment (1, 2, 4 or 8 row groups of up to 8) by 64 to
512 indices of the long dimension, in K chunks of 8 (FP64) or 16 (FP32): sizes around
those, and vectors that do not start on a 16-byte boundary.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle.superblock import Superblock  # noqa: E402
from paper_0707_0159_gb300 import dmrg2d, synth  # noqa: E402

from test_gpu_sectors import packed_map  # noqa: E402

pytestmark = pytest.mark.gpu

SECTORS = {
    "one_state": ((1,), (1,)),
    "row_groups": ((1, 8, 9, 16, 17, 7), (32, 33, 2, 24)),
    "chunks": ((63, 64, 65), (128, 129, 15)),
}


def rel(a, b):
    return np.linalg.norm(a - b) / np.linalg.norm(b)


@pytest.mark.parametrize("offset", [0, 1])
@pytest.mark.parametrize("prec,tol", [(dmrg2d.FP64, 1e-12), (dmrg2d.FP32, 1e-5)])
@pytest.mark.parametrize("name", sorted(SECTORS))
def test_sector_sizes(name, prec, tol, offset):
    left_sizes, right_sizes = SECTORS[name]

    def labels(sizes):
        return synth.labels_from_sectors((4,), [(q - len(sizes) // 2,) for q in range(len(sizes))],
                                         sizes)

    mdl = synth.model("heisenberg", 2)
    left = synth.heisenberg_block(sum(left_sizes), 2, 1, labels(left_sizes))
    right = synth.heisenberg_block(sum(right_sizes), 2, 2, labels(right_sizes))
    target = (10,)
    ops = dmrg2d.build_ops(mdl, left, right, target=target)
    sb = Superblock(mdl, left, right)
    pmap = packed_map(sb, target)
    valid = pmap >= 0
    vp = np.where(valid, synth.start_vector(len(pmap), 5), 0.0)
    vd = np.zeros(sb.n_vec)
    vd[pmap[valid]] = vp[valid]
    ref = np.zeros(len(pmap))
    ref[valid] = sb.apply(vd)[pmap[valid]]
    dt = torch.float64 if prec == dmrg2d.FP64 else torch.float32
    x = torch.zeros(len(pmap) + offset, dtype=dt, device="cuda")
    x[offset:] = torch.from_numpy(vp).to("cuda", dt)
    y = torch.full((len(pmap) + offset,), 7.0, dtype=dt, device="cuda")
    dmrg2d.apply_H(ops, x[offset:], y[offset:], prec)
    got = y.double().cpu().numpy()[offset:]
    assert np.all(got[~valid] == 0.0)
    assert rel(got, ref) <= tol
