"""The tensor-core configuration of a sector superblock that nobody tuned (GPU).

Narrow sectors default to the segment kernels, which store Y in 16-byte pieces: a Y off that
boundary takes the grouped kernel instead, and is refused only when the segment kernels were
asked for.  TF32 and BF16 bounds as for every tile configuration.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle.superblock import Superblock  # noqa: E402
from paper_0707_0159_gb300 import dmrg2d, synth  # noqa: E402

from test_gpu_sectors import packed_map  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def narrow():
    mdl, left, right, target = synth.workload_ladder3_hubbard_sectors(m=40, block_sites=6, n_up=6,
                                                                      n_dn=6)
    sb = Superblock(mdl, left, right)
    ops = dmrg2d.build_ops(mdl, left, right, target=target)
    pmap = packed_map(sb, target)
    valid = pmap >= 0
    vp = np.where(valid, synth.start_vector(len(pmap), 17), 0.0)
    vd = np.zeros(sb.n_vec)
    vd[pmap[valid]] = vp[valid]
    ref = np.zeros(len(pmap))
    ref[valid] = sb.apply(vd)[pmap[valid]]
    return ops, vp, ref, valid


@pytest.mark.parametrize("prec,tol", [(dmrg2d.TF32, 1e-3), (dmrg2d.BF16, 6e-3),
                                      (dmrg2d.BF16X3, 1e-4)])
@pytest.mark.parametrize("offset", [0, 1])
def test_default_configuration(narrow, prec, tol, offset):
    ops, vp, ref, valid = narrow
    v = dmrg2d.convert_input(torch.from_numpy(vp).cuda(), prec)
    buf = torch.full((len(vp) + offset,), 7.0, dtype=torch.float32, device="cuda")
    dmrg2d.apply_H(ops, v, buf[offset:], prec)
    got = buf.double().cpu().numpy()[offset:]
    assert np.all(got[~valid] == 0.0)
    assert np.linalg.norm(got - ref) <= tol * np.linalg.norm(ref)
    if offset:
        assert buf[0].item() == 7.0


def test_explicit_segment_kernels_refuse_unaligned_y(narrow):
    ops, vp, _, _ = narrow
    dmrg2d.set_tile_config(ops, "tf32", 22)
    v = dmrg2d.convert_input(torch.from_numpy(vp).cuda(), "tf32")
    buf = torch.zeros(len(vp) + 1, dtype=torch.float32, device="cuda")
    with pytest.raises(dmrg2d.Dmrg2dError):
        dmrg2d.apply_H(ops, v, buf[1:], "tf32")
