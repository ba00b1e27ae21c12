"""Split BF16 on the segment kernels at the edges of their boxes (GPU).

BF16X3 takes the BF16 configuration, here the segment kernels asked for by number: three
products, the last with the operators' low parts, the second with v's, whose matrices start
n_vec elements on, accumulated onto Y.  Sector extents as in test_gpu_segment_boxes.py (its
BF16X3 runs keep the default configuration, which for superblocks this small is the grouped
kernel); bound of every BF16X3 test.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_0707_0159_gb300 import dmrg2d, synth  # noqa: E402

from test_gpu_segment_boxes import spin_block  # noqa: E402

pytestmark = pytest.mark.gpu

SEGMENT = 22  # "segment kernels"


@pytest.mark.parametrize("left,right", [([1, 31, 33], [32, 64, 5]),
                                        ([95, 97, 3], [96, 127, 1]),
                                        ([129, 64], [257, 130]),
                                        ([8], [1]),
                                        ([40, 40, 40], [7, 65, 9])])
def test_split_bf16(left, right):
    assert "segment" in dmrg2d.tile_config_name(SEGMENT)
    mdl = synth.model(synth.HEISENBERG, 2)
    target = (2 * 4 + len(left) // 2 + len(right) // 2 + 2,)
    ops = dmrg2d.build_ops(mdl, spin_block(left, 2, 5), spin_block(right, 2, 6), target=target)
    rng = np.random.default_rng(9)
    n = ops.info["n_vec"]
    v0 = torch.from_numpy(rng.standard_normal(n)).cuda()
    y0 = torch.empty_like(v0)
    dmrg2d.apply_H(ops, v0, y0, dmrg2d.FP64)  # zero on the layout's padding
    ref = torch.empty_like(y0)
    dmrg2d.apply_H(ops, y0, ref, dmrg2d.FP64)
    v = dmrg2d.convert_input(y0, dmrg2d.BF16X3)
    dmrg2d.set_tile_config(ops, dmrg2d.BF16, SEGMENT)
    got = torch.full((n,), 7.0, dtype=torch.float32, device="cuda")
    dmrg2d.apply_H(ops, v, got, dmrg2d.BF16X3)
    assert torch.all(got.double()[ref == 0.0] == 0.0)
    assert float((got.double() - ref).norm()) <= 1e-4 * float(ref.norm())
    # the segment kernels, and no other, refuse a Y off the 16-byte boundary
    buf = torch.zeros(n + 1, dtype=torch.float32, device="cuda")
    with pytest.raises(dmrg2d.Dmrg2dError):
        dmrg2d.apply_H(ops, v, buf[1:], dmrg2d.BF16X3)
