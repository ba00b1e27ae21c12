"""The two-pass H·v (CUDA cores, and FP64X on tensor cores) at the edges of its items,
against the oracle (GPU).

An item is up to 64 indices of one segment (CUDA cores: 1, 2, 4 or 8 row groups of up to 8;
tensor cores: N = 16..64) by 64 to 512 (tensor cores: 128) indices of the long dimension, in
K chunks of 8, 16 or 32: sizes around those, and vectors that do not start on a 16-byte
boundary.  FP64X keeps 52 bits below the largest entry of each row of V and of the operator
blocks and leaves out products below 2^-52 of the largest one: with rows of entries within a
few hundred times their RMS that is well under the 1e-12 of the other FP64X tests.
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
@pytest.mark.parametrize("prec,tol", [(dmrg2d.FP64, 1e-12), (dmrg2d.FP64X, 1e-12),
                                      (dmrg2d.FP32, 1e-5)])
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
    dt = torch.float32 if prec == dmrg2d.FP32 else torch.float64
    x = torch.zeros(len(pmap) + offset, dtype=dt, device="cuda")
    x[offset:] = torch.from_numpy(vp).to("cuda", dt)
    y = torch.full((len(pmap) + offset,), 7.0, dtype=dt, device="cuda")
    dmrg2d.apply_H(ops, x[offset:], y[offset:], prec)
    got = y.double().cpu().numpy()[offset:]
    assert np.all(got[~valid] == 0.0)
    assert rel(got, ref) <= tol


def dense_apply(ops, v, prec):
    x = torch.from_numpy(v).cuda()
    y = torch.full_like(x, 7.0)
    dmrg2d.apply_H(ops, x, y, prec)
    return y.cpu().numpy()


@pytest.mark.parametrize("legs,m1,m4", [(1, 1, 1), (2, 15, 17), (2, 33, 129), (3, 64, 65),
                                        (2, 1400, 8)])   # the last: K above 4096
def test_fp64x_dense_sizes(legs, m1, m4):
    mdl = synth.model("heisenberg", legs)
    left, right = synth.heisenberg_block(m1, legs, 3), synth.heisenberg_block(m4, legs, 4)
    sb = Superblock(mdl, left, right)
    v = synth.start_vector(sb.n_vec, 9)
    got = dense_apply(dmrg2d.build_ops(mdl, left, right), v, dmrg2d.FP64X)
    assert rel(got, sb.apply(v)) <= 1e-12


@pytest.mark.parametrize("prec,tol", [(dmrg2d.FP64, 1e-12), (dmrg2d.FP32, 1e-5)])
@pytest.mark.parametrize("kind,legs,m1,m4", [
    ("heisenberg", 2, 7, 9), ("heisenberg", 2, 64, 64), ("heisenberg", 3, 70, 65),
    ("heisenberg", 3, 131, 100), ("hubbard", 2, 10, 10), ("hubbard", 2, 41, 38),
    ("heisenberg", 5, 33, 3)])
def test_dense_kernel_choice(kind, legs, m1, m4, prec, tol):
    """Every piece size and the two-pass kernel of the dense CUDA-core H.v."""
    make = synth.heisenberg_block if kind == "heisenberg" else synth.hubbard_block
    mdl, left, right = synth.model(kind, legs), make(m1, legs, 3), make(m4, legs, 4)
    sb = Superblock(mdl, left, right)
    v = synth.start_vector(sb.n_vec, 9)
    x = torch.from_numpy(v).to("cuda", torch.float64 if prec == dmrg2d.FP64 else torch.float32)
    y = torch.full_like(x, 7.0)
    dmrg2d.apply_H(dmrg2d.build_ops(mdl, left, right), x, y, prec)
    assert rel(y.double().cpu().numpy(), sb.apply(v)) <= tol


@pytest.fixture(scope="module")
def hubbard2():
    mdl = synth.model("hubbard", 2, t=1.0, U=6.0)
    left, right = synth.hubbard_block(24, 2, 5), synth.hubbard_block(40, 2, 6)
    return dmrg2d.build_ops(mdl, left, right), Superblock(mdl, left, right)


def test_fp64x_scales_exactly(hubbard2):
    """A power of two on the vector is a power of two on the result, bit for bit."""
    ops, sb = hubbard2
    v = synth.start_vector(sb.n_vec, 10)
    y = dense_apply(ops, v, dmrg2d.FP64X)
    for e in (-300, 41, 300):
        assert np.array_equal(dense_apply(ops, np.ldexp(v, e), dmrg2d.FP64X), np.ldexp(y, e))
    assert np.all(dense_apply(ops, np.zeros_like(v), dmrg2d.FP64X) == 0.0)


@pytest.mark.parametrize("up", [1, -1])
def test_fp64x_growing_scales(hubbard2, up):
    """Entries that grow (or fall) by 2^40 along both dimensions of V: the scales change from
    stage to stage; each column's and each row's error stays small against its own norm."""
    ops, sb = hubbard2
    rows, cols = sb.m1 * sb.d, sb.m4 * sb.d
    grade = np.exp2(up * 40.0 * np.arange(rows) / rows)[:, None] * np.exp2(
        up * 40.0 * np.arange(cols) / cols)[None, :]
    v = (synth.start_vector(sb.n_vec, 11).reshape(cols, rows).T * grade).T.ravel()
    d = dense_apply(ops, v, dmrg2d.FP64X) - sb.apply(v)
    ref = sb.apply(v)
    assert np.linalg.norm(d) <= 1e-12 * np.linalg.norm(ref)


def test_fp64x_not_finite(hubbard2):
    """Inf and NaN reach the outputs that FP64 arithmetic takes them to, and no others."""
    ops, sb = hubbard2
    v = synth.start_vector(sb.n_vec, 12)
    v[123], v[4567] = np.inf, np.nan
    a, b = dense_apply(ops, v, dmrg2d.FP64X), dense_apply(ops, v, dmrg2d.FP64)
    assert np.array_equal(np.isfinite(a), np.isfinite(b))
    v[123], v[4567] = 1.7e308, 0.0   # finite, at the top of the exponent range
    assert np.all(np.isfinite(dense_apply(ops, v * 1e-3, dmrg2d.FP64X)))
