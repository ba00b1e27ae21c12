"""FP64X output by output: against 80- or 128-bit arithmetic, in units of the largest operands
(GPU).

The operands are integers of 61 bits below a scale of each operator row and each line of V, at
most 8 times the product of the largest operator entry of the row and the largest entry of the
line (a line's scale is up to two bits above its largest entry, a row's up to one).  64-bit sums
take a unit of 2^-54 of that for K up to 256, as here: 2^-51 of the product of the two largest
entries at most, 2^-52 as a rule.  Each group of four stages (7 stages here, each its own group
when the scales grow) rounds twice to the unit, the digits' products left out add 0.2 units, a
sum that is shifted loses at most one more unit: three units, 2^-50.4, in the mean.  The bound
is 2^-49 in the root mean square over each row, each column and the whole, plus the rounding of
Y itself.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle.superblock import Superblock  # noqa: E402
from paper_0707_0159_gb300 import dmrg2d, synth  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def hubbard2():
    mdl = synth.model("hubbard", 2, t=1.0, U=6.0)
    left, right = synth.hubbard_block(16, 2, 5), synth.hubbard_block(24, 2, 6)
    return dmrg2d.build_ops(mdl, left, right), Superblock(mdl, left, right)


def parity_scale(sb, f):
    """1 on the even, f on the odd states of (block 1, column 2) and (column 3, block 4)."""
    col = np.array([(-1.0) ** bin(i).count("1") for i in range(sb.d)])
    rows = np.outer(col, sb.left["parity"]).ravel()
    cols = np.outer(col, sb.right["parity"]).ravel()
    return np.where(np.outer(rows, cols) > 0, 1.0, f)


def grades(sb):
    rows, cols = sb.m1 * sb.d, sb.m4 * sb.d
    i, j = np.arange(rows) / rows, np.arange(cols) / cols
    return {"even": np.ones((rows, cols)),
            "up": np.exp2(40.0 * i)[:, None] * np.exp2(40.0 * j)[None, :],
            "down": np.exp2(-40.0 * i)[:, None] * np.exp2(-40.0 * j)[None, :],
            "odd_small": parity_scale(sb, 2.0 ** -20)}


@pytest.mark.parametrize("grade", ["even", "up", "down", "odd_small"])
def test_error_in_units_of_the_largest_operands(hubbard2, grade):
    ops, sb = hubbard2
    rows, cols = sb.m1 * sb.d, sb.m4 * sb.d
    V = synth.start_vector(sb.n_vec, 13).reshape(cols, rows).T * grades(sb)[grade]
    v = np.ascontiguousarray(V.T).ravel()
    x = torch.from_numpy(v).cuda()
    y = torch.full_like(x, 7.0)
    dmrg2d.apply_H(ops, x, y, dmrg2d.FP64X)
    ref = sb.apply(v.astype(np.longdouble)).reshape(cols, rows).T
    err = np.abs(y.cpu().numpy().reshape(cols, rows).T - ref).astype(np.float64)
    aV = np.abs(V)
    unit = (np.abs(sb.H_left()).max(1)[:, None] * aV.max(0)[None, :] +
            aV.max(1)[:, None] * np.abs(sb.H_right()).max(1)[None, :])
    # three sums and the final conversions round Y: half a last place each
    bound = 2.0 ** -49 * unit + 2.0 ** -51 * np.abs(ref).astype(np.float64)
    rms = lambda a, ax=None: np.sqrt((a * a).mean(ax))  # noqa: E731
    assert rms(err) <= rms(bound)
    assert np.all(rms(err, 0) <= rms(bound, 0))
    assert np.all(rms(err, 1) <= rms(bound, 1))


@pytest.mark.parametrize("kind,legs,m1,m4", [("hubbard", 2, 16, 24), ("hubbard", 2, 7, 9),
                                             ("heisenberg", 3, 17, 9)])
def test_norm_error_below_48_bits(kind, legs, m1, m4):
    """As a whole the result is closer than 48-bit significands (float pairs) would be."""
    make = synth.heisenberg_block if kind == "heisenberg" else synth.hubbard_block
    mdl, left, right = synth.model(kind, legs), make(m1, legs, 3), make(m4, legs, 4)
    sb = Superblock(mdl, left, right)
    v = synth.start_vector(sb.n_vec, 9)
    x = torch.from_numpy(v).cuda()
    y = torch.full_like(x, 7.0)
    dmrg2d.apply_H(dmrg2d.build_ops(mdl, left, right), x, y, dmrg2d.FP64X)
    ref = sb.apply(v.astype(np.longdouble))
    err = (y.cpu().numpy() - ref).astype(np.float64)
    assert np.linalg.norm(err) <= 2.0 ** -48 * np.linalg.norm(ref.astype(np.float64))
