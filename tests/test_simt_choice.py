"""Which dense CUDA-core kernel a superblock takes, on the host (no GPU).

The rule (csrc/simt_choice.h) is compiled by itself and asked for superblocks that stand for
each branch on 152 SMs: `CASES` holds them with ragged sizes, and test_gpu_simt_branches.py
runs the H·v of each.  `items` is the number of two-pass items of pass 0, cut as the plan cuts
them: columns of one block in equal chunks of up to 64 (FP32: rounded to 4), by 64 long
indices per row group of 8 (FP32: 512, 256 or 128 for up to 16, 32 or 64 columns).
"""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CXX = shutil.which("g++")

# precision, model, legs, m1, m4, branch
CASES = [
    ("fp64", "heisenberg", 2, 1213, 63, "64"),
    ("fp64", "heisenberg", 2, 607, 31, "32"),
    ("fp64", "heisenberg", 2, 301, 16, "16"),
    ("fp64", "heisenberg", 2, 45, 50, "8"),
    ("fp64", "hubbard", 2, 50, 129, "two_pass"),
    ("fp64", "hubbard", 2, 67, 131, "two_pass"),
    ("fp32", "hubbard", 2, 11, 13, "64"),
    ("fp32", "heisenberg", 2, 99, 126, "32"),
    ("fp32", "heisenberg", 2, 45, 50, "16"),
    ("fp32", "hubbard", 2, 41, 38, "two_pass"),
]

MAIN = r"""
#include <cstdio>
#include "simt_choice.h"
int main() {
  int p, m1, m4, d, sms;
  long long items;
  while (scanf("%d %d %d %d %d %lld", &p, &m1, &m4, &d, &sms, &items) == 6) {
    const dmrg2d::SimtChoice c = p == 64 ? dmrg2d::simt_choice_f64(m1, m4, d, sms, items)
                                         : dmrg2d::simt_choice_f32(m1, m4, d, sms, items);
    if (c.two_pass) printf("two_pass\n");
    else printf("%d%s\n", c.piece, dmrg2d::simt_grid_fits(m1, m4, d, c.piece) ? "" : " refused");
  }
}
"""


def items(prec, m1, m4, d):
    chunks = -(-m4 // 64)
    per = -(-m4 // chunks)
    if prec == "fp32":
        per = -(-per // 4) * 4
    total = 0
    for s0 in range(0, m4, per):
        cnt = min(per, m4 - s0)
        if prec == "fp64":
            width = 64 * (8 if cnt <= 8 else 4 if cnt <= 16 else 2 if cnt <= 32 else 1)
        else:
            width = 512 if cnt <= 16 else 256 if cnt <= 32 else 128
        total += -(-m1 * d // width)
    return d * total


@pytest.fixture(scope="module")
def choose(tmp_path_factory):
    if CXX is None:
        pytest.skip("no g++")
    tmp = tmp_path_factory.mktemp("choice")
    (tmp / "main.cpp").write_text(MAIN)
    exe = str(tmp / "main")
    subprocess.run([CXX, "-std=c++17", "-O1", "-I", os.path.join(ROOT, "paper_0707_0159_gb300", "csrc"),
                    str(tmp / "main.cpp"), "-o", exe], check=True, capture_output=True)

    def ask(prec, m1, m4, d, sms=152):
        line = f"{prec[2:]} {m1} {m4} {d} {sms} {items(prec, m1, m4, d)}\n"
        return subprocess.run([exe], input=line, capture_output=True, text=True,
                              check=True).stdout.strip()
    return ask


@pytest.mark.parametrize("prec,kind,legs,m1,m4,branch", CASES)
def test_branch(choose, prec, kind, legs, m1, m4, branch):
    assert choose(prec, m1, m4, (2 if kind == "heisenberg" else 4) ** legs) == branch


def test_measured_superblocks(choose):
    """The superblocks whose times stand beside the rule."""
    assert choose("fp64", 250, 131, 8) == "two_pass"
    assert choose("fp64", 200, 200, 4) == "8"
    assert choose("fp64", 40, 40, 16) == "8"
    assert choose("fp64", 64, 64, 4) == "8"
    assert choose("fp32", 100, 128, 4) == "32"
    for m1, m4, d in ((40, 40, 16), (250, 131, 8), (128, 128, 64)):
        assert choose("fp32", m1, m4, d) == "two_pass"


@pytest.mark.parametrize("m1,m4,d", [(16, 4096, 256), (16, 4000, 1024), (16, 520, 1024),
                                     (8, 512, 1024), (3, 1000, 1024), (24, 2041, 1024)])
def test_piece_fits_the_launch_limits(choose, m1, m4, d):
    """Many tiles of many states: small pieces would need a grid above 65535 in y, where a
    larger piece or the two-pass kernel runs, as pieces of 64 always could."""
    assert "refused" not in choose("fp64", m1, m4, d)
