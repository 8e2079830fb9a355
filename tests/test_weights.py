"""The compile-time weights of the unrolled rows (constant viscosity, h = 1) are
the exact multiples of 1/360 rounded once, whichever compiler flags the
generator was built with: the tables and the diagonals of a level, which stand
beside them in the smoother, come from another compilation of the same source.
The C terms (segment 2, |T|^(2/3)) are no such multiples.
"""
import os
import re
import subprocess

import pytest

from paper_2010_13513_gb300 import build

FLAGS = [["-O1"], ["-O3", "-ffp-contract=off"], ["-O3", "-ffp-contract=fast"]]


def weights(text):
    """{(disc, op): (weights of B, B^T and A, weights of C)} of the constant-viscosity tables."""
    out = {}
    for m in re.finditer(r"struct S<(\d), 0, (\d)> \{(.*?)\n\};", text, re.S):
        rows = re.search(r"rows\[\d+\] = \{(.*?)\};", m[3])[1]
        w = [float(v) for v in re.search(r"wref\[\d+\] = \{(.*?)\};", m[3])[1].split(",")]
        ab, c = [], []
        for r in re.findall(r"\{([^{}]*)\}", "{" + rows + "}" if not rows.startswith("{") else rows):
            _, _, _, t0, n0, n1, n2 = (int(v) for v in r.split(","))
            ab += w[t0:t0 + n0 + n1]
            c += w[t0 + n0 + n1:t0 + n0 + n1 + n2]
        out[int(m[1]), int(m[2])] = ab, c
    return out


@pytest.mark.parametrize("flags", FLAGS, ids=" ".join)
def test_weights_are_exact(flags, tmp_path):
    exe = str(tmp_path / "gen")
    subprocess.run(["g++", *flags, "-std=c++17", "-I", os.path.join(build.ROOT, "include"),
                    os.path.join(build.CSRC, "gen_structure.cpp"), os.path.join(build.CSRC, "stencils.cpp"), "-o", exe],
                   check=True)
    tables = weights(subprocess.run([exe], check=True, capture_output=True, text=True).stdout)
    assert len(tables) == 8                        # P1-P1 and P2-P1: the full operator, A, B^T, (B, -C)
    for (disc, _), (ab, c) in tables.items():
        assert len(ab) > 20 and (disc == 1 or not c)
        assert all(v == round(v * 360) / 360 and v != 0 for v in ab)
