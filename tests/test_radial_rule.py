"""Which grids the tensor's radial tables are used for (csrc/radial.h, compiled
for the host): common integer ratios of the squared steps over a third, a half
or the whole of the smallest; a table of at most a quarter of the octant;
ratios equal to what the rounding of the half-widths allows, and no others."""
import math
import os
import random
import shutil
import subprocess
from fractions import Fraction

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def rule(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    exe = str(tmp_path_factory.mktemp("radial") / "radial_rule_check")
    r = subprocess.run([cxx, "-std=c++17", "-O1", os.path.join(HERE, "radial_rule_check.cpp"), "-o", exe],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr

    def ask(rows):
        text = "".join("%d %d %d %s %s %s %s\n" % (*n, *(v.hex() for v in L), kind) for n, L, kind in rows)
        out = subprocess.run([exe], input=text, capture_output=True, text=True, timeout=300)
        lines = out.stdout.split("\n")[:-1]
        assert out.returncode == 0 and len(lines) == len(rows)
        return [None if v == "no" else tuple(int(k) for k in v.split()) for v in lines]

    return ask


KNOWN = [  # n, L, steps -> m, r0, r1, r2 (None: per point)
    ((256, 256, 256), (16.0, 16.0, 16.0), "h", (1, 1, 1, 1)),
    ((256, 256, 256), (16.0, 16.0, 16.0), "c", (1, 1, 1, 1)),
    ((24, 48, 96), (1.55, 3.1, 6.2), "h", (1, 1, 1, 1)),
    ((64, 64, 64), (0.3, 0.1, 0.1), "h", (1, 9, 1, 1)),
    ((64, 64, 128), (4.0, 4.0, 4.0), "h", (1, 4, 4, 1)),
    ((128, 128, 128), (8.0, 8.0, 12.0), "h", (2, 4, 4, 9)),
    ((128, 128, 128), (8.0, 8.0, 12.0), "c", (2, 9, 9, 4)),
    ((192, 192, 96), (12.0, 12.0, 8.0), "h", (3, 9, 9, 16)),
    ((192, 192, 96), (16.0, 16.0, 12.0), "c", (3, 9, 9, 16)),
    ((64, 64, 64), (8.0, 8.0, 12.0), "h", None),      # halves: a table above a quarter of the octant
    ((32, 24, 16), (1.3, 1.7, 2.9), "h", None),       # no common ratio
    ((8, 8, 8), (1.0, 1.0, 1.0), "h", None),          # too small for a table
]


def test_known_grids(rule):
    for (n, L, kind, want), got in zip(KNOWN, rule([k[:3] for k in KNOWN])):
        assert (got[:4] if got else None) == want, (n, L, kind, got)
        if got:
            assert got[4] == 1 + sum(r * k * k for r, k in zip(got[1:4], n))
            assert got[4] <= math.prod(k + 1 for k in n) // 4


def test_rounded_multiples_of_one_length_are_accepted(rule):
    g = random.Random(5)
    rows = []
    for _ in range(20000):
        t = Fraction(g.uniform(0.01, 100.0))
        rows.append(((128, 128, 128), tuple(float(t * k) for k in g.choice(((1, 1, 1), (2, 1, 1), (2, 2, 3)))),
                     g.choice("hc")))
    assert all(rule(rows))


def test_boxes_that_are_not_multiples_are_refused(rule):
    """A half-width off by three to twelve units of 2^-53 (relative) against an
    exact multiple: the squared ratio is off by six units or more."""
    g = random.Random(6)
    rows = []
    for _ in range(5000):
        t = g.uniform(1.0, 1.9)
        off = math.ldexp(1.0, -52) * g.choice((3, 4, 6)) * g.choice((1, -1))
        rows.append(((128, 128, 128), (t, t, t + off), g.choice("hc")))
    assert not any(rule(rows))
