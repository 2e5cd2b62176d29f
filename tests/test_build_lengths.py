"""The build's list of compiled line lengths is the one of the sources."""
import os
import re

from paper_1807_04638_gb300 import build


def smooth(n):
    for r in (2, 3, 5):
        while n % r == 0:
            n //= r
    return n == 1


def test_a_unit_for_every_length_of_the_table():
    lengths = build.stage_lengths()
    assert sorted(lengths) == [n for n in range(16, 321) if smooth(n)] + [384]
    units = [name for _, name, _ in build.SOURCES]
    assert len(units) == len(set(units))
    assert [n for n in units if re.match(r"stage_n\d", n)] == [f"stage_n{n}.o" for n in lengths]


def test_radices_of_the_table():
    with open(os.path.join(build.CSRC, "stage.cuh")) as f:
        rows = re.findall(r"X\((\d+), (\d+), (\d+), (\d+)\)", f.read())
    assert len(rows) == len(build.stage_lengths())
    for n, a, b, c in (tuple(map(int, r)) for r in rows):
        assert n == a * b * c
