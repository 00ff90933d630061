"""The table of mixed-radix line lengths (csrc/line_lengths.h): every stored value of a line has a
place of its own inside the line, for the strides of both precisions, and the set is fine enough."""
import os
import re

import pytest

HEADER = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2008_02478_gb300", "csrc",
                      "line_lengths.h")


def entries():
    text = open(HEADER).read()
    fine = int(re.search(r"N_FINE = (\d+)", text).group(1))
    rows = [tuple(int(v) for v in m.split(",")) for m in re.findall(r"X\((\d[^)]*)\)", text)]
    assert [r[0] for r in rows] == list(range(len(rows)))
    return fine, rows


@pytest.mark.parametrize("row", entries()[1], ids=lambda r: "x".join(map(str, r[1:4])))
def test_positions_are_distinct_and_inside_the_line(row):
    _, r1, r2, r3, *strides = row
    for P2, P1, OFF, LS in (strides[:4], strides[4:]):
        pos = [p * OFF + k1 * P1 + k2 * P2 + k3
               for p in range(2) for k1 in range(r1) for k2 in range(r2) for k3 in range(r3)]
        assert len(set(pos)) == 2 * r1 * r2 * r3
        assert min(pos) == 0 and max(pos) < LS


def test_half_lengths_ascend_and_reach_the_largest_axis():
    fine, rows = entries()
    half = [a * b * c for _, a, b, c, *_ in rows[:fine]]
    assert half == sorted(set(half)) and half[0] == 2 and half[-1] == 2048
    # above the smallest ones no axis pays for more than a third beyond its own cells
    assert all(b <= 1.34 * a for a, b in zip(half, half[1:]) if a >= 12)
    coarse = [a * b * c for _, a, b, c, *_ in rows[fine:]]
    assert set(coarse) <= set(half)
