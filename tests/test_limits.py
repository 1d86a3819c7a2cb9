"""Sizes of trees that 32-bit indices cannot hold are refused (csrc/tree_limits.h): the arithmetic, on the CPU."""
import os
import subprocess
from fractions import Fraction

import pytest

from paper_2411_04975_b200 import build

SOURCE = r"""
#include <stdio.h>
#include <stdlib.h>
#include "tree_limits.h"
int main(int, char** a) {
    TreeTotals t = {atoll(a[1]), atoll(a[2]), atoll(a[3]), 0, 0, 0};
    printf("%lld", sd_pool_entries(t, atoll(a[4])));
}
"""
MOST = 2**31 - 3


@pytest.fixture(scope="module")
def entries(tmp_path_factory):
    d = tmp_path_factory.mktemp("limits")
    (d / "a.cpp").write_text(SOURCE)
    subprocess.check_call(["g++", "-std=c++17", "-fsanitize=undefined", "-fno-sanitize-recover", "-I", build.CSRC, str(d / "a.cpp"), "-o", str(d / "a")])
    return lambda *v: int(subprocess.check_output([str(d / "a"), *map(str, v)], text=True))


@pytest.mark.parametrize("below,top,wide,extra", [
    (0, 0, 0, 0), (0, 0, 0, -1), (10, 3, 0, 7), (41_000_000, 128_256, 900_000, -1), (5_000_000, 9, 70, -1), (3, 1, 200, -1),
    (MOST, 0, 0, 0), (MOST - 5, 2, 3, 0), (MOST, 1, 0, 0), (MOST - 5, 2, 3, 1), (2**30, 0, 0, -1), (2**30 - 2, 0, 0, -1),
    # what 32-bit sums made small again
    (2**31, 0, 0, 0), (2**32 + 5, 100, 0, 0), (2**32, 2**20, 2**32 + 9, -1), (2**36, 0, 0, 0), (100, 10, 2**32 + 77, 0),
    (100, 10, 0, 2**63 - 1), (MOST, MOST, MOST, MOST), (100, 10, 0, 2**32 + 1)])
def test_entries_of_the_pool(entries, below, top, wide, extra):
    nodes = below + top
    want = nodes + wide + (extra if extra >= 0 else max(2**22, nodes))
    assert entries(below, top, wide, extra) == (want if want <= MOST else -1)


def test_quotient_from_a_rounded_reciprocal_is_rounded_right():
    """The drafts' quotients for sums up to 511: q = RN(a r), then RN(q + r RN(a - b q)), with exact sums rounded once."""
    for b in range(1, 512):
        r = 1.0 / b
        for a in range(1, b + 1):
            q = a * r
            rest = float(Fraction(a) - b * Fraction(q))
            assert float(Fraction(q) + Fraction(r) * Fraction(rest)) == a / b
