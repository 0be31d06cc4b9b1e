"""Host model of the folded division by 2^log N at the largest sums that the kernels' static
assertion lets through: the window next to the bound, where y - k c is furthest below y."""
import os
import re

import pytest

from paper_2506_11586_gb300.inputs import CANONICAL_PRIMES

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2506_11586_gb300", "csrc")


def asserted_bound():
    """b of the assertion that a folded stage's inputs stay within b q in magnitude."""
    text = open(os.path.join(CSRC, "hc_ntt.cuh")).read()
    name = re.search(r"static_assert\(bound <= \(SP \? (\w+) :", text).group(1)
    if name.isdigit():
        return int(name)
    return int(re.search(r"%s = (\d+)" % name, open(os.path.join(CSRC, "hc_arith.cuh")).read()).group(1))


@pytest.mark.parametrize("logn", [12, 13, 14])
@pytest.mark.parametrize("q", CANONICAL_PRIMES + ((1 << 50) - (1 << 22) + 1, (1 << 50) - 1))
def test_division_next_to_the_bound(q, logn):
    c, n = (1 << 50) - q, 1 << logn
    top = 2 * asserted_bound() * q          # |X + Y| and |X - Y| of such inputs
    assert top < 1 << 63
    for d in (0, 1, 2, n // 2, n // 2 + 1, n - 2, n - 1):
        for y in (d - top, top - d):
            if c % n == n - 1:              # 2^log N divides q - 1, as in a context
                k = -y % n
                t = y - k * c
                assert -(1 << 63) <= t < 1 << 63, (y, k)
                r = (t >> logn) + (k << (50 - logn)) + 4 * q
                assert t % n == 0 and r >= 0
                r = (r & ((1 << 50) - 1)) + (r >> 50) * c
                assert r < 2 * q and (r - q if r >= q else r) == y * pow(n, -1, q) % q
            for k in (n - 1, n // 2):       # any q: the product does not wrap
                assert y - k * c >= -(1 << 63)
