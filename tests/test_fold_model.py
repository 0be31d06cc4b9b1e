"""Host model of the folded twiddle product (q = 2^50 - c, c < 2^22): congruence and the
bounds that the transforms' lazy arithmetic relies on, at the extremes of both operands."""
import itertools

import pytest

from paper_2506_11586_gb300.inputs import CANONICAL_PRIMES, Stream

FOLD_MAX = 35  # |product| <= 35 q
# smallest and largest c, and the canonical primes (the identity needs no primality)
QS = CANONICAL_PRIMES + ((1 << 50) - 1, (1 << 50) - (1 << 22) + 1)


def fold_mul(y, w, q):
    """y: signed 64-bit, w < q; the kernels' six wide products."""
    c = (1 << 50) - q
    v = (w << 32) % q
    yl, yh = y & 0xFFFFFFFF, y >> 32
    mask = (1 << 20) - 1
    mid = yl * (w >> 20) + yh * (v >> 20)
    lo = yl * (w & mask) + yh * (v & mask)
    assert -(1 << 63) <= mid < 1 << 63 and -(1 << 63) <= lo < 1 << 63
    t = lo + ((mid & 0xFFFFFFFF) << 20) + (mid >> 32) * 4 * c
    assert -(1 << 63) <= t < 1 << 63
    return t


@pytest.mark.parametrize("q", QS)
def test_fold_product(q):
    s = Stream(3, q & 0xFFFF)
    ys = [0, 1, -1, (1 << 63) - 1, -(1 << 63), (1 << 32) - 1, -(1 << 32), q - 1, 4095 * q, -4095 * q]
    ys += [int(x) - (1 << 63) for x in s.u64(40)]
    ws = [0, 1, (1 << 20) - 1, 1 << 20, q - 1, q - (1 << 20), q // 2] + [int(x) for x in s.below(q, 40)]
    for y, w in itertools.product(ys, ws):
        t = fold_mul(y, w, q)
        assert (t - y * w) % q == 0
        assert -10 * (1 << 50) <= t < 34 * (1 << 50) and abs(t) <= FOLD_MAX * q
        assert t + 16 * q > 0


@pytest.mark.parametrize("rounds", [(5, 5, 3), (5, 5, 4), (5, 5, 2), (4, 4, 4), (4, 4, 4, 1), (4, 4, 4, 2),
                                    (3, 3, 3, 3), (3, 3, 3, 3, 1)])
@pytest.mark.parametrize("half", [False, True])
def test_inverse_bounds(rounds, half):
    """The inverse's bounds round by round: differences stay below 2^63 and few registers fold."""
    b = 1
    for r, k in enumerate(rounds):
        last = r + 1 == len(rounds)
        limit = 4096 if last else 4096 >> (rounds[r + 1] - 1)
        regs = [b] * (1 << k)
        for sig in range(k):
            for j in range(1 << k):
                if not j >> sig & 1:
                    hi = regs[j] + regs[j | 1 << sig]
                    assert hi * (1 << 50) <= 1 << 63
                    regs[j], regs[j | 1 << sig] = hi, FOLD_MAX
        model = [b << k if j == 0 else FOLD_MAX << (k - 1 - (j.bit_length() - 1)) for j in range(1 << k)]
        assert all(a <= m for a, m in zip(regs, model))
        if last and not half:
            break
        folds = sum(m > limit for m in model)
        assert folds <= 4
        b = max(5 if m > limit else m for m in model)
        assert b <= 4096


@pytest.mark.parametrize("logn", [12, 13, 14])
@pytest.mark.parametrize("q", CANONICAL_PRIMES)
def test_division_by_the_degree(q, logn):
    """y / 2^logn mod q by one product: exact shifts, a non-negative value below 2^53 that
    one fold at 2^50 and one subtraction make canonical."""
    c, ninv = (1 << 50) - q, pow(1 << logn, -1, q)
    ys = [0, 1, -1, 8192 * q, -8192 * q, 8192 * q - 1, 1 - 8192 * q, q, -q, (1 << logn) - 1, -(1 << logn)]
    ys += [(int(x) - (1 << 63)) // (1 << 63) * 8192 * q + int(x) % (8192 * q) for x in Stream(5, logn).u64(200)]
    for y in ys:
        assert abs(y) <= 8192 * q
        k = -y % (1 << logn)
        t = y - k * c
        assert -(1 << 63) <= t < 1 << 63 and t % (1 << logn) == 0
        r = (t >> logn) + (k << (50 - logn)) + 4 * q
        assert 0 <= r < 1 << 53
        r = (r & ((1 << 50) - 1)) + (r >> 50) * c
        assert r < 2 * q and (r - q if r >= q else r) == y * ninv % q
