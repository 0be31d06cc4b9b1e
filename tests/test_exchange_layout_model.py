"""Host model of the transforms' shared-memory layout: a thread's positions are its first
one plus constants where words are padded, every element has a place of its own, and the
sixteen threads of each half-warp touch sixteen bank pairs in every access pattern."""
import pytest

SHAPES = [(12, 3), (12, 4), (13, 4), (13, 5), (14, 4), (14, 5), (9, 3), (10, 3), (11, 3)]


def spos(e, logc, padded):
    return e + (e >> logc) if padded else e ^ ((e >> logc) & 15)


def patterns(logn, logc):
    """(name, base(tid), offsets) of the register rounds' layouts."""
    n, c = 1 << logn, 1 << logc
    t, rounds = n // c, -(-logn // logc)
    for r in range(rounds):
        s0 = r * logc
        k = min(logc, logn - s0)
        kk = 1 << k
        s = n >> (s0 + k)
        if s == 1:
            yield "fwd%d" % r, lambda tid: tid * c, list(range(c))
        else:
            assert kk == c
            yield "fwd%d" % r, lambda tid, s=s, s0=s0: tid // s * (n >> s0) + tid % s, [j * s for j in range(c)]
        s = 1 << s0
        assert t % s == 0 or s == n >> k
        step = t << k if t % s == 0 else t
        yield "inv%d" % r, lambda tid, s=s, k=k: tid // s * (s << k) + tid % s, \
            [(q >> k) * step + (q & (kk - 1)) * s for q in range(c)]


@pytest.mark.parametrize("logn,logc", SHAPES)
def test_layout(logn, logc):
    n, c = 1 << logn, 1 << logc
    t, padded = n // c, logn >= 14 and logc >= 4
    assert len({spos(e, logc, padded) for e in range(n)}) == n and t % c in (0, t)
    for name, base, offs in patterns(logn, logc):
        seen = set()
        for tid in range(t):
            for o in offs:
                e = base(tid) + o
                seen.add(e)
                if padded:
                    assert base(tid) % c + o % c < c
                    assert spos(e, logc, padded) == spos(base(tid), logc, padded) + spos(o, logc, padded), name
        assert len(seen) == n, name
        for half in range(0, t, 16):
            for o in offs:
                assert len({spos(base(tid) + o, logc, padded) % 16 for tid in range(half, half + 16)}) == 16, (name, half, o)
