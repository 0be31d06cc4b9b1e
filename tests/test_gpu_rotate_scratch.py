"""Device scratch of the rotation calls stays within what the header states, at every limb count and
with more outputs than inputs, counted by an allocator hook in a child process."""
import os
import subprocess
import sys
import textwrap

import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

CHILD = textwrap.dedent("""
    import ctypes as C, sys
    import numpy as np, torch
    sys.path.insert(0, sys.argv[1])
    sys.path.insert(0, sys.argv[1] + "/tests")
    from gpu_util import to_dev
    from paper_2506_11586_gb300 import _lib as L
    from paper_2506_11586_gb300.inputs import CANONICAL_PRIMES, Stream, uniform_residues

    ALLOC = C.CFUNCTYPE(C.c_void_p, C.c_size_t, C.c_void_p, C.c_void_p)
    FREE = C.CFUNCTYPE(None, C.c_void_p, C.c_void_p, C.c_void_p)
    live, stats = {}, {"now": 0, "peak": 0}

    def alloc(nbytes, stream, user):
        p = torch.cuda.caching_allocator_alloc(nbytes, 0, stream or 0)
        live[p] = nbytes
        stats["now"] += nbytes
        stats["peak"] = max(stats["peak"], stats["now"])
        return p

    def free(ptr, stream, user):
        stats["now"] -= live.pop(ptr)
        torch.cuda.caching_allocator_delete(ptr)

    a, f = ALLOC(alloc), FREE(free)
    L.lib().hc_set_allocator(C.cast(a, C.c_void_p), C.cast(f, C.c_void_p), None)
    N = 4096
    for nl in (1, 2, 3):
        moduli = CANONICAL_PRIMES[:nl]
        s = Stream(93, nl)
        gk = np.stack([np.stack([np.stack([s.below(q, N) for q in CANONICAL_PRIMES[:nl + 1]]) for _ in range(2)])
                       for _ in range(nl)])
        ctx = L.hc_ctx_create(N, moduli, 65537)
        Wp, k = 8, 3
        key = L.hc_galois_key_create(ctx, CANONICAL_PRIMES[nl], 5, gk)
        row = L.hc_galois_key_create(ctx, CANONICAL_PRIMES[nl], pow(5, Wp - k + 1, 2 * N), gk)
        words = nl * N * 8
        rot = (4 * nl + 2) * N * 8

        def peak(call):
            torch.cuda.synchronize()
            base = stats["now"]
            stats["peak"] = base
            call()
            torch.cuda.synchronize()
            assert stats["now"] == base
            return stats["peak"] - base

        def res(*shape):
            return to_dev(uniform_residues(s, moduli, shape, N))

        out = torch.empty(40 * 2 * nl * N, dtype=torch.int64, device="cuda")
        for n in (1, 5):
            got = peak(lambda: L.hc_ct_rotate(ctx, key, res(n, 2), out[:n * 2 * nl * N]))
            assert got <= n * rot, (nl, n, got, n * rot)
        for m, n in ((1, 2), (1, 5), (4, 3)):
            got = peak(lambda: L.hc_mac_rotate_many(ctx, key, res(m, 2), res(n), out[:m * 2 * nl * N]))
            assert got <= (m * n + m) * 2 * words + m * rot, (nl, m, n, got)
        for Cin, M in ((1, 16), (3, 2), (2, 7)):
            desc, Y = L.make_desc(Cin, 6, 6, M, k, k, pad=1), (M + 1) // 2
            got = peak(lambda: L.hc_zp_conv(ctx, desc, key, row, res(Y * k * k * Cin), res(Cin, 2), out[:Y * 2 * nl * N]))
            assert got <= (Cin + Y * k * k) * 2 * words + Y * rot, (nl, Cin, M, got)
        row.close(); key.close(); ctx.close()
    L.lib().hc_set_allocator(None, None, None)
    print("ok")
""")


def test_peak_scratch_in_child():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2506_11586_gb300.build import build
    build()
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", CHILD, root], capture_output=True, text=True, timeout=600)
    assert r.returncode == 0 and "ok" in r.stdout, (r.stdout[-2000:], r.stderr[-4000:])
