"""The key switch at its largest digit counts, in both twiddle forms, against the oracle's rotation:
seven digits at N <= 8192, and odd counts at
N = 16384 with a 45-bit prime among them."""
import numpy as np
import pytest

from gpu_util import to_dev, to_host
from oracle import core, zp
from paper_2506_11586_gb300.inputs import Stream

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

P45 = 35184371138561  # prime, 1 mod 2^15: no folded twiddles


def _primes(N, n):
    """The largest n primes below 2^50 that are 1 mod 2N; all of the folded form at N <= 8192."""
    out, q = [], (1 << 50) + 1
    while len(out) < n:
        q -= 2 * N
        if core.is_prime(q):
            out.append(q)
    return tuple(out)


A, B, C = _primes(4096, 8), _primes(8192, 8), _primes(16384, 8)
assert max((1 << 50) - q for q in A + B + C[:6]) < 1 << 22 <= (1 << 50) - C[6]


@pytest.fixture(scope="module")
def L():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2506_11586_gb300 import _lib
    from paper_2506_11586_gb300.build import build
    build()
    return _lib


@pytest.mark.parametrize("N,moduli,special,g", [
    (4096, A[:7], A[7], 5),
    (8192, B[:7], B[7], 5),
    (8192, B[:6] + (P45,), B[7], 3),
    (16384, C[:3], C[5], 5),
    (16384, (C[0], P45, C[2]), C[7], 32767),
    (16384, C[:1], P45, 5),
])
def test_digit_counts(L, N, moduli, special, g):
    nl = len(moduli)
    kp = zp.KsParams(N, tuple(moduli), special)
    s = Stream(92, N + nl)
    gk = np.stack([np.stack([np.stack([s.below(q, N) for q in kp.qp]) for _ in range(2)]) for _ in range(nl)])
    ctx = L.hc_ctx_create(N, moduli, 65537)
    key = L.hc_galois_key_create(ctx, special, g, gk)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    n = 2 * sms // (8 * (nl + 1)) + 1        # the first size on the throughput shape
    ct = np.stack([np.stack([s.below(q, N) for q in moduli]) for _ in range(2)])
    for i, q in enumerate(moduli):
        ct[:, i, :4] = [0, q - 1, 1, q - 2]
    ct[:, :, 4:64] = np.array(moduli, dtype=np.uint64)[None, :, None] - np.uint64(1)
    want = zp.rotate(ct, gk, g, kp)
    src = to_dev(np.stack([ct] * n))
    out = torch.full((n * 2 * nl * N,), -1, dtype=torch.int64, device="cuda")
    L.hc_ct_rotate(ctx, key, src, out)
    many = to_host(out).reshape(n, 2, nl, N)
    assert np.array_equal(many[0], want) and all(np.array_equal(m, many[0]) for m in many)
    one = torch.empty(2 * nl * N, dtype=torch.int64, device="cuda")
    L.hc_ct_rotate(ctx, key, src[0].contiguous(), one)
    assert np.array_equal(to_host(one).reshape(2, nl, N), want)
