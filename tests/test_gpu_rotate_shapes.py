"""The key switch's launch shapes (few units: a thread group per digit; many: two
digits per thread) against the oracle's rotation, at every ring degree, with one digit,
odd and even digit counts, both twiddle forms (canonical primes; a 45-bit prime among
them), residues at both ends of their range, and buffers on odd words."""
import numpy as np
import pytest

from gpu_util import to_dev, to_host
from oracle import zp
from paper_2506_11586_gb300.inputs import CANONICAL_PRIMES, Stream

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

P45 = 35184371138561  # prime, 1 mod 2^15: no folded twiddles


@pytest.fixture(scope="module")
def L():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2506_11586_gb300 import _lib
    from paper_2506_11586_gb300.build import build
    build()
    return _lib


@pytest.mark.parametrize("N,moduli,special,g", [
    (4096, CANONICAL_PRIMES[:1], CANONICAL_PRIMES[1], 5),
    (4096, CANONICAL_PRIMES[:2], P45, 8191),
    (4096, CANONICAL_PRIMES[:5], CANONICAL_PRIMES[5], 1),
    (8192, CANONICAL_PRIMES[:3], CANONICAL_PRIMES[3], 3277),
    (8192, (CANONICAL_PRIMES[0], P45), CANONICAL_PRIMES[3], 5),
    (16384, CANONICAL_PRIMES[:2], CANONICAL_PRIMES[2], 25),
])
def test_both_shapes_match_the_oracle(L, N, moduli, special, g):
    nl = len(moduli)
    kp = zp.KsParams(N, tuple(moduli), special)
    s = Stream(191, N + nl)
    gk = np.stack([np.stack([np.stack([s.below(q, N) for q in kp.qp]) for _ in range(2)]) for _ in range(nl)])
    ctx = L.hc_ctx_create(N, moduli, 65537)
    key = L.hc_galois_key_create(ctx, special, g, gk)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    n = 2 * sms // (8 * (nl + 1)) + 1        # the first size on the throughput shape
    cts = np.stack([np.stack([np.stack([s.below(q, N) for q in moduli]) for _ in range(2)]) for _ in range(n)])
    for i, q in enumerate(moduli):
        cts[0, :, i, :4] = [0, q - 1, 1, q - 2]
    cts[-1] = cts[0]                     # first and last unit of the launch: the same answer
    want = zp.rotate(cts[0], gk, g, kp)
    words = 2 * nl * N
    d = to_dev(cts)
    for off in (0, 1):                   # 16-byte aligned and not
        src = torch.empty(n * words + 1, dtype=torch.int64, device="cuda")[off:off + n * words]
        src.copy_(d.reshape(-1))
        out = torch.full((n * words + 2,), -1, dtype=torch.int64, device="cuda")
        L.hc_ct_rotate(ctx, key, src, out[off:off + n * words])
        L.hc_ctx_device_status(ctx)
        many = to_host(out)
        assert many[off + n * words] == 2**64 - 1
        many = many[off:off + n * words].reshape(n, 2, nl, N)
        assert np.array_equal(many[0], want) and np.array_equal(many[-1], want)
        one = torch.empty(words, dtype=torch.int64, device="cuda")
        for c in (0, 1, n // 2):         # the latency shape, one ciphertext at a time
            L.hc_ct_rotate(ctx, key, d.reshape(n, words)[c], one)
            assert np.array_equal(to_host(one).reshape(2, nl, N), many[c]), c
