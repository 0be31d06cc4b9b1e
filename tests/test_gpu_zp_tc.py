"""The Z_P calls' products take the blocked MAC, and with it the tensor-core MAC where a context is set
to it: the same bits as with the integer MAC, for one and several ciphertexts, more plaintexts than
one tile of channels, and sums of several terms."""
import numpy as np
import pytest

from gpu_util import to_dev
from paper_2506_11586_gb300.inputs import CANONICAL_PRIMES, Stream, uniform_residues

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


@pytest.mark.parametrize("N,moduli", [(4096, CANONICAL_PRIMES[:2]), (8192, (CANONICAL_PRIMES[0], P45)),
                                      (16384, CANONICAL_PRIMES[:1])])
def test_products_through_either_mac(L, N, moduli):
    nl, special = len(moduli), CANONICAL_PRIMES[4]
    s = Stream(97, N)
    gk = np.stack([np.stack([np.stack([s.below(q, N) for q in tuple(moduli) + (special,)]) for _ in range(2)])
                   for _ in range(nl)])

    def res(*shape):
        a = uniform_residues(s, moduli, shape, N)
        for i, q in enumerate(moduli):
            a[..., i, :4] = [0, q - 1, q - 1, 1]
        return to_dev(a)

    cts, ws, step = res(4, 2), res(70), 8 - 3 + 1
    wz = {c: res(3 * 9 * c) for c in (1, 8)}
    got = []
    for variant in (0, 3):
        ctx = L.hc_ctx_create(N, moduli, 65537)
        L.hc_ctx_set_variant(ctx, L.KIND_MAC_CONV, variant)
        key = L.hc_galois_key_create(ctx, special, 5, gk)
        row = L.hc_galois_key_create(ctx, special, pow(5, step, 2 * N), gk)
        outs = []
        for m, n in ((1, 1), (1, 70), (4, 5), (3, 2)):
            out = torch.full((m * 2 * nl * N,), -1, dtype=torch.int64, device="cuda")
            L.hc_mac_rotate_many(ctx, key, cts[:m].contiguous(), ws[:n].contiguous(), out)
            outs.append(out)
        for c in (1, 8):
            ct = torch.cat([cts, cts])[:c].contiguous()
            out = torch.full((3 * 2 * nl * N,), -1, dtype=torch.int64, device="cuda")
            L.hc_zp_conv(ctx, L.make_desc(c, 6, 6, 5, 3, 3, pad=1), key, row, wz[c], ct, out)
            outs.append(out)
        L.hc_ctx_device_status(ctx)
        got.append(outs)
    assert all(torch.equal(a, b) for a, b in zip(*got))
