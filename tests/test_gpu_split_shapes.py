"""Transforms and products of few polynomials run split over clusters; around the last size
that does and with both twiddle forms they must give the bits of the one-CTA shapes, and a
round trip returns the input.  (The one-CTA shapes are checked against the oracle in
test_gpu_ntt and test_gpu_mac.)"""
import numpy as np
import pytest

from gpu_util import to_dev, to_host
from paper_2506_11586_gb300.inputs import CANONICAL_PRIMES, T_PLAIN, Stream, uniform_residues

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

P45 = 35184371138561  # prime, 1 mod 2^15: no folded twiddles
NTT_LIMBS = {4096: 7, 8192: 8, 16384: 4}      # eighths of the SM count
PRODUCT_LIMBS = {4096: 3, 8192: 4, 16384: 2}


@pytest.fixture(scope="module")
def L():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2506_11586_gb300 import _lib
    from paper_2506_11586_gb300.build import build
    build()
    return _lib


def _sms():
    return torch.cuda.get_device_properties(0).multi_processor_count


def _residues(seed, moduli, before, N):
    a = uniform_residues(Stream(seed, N), moduli, before, N)
    for i, q in enumerate(moduli):
        a[..., i, :3] = [0, q - 1, 1]
    return a


@pytest.mark.parametrize("moduli", [CANONICAL_PRIMES[:1], (CANONICAL_PRIMES[1], P45)])
@pytest.mark.parametrize("N", [4096, 8192, 16384])
def test_transforms(L, N, moduli):
    nl = len(moduli)
    last = _sms() * NTT_LIMBS[N] // 8 // nl
    for n in (1, last, last + 1):
        a = _residues(7, moduli, (n,), N)
        ctx, one = L.hc_ctx_create(N, moduli, T_PLAIN), L.hc_ctx_create(N, moduli, T_PLAIN)
        for kind in (L.KIND_NTT_FWD, L.KIND_NTT_INV):
            L.hc_ctx_set_variant(one, kind, 1 if N == 4096 else 0)
        d, e = to_dev(a), to_dev(a)
        L.hc_ntt_fwd(ctx, d)
        L.hc_ntt_fwd(one, e)
        assert torch.equal(d, e), n
        L.hc_ntt_inv(one, e)
        L.hc_ntt_inv(ctx, d)
        assert torch.equal(d, e) and np.array_equal(to_host(d).reshape(a.shape), a), n


@pytest.mark.parametrize("moduli", [CANONICAL_PRIMES[:1], (CANONICAL_PRIMES[1], P45)])
@pytest.mark.parametrize("N", [4096, 8192, 16384])
def test_products(L, N, moduli):
    nl = len(moduli)
    last = _sms() * PRODUCT_LIMBS[N] // 8 // nl
    for n in (1, last, last + 1):
        ct, pt = to_dev(_residues(8, moduli, (n, 2), N)), to_dev(_residues(9, moduli, (n,), N))
        slots = (np.arange(n) * 5 + 2) % (n + 3 if (n + 3) % 5 else n + 4)   # distinct, not every slot
        n_out = int(slots.max()) + 2
        got = []
        for variant in (0, 1):           # split where few enough, one CTA per limb
            ctx = L.hc_ctx_create(N, moduli, T_PLAIN)
            L.hc_ctx_set_variant(ctx, L.KIND_PRODUCT, variant)
            out = torch.full((n_out * 2 * nl * N,), -1, dtype=torch.int64, device="cuda")
            L.hc_ctpt_mac(ctx, ct, pt, slots.astype(np.uint32), out)
            got.append(out)
        assert torch.equal(*got), n
        empty = sorted(set(range(n_out)) - set(slots.tolist()))
        assert not got[0].reshape(n_out, -1)[empty].any()
