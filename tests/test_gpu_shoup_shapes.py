"""Contexts without folded twiddles (a modulus that is not 2^50 - c) take other launch shapes than
the default variants' for some sizes.  Around each line: forward transforms as plain and as
ciphertext transforms, products and sums give the bits of a variant chosen explicitly."""
import numpy as np
import pytest

from gpu_util import to_dev, to_host
from paper_2506_11586_gb300.inputs import CANONICAL_PRIMES, T_PLAIN, Stream, uniform_residues

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

P45 = 35184371138561  # prime, 1 mod 2^15: no folded twiddles
EXPLICIT = {4096: 1, 8192: 0, 16384: 1}  # forward variants that no rule redirects


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


@pytest.mark.parametrize("moduli", [(P45,), (CANONICAL_PRIMES[1], P45)])
@pytest.mark.parametrize("N", [4096, 8192, 16384])
def test_forward(L, N, moduli):
    nl, sms = len(moduli), _sms()
    lines = {4096: (sms * 7 // 8, sms, 2 * sms), 8192: (sms * 3 // 4, sms, 3 * sms // 2, 2 * sms), 16384: (sms // 2, sms)}[N]
    ctx, one = (L.hc_ctx_create(N, moduli, T_PLAIN) for _ in range(2))
    for kind in (L.KIND_NTT_FWD, L.KIND_NTT_INV):
        L.hc_ctx_set_variant(one, kind, EXPLICIT[N])
    for n in sorted({max(1, x // nl + d) for x in lines for d in (0, 1)}):
        a = to_dev(_residues(41, moduli, (n,), N))
        d, e = a.clone(), a.clone()
        L.hc_ntt_fwd(ctx, d)
        L.hc_ntt_fwd(one, e)
        assert torch.equal(d, e), n
        L.hc_ntt_inv(ctx, d)
        assert torch.equal(d, a), n


@pytest.mark.parametrize("N", [4096, 8192])
def test_products_and_sums(L, N):
    moduli, sms = (P45,), _sms()
    lines = {4096: (sms // 2, sms, 3 * sms // 2, 3 * sms), 8192: (sms, 7 * sms // 4, 2 * sms)}[N]
    for n in [1] + [x + d for x in lines for d in (0, 1)]:
        ct, pt = to_dev(_residues(42, moduli, (n, 2), N)), to_dev(_residues(43, moduli, (n,), N))
        slots = (np.arange(n) * 7 + 3) % n if n % 7 else np.arange(n)[::-1]
        got = []
        for v in (0, 2 if N == 4096 else 1):
            ctx = L.hc_ctx_create(N, moduli, T_PLAIN)
            L.hc_ctx_set_variant(ctx, L.KIND_PRODUCT, v)
            out = torch.full((n * 2 * N,), -1, dtype=torch.int64, device="cuda")
            L.hc_ctpt_mac(ctx, ct, pt, slots.astype(np.uint32), out)
            got.append(out)
        assert torch.equal(*got), n
    for n, terms in ((1, 9), (5, 4), (7, 3), (2 * sms, 1), (2 * sms + 1, 2)):   # four terms at a time, and rests
        n_prod = n * terms + (1 if terms == 1 else 0)                           # one slot of two at least
        slots = np.arange(n_prod) % n
        ct, pt = to_dev(_residues(44, moduli, (n_prod, 2), N)), to_dev(_residues(45, moduli, (n_prod,), N))
        single = torch.empty(n_prod * 2 * N, dtype=torch.int64, device="cuda")
        ctx = L.hc_ctx_create(N, moduli, T_PLAIN)
        L.hc_ctpt_mac(ctx, ct, pt, np.arange(n_prod, dtype=np.uint32), single)
        want = torch.zeros(n, 2 * N, dtype=torch.int64, device="cuda")
        for j in range(0, n_prod, n):
            part = single.reshape(n_prod, -1)[j:j + n]
            want[:part.shape[0]] = (want[:part.shape[0]] + part) % P45
        for v in range(L.N_VARIANTS):
            L.hc_ctx_set_variant(ctx, L.KIND_MAC_INTT, v)
            out = torch.full((n * 2 * N,), -1, dtype=torch.int64, device="cuda")
            L.hc_ctpt_mac(ctx, ct, pt, slots.astype(np.uint32), out)
            assert torch.equal(out.reshape(n, -1), want), (n, terms, v)


@pytest.mark.parametrize("N", [4096, 8192])
def test_layer_transforms(L, N):
    """A layer with as many input limbs as the redirected sizes, alone and in a two-layer plan."""
    moduli = (P45, CANONICAL_PRIMES[0])
    ctx, one = (L.hc_ctx_create(N, moduli, T_PLAIN) for _ in range(2))
    for kind in (L.KIND_NTT_FWD_CT, L.KIND_NTT_INV_CT):
        L.hc_ctx_set_variant(one, kind, EXPLICIT[N])
    s = Stream(46, N)
    C_, side, M = 200, 28 if N == 4096 else 40, 2
    K = s.int8(M * C_).reshape(M, C_, 1, 1)
    ws = [L.hc_weights_preprocess(c, L.make_desc(C_, side, side, M, 1, 1), K) for c in (ctx, one)]
    w = ws[0]
    assert _sms() * 3 // 4 < 4 * w.I < 4 * _sms()
    ct = to_dev(uniform_residues(s, moduli, (w.I, 2), N))
    outs = [torch.full((w.O * 4 * N,), -1, dtype=torch.int64, device="cuda") for _ in range(4)]
    L.hc_conv_ct_pt(ctx, w, ct, outs[0])
    L.hc_conv_ct_pt(one, ws[1], ct, outs[1])
    plan = L.hc_plan_create([L.work_conv(ctx, w, ct, outs[2]), L.work_conv(ctx, w, ct, outs[3])])
    L.hc_plan_run(plan)
    assert all(torch.equal(outs[0], o) for o in outs[1:])
    assert to_host(outs[0]).max() < CANONICAL_PRIMES[0]
