"""Device buffers on odd words (8 bytes past a 16-byte boundary): inverse transforms at N >= 8192
and convolutions give the bits of aligned buffers, and operands that the kernels read or store in
pairs are refused before any kernel takes them."""
import numpy as np
import pytest

from gpu_util import to_dev
from paper_2506_11586_gb300.inputs import CANONICAL_PRIMES, T_PLAIN, Stream, uniform_residues

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


def _odd(words, src=None):
    t = torch.full((words + 2,), -1, dtype=torch.int64, device="cuda")
    v = t[1:words + 1]
    assert v.data_ptr() % 16 == 8
    if src is not None:
        v.copy_(src.reshape(-1))
    return t, v


@pytest.mark.parametrize("N,nl", [(8192, 3), (16384, 4)])
@pytest.mark.parametrize("last", [CANONICAL_PRIMES[-1], P45])
def test_inverse_on_odd_words(L, N, nl, last):
    moduli = CANONICAL_PRIMES[:nl - 1] + (last,)
    for n in (1, 60, 340 // nl + 1):     # one unit, fewer and more than the resident CTAs
        a = to_dev(uniform_residues(Stream(31, n), moduli, (n,), N))
        for variant in range(L.N_VARIANTS):
            ctx = L.hc_ctx_create(N, moduli, T_PLAIN)
            L.hc_ctx_set_variant(ctx, L.KIND_NTT_INV, variant)
            d = a.clone()
            L.hc_ntt_fwd(ctx, d)
            t, v = _odd(n * nl * N, d)
            L.hc_ntt_inv(ctx, v)
            assert torch.equal(v, a.reshape(-1)), (n, variant)
            assert t[0] == -1 and t[-1] == -1


@pytest.mark.parametrize("N,nl", [(8192, 3), (16384, 4)])
@pytest.mark.parametrize("M", [5, 60])
def test_layer_on_odd_words(L, N, nl, M):
    ctx = L.hc_ctx_create(N, CANONICAL_PRIMES[:nl], T_PLAIN)
    s = Stream(32, M)
    w = L.hc_weights_preprocess(ctx, L.make_desc(8, 12, 12, M, 3, 3, pad=1), s.int8(M * 8 * 9).reshape(M, 8, 3, 3))
    ct = to_dev(uniform_residues(s, CANONICAL_PRIMES[:nl], (w.I, 2), N))
    words = w.O * 2 * nl * N
    ref = torch.empty(words, dtype=torch.int64, device="cuda")
    L.hc_conv_ct_pt(ctx, w, ct, ref)
    _, cin = _odd(ct.numel(), ct)
    for form in range(3):
        for mac in (0, 3):               # integer and tensor-core MAC
            L.hc_ctx_set_variant(ctx, L.KIND_CONV_FORM, form)
            L.hc_ctx_set_variant(ctx, L.KIND_MAC_CONV, mac)
            t, out = _odd(words)
            L.hc_conv_ct_pt(ctx, w, cin, out)
            L.hc_ctx_device_status(ctx)
            assert torch.equal(out, ref), (form, mac)
            assert t[0] == -1 and t[-1] == -1


def test_operands_taken_in_pairs_are_refused(L):
    """Odd words where the kernels take pairs: an error before the launch, and the context goes on."""
    N, moduli = 4096, CANONICAL_PRIMES[:2]
    ctx = L.hc_ctx_create(N, moduli, T_PLAIN)
    s = Stream(33, 1)
    ct = to_dev(uniform_residues(s, moduli, (2, 2), N))
    pt = to_dev(uniform_residues(s, moduli, (2,), N))
    _, pt_odd = _odd(pt.numel(), pt)
    _, ct_odd = _odd(ct.numel(), ct)
    out = torch.full((ct.numel(),), 7, dtype=torch.int64, device="cuda")
    gk = np.stack([np.stack([np.stack([s.below(q, N) for q in CANONICAL_PRIMES[:3]]) for _ in range(2)]) for _ in range(2)])
    key = L.hc_galois_key_create(ctx, CANONICAL_PRIMES[2], 5, gk)
    desc = L.make_desc(1, 4, 4, 2, 1, 2)
    w = L.hc_weights_preprocess(ctx, L.make_desc(2, 6, 6, 3, 3, 3), s.int8(54).reshape(3, 2, 3, 3))
    wi = to_dev(uniform_residues(s, moduli, (w.I, 2), N))
    _, w_out = _odd(w.O * 4 * N)
    calls = {
        "fwd": lambda: L.hc_ntt_fwd(ctx, pt_odd),
        "inv": lambda: L.hc_ntt_inv(ctx, pt_odd),
        "products": lambda: L.hc_ctpt_mac(ctx, ct, pt_odd, np.array([0, 1]), out),
        "sums": lambda: L.hc_ctpt_mac(ctx, ct, pt_odd, np.array([0, 0]), out),
        "iteration": lambda: L.hc_mac_rotate(ctx, key, ct[0], pt_odd, out[:4 * N]),
        "zp conv": lambda: L.hc_zp_conv(ctx, desc, key, None, pt_odd, ct[0], out[:4 * N]),
        "plan": lambda: L.hc_plan_create([L.work_products(ctx, ct, pt_odd, out)]),
        "layer": lambda: L.hc_conv_ct_pt(ctx, w, wi, w_out),
    }
    for name, call in calls.items():
        with pytest.raises(L.HcError) as e:
            call()
        assert e.value.status == L.HC_ERR_INVALID_ARG, name
    torch.cuda.synchronize()
    assert torch.all(out == 7) and torch.all(w_out == -1)
    # ciphertexts may lie anywhere
    ref = torch.empty_like(out)
    L.hc_ctpt_mac(ctx, ct, pt, np.array([0, 1]), ref)
    t, out_odd = _odd(ct.numel())
    L.hc_ctpt_mac(ctx, ct_odd, pt, np.array([0, 1]), out_odd)
    assert torch.equal(out_odd, ref) and t[0] == -1 and t[-1] == -1
    L.hc_mac_rotate(ctx, key, ct[0], pt, ref[:4 * N])
    L.hc_mac_rotate(ctx, key, ct_odd[:4 * N], pt, out_odd[:4 * N])
    assert torch.equal(out_odd[:4 * N], ref[:4 * N])
