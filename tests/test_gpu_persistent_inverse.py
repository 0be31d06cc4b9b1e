"""The persistent inverse transforms (variant 2 at N = 4096 and 16384, variant 1 at N = 8192), whose
CTAs load their next limb while they finish one, with more limbs than resident CTAs: every variant
gives the same bits, as a plain inverse, as the inverse of a layer's ciphertexts and of two layers
in one launch, in both twiddle forms."""
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


@pytest.mark.parametrize("last", [CANONICAL_PRIMES[1], P45])
@pytest.mark.parametrize("N", [4096, 8192, 16384])
def test_many_limbs(L, N, last):
    moduli = (CANONICAL_PRIMES[0], last)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    n = sms + 40 + sms // 3 if N < 16384 else sms // 2 + 60    # limbs: above two (one) CTAs an SM, not a multiple
    ctx = L.hc_ctx_create(N, moduli, T_PLAIN)
    a = uniform_residues(Stream(51, N), moduli, (n,), N)
    for i, q in enumerate(moduli):
        a[:, i, :2] = [0, q - 1]
    a = to_dev(a)
    fwd = a.clone()
    L.hc_ntt_fwd(ctx, fwd)
    # a 1x1 layer whose outputs are as many limbs, alone and twice in a plan
    s = Stream(52, N)
    C_, M = 8, (n + 1) // 2
    w = L.hc_weights_preprocess(ctx, L.make_desc(C_, 12, 12, M, 1, 1), s.int8(M * C_).reshape(M, C_, 1, 1))
    assert w.O * 4 >= 2 * n - 2
    ct = to_dev(uniform_residues(s, moduli, (w.I, 2), N))
    ref = torch.empty(w.O * 4 * N, dtype=torch.int64, device="cuda")
    L.hc_conv_ct_pt_plain(ctx, w, ct, ref)
    outs = [torch.empty_like(ref) for _ in range(3)]
    plan = L.hc_plan_create([L.work_conv(ctx, w, ct, o) for o in outs[1:]])
    for v in range(L.N_VARIANTS):
        L.hc_ctx_set_variant(ctx, L.KIND_NTT_INV, v)
        L.hc_ctx_set_variant(ctx, L.KIND_NTT_INV_CT, v)
        d = fwd.clone()
        L.hc_ntt_inv(ctx, d)
        assert torch.equal(d, a), v
        for o in outs:
            o.fill_(-1)
        L.hc_conv_ct_pt(ctx, w, ct, outs[0])
        L.hc_profile_enable(True)           # launches directly, in the variants as they are now
        L.hc_plan_run(plan)
        L.hc_profile_enable(False)
        L.hc_profile_collect()
        L.hc_ctx_device_status(ctx)
        assert all(torch.equal(o, ref) for o in outs), v
