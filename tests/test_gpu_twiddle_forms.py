"""Kernels exist in two twiddle forms, and launches over several contexts split by form.  Contexts
without folded twiddles through every kernel family, and plans that mix both kinds of contexts,
against the oracle and against the calls one by one."""
import numpy as np
import pytest

from gpu_util import sample_indices, to_dev, to_host
from oracle import conv, core
from paper_2506_11586_gb300.inputs import CANONICAL_PRIMES, T_PLAIN, Stream, uniform_residues

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

P45 = 35184371138561  # prime, 1 mod 2^15: no folded twiddles
DEGREES = (4096, 8192, 16384)
FORMS = (CANONICAL_PRIMES[:2], (P45, CANONICAL_PRIMES[2]))


@pytest.fixture(scope="module")
def L():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2506_11586_gb300 import _lib
    from paper_2506_11586_gb300.build import build
    build()
    return _lib


def _layer(L, ctx, seed, C_=6, side=9, M=5):
    N, moduli = ctx.N, ctx.moduli
    s = Stream(seed, N)
    K = s.int8(M * C_ * 9).astype(np.int64).reshape(M, C_, 3, 3)
    w = L.hc_weights_preprocess(ctx, L.make_desc(C_, side, side, M, 3, 3, pad=1), K.astype(np.int8))
    ct = uniform_residues(s, moduli, (w.I, 2), N)
    p = conv.canonical_partition(C_, side, side, M, 3, 3, 1, N)
    ks = sample_indices(N, 8, seed)
    want = conv.conv_ct_pt(ct, conv.pack_weights(K, p), p, moduli, ks)
    out = torch.full((w.O * 2 * len(moduli) * N,), -1, dtype=torch.int64, device="cuda")
    return dict(ctx=ctx, w=w, d_in=to_dev(ct), out=out, ks=ks, want=want)


def _check_layer(it):
    got = to_host(it["out"]).reshape(it["w"].O, 2, len(it["ctx"].moduli), it["ctx"].N)
    assert np.array_equal(got[..., it["ks"]], it["want"])


def _products(L, ctx, seed, n=5):
    N, moduli = ctx.N, ctx.moduli
    s = Stream(seed, N)
    ct, pt = uniform_residues(s, moduli, (n, 2), N), uniform_residues(s, moduli, (n,), N)
    d_pt = to_dev(pt)
    L.hc_ntt_fwd(ctx, d_pt)
    ks = sample_indices(N, 8, seed)
    want = np.stack([np.stack([np.stack([core.negacyclic(ct[j, c, i], pt[j, i], q, ks) for i, q in enumerate(moduli)])
                               for c in range(2)]) for j in range(n)])
    out = torch.full((n * 2 * len(moduli) * N,), -1, dtype=torch.int64, device="cuda")
    return dict(ctx=ctx, d_ct=to_dev(ct), d_pt=d_pt, out=out, ks=ks, want=want, n=n)


def _check_products(it):
    got = to_host(it["out"]).reshape(it["n"], 2, len(it["ctx"].moduli), it["ctx"].N)
    assert np.array_equal(got[..., it["ks"]], it["want"])


def _launches(L, plan):
    L.hc_profile_enable(True)
    L.hc_profile_collect()
    L.hc_plan_run(plan)
    got = sum(n for n, _ in L.hc_profile_collect().values())
    L.hc_profile_enable(False)
    return got


@pytest.mark.parametrize("form", [0, 1, 2])
def test_plan_of_both_forms(L, form):
    """Layers and products of both forms at the three degrees: one launch per form that occurs."""
    layers, prods = [], []
    for N in DEGREES:
        for moduli in FORMS:
            ctx = L.hc_ctx_create(N, moduli, T_PLAIN)
            L.hc_ctx_set_variant(ctx, L.KIND_CONV_FORM, form)
            layers.append(_layer(L, ctx, 61 + form))
            prods.append(_products(L, ctx, 64))
    plan = L.hc_plan_create([L.work_conv(it["ctx"], it["w"], it["d_in"], it["out"]) for it in layers]
                            + [L.work_products(it["ctx"], it["d_ct"], it["d_pt"], it["out"]) for it in prods])
    for _ in range(3):             # direct, captured, replayed
        for it in layers + prods:
            it["out"].fill_(-1)
        L.hc_plan_run(plan)
        for it in layers:
            _check_layer(it)
        for it in prods:
            _check_products(it)
    for it in layers:
        L.hc_ctx_device_status(it["ctx"])
    assert _launches(L, plan) == L.hc_plan_info(plan)[2]


@pytest.mark.parametrize("N", DEGREES)
def test_every_launch_shape_without_folded_twiddles(L, N):
    ctx = L.hc_ctx_create(N, FORMS[1], T_PLAIN)
    it, pr = _layer(L, ctx, 71, C_=7, side=11, M=6), _products(L, ctx, 72)
    share, mask = (Stream(73, N).below(T_PLAIN, n).astype(np.uint64) for n in (7 * 121, 6 * 121))
    d_share, d_mask = to_dev(share), to_dev(mask)
    S, nl = L.slot_count(it["w"]), 2
    plan = L.hc_plan_create([L.work_products(ctx, pr["d_ct"], pr["d_pt"], pr["out"])])
    L.hc_plan_run(plan)
    _check_products(pr)
    for v in range(L.N_VARIANTS):
        for kind in (L.KIND_NTT_FWD, L.KIND_NTT_INV, L.KIND_NTT_FWD_CT, L.KIND_NTT_INV_CT, L.KIND_MAC_INTT,
                     L.KIND_PRODUCT, L.KIND_MAC_CONV):
            L.hc_ctx_set_variant(ctx, kind, v)
        for form in (0, 1, 2):
            L.hc_ctx_set_variant(ctx, L.KIND_CONV_FORM, form)
            it["out"].fill_(-1)
            L.hc_conv_ct_pt(ctx, it["w"], it["d_in"], it["out"])
            _check_layer(it)
            full = torch.full_like(it["out"], -1)
            slots = torch.full((it["w"].O * nl * S,), -1, dtype=torch.int64, device="cuda")
            c1, slots2 = torch.full((it["w"].O * nl * N,), -1, dtype=torch.int64, device="cuda"), slots.clone()
            L.hc_conv_server_step(ctx, it["w"], it["d_in"], d_share, d_mask, full, slots)
            L.hc_conv_server_step_sparse(ctx, it["w"], it["d_in"], d_share, d_mask, c1, slots2)
            assert torch.equal(slots, slots2)
            assert torch.equal(c1.view(it["w"].O, -1), full.view(it["w"].O, 2, -1)[:, 1])
        pr["out"].fill_(-1)
        L.hc_ctpt_mac(ctx, pr["d_ct"], pr["d_pt"], np.arange(pr["n"], dtype=np.uint32), pr["out"])
        _check_products(pr)
        L.hc_ctx_device_status(ctx)
