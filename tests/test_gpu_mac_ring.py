"""The blocked MAC's two ways to its weights: layers whose input chunk of 64 slots exceeds 50 KB take
them through the shared-memory ring, in stages of several channels or, where two do not fit, of one;
the others stream them.  On both sides of that line, with even and odd channel counts per stage and
tile, every residue equals the oracle's."""
import numpy as np
import pytest

from gpu_util import sample_indices, to_dev, to_host
from oracle import conv
from paper_2506_11586_gb300.inputs import CANONICAL_PRIMES, T_PLAIN, Stream, uniform_residues

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

P45 = 35184371138561  # prime, 1 mod 2^15: no folded twiddles
# (G, B, M): G*B > 50 through the ring, in stages of 16 / G channels or so (two at least)
SHAPES = [(10, 5, 7), (50, 1, 5), (51, 1, 4),                     # the line: streamed, streamed, ring
          (8, 7, 9), (4, 13, 11), (2, 26, 7), (1, 51, 19),        # stages of 2, 4, 8 and 16 channels
          (17, 9, 5), (16, 10, 1), (30, 2, 3),                    # one-channel stages; one channel; G = 30
          (5, 1, 13), (3, 2, 5), (3, 3, 6), (1, 4, 3)]            # streamed: each tile shape


@pytest.fixture(scope="module")
def L():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2506_11586_gb300 import _lib
    from paper_2506_11586_gb300.build import build
    build()
    return _lib


@pytest.mark.parametrize("moduli", [CANONICAL_PRIMES[:1], (P45,)])
@pytest.mark.parametrize("G,B,M", SHAPES)
def test_ring_and_streamed_layers(L, G, B, M, moduli):
    N, Cw, W = 4096, 2, 5
    C_, H = max(G * Cw - 1, Cw), B                 # blocks of one row; the last of several groups short of a channel
    p = conv.Partition(C_, H, W, M, 1, 1, 0, N, Cw, 1, W)
    assert (p.G, p.B) == (G, B)
    s = Stream(81, G * 64 + B)
    K = s.int8(M * C_).astype(np.int64).reshape(M, C_, 1, 1)
    ct = uniform_residues(s, moduli, (p.I, 2), N)
    ct[..., :2] = moduli[0] - 1
    ks = sample_indices(N, 16, G)
    want = conv.conv_ct_pt(ct, conv.pack_weights(K, p), p, moduli, ks)
    ctx = L.hc_ctx_create(N, moduli, T_PLAIN)
    w = L.hc_weights_preprocess(ctx, L.make_desc(C_, H, W, M, 1, 1, Cw=Cw, Hw=1, Ww=W), K.astype(np.int8))
    d_in = to_dev(ct)
    ref = None
    for v in range(L.N_VARIANTS):
        L.hc_ctx_set_variant(ctx, L.KIND_MAC_CONV, v)
        for form in (0, 2, 1):                     # launches by phase, chains per limb, fused (always the ring)
            L.hc_ctx_set_variant(ctx, L.KIND_CONV_FORM, form)
            out = torch.full((p.O * 2 * N,), -1, dtype=torch.int64, device="cuda")
            L.hc_conv_ct_pt(ctx, w, d_in, out)
            L.hc_ctx_device_status(ctx)
            assert np.array_equal(to_host(out).reshape(p.O, 2, 1, N)[..., ks], want), (v, form)
            ref = out if ref is None else ref
            assert torch.equal(out, ref), (v, form)
