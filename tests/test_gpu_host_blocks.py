"""The host-buffer layer's blocks of output channels: every channel count from one block to seven
gives the bits of the device-buffer call, with several spatial blocks and a ragged last block, in
layers whose MAC streams its weights (blocks double to the end) and in others (up to a quarter)."""
import numpy as np
import pytest

from gpu_util import to_dev, to_host
from paper_2506_11586_gb300.inputs import CANONICAL_PRIMES, T_PLAIN, Stream, uniform_residues

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def L():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2506_11586_gb300 import _lib
    from paper_2506_11586_gb300.build import build
    build()
    return _lib


@pytest.mark.parametrize("M", [1, 2, 3, 4, 5, 7, 15, 16, 17, 19, 31, 33, 64, 67])
@pytest.mark.parametrize("streams", [True, False])
def test_blocks(L, M, streams):
    N, moduli = 4096, CANONICAL_PRIMES[:2]
    ctx = L.hc_ctx_create(N, moduli, T_PLAIN)
    s = Stream(85, M)
    if streams:      # three channel groups by two spatial blocks
        w = L.hc_weights_preprocess(ctx, L.make_desc(5, 30, 31, M, 3, 3, pad=1, Cw=2, Hw=18, Ww=33),
                                    s.int8(M * 45).reshape(M, 5, 3, 3))
    else:            # eleven by five
        w = L.hc_weights_preprocess(ctx, L.make_desc(22, 5, 6, M, 1, 1, Cw=2, Hw=1, Ww=6),
                                    s.int8(M * 22).reshape(M, 22, 1, 1))
    ct = uniform_residues(s, moduli, (w.I, 2), N)
    ref = torch.empty(w.O * 4 * N, dtype=torch.int64, device="cuda")
    L.hc_conv_ct_pt(ctx, w, to_dev(ct), ref)
    h_in, h_out = torch.from_numpy(ct.view(np.int64)).pin_memory(), torch.full((w.O * 4 * N,), -1, dtype=torch.int64).pin_memory()
    for _ in range(2):
        h_out.fill_(-1)
        L.hc_conv_ct_pt_host(ctx, w, h_in, h_out)
        assert np.array_equal(to_host(h_out), to_host(ref))
