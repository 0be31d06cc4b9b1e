"""Integer-pipe work of bench.py in the folded form, which its workloads' moduli take: six wide
multiply-adds a butterfly, three a term of a blocked sum and six a reduction, against independent
statements (no GPU)."""
import os
import sys

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
import bench  # noqa: E402


def test_folded_work():
    assert bench.FORM == "folded"
    # the 56x56x64 layer: I = 32, P = 512, O = 256, 2048 products, N = 8192, L = 3
    geo = dict(I=32, P=512, O=256, products=2048)
    N, L = 8192, 3
    bfly = 4096 * 13
    fwd, inv = 2 * 32 * L * bfly * 12, 2 * 256 * L * bfly * 12
    mac = 2048 * 2 * L * N * 6 + 256 * 2 * L * N * 12
    assert bench.conv_imad_eq(32, 256, 2048, N, L, "folded") == fwd + mac + inv
    assert bench.kernel_work("k_ntt_inv/N8192", geo, N, L, "folded")["imad_eq"] == inv
    assert bench.kernel_work("k_mac_conv", geo, N, L, "folded")["imad_eq"] == mac
    assert bench.product_imad_eq(4096, 2, "folded") == 2 * 2 * (2 * 2048 * 12 * 12 + 4096 * 16)
    # one rotation: 12 digit transforms and 8 inverse ones of N = 8192, L = 3
    assert bench.zp_rotation_imad_eq(N, L) == 20 * bfly * 12 + 24 * N * 8 + 8 * N * 6 + 6 * N * 14
