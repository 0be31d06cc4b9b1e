"""Host model of the folded inverse split over clusters: a part's register rounds, folded down to what
the cross stages may take, then the cross stages, register by register, up to the last sums and
differences."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2506_11586_gb300", "csrc")
FOLD_MAX, FOLDED = 35, 5      # products, folded values: multiples of q


def _limit():
    """What the cross stages are asserted to take: their last stage's inputs, in multiples of q."""
    text = open(os.path.join(CSRC, "hc_split.cuh")).read()
    assert re.search(r"static_assert\(sums <= kFoldStage && \(kFoldMax << LOGP\) <= kFoldStage", text)
    return int(re.search(r"kFoldStage = (\d+)", open(os.path.join(CSRC, "hc_arith.cuh")).read()).group(1))


def _stages(regs, k, q_bits=50):
    for sig in range(k):
        for j in range(len(regs)):
            if not j >> sig & 1:
                hi = regs[j] + regs[j | 1 << sig]
                assert hi << q_bits < 1 << 63
                regs[j], regs[j | 1 << sig] = hi, FOLD_MAX
    return regs


@pytest.mark.parametrize("logn", [12, 13, 14])
@pytest.mark.parametrize("logp", [1, 2, 3])
def test_part_and_cross_stages(logn, logp):
    limit_last = _limit()
    nl = logn - logp
    rounds = [3] * (nl // 3) + ([nl % 3] if nl % 3 else [])
    b = 1
    for r, k in enumerate(rounds):
        limit = 4096 >> (rounds[r + 1] - 1 if r + 1 < len(rounds) else logp - 1)
        regs = _stages([b] * (1 << k), k)
        model = [b << k if j == 0 else FOLD_MAX << (k - 1 - (j.bit_length() - 1)) for j in range(1 << k)]
        assert all(x <= m for x, m in zip(regs, model))
        b = max(FOLDED if m > limit else m for m in model)
        assert b <= limit
    assert b << (logp - 1) <= limit_last and FOLD_MAX << logp <= limit_last
    regs = _stages([b] * (1 << logp), logp - 1)       # inputs of the last cross stage
    assert max(regs) <= limit_last
    assert 2 * max(regs) * ((1 << 50) - 1) + (1 << 36) < 1 << 63
