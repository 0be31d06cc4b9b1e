"""Autotuner caches written before the variant numbers came to stand for other launch shapes are
timed again instead of applied."""
import re

import pytest

from gpu_util import to_dev
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


def test_choices_of_other_shape_tables_are_not_applied(L, tmp_path):
    N, moduli = 4096, CANONICAL_PRIMES[:2]
    ctx = L.hc_ctx_create(N, moduli, T_PLAIN)
    s = Stream(95, 1)
    w = L.hc_weights_preprocess(ctx, L.make_desc(4, 9, 9, 3, 3, 3, pad=1), s.int8(108).reshape(3, 4, 3, 3))
    ct = to_dev(uniform_residues(s, moduli, (w.I, 2), N))
    out = torch.empty(w.O * 4 * N, dtype=torch.int64, device="cuda")
    plan = L.hc_plan_create([L.work_conv(ctx, w, ct, out)])

    def lines(path):
        return [x for x in path.read_text().split("\n") if x]

    new = tmp_path / "new.txt"
    L.hc_plan_autotune(plan, str(new))
    made = lines(new)
    assert made
    # the same file as written by a library without a shape version in its keys
    old = tmp_path / "old.txt"
    old.write_text("".join(re.sub(r"\|shapes\d+", "", x).rsplit(" ", 1)[0] + " 1\n" for x in made))
    L.hc_plan_autotune(plan, str(old))
    assert len(lines(old)) == 2 * len(made)          # every choice timed and appended
    L.hc_plan_autotune(plan, str(old))
    assert len(lines(old)) == 2 * len(made)          # and read from then on
