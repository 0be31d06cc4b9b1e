"""Kernels that may start before their predecessors have ended: every load of what those wrote must
stay behind the wait.  The compiler may move the L2 load intrinsic (ld_data), which it does not see
touching memory, and loads through __restrict__ parameters, so their addresses come from after_wait
and ordinary loads (ld_near) from plain parameters.  Checked in the sources."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2506_11586_gb300", "csrc")
# functions whose address argument was taken behind the wait by their caller
CALLER_WAITS = {"split_fwd_cross": r"split_fwd_cross<[^;]*?>\(\s*(after_wait\(|c1\b)"}


def _functions():
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        if os.path.basename(path) == "hc_async.cuh":
            continue
        text = re.sub(r"//[^\n]*", "", open(path).read())
        for m in re.finditer(r"\n(?:template[^;{]*\n)?(?:__device__|__global__|[a-z_]\w*\()[^;{}]*\)\s*\n\{.*?\n\}", text, re.S):
            yield os.path.basename(path), m.group(0)


def test_loads_stay_behind_the_wait():
    seen = 0
    for path, body in _functions():
        name = re.search(r"(\w+)\s*\(", re.sub(r"__launch_bounds__\([^)]*\)+|__cluster_dims__\([^)]*\)|__align__\(\d+\)", "", body)).group(1)
        assert "__ldca" not in body and ("__ldcg" not in body), (path, name)
        if "ld_data(" in body:
            seen += 1
            assert "after_wait(" in body or name in CALLER_WAITS, (path, name)
        if "ld_near(" in body:
            for arg in re.findall(r"ld_near\((?:reinterpret_cast<[^>]*>\()?\s*(\w+)", body):
                assert not re.search(r"__restrict__ %s\b" % arg, body), (path, name, arg)
    assert seen >= 6


def test_split_callers_wait():
    for f in ("hc_split.cuh", "hc_keyswitch.cuh"):
        text = open(os.path.join(CSRC, f)).read()
        calls = re.findall(r"split_fwd_cross<S, \w+, SP>\(([^,]*),", text)
        assert calls
        for arg in calls:
            base = arg.strip().split(" ")[0].split("(")[0]
            assert base == "after_wait" or re.search(r"\*%s = after_wait\(" % base, text), (f, arg)
