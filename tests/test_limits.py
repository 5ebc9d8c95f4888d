"""Sizes that tests place on both sides of a line are tied to the line's own
constant in the source, so that a moved line fails here instead of leaving the
tests on one side of it."""
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _source(name):
    return open(os.path.join(ROOT, "paper_1212_1639_gb300", "csrc", name)).read()


def _const(src, name):
    m = re.search(r"\b%s = (\d+)" % name, src)
    assert m, name
    return int(m.group(1))


def test_ticket_edges_follow_the_launch_rule():
    import test_gpu_prop_ticket as t
    src = _source("kernels.cuh")
    assert t.UNITS_PER_WARP == {"plain": _const(src, "PROP_DYN"), "adaptive": _const(src, "PROP_DYN_ESS")}
    # _edge: 3 CTAs of 8 warps per SM
    assert re.search(r"__launch_bounds__\(BLOCK, 3\) k_propagate2", src) and _const(src, "BLOCK") == 256


def test_sizes_follow_the_cluster_launches():
    import test_gpu_small as s
    import test_gpu_resample_small as r
    src = _source("small.cuh")
    n32 = _const(src, "SMALL_M") * _const(src, "SMALL_GMAX")
    assert {n32 - 1, n32, n32 + 1} <= set(s.SIZES["fp32"]) and {n32 // 2, n32 // 2 + 1} <= set(s.SIZES["fp64"])
    top = _const(src, "RES_K") * 256 * _const(src, "SMALL_GMAX")
    assert {top, top + 1} <= set(r.SIZES)


def test_sizes_follow_the_heavy_rule():
    src = _source("slots.cuh")
    own = int(re.search(r"OWN = SRC == SRC_E64 \? (\d+) : 0", src).group(1))
    line = (own + 1) * 4096
    text = open(os.path.join(ROOT, "tests", "test_gpu_heavy.py")).read().replace("_", "")
    for n in (line - 64, line - 63, line, line + 1):
        assert str(n) in text, n
