"""Orderings in the kernels' source that no run can show to be missing: where one is left
out, results are right until timing makes them wrong."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1509_07925_gb300", "csrc")


def _between(text, first, last):
    """The text after `first` up to the next `last`."""
    assert text.count(first) >= 1, first
    rest = text.split(first, 1)[1]
    assert last in rest, last
    return rest.split(last, 1)[0]


def _in_order(text, *parts):
    at = 0
    for p in parts:
        at = text.find(p, at)
        if at < 0:
            return False
        at += len(p)
    return True


def test_stage_vectors_cross_proxies_behind_a_fence():
    """The tensor kernel's epilogue writes a stage's blocks with generic stores, and another
    CTA reads them with bulk copies, which belong to the async proxy: both ends of the
    dependency counters carry a proxy fence, and the panel warp's copying lanes are
    ordered behind the lane that acquired the counter."""
    with open(os.path.join(CSRC, "apply_tc.cu")) as f:
        src = f.read()
    panel = _between(src, "X panels", "L2 discards")
    assert _in_order(panel, "ld_acquire(cp)", "__syncwarp();", "fence_proxy_async_global();", "bulk_g2s(")
    signal = _between(src, "- signal warps", "teardown")
    assert _in_order(signal, "__threadfence();", "fence_proxy_async_global();", "atomicAdd(cnt_out")


def test_no_clear_on_the_default_stream():
    """A clear on the default stream may return before it has run and streams that do not
    block on that stream overtake it: a workspace's status word cleared so late loses the
    timeout that an apply has just recorded, or reads as one before."""
    for path in glob.glob(os.path.join(CSRC, "*.c*")):
        with open(path) as f:
            assert not re.search(r"\bcudaMemset\(", f.read()), os.path.basename(path)
