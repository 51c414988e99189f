"""Ordering rules of the device code that hold by the source alone: a run on a
GPU that happens to keep the order cannot show that a rule is broken."""
import os
import re

from paper_2505_23970_gb300 import build as gbuild


def source(name):
    text = open(os.path.join(gbuild.CSRC, name)).read()
    return re.sub(r"//[^\n]*", "", text)


def body(text, function):
    """The function's definition, from its name to the brace that closes it."""
    at = re.search(r"\b%s\s*\([^;{]*\)\s*\{" % function, text)
    depth = 0
    for i in range(text.index("{", at.start()), len(text)):
        depth += {"{": 1, "}": -1}.get(text[i], 0)
        if depth == 0:
            return text[at.start():i + 1]
    raise AssertionError(function)


def test_item_slot_is_released_on_every_lanes_values():
    """The pair kernel's item slots are overwritten from the other CTA without a
    cluster-wide fence, so a warp may release one only once every lane has its
    values: a lane that has not read yet could see the next item."""
    text = source("attn_tc2.cu")
    vote = body(text, "item_read_warp")
    assert re.search(r"__all_sync\(0xffffffffu, w\.read\)", vote)
    for warp_wide in ("producer2", "softmax2h"):
        text_of = body(text, warp_wide)
        assert "item_read_warp(" in text_of
        assert not re.search(r"\bitem_read\(", text_of), warp_wide


def test_dependent_kernels_take_no_read_only_loads():
    """A kernel launched as a programmatic dependent is resident while the one
    before it still writes what it will read, so nothing may say that its inputs
    do not change: no read-only loads, no __restrict__."""
    dependent = [f for f in sorted(os.listdir(gbuild.CSRC))
                 if f.endswith(".cu") and "dependent_begin()" in source(f)]
    assert len(dependent) >= 6
    for name in dependent + ["gc_internal.cuh", "sm103_ptx.cuh"]:
        for word in ("__ldg", r"ld\.global\.nc", "__restrict__"):
            assert not re.search(word, source(name)), (name, word)
