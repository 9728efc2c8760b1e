"""Orders that the decode kernel's memory accesses need and that no run shows reliably, read from its source (CPU)."""
import os
import re

import paper_2608_02901_gb300 as akv

SRC = open(os.path.join(os.path.dirname(akv.__file__), "csrc", "akv_decode.cuh")).read()
SRC = re.sub(r"//[^\n]*", "", SRC)
KERNEL = SRC[SRC.index("akv_decode_kernel(const DecodeParams P)"):]


def _before(text, what, mark):
    """The part of `text` from the last `mark` before the only `what` to it."""
    assert text.count(what) == 1
    head = text[:text.index(what)]
    return head[head.rindex(mark):]


def test_key_terms_are_ordered_before_the_copy_that_takes_their_place():
    """Product warps write key terms into the ring with ordinary stores and release the tile on bar_empty, after which
    a bulk copy (the asynchronous proxy) writes the same bytes: the writers need a proxy fence before that arrival."""
    arrive = "mbar_arrive(bar_empty(lt % NSG))"
    assert "fence.proxy.async.shared::cta" in _before(KERNEL, arrive, "residual(g16")
