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


def test_a_tile_without_its_shape_is_left_alone():
    """A tile's shape (fast, nVs, offsets) is written by the product warp that waited for it.  If that wait runs out, the
    descriptor holds the shape of an older tile, which must not be used with the bytes of one that lands late: the
    warp marks it before it arrives on bar_kdone, and both roles look at the mark before they touch the tile."""
    phase = KERNEL[KERNEL.index("auto key_phase"):KERNEL.index("mbar_arrive(bar_kdone(b))")]
    assert re.search(r"else if \(wi8 == 0 && lane == 0\) \{\s*meta\[t % NSG\]\.fast = kNoShape;", phase)
    uses = re.findall(r"const bool go = [^;]*;", KERNEL)
    assert len(uses) == 3  # the key phase's own, the token warps' and the product warps'
    for go in uses:
        assert "landed" in go or "kNoShape" in go, go
