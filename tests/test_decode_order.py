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
    """A tile's shape (tokens, fast, nVs, offsets) is written by the product warp that waited for it.  If that wait runs
    out, the descriptor holds the shape of an older tile, which must not be used with the bytes of one that lands late: the
    warp takes its tokens away and marks it before it arrives on bar_kdone; the token warps have nothing to do then, and
    the product warps look at the mark before they touch the tile."""
    phase = KERNEL[KERNEL.index("auto key_phase"):KERNEL.index("mbar_arrive(bar_kdone(b))")]
    assert re.search(r"else if \(wi8 == 0 && lane == 0\) \{\s*meta\[t % NSG\]\.fast = kNoShape;\s*meta\[t % NSG\]\.n = 0;", phase)
    tokens = KERNEL[KERNEL.index("mt.fast & 1u"):KERNEL.index("mbar_arrive(bar_tdone(b))")]
    assert re.search(r"constexpr uint32_t kNoShape = 4u;", SRC) and re.search(r"else if \(t0 < tv\.n\)", tokens)
    assert re.search(r"const bool go = waited && !\(mt\.fast & kNoShape\);", KERNEL)
