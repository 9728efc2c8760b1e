"""Decode launch plans: calls whose plans must differ, and the paths that a rule on sizes picks (GPU)."""
import pytest

import paper_2608_02901_gb300 as akv
from test_decode_parity import _run_seeded, dev  # noqa: F401

pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_order_of_lengths(dev):  # noqa: F811
    """The same lengths in another order: same totals and maxima, other ranges per CTA."""
    p = akv.Params(batch=4, n_kv_heads=2, n_q_heads=8, seed=3)
    for lens in ([8192, 3000, 6001, 700], [700, 8192, 6001, 3000], [6001, 700, 3000, 8192]):
        _run_seeded(dev, p, lens)


@pytest.mark.parametrize("G", [1, 2, 4, 8])
@pytest.mark.parametrize("B,k", [(1, 1), (1, 15), (1, 16), (1, 17), (1, 63), (1, 64), (1, 65), (16, 1024), (16, 1025)])
def test_anchor_counts_around_the_score_paths(dev, G, B, k):  # noqa: F811
    """Anchor counts at the edges of the score launches' blocks, and on both sides of the line between them (64 units:
    16 and 17 chunks of 64 anchors each)."""
    S = max(2 * k, 1500) + 1
    p = akv.Params(batch=B, n_kv_heads=4, n_q_heads=4 * G, anchor_frac=(k - 0.5) / S, window=0, seed=4)
    assert akv.akv_unit_shapes(p, [S] * B)[0][1] == k
    _run_seeded(dev, p, [S] * B)


@pytest.mark.parametrize("S", [7, 8, 9, 57, 63, 65, 255, 257, 1016, 1017, 1023, 1025, 1032, 2047])
@pytest.mark.parametrize("lloyd", [False, True])
def test_partial_tiles(dev, S, lloyd):  # noqa: F811
    """A unit's last tile at the edges of lanes (8 tokens), bitmap words (64) and warps (256)."""
    p = akv.Params(batch=1, n_kv_heads=2, n_q_heads=8, res_frac_k=0.15, res_frac_v=0.15, window=4, seed=5, lloyd=lloyd)
    from helpers import seeded_units  # noqa: F401

    def mutate(u, d):
        if lloyd:
            d["min_k"] = d["min_k"] * 0
            d["min_v"] = d["min_v"] * 0
    _run_seeded(dev, p, [S], mutate=mutate)


@pytest.mark.parametrize("S", [1, 8, 9, 15, 16, 17, 48, 64, 65, 255, 256, 257, 1023, 1025, 1281])
@pytest.mark.parametrize("G,fr,rotate", [(1, 0.1, True), (2, 1.0, True), (4, 0.0, True), (4, 0.3, False), (8, 0.5, True)])
def test_rope_chunks(dev, S, G, fr, rotate):  # noqa: F811
    """Rotary keys at the edges of a warp's pieces (16 tokens), its bitmap word (64), a block (256) and a tile (1024),
    with no, some and only residual tokens, beside a longer request."""
    p = akv.Params(batch=2, n_kv_heads=2, n_q_heads=2 * G, res_frac_k=fr, res_frac_v=0.1, window=4, seed=6, rotate=rotate,
                   rope=True, rope_theta=10000.0)
    _run_seeded(dev, p, [S, 1300], sm_scale=0.1)
