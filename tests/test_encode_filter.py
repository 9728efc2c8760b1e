"""The encoder's fp32 and tensor-core filters where they can go wrong: edges of the position tiles and anchor
chunks, duplicates and equal energies, rows outside the filters' range.  Bit for bit against the fp64 oracle (GPU)."""
import numpy as np
import pytest

import gen
import paper_2608_02901_gb300 as akv
from test_encode_parity import _encode_both, dev  # noqa: F401

pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _scaled(x, e):
    return gen.bf16_bits(np.ldexp(gen.bf16_to_f64(x), e))


@pytest.mark.parametrize("lens", [[127, 128, 129], [255, 256, 257], [384, 385, 386]])
@pytest.mark.parametrize("fa", [0.1, 0.5, 1.0])
def test_tile_and_chunk_edges(dev, lens, fa):  # noqa: F811
    p = akv.Params(batch=3, n_kv_heads=2, n_q_heads=2, anchor_frac=fa, res_frac_k=0.3, res_frac_v=0.1, window=8, seed=5)
    K, V = gen.clustered_batch(3, 2, lens, seed=lens[0])
    _encode_both(dev, p, lens, K, V)


@pytest.mark.parametrize("e", [-70, -40, 33, 60])
def test_rows_outside_the_filter_range(dev, e):  # noqa: F811
    """Whole sides, single positions and single anchors scaled by 2^e, and rows of zeros."""
    lens = [700]
    p = akv.Params(batch=1, n_kv_heads=3, n_q_heads=3, anchor_frac=0.05, res_frac_k=0.2, res_frac_v=0.2, seed=6)
    K, V = gen.clustered_batch(1, 3, lens, seed=9)
    K[0, 0] = _scaled(K[0, 0], e)
    K[0, 1, 5:300:7] = _scaled(K[0, 1, 5:300:7], e)
    V[0, 1, 690:] = _scaled(V[0, 1, 690:], e)  # window positions: anchors
    V[0, 2, ::3] = 0
    _encode_both(dev, p, lens, K, V)


@pytest.mark.parametrize("kinds,k1", [(1, False), (4, True), (4, False), (40, False)])
def test_equal_rows(dev, kinds, k1):  # noqa: F811
    """Positions drawn from a few distinct rows: equal scores (the lowest slot wins), energies that are exactly 0, and
    thousands of equal energies other than 0 (one anchor)."""
    S = 4500
    p = akv.Params(batch=1, n_kv_heads=1, n_q_heads=1, anchor_frac=0.0 if k1 else 0.04, window=1 if k1 else 32,
                   res_frac_k=0.3, res_frac_v=0.9, seed=8)
    K, V = gen.clustered_batch(1, 1, [S], seed=10)
    pick = np.random.Generator(np.random.PCG64(3)).integers(0, kinds, size=S)
    _encode_both(dev, p, [S], K[:, :, pick], V[:, :, pick])
