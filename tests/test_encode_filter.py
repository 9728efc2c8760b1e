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


@pytest.mark.parametrize("lloyd,rotate", [(True, True), (True, False), (False, True)])
@pytest.mark.parametrize("e", [-60, -46, -44, -42, -40, 20, 52])
def test_record_magnitudes(dev, e, lloyd, rotate):  # noqa: F811
    """Residuals on both sides of the range in which the fp32 quantiser's sums of squares stay normal."""
    lens = [400]
    p = akv.Params(batch=1, n_kv_heads=1, n_q_heads=1, anchor_frac=0.05, res_frac_k=0.5, res_frac_v=0.5, seed=16,
                   lloyd=lloyd, rotate=rotate)
    K, V = gen.clustered_batch(1, 1, lens, seed=17)
    K[0, 0] = _scaled(K[0, 0], e)
    V[0, 0, ::2] = _scaled(V[0, 0, ::2], e)
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


@pytest.mark.parametrize("k", [1, 31, 33, 127, 129, 256, 300, 640])
def test_near_ties_across_anchor_chunks(dev, k):  # noqa: F811
    """Every row again half the positions later, one bit apart in one dimension: the nearest anchors' scores differ by
    less than the filter tells, mostly in different anchor chunks (of 128, in turn to two accumulators)."""
    S = 1300
    p = akv.Params(batch=1, n_kv_heads=1, n_q_heads=1, anchor_frac=(k - 0.5) / S, window=0, res_frac_k=0.1,
                   res_frac_v=0.1, seed=14)
    assert akv.akv_unit_shapes(p, [S])[0][1] == k
    K, V = gen.clustered_batch(1, 1, [S], seed=15)
    for X in (K, V):
        X[:, :, S // 2:] = X[:, :, :S // 2]
        X[:, :, S // 2:, 7] ^= 1
    _encode_both(dev, p, [S], K, V)


@pytest.mark.parametrize("kinds,e", [(30, 0), (0, 40), (300, 0)])
def test_selection_left_to_fp64(dev, kinds, e):  # noqa: F811
    """The full selection where the paired sums cannot rank: positions drawn from a few distinct rows (equal scores
    and utilities, ties to the lower head and position), and keys whose norms leave the fp32 range."""
    import oracle
    import torch
    from helpers import assert_same_unit, stored_order, to_dev_u16
    lens, H, G, W = [900, 333], 2, 2, 16
    p = akv.Params(batch=2, n_kv_heads=H, n_q_heads=H * G, anchor_frac=0.06, res_frac_k=0.0, res_frac_v=0.0, window=W,
                   seed=12, rot_seed=13)
    sel = akv.SelectParams(theta=0.3, rho=0.7, kappa=3)
    K, V = gen.clustered_batch(2, H, lens, seed=14)
    if kinds:
        pick = np.random.Generator(np.random.PCG64(4)).integers(0, min(kinds, 300), size=K.shape[2])
        K, V = K[:, :, pick].copy(), V[:, :, pick].copy()
        for b, S in enumerate(lens):
            K[b, :, S:] = V[b, :, S:] = 0
    K = _scaled(K, e)
    Q = gen.observation_queries(_scaled(K, -e), lens, W * G, seed=15)
    a_bytes, w_bytes = akv.akv_cache_size_select(p, sel, lens)
    arena = torch.empty(a_bytes, dtype=torch.uint8, device=dev)
    ws = torch.full((w_bytes,), 0xAB, dtype=torch.uint8, device=dev)
    akv.akv_encode_select(p, sel, lens, to_dev_u16(K, torch, dev), to_dev_u16(V, torch, dev), to_dev_u16(Q, torch, dev), arena, ws)
    got = oracle.unpack_arena(arena.cpu().numpy())
    want = oracle.encode_select(K, V, Q, lens, H, p.anchor_frac, W, sel.theta, sel.rho, sel.kappa, p.seed, p.rot_seed, True)
    for u, (g, w) in enumerate(zip(got, want)):
        assert (g.S, g.k, g.nk, g.nv) == (w.S, w.k, w.nk, w.nv), u
        assert_same_unit(g, stored_order(w), f"unit {u}")


@pytest.mark.parametrize("e", [-125, -90, 62, 64, 110])
def test_rows_far_outside_the_filter_range(dev, e):  # noqa: F811
    """The same with rows whose products fp32 does not hold unscaled, of subnormal components among them, both sides at
    once, near ties (rows that differ by a bit), and one such anchor in a unit of ordinary rows."""
    lens = [700]
    p = akv.Params(batch=1, n_kv_heads=4, n_q_heads=4, anchor_frac=0.1, res_frac_k=0.2, res_frac_v=0.2, seed=21)
    K, V = gen.clustered_batch(1, 4, lens, seed=22)
    K[0, 0], V[0, 0] = _scaled(K[0, 0], e), _scaled(V[0, 0], e)
    K[0, 1, 350:] = K[0, 1, :350]
    K[0, 1, 350:, 5] ^= 1
    K[0, 1] = _scaled(K[0, 1], e)
    K[0, 2, 5:300:7] = _scaled(K[0, 2, 5:300:7], e)
    V[0, 2, 699:] = _scaled(V[0, 2, 699:], e)
    V[0, 3, ::3] = _scaled(V[0, 3, ::3], -e // 2)
    V[0, 3, 1::3] = _scaled(V[0, 3, 1::3], e)
    _encode_both(dev, p, lens, K, V)


def test_time_with_an_anchor_outside_the_filter_range(dev):  # noqa: F811
    """One tiny anchor per unit turns the filter off for it: the scores are then fp32 of scaled rows (some 25 times the
    call's time), not fp64 (350 times)."""
    import torch
    p = akv.Params(batch=1, n_kv_heads=8, n_q_heads=8, seed=23)
    lens = [32768]
    K = torch.randn((1, 8, lens[0], 128), device=dev).to(torch.bfloat16)
    V = torch.randn_like(K)
    a, w = akv.akv_cache_size(p, lens)
    arena, ws = torch.empty(a, dtype=torch.uint8, device=dev), torch.empty(w, dtype=torch.uint8, device=dev)

    def ms():
        best = 1e9
        for _ in range(3):
            x, y = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            x.record()
            akv.akv_encode(p, lens, K, V, arena, ws)
            y.record()
            torch.cuda.synchronize()
            best = min(best, x.elapsed_time(y))
        return best

    plain = ms()
    K[:, :, -1] *= 1e-11  # (a window position)
    assert ms() < 100 * plain
