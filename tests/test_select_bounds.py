"""The full selection's error bounds where its utilities nearly vanish or its products leave the fp32 range: the
chosen slots and every byte are those of the fp64 oracle (GPU)."""
import numpy as np
import pytest

import gen
import oracle
import paper_2608_02901_gb300 as akv
from helpers import assert_same_unit, stored_order, to_dev_u16
from test_encode_parity import dev  # noqa: F401

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

H, G, W = 2, 2, 8


def _encode_both(dev, K, V, Q, lens, theta, anchor_frac=0.001, rho=0.0):  # noqa: F811
    """K, V, Q as fp64, rounded to bf16; anchors: the window alone, unless anchor_frac says more."""
    K, V, Q = (gen.bf16_bits(x) for x in (K, V, Q))
    p = akv.Params(batch=len(lens), n_kv_heads=H, n_q_heads=H * G, anchor_frac=anchor_frac, res_frac_k=0.0, res_frac_v=0.0,
                   window=W, seed=12, rot_seed=13)
    sel = akv.SelectParams(theta=theta, rho=rho, kappa=3)
    a_bytes, w_bytes = akv.akv_cache_size_select(p, sel, lens)
    arena = torch.empty(a_bytes, dtype=torch.uint8, device=dev)
    ws = torch.full((w_bytes,), 0xAB, dtype=torch.uint8, device=dev)
    akv.akv_encode_select(p, sel, lens, to_dev_u16(K, torch, dev), to_dev_u16(V, torch, dev), to_dev_u16(Q, torch, dev), arena, ws)
    got = oracle.unpack_arena(arena.cpu().numpy())
    want = oracle.encode_select(K, V, Q, lens, H, p.anchor_frac, W, sel.theta, sel.rho, sel.kappa, p.seed, p.rot_seed, True)
    room = sum(w.S - w.k for w in want)
    assert 0 < sum(w.nk for w in want) < room and 0 < sum(w.nv for w in want) < room  # the budget cuts among the candidates
    for u, (g, w) in enumerate(zip(got, want)):
        assert (g.S, g.k, g.nk, g.nv) == (w.S, w.k, w.nk, w.nv), u
        assert_same_unit(g, stored_order(w), f"unit {u}")


@pytest.mark.parametrize("seed", range(8))
def test_token_that_takes_all_the_attention(dev, seed):  # noqa: F811
    """One position outside the window takes all but about 1e-11 of every row's attention, so its |V - y|^2, and with it
    u^K, is a difference of nearly equal sums that may come out on either side of 0; in fp64 it ranks high."""
    S, r = 500, np.random.Generator(np.random.PCG64(100 + seed))
    K, V = r.standard_normal((2, 1, H, S, 128))
    at = 17 + 31 * seed
    K[:, :, at] *= np.sqrt(128.0) / np.linalg.norm(K[:, :, at], axis=-1, keepdims=True)
    Q = 3.2 * K[:, :, at:at + 1] + 0.1 * r.standard_normal((1, H, W * G, 128))
    _encode_both(dev, K, V, Q, [S], theta=0.12)


@pytest.mark.parametrize("eq,ek", [(-126, -18), (-66, -79)])
def test_products_below_the_fp32_range(dev, eq, ek):  # noqa: F811
    """Queries and key residuals whose products, or whose squares, fall below what fp32 holds: the sums of q . r are
    then off by far more than their relative error."""
    S, r = 500, np.random.Generator(np.random.PCG64(7))
    K, V = r.standard_normal((2, 1, H, S, 128))
    Q = r.standard_normal((1, H, W * G, 128))
    _encode_both(dev, np.ldexp(K, ek), V, np.ldexp(Q, eq), [S], theta=0.08)


@pytest.mark.parametrize("e", [-73, -74])
def test_value_residuals_below_the_fp32_range(dev, e):  # noqa: F811
    """Values of ordinary norm that differ from their anchors by amounts whose squares fp32 does not hold."""
    S, r = 500, np.random.Generator(np.random.PCG64(8))
    K, V = r.standard_normal((2, 1, H, S, 128))
    V = np.ldexp(V, e)
    V[..., 0] = 4.0
    Q = 1e-3 * r.standard_normal((1, H, W * G, 128))
    _encode_both(dev, K, V, Q, [S], theta=0.08)


def test_attention_taken_in_fp64_once(dev):  # noqa: F811
    """Where the scores and the utilities are both left to fp64 (keys whose norms leave the fp32 range), the attention is
    taken in fp64 once: the call takes little longer than one without scored anchors."""
    S, heads = 4096, 8
    p = akv.Params(batch=1, n_kv_heads=heads, n_q_heads=4 * heads, anchor_frac=0.02, res_frac_k=0.0, res_frac_v=0.0, seed=3)
    g = torch.Generator(device=dev).manual_seed(5)
    K, V = ((torch.randn((1, heads, S, 128), generator=g, device=dev) * f).to(torch.bfloat16) for f in (1e12, 1.0))
    Q = torch.randn((1, heads, 128, 128), generator=g, device=dev).to(torch.bfloat16)

    def ms(rho):
        sel = akv.SelectParams(theta=0.05, rho=rho, kappa=7)
        a, w = akv.akv_cache_size_select(p, sel, [S])
        arena, ws = torch.empty(a, dtype=torch.uint8, device=dev), torch.empty(w, dtype=torch.uint8, device=dev)
        best = 1e9
        for _ in range(3):
            x, y = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            x.record()
            akv.akv_encode_select(p, sel, [S], K, V, Q, arena, ws)
            y.record()
            torch.cuda.synchronize()
            best = min(best, x.elapsed_time(y))
        return best

    assert ms(0.7) < 1.08 * ms(0.0)  # (1.00; 1.17 with it taken twice)
