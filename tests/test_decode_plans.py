"""Decode launch plans: calls whose plans must differ, and the paths that a rule on sizes picks (GPU)."""
import pytest

import paper_2608_02901_gb300 as akv
from test_decode_parity import _run_seeded, debug_controls, dev  # noqa: F401

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


@pytest.mark.parametrize("before", ["nothing", "copy", "kernel", "join"])
@pytest.mark.parametrize("rope,lens", [(False, [3000]), (False, [9000] * 20), (True, [2500, 700])])
def test_queries_written_just_before(dev, before, rope, lens):  # noqa: F811
    """Calls in a row on one workspace, each behind what writes its queries (a copy, a kernel, another stream's
    kernel): every launch may be set up while the one before it runs, and must see all of it.  In the stream and as
    a replayed graph, where each kind of predecessor is another kind of edge."""
    import gen
    import torch
    from helpers import seeded_units, to_dev_u16
    p = akv.Params(batch=len(lens), n_kv_heads=4, n_q_heads=16, seed=9, anchor_frac=0.04, rope=rope, rope_theta=10000.0)
    units = seeded_units(p, lens, seed=3)
    arena = torch.from_numpy(akv.akv_cache_pack_host(p, lens, [akv.unit_host_from_logical(u) for u in units])).to(dev)
    shape = (p.batch, p.n_q_heads, 128)
    qs = [to_dev_u16(gen.queries(p.batch * p.n_q_heads, seed=s).reshape(shape), torch, dev) for s in (1, 2)]
    ws = torch.empty(akv.akv_decode_workspace_size(p, lens), dtype=torch.uint8, device=dev)
    q = torch.empty_like(qs[0])
    outs = [torch.empty(shape, dtype=torch.float32, device=dev) for _ in range(6)]
    out = torch.empty(shape, dtype=torch.bfloat16, device=dev)
    want = []
    for x in qs:
        o = torch.empty_like(outs[0])
        akv.akv_decode_attn(p, lens, arena, x, out, o, sm_scale=1.0, ws=ws)
        torch.cuda.synchronize()
        want.append(o)
    assert (want[0] - want[1]).abs().max() > 0.1
    main, other = torch.cuda.Stream(device=dev), torch.cuda.Stream(device=dev)

    def calls():
        for i, o in enumerate(outs):
            x = qs[i & 1]
            if before == "copy":
                q.copy_(x)
            elif before == "kernel":
                torch.mul(x, 1.0, out=q)
            elif before == "join":
                other.wait_stream(main)
                with torch.cuda.stream(other):
                    torch.mul(x, 1.0, out=q)
                main.wait_stream(other)
            akv.akv_decode_attn(p, lens, arena, x if before == "nothing" else q, out, o, sm_scale=1.0, ws=ws, stream=main)

    def check():
        torch.cuda.synchronize()
        for i, o in enumerate(outs):
            assert torch.allclose(o, want[i & 1], rtol=1e-4, atol=1e-4)
            o.zero_()
        torch.cuda.synchronize()

    with torch.cuda.stream(main):
        for _ in range(5):
            calls()
    check()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=main):
        calls()
    for _ in range(3):
        with torch.cuda.stream(main):
            g.replay()
        check()


@pytest.mark.parametrize("G", [1, 4, 8])
@pytest.mark.parametrize("fa,fr", [(0.01, 0.0), (0.02, 0.3), (0.04, 0.2), (0.08, 0.1), (0.15, 0.2), (0.27, 0.1)])
def test_plans_by_anchor_share(dev, G, fa, fr):  # noqa: F811
    """From rings of five mean tiles with the score table in shared memory to two tiles with the table in global
    memory, and tiles with more runs than the staged anchor-value rows; two units, so that ranges cross them."""
    p = akv.Params(batch=2, n_kv_heads=1, n_q_heads=G, anchor_frac=fa, res_frac_k=fr, res_frac_v=fr, seed=8)
    _run_seeded(dev, p, [41000, 20011], sm_scale=0.2)


@pytest.mark.parametrize("G", [2, 8])
@pytest.mark.parametrize("nv", [1, 15, 16, 17, 31, 33, 200])
def test_lloyd_max_record_groups(dev, G, nv):  # noqa: F811
    """Value records around the edges of their groups of 16, Lloyd-Max levels."""
    S = 1000
    p = akv.Params(batch=1, n_kv_heads=1, n_q_heads=G, res_frac_k=0.05, res_frac_v=(nv + 0.5) / S, seed=10, lloyd=True)
    assert akv.akv_unit_shapes(p, [S])[0][3] == nv

    def mutate(u, d):
        d["min_k"] = d["min_k"] * 0
        d["min_v"] = d["min_v"] * 0
    _run_seeded(dev, p, [S], mutate=mutate)


@pytest.mark.parametrize("G", [1, 4, 8])
@pytest.mark.parametrize("fa,fr", [(0.12, 0.1), (0.1, 0.4), (0.33, 0.1), (0.6, 0.3), (1.0, 0.0), (0.02, 0.35), (0.02, 0.5), (0.02, 0.95)])
@pytest.mark.parametrize("rope", [False, True])
def test_plans_at_large_shares(dev, G, fa, fr, rope):  # noqa: F811
    """Tiles that cover more value slots than have their anchor-value rows staged, up to one per token, and records up to
    one per token; lengths that end tiles early, a range that crosses units."""
    p = akv.Params(batch=2, n_kv_heads=2, n_q_heads=2 * G, anchor_frac=fa, res_frac_k=fr, res_frac_v=fr, seed=11, rope=rope,
                   rope_theta=10000.0)
    _run_seeded(dev, p, [9001, 3333], sm_scale=0.2)


@pytest.mark.parametrize("G", [1, 2])
@pytest.mark.parametrize("fa", [0.01, 0.04, 0.15])
@pytest.mark.parametrize("ctas", [1, 2, 5, 6])
def test_copies_in_turn(dev, debug_controls, G, fa, ctas):  # noqa: F811
    """Small query groups, no records and many tiles per CTA: the token warps copy in turn; ranges that cross units, rings of
    a dozen tiles and of two or three (whose first three do not fit at once), on both sides of the line (63 tiles, 12 per
    CTA)."""
    p = akv.Params(batch=3, n_kv_heads=1, n_q_heads=G, anchor_frac=fa, res_frac_k=0.0, res_frac_v=0.0, seed=14)
    akv.akv_decode_set_debug(ctas=ctas)
    _run_seeded(dev, p, [33333, 3000, 27000], sm_scale=0.2)


@pytest.mark.parametrize("lloyd", [False, True])
def test_copies_in_turn_with_records(dev, debug_controls, lloyd):  # noqa: F811
    """An arena of the full selection holds records that the parameters do not tell of."""
    import gen
    import oracle
    import torch
    from helpers import check_outputs, decode_on_gpu, oracle_decode, to_dev_u16
    lens, W = [14000], 32
    p = akv.Params(batch=1, n_kv_heads=1, n_q_heads=1, res_frac_k=0.0, res_frac_v=0.0, window=W, seed=16, lloyd=lloyd)
    sel = akv.SelectParams(theta=0.1)
    K, V = gen.clustered_batch(1, 1, lens, seed=17)
    Q = gen.observation_queries(K, lens, W, seed=18)
    a, w = akv.akv_cache_size_select(p, sel, lens)
    arena, ws = (torch.empty(n, dtype=torch.uint8, device=dev) for n in (a, w))
    akv.akv_encode_select(p, sel, lens, to_dev_u16(K, torch, dev), to_dev_u16(V, torch, dev), to_dev_u16(Q, torch, dev), arena, ws)
    units = oracle.unpack_arena(arena.cpu().numpy())
    assert units[0].nk > 1000 and units[0].nv > 1000
    q = gen.queries(1, seed=19)
    akv.akv_decode_set_debug(ctas=1)
    out, out32 = decode_on_gpu(torch, p, lens, arena, q, 0.2)
    check_outputs(out, out32, oracle_decode(p, units, q, 0.2), where="in turn with records")


def test_withheld_tile_with_copies_in_turn(dev, debug_controls):  # noqa: F811
    """The last tile of each range withheld: NaN outputs after the bounded wait, and the next call is right."""
    import numpy as np
    import torch
    from helpers import check_outputs, decode_on_gpu, oracle_decode, oracle_unit, seeded_units
    import gen
    p = akv.Params(batch=1, n_kv_heads=1, n_q_heads=1, res_frac_k=0.0, res_frac_v=0.0, seed=15)
    lens = [40000]
    units = seeded_units(p, lens, seed=5)
    arena = torch.from_numpy(akv.akv_cache_pack_host(p, lens, [akv.unit_host_from_logical(u) for u in units])).to(dev)
    q = gen.queries(1, seed=17)
    akv.akv_decode_set_debug(ctas=2, withhold_last=1)
    out, out32 = decode_on_gpu(torch, p, lens, arena, q, 1.0)
    assert np.all(np.isnan(out32)) and np.all(np.isnan(out))
    akv.akv_decode_set_debug(ctas=2)
    out, out32 = decode_on_gpu(torch, p, lens, arena, q, 1.0)
    check_outputs(out, out32, oracle_decode(p, [oracle_unit(u) for u in units], q, 1.0), where="after the timed-out call in turn")


@pytest.mark.parametrize("S", [60001, 70000])
@pytest.mark.parametrize("lloyd", [False, True])
@pytest.mark.parametrize("fa,fr", [(0.08, 0.2), (0.06, 0.3)])
def test_half_of_the_score_table_in_shared_memory(dev, S, lloyd, fa, fr):  # noqa: F811
    """Eight query heads, a score table that does not fit into shared memory and many records: heads 0-3 gather from shared,
    heads 4-7 from global memory; anchor counts that are and are not a multiple of four."""
    p = akv.Params(batch=1, n_kv_heads=2, n_q_heads=16, anchor_frac=fa, res_frac_k=fr, res_frac_v=fr, seed=13, lloyd=lloyd)

    def mutate(u, d):
        if lloyd:
            d["min_k"] = d["min_k"] * 0
            d["min_v"] = d["min_v"] * 0
    _run_seeded(dev, p, [S], mutate=mutate, sm_scale=0.2)


@pytest.mark.parametrize("G", [2, 8])
def test_time_at_large_shares(dev, G):  # noqa: F811
    """No cliff: a call with many anchors or many records takes a few times what one at 20 % anchors takes, as its bytes
    do (at most 2.3 times as many), not a hundred times (tiles off the tensor-core paths)."""
    import torch
    from helpers import seeded_units

    def us(fa, fr):
        p = akv.Params(batch=1, n_kv_heads=8, n_q_heads=8 * G, anchor_frac=fa, res_frac_k=fr, res_frac_v=fr, seed=12)
        lens = [20000]
        units = [akv.unit_host_from_logical(u) for u in seeded_units(p, lens)]
        arena = torch.from_numpy(akv.akv_cache_pack_host(p, lens, units)).to(dev)
        q = torch.randn((1, 8 * G, 128), device=dev).to(torch.bfloat16)
        out, ws = torch.empty_like(q), torch.empty(akv.akv_decode_workspace_size(p, lens), dtype=torch.uint8, device=dev)
        best = 1e9
        for _ in range(4):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            for _ in range(5):
                akv.akv_decode_attn(p, lens, arena, q, out, ws=ws)
            b.record()
            torch.cuda.synchronize()
            best = min(best, a.elapsed_time(b) / 5 * 1e3)
        return best

    base = us(0.2, 0.1)
    for fa, fr in ((0.12, 0.1), (0.25, 0.0), (0.3, 0.1), (0.5, 0.0), (0.02, 0.35), (0.02, 0.5)):
        assert us(fa, fr) < 8 * base, (fa, fr)
