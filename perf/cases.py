"""What a user of this library has it do, as cases that can be timed and compared.

Every case is one call (or the calls of one generation step) through the public entry points of
paper_2608_02901_gb300 on one layer's cache:

decode   akv_decode_attn on a cache that the program holds on the GPU, with its options: the query
         group size, the residual codec, pre-RoPE keys, the exact dense suffix of generated tokens
step     one generation step: akv_suffix_append of the new token, then akv_decode_attn with the suffix
encode   akv_encode of a prompt's dense keys and values
select   akv_encode_select, the same with the paper's full selection

Sizes: 1 to 16 requests of 200 to 131072 tokens, 1 to 8 KV heads (the heads one GPU holds), 1 to 8
query heads each, 1 to 4 % anchors, 0 to 20 % residuals, as in the benchmark's workloads and the tests.
"""
import math

import numpy as np
import torch

import paper_2608_02901_gb300 as akv

D = 128
WINDOW = 32
THETA = 500000.0  # RoPE base
LEVELS = (-1.5078125, -0.453125, 0.453125, 1.5078125)  # Lloyd-Max levels


def _case(name, kind, lens, H, G, fa=0.02, fr=0.10, lloyd=False, rope=False, suffix=0, encoded=False, f32=False):
    return dict(name=name, kind=kind, lens=",".join(str(s) for s in lens), H=H, G=G, fa=fa, fr=fr, lloyd=lloyd, rope=rope,
                suffix=suffix, encoded=encoded, f32=f32)


def listed():
    return [
        # a short chat prompt on one GPU: the smallest call, all launch and latency
        _case("decode-1k", "decode", [1021], 8, 4),
        # Llama-3.1-8B layer, one request at 32K, the cache as the encoder writes it
        _case("decode-8b-32k", "decode", [32768], 8, 4, encoded=True),
        # Llama-3.1-8B layer, a batch of ragged requests, fp32 results asked for as well
        _case("decode-8b-ragged", "decode", [131072, 8193, 50021, 23456, 100003, 12345], 8, 4, fr=0.20, f32=True),
        # Llama-3-70B layer, eight requests at 128K: the largest decode
        _case("decode-70b-128k", "decode", [131072] * 8, 8, 8),
        # plain multi-head and two-head groups, mid-size ragged requests, few residuals
        _case("decode-mha", "decode", [16001, 9000, 4173], 8, 1, fr=0.05),
        # a generation step at 32K with the tokens generated so far exact, Lloyd-Max codec
        _case("step-70b-32k", "step", [32768, 30011, 32000, 28673], 8, 8, lloyd=True, suffix=200),
        # pre-RoPE keys, RoPE applied at decode, one request at 32K, then a batch with a suffix
        _case("rope-8b-32k", "decode", [32768], 8, 4, rope=True),
        _case("rope-8b-batch", "decode", [40960, 20011, 65536, 9001], 8, 4, rope=True, lloyd=True, suffix=60),
        # prompts compressed after prefill: 32K on one GPU, a ragged batch of short ones, and 128K on the two KV
        # heads that one of four GPUs holds
        _case("encode-8b-32k", "encode", [32768], 8, 4),
        _case("encode-batch", "encode", [4173, 700, 8192, 2500, 6001, 333], 4, 4, fr=0.05, lloyd=True, rope=True),
        _case("encode-128k", "encode", [131072], 2, 8),
        # the paper's full selection on a 4K prompt
        _case("select-4k", "select", [4096], 8, 4),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["decode"] * 6 + ["step", "step", "encode", "encode", "select"])
    H, G = rng.choice([1, 2, 4, 8, 8, 8]), rng.choice([1, 2, 4, 4, 8, 8])
    fa, fr = rng.choice([0.01, 0.02, 0.02, 0.04]), rng.choice([0.0, 0.05, 0.10, 0.10, 0.20])
    rope = kind in ("decode", "encode") and rng.random() < 0.25
    # tokens of all units together: no more than the largest listed case of the kind takes
    room = {"decode": 1 << 20 if rope else 1 << 22, "step": 1 << 20, "encode": 1 << 18, "select": 1 << 15}[kind]
    most = {"decode": 131072, "step": 65536, "encode": 65536, "select": 4096}[kind]
    B = _log_int(rng, 1, 16)
    top = max(256, min(most, room // (H * B)))
    S = _log_int(rng, 256, top)
    lens = [S] * B if rng.random() < 0.4 else [rng.randint(max(200, S // 4), S) for _ in range(B)]
    suffix = rng.randint(1, 256) if kind == "step" or (kind == "decode" and rng.random() < 0.25) else 0
    c = _case("", kind, lens, H, G, fa=fa, fr=fr, lloyd=rng.random() < 0.3, rope=rope, suffix=suffix,
              encoded=kind == "decode" and sum(lens) * H <= 1 << 18 and rng.random() < 0.3)
    del c["name"]
    return c


# ---- inputs ------------------------------------------------------------------------------


def _lens(case):
    return [int(s) for s in case["lens"].split(",")]


def _params(case, seed):
    return akv.Params(batch=len(_lens(case)), n_kv_heads=case["H"], n_q_heads=case["H"] * case["G"], anchor_frac=case["fa"],
                      res_frac_k=case["fr"], res_frac_v=case["fr"], window=WINDOW, seed=seed, rot_seed=0x5EED,
                      lloyd=case["lloyd"], rope=case["rope"], rope_theta=THETA)


def _gen(seed, what):
    return torch.Generator(device="cuda").manual_seed((seed * 1000003 + what * 7919) & 0x7FFFFFFFFFFFFFFF)


def _rows(gen, *shape, scale=1.0):
    return (torch.randn(shape, generator=gen, device="cuda") * scale).to(torch.bfloat16)


def _clustered(gen, S):
    """One unit's keys and values: 64 clusters, four outlier channels among the keys (bf16 [S][128])."""
    ck, cv = torch.randn((2, 64, D), generator=gen, device="cuda")
    cid = torch.randint(0, 64, (S,), generator=gen, device="cuda")
    nk, nv = 1.0 + 0.2 * torch.randn((2, S, 1), generator=gen, device="cuda")
    k = nk * (ck[cid] + 0.3 * torch.randn((S, D), generator=gen, device="cuda"))
    v = nv * (cv[cid] + 0.3 * torch.randn((S, D), generator=gen, device="cuda"))
    k[:, torch.randperm(D, generator=gen, device="cuda")[:4]] *= 8
    return k.to(torch.bfloat16), v.to(torch.bfloat16)


def _dense(case, seed):
    """Keys and values of a whole layer, bf16 [B][H][longest][128], rows past a request's end zero."""
    lens, H, gen = _lens(case), case["H"], _gen(seed, 1)
    K = torch.zeros((len(lens), H, max(lens), D), dtype=torch.bfloat16, device="cuda")
    V = torch.zeros_like(K)
    for b, S in enumerate(lens):
        for h in range(H):
            K[b, h, :S], V[b, h, :S] = _clustered(gen, S)
    return K, V


def _shape(case, S):
    """Anchors and residual records of one unit (the formulas of akv_params)."""
    w = min(WINDOW, S)
    k = min(S, max(w, math.ceil(float(np.float32(case["fa"])) * S)))
    return w, k, min(int(float(np.float32(case["fr"])) * S), S - k)


def _logical(case, gen, S):
    """One unit's compressed cache drawn directly: dict of device arrays, by position."""
    w, k, n = _shape(case, S)
    u = {}
    at = torch.randperm(S - w, generator=gen, device="cuda")[:k - w]
    u["anchor_pos"] = torch.cat([at.sort().values, torch.arange(S - w, S, device="cuda")])
    u["anchor_k"], u["anchor_v"] = _clustered(gen, k)
    free = torch.ones(S, dtype=torch.bool, device="cuda")
    free[u["anchor_pos"]] = False
    free = free.nonzero()[:, 0]
    for side in "kv":
        idx = torch.randint(0, k, (S,), generator=gen, device="cuda")
        gam = (1.0 + 0.1 * torch.randn(S, generator=gen, device="cuda")).to(torch.float16)
        idx[u["anchor_pos"]] = torch.arange(k, device="cuda")
        gam[u["anchor_pos"]] = 1.0
        sc = (0.01 + 0.09 * torch.rand(n, generator=gen, device="cuda")).to(torch.float16)
        u["idx_" + side], u["gamma_" + side] = idx, gam
        u["res_pos_" + side] = free[torch.randperm(len(free), generator=gen, device="cuda")[:n]].sort().values
        u["codes_" + side] = torch.randint(0, 256, (n, 32), generator=gen, device="cuda", dtype=torch.uint8)
        u["scale_" + side] = sc
        u["min_" + side] = torch.zeros_like(sc) if case["lloyd"] else (-1.5 * sc.float()).to(torch.float16)
    return u


def _bits(t):
    if t.dtype in (torch.bfloat16, torch.float16):
        return t.view(torch.int16).cpu().numpy().view(np.uint16)
    return t.cpu().numpy()


def _inputs(case, seed):
    """Query rows [B][H_q][128], and the generated tokens: held rows [B][H][cap][128] per side, the lengths held, the new token's rows."""
    lens, H = _lens(case), case["H"]
    B, n, gen = len(lens), case["suffix"], _gen(seed, 2)
    x = {"q": _rows(gen, B, H * case["G"], D, scale=D ** -0.5)}
    if n:
        cap = (n + 1 + 63) // 64 * 64
        x["ks"], x["vs"] = _rows(gen, B, H, cap, D, scale=D ** -0.5), _rows(gen, B, H, cap, D)
        x["held"] = torch.tensor([max(0, n - 5 * b) for b in range(B)], dtype=torch.int32, device="cuda")
        x["k_new"], x["v_new"] = _rows(gen, B, H, D, scale=D ** -0.5), _rows(gen, B, H, D)
    return x


def prepare(case, seed):
    lens, p = _lens(case), _params(case, seed)
    st = {"case": case, "p": p, "lens": lens}
    if case["kind"] in ("encode", "select"):
        st["K"], st["V"] = _dense(case, seed)
        if case["kind"] == "select":
            # observation rows: the last positions' queries, each near one of the keys it attends to
            gen, m = _gen(seed, 3), WINDOW * case["G"]
            st["sel"] = akv.SelectParams(theta=0.05, rho=0.7, kappa=7)
            Q = torch.randn((len(lens), case["H"], m, D), generator=gen, device="cuda")
            for b, S in enumerate(lens):
                for h in range(case["H"]):
                    Q[b, h] += 0.25 * st["K"][b, h, torch.randint(0, S, (m,), generator=gen, device="cuda")].float()
            st["Q"] = Q.to(torch.bfloat16)
            a, w = akv.akv_cache_size_select(p, st["sel"], lens)
        else:
            a, w = akv.akv_cache_size(p, lens)
        st["arena"] = torch.empty(a, dtype=torch.uint8, device="cuda")
        st["ws"] = torch.empty(w, dtype=torch.uint8, device="cuda")
        return st
    if case["encoded"]:
        K, V = _dense(case, seed)
        a, w = akv.akv_cache_size(p, lens)
        st["arena"] = torch.empty(a, dtype=torch.uint8, device="cuda")
        akv.akv_encode(p, lens, K, V, st["arena"], torch.empty(w, dtype=torch.uint8, device="cuda"))
    else:
        gen = _gen(seed, 1)
        units = []
        for S in lens:
            for _ in range(case["H"]):
                units.append({n: _bits(t) for n, t in _logical(case, gen, S).items()})
        st["arena"] = torch.from_numpy(akv.akv_cache_pack_host(p, lens, units)).cuda()
    st.update(_inputs(case, seed))
    st["out"] = torch.empty_like(st["q"])
    st["out32"] = torch.empty(st["q"].shape, dtype=torch.float32, device="cuda") if case["f32"] else None
    st["suffix"] = None
    if case["suffix"]:
        st["len"] = st["held"].clone()
        st["suffix"] = akv.Suffix(st["ks"], st["vs"], st["len"])
    cap = st["suffix"].cap if st["suffix"] else 0
    st["ws"] = torch.empty(akv.akv_decode_workspace_size(p, lens, cap), dtype=torch.uint8, device="cuda")
    return st


def run(st):
    p, lens, kind = st["p"], st["lens"], st["case"]["kind"]
    if kind == "encode":
        akv.akv_encode(p, lens, st["K"], st["V"], st["arena"], st["ws"])
        return st["arena"]
    if kind == "select":
        akv.akv_encode_select(p, st["sel"], lens, st["K"], st["V"], st["Q"], st["arena"], st["ws"])
        return st["arena"]
    if kind == "step":
        st["len"].copy_(st["held"])  # the tokens accepted so far: a drafted one is rolled back before the next
        akv.akv_suffix_append(p, st["k_new"], st["v_new"], st["suffix"])
    akv.akv_decode_attn(p, lens, st["arena"], st["q"], st["out"], st["out32"], sm_scale=1.0, ws=st["ws"], suffix=st["suffix"])
    got = {"out": st["out"]}
    if st["out32"] is not None:
        got["out32"] = st["out32"]
    if kind == "step":
        got.update(len=st["len"], ks=st["ks"], vs=st["vs"])
    return got


# ---- what a pass cannot do without ---------------------------------------------------------


def work(case):
    lens, H, G, kind = _lens(case), case["H"], case["G"], case["kind"]
    total, flops = 0, 0
    for b, S in enumerate(lens):
        w, k, n = _shape(case, S)
        held = max(0, case["suffix"] - 5 * b) + (kind == "step") if case["suffix"] else 0
        # anchors, one index and coefficient word per token and side, residual flags, records
        cache = 512 * k + 8 * S + S // 4 + 72 * n + (4 * S if case["rope"] else 0)
        if kind in ("encode", "select"):
            total += H * (512 * S + cache)
            flops += H * 2 * 2 * D * S * k
            if kind == "select":
                total += H * 2 * D * WINDOW * G
                flops += H * 2 * 2 * D * S * WINDOW * G
        else:
            total += H * (cache + 512 * held + 4 * D * G + (4 * D * G if case["f32"] else 0))
            flops += H * 2 * G * (D * (2 * k + 2 * n + 2 * held + (S if case["rope"] else 0)) + 2 * S)
    return {"bytes": total, "flops": flops}


# ---- the same in 64 bits -------------------------------------------------------------------


def _wht():
    h = torch.ones((1, 1), dtype=torch.float64, device="cuda")
    while h.shape[0] < D:
        h = torch.cat([torch.cat([h, h], 1), torch.cat([h, -h], 1)], 0)
    return h


def _signs(rot_seed):
    mask, out = (1 << 64) - 1, []
    for half in range(2):
        z = (rot_seed + half + 0x9E3779B97F4A7C15) & mask
        z = ((z ^ (z >> 30)) * 0xBF58476D1CE4E5B9) & mask
        z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & mask
        z ^= z >> 31
        out += [-1.0 if (z >> j) & 1 else 1.0 for j in range(64)]
    return torch.tensor(out, dtype=torch.float64, device="cuda")


def _rebuilt(case, u, side, turn):
    """Every token's key or value row (Eq. 3), by position."""
    x = u["gamma_" + side].double()[:, None] * u["anchor_" + side].double()[u["idx_" + side]]
    codes = torch.stack([(u["codes_" + side] >> (2 * j)) & 3 for j in range(4)], dim=2).reshape(-1, D).long()
    c = torch.tensor(LEVELS, dtype=torch.float64, device="cuda")[codes] if case["lloyd"] else codes.double()
    c = u["min_" + side].double()[:, None] + u["scale_" + side].double()[:, None] * c
    x[u["res_pos_" + side]] += c @ turn
    return x


def _rope(x, pos):
    a = pos.double()[:, None] * THETA ** (-2.0 * torch.arange(64, dtype=torch.float64, device="cuda") / D)
    lo, hi = x[:, :64], x[:, 64:]
    return torch.cat([lo * a.cos() - hi * a.sin(), hi * a.cos() + lo * a.sin()], 1)


def exact(case, seed):
    if case["kind"] in ("encode", "select") or case["encoded"]:
        return None
    lens, H, G = _lens(case), case["H"], case["G"]
    gen, x = _gen(seed, 1), _inputs(case, seed)
    turn = _wht() * _signs(0x5EED)[None, :] / D
    length = None
    if case["suffix"]:
        length = x["held"].clone()
        if case["kind"] == "step":
            for b in range(len(lens)):
                x["ks"][b, :, int(length[b])] = x["k_new"][b]
                x["vs"][b, :, int(length[b])] = x["v_new"][b]
            length += 1
    out = torch.empty(x["q"].shape, dtype=torch.float64, device="cuda")
    for b, S in enumerate(lens):
        for h in range(H):
            u = _logical(case, gen, S)
            k, v = _rebuilt(case, u, "k", turn), _rebuilt(case, u, "v", turn)
            if length is not None:
                n = int(length[b])
                k = torch.cat([k, x["ks"][b, h, :n].double()])
                v = torch.cat([v, x["vs"][b, h, :n].double()])
            if case["rope"]:
                k = _rope(k, torch.arange(len(k), device="cuda"))
            q = x["q"][b, h * G:(h + 1) * G].double()
            out[b, h * G:(h + 1) * G] = torch.softmax(q @ k.T, dim=1) @ v
    got = {"out": out}
    if case["f32"]:
        got["out32"] = out
    if case["kind"] == "step":
        got.update(len=None, ks=x["ks"].double(), vs=x["vs"].double())
    return got
