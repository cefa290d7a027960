"""What the performance of this framework is measured on.

A user of the framework serves a WhiteMatter model: prompts go through the
causal channel attention (Jacobi passes and cyclic Gauss-Seidel groups) and the
cross-layer KV pool over groups of tokens; generation is one decode step per
token, L decode-attention calls and one pool call.  Every case calls those
entry points through ``DecodeSession`` as such a program does: the session
(cache, workspaces, weights) and the tensors of the call are in hand before it.

``listed`` holds the calls with the sizes of this repository's workloads and
tests, ``draw`` spreads the same calls over the ranges these stand for.
"""
from __future__ import annotations

import math
from types import SimpleNamespace

import numpy as np
import torch

from paper_2608_18486_gb300 import _lib as W
from paper_2608_18486_gb300.session import DecodeSession

DEV = "cuda:0"
THETA = 1e6
EPS = 1e-6
ROUTER_STRIDE = 2  # the router reads every second layer


# ------------------------------------------------------------------ the cases
def _attn(name, B, Hq, Hkv, d, ctx, ctx_lo=0, page=16, dtype="bf16"):
    return dict(name=name, kind="attn", B=B, Hq=Hq, Hkv=Hkv, d=d, ctx=ctx, ctx_lo=ctx_lo, page=page,
                dtype=dtype)


def _prefill(name, B, T, g, q, Hq, Hkv, d, page=16):
    return dict(name=name, kind="prefill", B=B, T=T, g=g, q=q, Hq=Hq, Hkv=Hkv, d=d, page=page,
                dtype="bf16")


def _pool(name, L, k, D, Hkv, d, B, ctx, ctx_lo=0, g=0, q=0, page=16, dtype="bf16"):
    return dict(name=name, kind="pool", L=L, k=k, D=D, Hq=Hkv, Hkv=Hkv, d=d, B=B, ctx=ctx,
                ctx_lo=ctx_lo, g=g, q=q, page=page, dtype=dtype)


def _step(name, L, k, D, Hq, Hkv, d, B, ctx, ctx_lo=0, page=16, dtype="bf16", graph=True):
    return dict(name=name, kind="step", L=L, k=k, D=D, Hq=Hq, Hkv=Hkv, d=d, B=B, ctx=ctx,
                ctx_lo=ctx_lo, page=page, dtype=dtype, graph=graph)


def listed():
    return [
        # The smallest calls: a whole fp32 decode step of a toy model, called
        # eagerly (a debugging or accuracy run): nine launches of a few
        # microseconds each.
        _step("step_tiny_f32", L=4, k=2, D=256, Hq=4, Hkv=4, d=64, B=2, ctx=128, dtype="f32",
              graph=False),
        # Generation with the paper's own model (6/3 heads of 96, 16 layers and
        # channels): one whole decode step for 16 sequences, replayed from a
        # CUDA graph as a server does.
        _step("step_paper_k16", L=16, k=16, D=512, Hq=6, Hkv=3, d=96, B=16, ctx=2048),
        # One layer's decode attention at an ordinary size: 12 heads of 64.
        _attn("attn_mha64", B=16, Hq=12, Hkv=12, d=64, ctx=2048),
        # Grouped-query decode, few ragged sequences, eight query heads per kv head.
        _attn("attn_gqa8_64", B=8, Hq=64, Hkv=8, d=64, ctx=4096, ctx_lo=2),
        # Grouped-query decode of a wide model over a full batch of long prompts.
        _attn("attn_gqa4_128", B=32, Hq=32, Hkv=8, d=128, ctx=8192, ctx_lo=4096),
        # Multi-head decode of a wide model, ragged batch.
        _attn("attn_large", B=32, Hq=32, Hkv=32, d=128, ctx=8192, ctx_lo=4096),
        # Long-context decode, the largest launch: 17 GB of cache per layer.
        _attn("attn_long128k", B=8, Hq=32, Hkv=32, d=128, ctx=131072, page=64),
        # Prompt processing of the paper's model: a Jacobi pass over 16 prompts,
        # and one Gauss-Seidel group (every eighth position) of the same prompts.
        _prefill("prefill_paper", B=16, T=2048, g=1, q=0, Hq=6, Hkv=3, d=96),
        _prefill("prefill_paper_g8", B=16, T=2048, g=8, q=3, Hq=6, Hkv=3, d=96),
        # Prompt processing of a wide model: a Jacobi pass over two long prompts.
        _prefill("prefill_large", B=2, T=8192, g=1, q=0, Hq=32, Hkv=32, d=128),
        # The pool of a decode step of a wide model (weight streaming), and of
        # one Gauss-Seidel group of prompt tokens of the paper's model.
        _pool("pool_large", L=32, k=16, D=4096, Hkv=32, d=128, B=32, ctx=64, ctx_lo=32),
        _pool("pool_group", L=16, k=16, D=512, Hkv=3, d=96, B=16, ctx=2048, g=8, q=3),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


# A drawn case takes no longer than the largest listed ones: at most these
# bytes (times half the query heads per kv head) and these operations.
_MAX_BYTES = 1.7e10
_MAX_FLOPS = {"attn": 1e12, "prefill": 4e11, "pool": 2e11, "step": 2e11}


def draw(rng):
    while True:
        c = _draw(rng)
        w = work(c)
        scale = max(1.0, c["Hq"] / c["Hkv"] / 2)
        flops = _MAX_FLOPS[c["kind"]] / (8 if c["dtype"] == "f32" else 1)
        if w["bytes"] * scale <= _MAX_BYTES and w["flops"] <= flops:
            return c


def _draw(rng):
    kind = rng.choice(["attn", "attn", "prefill", "pool", "pool", "step"])
    d = rng.choice([64, 96, 128])
    page = rng.choice([16, 16, 32, 64, 128])
    if kind == "attn":
        G = rng.choice([1, 1, 2, 4, 8])
        Hkv = rng.choice([2, 3, 4, 8, 12, 16, 32])
        ctx = _log_int(rng, 100, 131072)
        c = _attn("", B=_log_int(rng, 1, 64), Hq=Hkv * G, Hkv=Hkv, d=d, ctx=ctx,
                  ctx_lo=rng.choice([0, max(1, ctx // 2), max(1, ctx // 4)]), page=page,
                  dtype=rng.choice(["bf16", "bf16", "bf16", "f32"]))
    elif kind == "prefill":
        G = rng.choice([1, 2, 4])
        Hkv = rng.choice([2, 3, 8, 16, 32])
        g = rng.choice([1, 1, 2, 4, 8, 16])
        c = _prefill("", B=_log_int(rng, 1, 16), T=_log_int(rng, 200, 8192), g=g, q=rng.randrange(g),
                     Hq=Hkv * G, Hkv=Hkv, d=d, page=page)
    elif kind == "pool":
        L = rng.randint(6, 32)
        k = rng.randint(1, min(L, 16))
        D = rng.choice([512, 768, 1024, 2048, 4096])
        Hkv = rng.choice([2, 3, 4, 8]) if D < 2048 else rng.choice([8, 16, 32])
        if rng.random() < 0.5:  # one decode step
            c = _pool("", L=L, k=k, D=D, Hkv=Hkv, d=d, B=_log_int(rng, 1, 64), ctx=64, ctx_lo=1,
                      page=page, dtype=rng.choice(["bf16", "bf16", "bf16", "f32"]))
        else:  # a group of prompt tokens
            g = rng.choice([1, 2, 4, 8])
            c = _pool("", L=L, k=k, D=min(D, 1024), Hkv=min(Hkv, 8), d=d, B=_log_int(rng, 1, 16),
                      ctx=_log_int(rng, 100, 2048), g=g, q=rng.randrange(g), page=page)
    else:
        L = rng.randint(4, 16)
        k = rng.randint(1, L)
        G = rng.choice([1, 2, 4])
        Hkv = rng.choice([2, 3, 4, 8, 12])
        ctx = _log_int(rng, 100, 4096)
        c = _step("", L=L, k=k, D=rng.choice([256, 512, 768, 1024]), Hq=Hkv * G, Hkv=Hkv, d=d,
                  B=_log_int(rng, 1, 32), ctx=ctx, ctx_lo=rng.choice([0, max(1, ctx // 2)]), page=page,
                  dtype=rng.choice(["bf16", "bf16", "bf16", "f32"]), graph=rng.choice([True, True, False]))
    del c["name"]
    return c


# ------------------------------------------------------------------ the work
def _esz(c):
    return 4 if c["dtype"] == "f32" else 2


def _lens(c, seed):
    """Cache slots of every sequence, the dummy included."""
    B = c["B"]
    if c["kind"] == "prefill" or c.get("g", 0) > 0:
        T = c.get("T", c.get("ctx"))
        return np.full(B, T, np.int64)
    if c["ctx_lo"] <= 0:
        return np.full(B, c["ctx"], np.int64)
    return np.random.RandomState(seed & 0x7FFFFFFF).randint(c["ctx_lo"], c["ctx"] + 1, B).astype(np.int64)


def _mean_slots(c):
    return c["ctx"] if c["ctx_lo"] <= 0 else (c["ctx"] + c["ctx_lo"]) / 2


def _attn_work(c):
    slots = c["B"] * _mean_slots(c)
    return {"bytes": (slots * c["Hkv"] * 2 + 2 * c["B"] * c["Hq"]) * c["d"] * _esz(c),
            "flops": slots * c["Hq"] * 4 * c["d"]}


def _tokens(c):
    return c["B"] * len(range(c["q"], c["ctx"], c["g"])) if c.get("g", 0) > 0 else c["B"]


def _pool_work(c, n):
    L, k, D, e = c["L"], c["k"], c["D"], _esz(c)
    Lp = -(-L // ROUTER_STRIDE)
    nout = c["Hkv"] * c["d"]
    weights = 2 * (k * L * Lp * D + k * L + k * nout * D + D + k * D) + k * c["d"]
    return {"bytes": (weights + n * L * D + 2 * n * k * nout) * e,
            "flops": 2.0 * n * 2 * (k * L * Lp * D + k * L * D + k * nout * D)}


def work(c):
    if c["kind"] == "attn":
        return _attn_work(c)
    if c["kind"] == "prefill":
        rows = range(c["q"], c["T"], c["g"])
        pairs = c["B"] * sum(i + 1 for i in rows)
        return {"bytes": c["B"] * c["d"] * 2.0 * (2 * len(rows) * c["Hq"] + 2 * c["T"] * c["Hkv"]),
                "flops": pairs * c["Hq"] * 4.0 * c["d"]}
    if c["kind"] == "pool":
        return _pool_work(c, _tokens(c))
    a, p = _attn_work(c), _pool_work(c, c["B"])
    # every layer reads its channel once; a channel several layers share counts once
    qo = 2 * c["B"] * c["Hq"] * c["d"] * _esz(c)
    return {"bytes": c["k"] * (a["bytes"] - qo) + c["L"] * qo + p["bytes"],
            "flops": c["L"] * a["flops"] + p["flops"]}


# ------------------------------------------------------------------ the inputs
def _tdt(c):
    return torch.float32 if c["dtype"] == "f32" else torch.bfloat16


def _shape(c):
    """Layers, channels and width (one of each where the call reads one layer)."""
    return c.get("L", 1), c.get("k", 1), c.get("D", 512)


def _pages(c, seed):
    """Page table and page count.  Slots 0..S of a sequence have pages (slot S
    receives a step's new token); the pages that receive new tokens are
    physical pages 0..B-1, all others a random permutation of the rest."""
    lens = _lens(c, seed)
    npg = lens // c["page"] + 1
    B, total = len(lens), int(npg.sum())
    perm = np.random.RandomState((seed + 7) & 0x7FFFFFFF).permutation(total - B) + B
    pt = np.full((B, int(npg.max())), -1, np.int32)
    o = 0
    for b in range(B):
        n = int(npg[b]) - 1
        pt[b, :n] = perm[o:o + n]
        pt[b, n] = b
        o += n
    return lens, pt, total


def _fill(gen, shape, dtype, std=1.0, mean=0.0):
    return torch.empty(shape, dtype=dtype, device=DEV).normal_(mean, std, generator=gen)


def _inputs(c, seed):
    """Every input of the case but the cache, which `_fill_cache` draws."""
    gen = torch.Generator(device=DEV).manual_seed(int(seed) * 2 + 1)
    L, k, D = _shape(c)
    dt, B, Hq, Hkv, d = _tdt(c), c["B"], c["Hq"], c["Hkv"], c["d"]
    lens, pt, total = _pages(c, seed)
    s = SimpleNamespace(lens=lens, pt=pt, num_pages=total, max_pages=pt.shape[1],
                        chan=[l % k for l in range(L)])
    s.page_table = torch.from_numpy(pt).to(DEV)
    if c["kind"] == "attn":
        s.q = _fill(gen, (1, B, Hq, d), dt)
    elif c["kind"] == "step":
        s.q = _fill(gen, (L, B, Hq, d), dt)
    elif c["kind"] == "prefill":
        pos = np.tile(np.arange(c["q"], c["T"], c["g"], dtype=np.int32), (B, 1))
        s.pos = torch.from_numpy(pos).to(DEV)
        s.q = _fill(gen, (B, pos.shape[1], Hq, d), dt)
    if c["kind"] in ("pool", "step"):
        if c.get("g", 0) > 0:  # the tokens of a group: sequence and position of each
            rows = np.arange(c["q"], c["ctx"], c["g"])
            s.tok_seq, tok_pos = np.repeat(np.arange(B), len(rows)), np.tile(rows, B)
            s.tok_slot = tok_pos + 1
        else:  # the next token of every sequence
            s.tok_seq, s.tok_slot = np.arange(B), lens
        n = len(s.tok_seq)
        s.tok_pages = torch.from_numpy(np.ascontiguousarray(pt[s.tok_seq])).to(DEV)
        s.slot = torch.from_numpy(s.tok_slot.astype(np.int32)).to(DEV)
        Lp = -(-L // ROUTER_STRIDE)
        # hidden states grow with depth; gains are near one, as trained
        h = _fill(gen, (n, L, D), torch.float32)
        s.h = (h * (1 + 0.1 * torch.arange(L, device=DEV))[None, :, None]).to(dt)
        del h
        bias = torch.zeros(k, L)
        for l in range(L):
            bias[s.chan[l], l] = 1.0
        s.weights = ([_fill(gen, (D,), dt, 0.1, 1.0) for _ in range(2)],
                     [_fill(gen, (k * L, Lp * D), dt, (Lp * D) ** -0.5) for _ in range(2)],
                     [bias.reshape(-1).to(dt).to(DEV) for _ in range(2)],
                     [_fill(gen, (k, D), dt, 0.1, 1.0) for _ in range(2)],
                     [_fill(gen, (k, Hkv * d, D), dt, D ** -0.5) for _ in range(2)],
                     _fill(gen, (k, d), dt, 0.1, 1.0))
    return s


def _fill_cache(c, seed, k_pool, v_pool):
    gen = torch.Generator(device=DEV).manual_seed(int(seed) * 2 + 2)
    k_pool.normal_(generator=gen)
    v_pool.normal_(generator=gen)


def prepare(c, seed):
    L, k, D = _shape(c)
    s = _inputs(c, seed)
    cfg = W.make_config(L, k, D, c["Hq"], c["Hkv"], c["d"], ROUTER_STRIDE, c["page"], c["dtype"], s.chan,
                        EPS, EPS, THETA)
    s.case = c
    s.B = len(s.tok_seq) if c["kind"] == "pool" else c["B"]
    s.sess = DecodeSession(cfg, s.B, s.num_pages, s.max_pages, DEV)
    _fill_cache(c, seed, s.sess.k_pool, s.sess.v_pool)
    if c["kind"] in ("pool", "step"):
        s.sess.set_weights(*s.weights)
        # the pages the pool writes to: every page for a group of prompt
        # tokens, else the pages that hold each sequence's next slot
        pages = s.num_pages if c.get("g", 0) > 0 else c["B"]
        s.new = [s.sess.k_pool[:, :pages], s.sess.v_pool[:, :pages]]
    if c["kind"] in ("attn", "step"):
        s.seq_lens = torch.from_numpy(s.lens.astype(np.int32)).to(DEV)
    if c["kind"] != "pool":
        s.out = torch.empty_like(s.q)
    if c["kind"] == "step" and c["graph"]:
        stream = torch.cuda.Stream()
        stream.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(stream):
            _step_calls(s)
        stream.synchronize()
        s.graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(s.graph, stream=stream):
            _step_calls(s)
    return s


def _step_calls(s):
    """One decode step: every layer's attention, then the pool."""
    for layer in range(s.case["L"]):
        s.sess.decode_attn(layer, s.q[layer], s.page_table, s.seq_lens, s.out[layer],
                           inputs_ready=layer > 0)
    s.sess.kv_mix(s.h, s.page_table, s.slot)


def run(s):
    kind = s.case["kind"]
    if kind == "attn":
        s.sess.decode_attn(0, s.q[0], s.page_table, s.seq_lens, s.out[0])
        return s.out[0]
    if kind == "prefill":
        s.sess.prefill_attn(0, s.q, s.pos, s.page_table, s.out)
        return s.out
    if kind == "pool":
        s.sess.kv_mix(s.h, s.tok_pages, s.slot)
        return s.new
    if s.case["graph"]:
        s.graph.replay()
    else:
        _step_calls(s)
    return [s.out] + s.new


# ------------------------------------------------------------------ the exact results
def _rows(pool_c, pt, n, page):
    """Slots 0..n-1 of one sequence, [Hkv][n][d] in 64 bits; pool_c [pages][Hkv][P][d]."""
    pg = torch.from_numpy(pt[:(n + page - 1) // page].astype(np.int64)).to(pool_c.device)
    x = pool_c[pg].permute(1, 0, 2, 3)
    return x.reshape(x.shape[0], -1, x.shape[3])[:, :n]


def _attn_exact(c, s, q, kc, vc):
    out = torch.empty(q.shape, dtype=torch.float64, device=DEV)
    Hkv, d = c["Hkv"], c["d"]
    G = c["Hq"] // Hkv
    for b in range(c["B"]):
        n = int(s.lens[b])
        K, V = _rows(kc, s.pt[b], n, c["page"]), _rows(vc, s.pt[b], n, c["page"])
        for h in range(Hkv):
            p = (q[b, h * G:(h + 1) * G].double() @ K[h].double().T) / math.sqrt(d)
            out[b, h * G:(h + 1) * G] = torch.softmax(p, -1) @ V[h].double()
    return out


def _prefill_exact(c, s, kc, vc):
    q, Hkv, d = s.q, c["Hkv"], c["d"]
    G, n = c["Hq"] // Hkv, c["T"]
    out = torch.empty(q.shape, dtype=torch.float64, device=DEV)
    hidden = torch.arange(n, device=DEV)[None, :] > s.pos[0].long()[:, None]
    for b in range(c["B"]):
        K, V = _rows(kc, s.pt[b], n, c["page"]), _rows(vc, s.pt[b], n, c["page"])
        for h in range(c["Hq"]):
            p = (q[b, :, h].double() @ K[h // G].double().T) / math.sqrt(d)
            p.masked_fill_(hidden, -math.inf)
            out[b, :, h] = torch.softmax(p, -1) @ V[h // G].double()
            del p
    return out


def _rms(x):
    return x / torch.sqrt((x * x).mean(-1, keepdim=True) + EPS)


def _pool_exact(c, s, kp, vp):
    """The pools (k first, v second, 64 bits) with the new tokens written."""
    L, k, D = _shape(c)
    Hkv, d, P = c["Hkv"], c["d"], c["page"]
    pre_g, Wr, br, ch_g, Wkv, qk_g = s.weights
    n = len(s.tok_seq)
    slot = torch.from_numpy(s.tok_slot.astype(np.int64)).to(DEV)
    page = torch.from_numpy(s.pt[s.tok_seq, s.tok_slot // P].astype(np.int64)).to(DEV)
    half = d // 2
    freq = THETA ** (-2.0 * torch.arange(half, dtype=torch.float64, device=DEV) / d)
    for X, pool in enumerate((kp, vp)):
        for t0 in range(0, n, 1024):
            t = slice(t0, min(n, t0 + 1024))
            hh = _rms(s.h[t].double()) * pre_g[X].double()
            xi = torch.cat([hh[:, l] for l in range(L - 1, -1, -ROUTER_STRIDE)], -1)
            z = torch.cat([xi @ Wr[X][r:r + 256].double().T for r in range(0, k * L, 256)], -1)
            alpha = (z + br[X].double()).view(-1, k, L)
            for j in range(k):
                x = _rms(torch.einsum("nl,nld->nd", alpha[:, j], hh)) * ch_g[X][j].double()
                y = (x @ Wkv[X][j].double().T).view(-1, Hkv, d)
                if X == 0:
                    y = _rms(y) * qk_g[j].double()
                    ang = (slot[t] - 1).double()[:, None, None] * freq
                    cs, sn = torch.cos(ang), torch.sin(ang)
                    y0, y1 = y[..., :half], y[..., half:]
                    y = torch.cat([y0 * cs - y1 * sn, y1 * cs + y0 * sn], -1)
                pool[j, page[t], :, slot[t] % P] = y
    return kp, vp


def exact(c, seed):
    L, k, _ = _shape(c)
    s = _inputs(c, seed)
    shape = (k, s.num_pages, c["Hkv"], c["page"], c["d"])
    kp, vp = (torch.empty(shape, dtype=_tdt(c), device=DEV) for _ in range(2))
    _fill_cache(c, seed, kp, vp)
    if c["kind"] == "attn":
        return _attn_exact(c, s, s.q[0], kp[0], vp[0])
    if c["kind"] == "prefill":
        return _prefill_exact(c, s, kp[0], vp[0])
    pages = s.num_pages if c.get("g", 0) > 0 else c["B"]
    new = list(_pool_exact(c, s, kp[:, :pages].double(), vp[:, :pages].double()))
    if c["kind"] == "pool":
        return new
    return [torch.stack([_attn_exact(c, s, s.q[l], kp[s.chan[l]], vp[s.chan[l]]) for l in range(L)])] + new
