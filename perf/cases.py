"""The work that performance is measured on: calls that programs make through the public binding.

Kinds of case (``kind``):

- ``prefill``: steps (a)-(d) of one attention layer. ``calls`` is ``whole`` (one call per step over
  the sequence, ``run_path``) or ``loop`` (chunked prefill in the order of Algorithm 2: per outer
  chunk step (a), then one selection and one attention call per unit);
- ``build``: step (a) alone over a sequence, with a real clustering threshold;
- ``select``: steps (b)-(c) alone over the last ``span`` tokens (block level, or token level when
  the block size is 1), scores returned;
- ``attend``: step (d) alone over the last ``span`` tokens on a given selection, with K and V
  contiguous or in a paged cache (``page`` > 0);
- ``decode``: ``steps`` consecutive decode steps at the end of a sequence, the first of which
  retrieves while the others reuse its selection.

``hq`` / ``hkv`` query and KV heads (head size 128, bf16), ``n`` tokens, ``sub`` / ``cap`` /
``outer`` the sub-chunk length, the cluster cap in sub-chunks and the outer chunk, ``block`` /
``topk`` / ``sink`` / ``local`` the selection's block size, picks, sinks and window, ``mode``
``cluster`` (one selection per cluster) or ``subchunk`` (one per sub-chunk).

Left out: ``scale_prefill_host`` runs the same kernels behind host-link copies, whose speed
varies with the machine's other users.
"""

from __future__ import annotations

import math

import torch

import paper_2609_31568_gb300 as pkg
from paper_2609_31568_gb300 import scale as S

DH = 128
ROPE_BASE = 500000.0


def listed():
    llama = dict(hq=32, hkv=8, theta=-1.0, page=0)
    return [
        # The smallest layer: a 4K prompt on 4 query heads, all units in one call per step.
        dict(name="prefill-4k", kind="prefill", calls="whole", mode="cluster", hq=4, hkv=1, n=4096, sub=256, cap=4,
             outer=1024, block=64, topk=8, sink=64, local=256, theta=-1.0, page=0),
        # A 32K prompt on a Llama-3-8B layer, chunk by chunk.
        dict(name="prefill-32k-loop", kind="prefill", calls="loop", mode="cluster", n=32768, sub=1024, cap=8,
             outer=8192, block=128, topk=32, sink=128, local=1024, **llama),
        # The same layer with a selection per sub-chunk (many small calls), a prompt of odd length.
        dict(name="prefill-32k-loop-subchunk", kind="prefill", calls="loop", mode="subchunk", n=32309, sub=1024,
             cap=8, outer=8192, block=128, topk=32, sink=128, local=1024, **llama),
        # The benchmark's layer: 128K tokens, one cluster per outer chunk.
        dict(name="prefill-128k-loop", kind="prefill", calls="loop", mode="cluster", n=131072, sub=2048, cap=8,
             outer=16384, block=128, topk=64, sink=128, local=1024, **llama),
        # Token-level selection (the paper's granularity and budget) over a 64K prompt of odd length.
        dict(name="prefill-64k-loop-tokens", kind="prefill", calls="loop", mode="cluster", n=64123, sub=2048, cap=8,
             outer=16384, block=1, topk=8192, sink=128, local=1024, **llama),
        # Step (a) with a threshold that closes clusters at topic changes (the paper's sub-chunk of 512).
        dict(name="build-128k-topics", kind="build", mode="cluster", hq=32, hkv=8, n=131072, sub=512, cap=8,
             outer=8192, block=128, topk=64, sink=128, local=512, theta=0.95, page=0),
        # One cluster's selection late in a 128K prompt: latency.
        dict(name="select-128k", kind="select", mode="cluster", n=131072, span=16384, sub=2048, cap=8, outer=16384,
             block=128, topk=64, sink=128, local=1024, **llama),
        # Every sub-chunk's selection of a 1M-token layer in one call: the largest block-level selection.
        dict(name="select-1m-batch", kind="select", mode="subchunk", n=1048576, span=1048576, sub=4096, cap=16,
             outer=65536, block=256, topk=128, sink=128, local=1024, **llama),
        # One cluster's token-level selection at the end of a 1M-token layer.
        dict(name="select-1m-tokens", kind="select", mode="cluster", n=1048576, span=65536, sub=4096, cap=16,
             outer=65536, block=1, topk=8192, sink=128, local=1024, **llama),
        # Attention of a Qwen2-7B layer (28 query heads on 4 KV heads) over a paged cache: one outer
        # chunk of 8192 tokens with a selection per sub-chunk of 512.
        dict(name="attend-64k-paged", kind="attend", mode="subchunk", hq=28, hkv=4, n=65472, span=8128, sub=512,
             cap=8, outer=8192, block=128, topk=64, sink=128, local=512, theta=-1.0, page=64),
        # A decode step that retrieves, at 1M tokens.
        dict(name="decode-1m", kind="decode", mode="cluster", n=1048576, steps=1, sub=512, cap=1, outer=512, block=1,
             topk=8192, sink=128, local=512, hq=32, hkv=8, theta=0.95, page=0),
        # Sixteen decode steps at 128K tokens sharing one retrieval.
        dict(name="decode-128k-cached", kind="decode", mode="cluster", n=131072, steps=16, sub=512, cap=16,
             outer=8192, block=1, topk=8192, sink=128, local=512, hq=32, hkv=8, theta=0.95, page=0),
    ]


def draw(rng):
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["prefill", "prefill", "prefill", "build", "select", "select", "attend", "decode"])
    hq, hkv = rng.choice([(32, 8), (32, 8), (28, 4), (16, 8), (8, 1), (6, 2), (4, 4)])
    c = dict(kind=kind, mode=rng.choice(["cluster", "subchunk"]), hq=hq, hkv=hkv, theta=-1.0, page=0)
    if kind == "decode":
        steps = rng.choice([1, 1, 4, 16])
        c.update(mode="cluster", n=size(3000, 900000), steps=steps, sub=512, cap=steps, outer=512 * steps, block=1,
                 topk=rng.choice([64, 1024, 2048, 8192]), sink=rng.choice([0, 64, 128]),
                 local=rng.choice([256, 512, 1000]), theta=0.95)
        return c
    sub = rng.choice([256, 512, 1024, 2048])
    cap = rng.choice([4, 8])
    c.update(sub=sub, cap=cap, outer=sub * cap, local=rng.choice([256, 512, 1024]), sink=rng.choice([0, 64, 128]))
    tokens = kind != "build" and rng.random() < 0.3
    if tokens and kind == "select":  # the workspace packs topk keys for every sub-chunk
        sub = max(sub, 1024)
        c.update(sub=sub, outer=sub * cap)
    if tokens:
        c.update(block=1, topk=rng.choice([512, 2048, 8192]))
    else:
        block = rng.choice([64, 128, 256])
        c.update(block=block, topk=rng.choice([8, 32, 64]))
    if kind == "prefill":
        c.update(calls=rng.choice(["whole", "loop"]), n=size(2000, 70000))
    elif kind == "build":
        c.update(n=size(2000, 160000), theta=rng.choice([-1.0, 0.95]))
    elif kind == "select":
        c.update(n=size(4000, 500000), span=0)
    else:
        c.update(n=size(4000, 120000), span=0, page=rng.choice([0, 64, 256]))
    if "span" in c:  # from a multiple of the outer chunk to the end
        outer = c["outer"]
        chunks = -(-c["n"] // outer)
        c["span"] = c["n"] - outer * (chunks - (1 if kind == "attend" else rng.randint(1, min(chunks, 4))))
    return c


# ---------------------------------------------------------------- inputs


def _centroids(gen, hkv, count):
    x = torch.randn(hkv, count, DH, generator=gen, device="cuda")
    return 3.0 * x / x.norm(dim=-1, keepdim=True)


def _rope(x, t0):
    half = DH // 2
    inv = ROPE_BASE ** (-torch.arange(half, dtype=torch.float64, device="cuda") * 2.0 / DH)
    ang = torch.arange(t0, t0 + x.shape[0], dtype=torch.float64, device="cuda")[:, None] * inv
    cos, sin = ang.cos().float()[:, None], ang.sin().float()[:, None]
    lo, hi = x[..., :half], x[..., half:]
    return torch.cat([lo * cos - hi * sin, hi * cos + lo * sin], dim=-1)


def _mixture(gen, out, cents, t0, shift=None):
    """Fill out [T, H, 128] (bf16, tokens from t0): a component of the head's KV head plus N(0, 1), then
    rotary positions; `shift(a, b)` adds a direction to the tokens [a, b)."""
    heads, hkv = out.shape[1], cents.shape[0]
    kvh = torch.arange(heads, device="cuda") // (heads // hkv)
    for a in range(0, out.shape[0], 8192):
        b = min(out.shape[0], a + 8192)
        ids = torch.randint(0, cents.shape[1], (b - a, heads), generator=gen, device="cuda")
        x = cents[kvh, ids]
        x += torch.randn(x.shape, generator=gen, device="cuda")
        if shift is not None:
            x += shift(a, b)
        out[a:b] = _rope(x, t0 + a)
    return out


def _empty(*shape):
    return torch.empty(shape, dtype=torch.bfloat16, device="cuda")


def _kv(gen, c, cents):
    k = _mixture(gen, _empty(c["n"], c["hkv"], DH), cents, 0)
    v = torch.randn(c["n"], c["hkv"], DH, generator=gen, device="cuda", dtype=torch.bfloat16)
    return k, v


def _topic_shift(gen, c):
    """A shared direction of norm 6 per query head and one of norm 3 for the segment's topic, in the lowest
    rotary frequencies, as the queries of trained models have; segments of about 16K tokens."""
    band = torch.cat([torch.arange(48, 64), torch.arange(112, 128)]).cuda()
    shared = torch.zeros(c["hq"], DH, device="cuda")
    topic = torch.zeros(16, DH, device="cuda")
    shared[:, band] = torch.randn(c["hq"], band.numel(), generator=gen, device="cuda")
    topic[:, band] = torch.randn(16, band.numel(), generator=gen, device="cuda")
    shared *= 6.0 / shared.norm(dim=-1, keepdim=True)
    topic *= 3.0 / topic.norm(dim=-1, keepdim=True)
    jump = torch.rand(c["n"], generator=gen, device="cuda") < 1.0 / 16384
    of = (jump.long().cumsum(0) * 7 + 1) % 16
    return lambda a, b: shared[None] + topic[of[a:b]][:, None]


def _units(c):
    """(first token, end) of every unit when the threshold admits every sub-chunk."""
    step = c["sub"] * (c["cap"] if c["mode"] == "cluster" else 1)
    out = []
    for o in range(0, c["n"], c["outer"]):
        end = min(c["n"], o + c["outer"])
        out += [(s, min(end, s + step)) for s in range(o, end, step)]
    return out


def _candidates(c, s):
    """The first and one past the last candidate block of a unit that starts at token s."""
    w = max(0, s - c["local"])
    lo = c["sink"] // c["block"]
    return lo, max(lo, -(-w // c["block"]))


def _inputs(c, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    cents = _centroids(gen, c["hkv"], 256)
    x = {}
    if c["kind"] in ("prefill", "build"):
        shift = _topic_shift(gen, c) if c["kind"] == "build" else None
        x["q"] = _mixture(gen, _empty(c["n"], c["hq"], DH), cents, 0, shift)
        x["k"], x["v"] = _kv(gen, c, cents)
    elif c["kind"] == "select":
        k = _mixture(gen, _empty(c["n"], c["hkv"], DH), cents, 0)
        m = -(-c["n"] // c["sub"])
        x["fp"] = torch.zeros(m, c["hq"] * DH, device="cuda")
        for s, _ in _units(c):
            if s >= c["n"] - c["span"]:
                rows = min(c["sub"], c["n"] - s)
                q = _mixture(gen, _empty(rows, c["hq"], DH), cents, s)
                x["fp"][s // c["sub"]] = q.float().mean(0).flatten()
        if c["block"] == 1:
            x["k"] = k
        else:
            nb = -(-c["n"] // c["block"])
            full = c["n"] // c["block"]
            reps = torch.empty(c["hkv"], nb, DH, device="cuda")
            for a in range(0, full, 512):
                b = min(full, a + 512)
                rows = k[a * c["block"]: b * c["block"]].view(b - a, c["block"], c["hkv"], DH)
                reps[:, a:b] = rows.float().mean(1).transpose(0, 1)
            if nb > full:
                reps[:, full] = k[full * c["block"]:].float().mean(0)
            x["reps"] = reps
    elif c["kind"] == "attend":
        b0 = c["n"] - c["span"]
        x["q"] = torch.zeros(c["n"], c["hq"], DH, dtype=torch.bfloat16, device="cuda")
        _mixture(gen, x["q"][b0:], cents, b0)
        x["k"], x["v"] = _kv(gen, c, cents)
        units = _units(c)
        sel = torch.full((-(-c["n"] // c["sub"]), c["topk"]), -1, dtype=torch.int32, device="cuda")
        cnt = torch.zeros(sel.shape[0], dtype=torch.int32, device="cuda")
        for u, (s, _) in enumerate(units):
            lo, hi = _candidates(c, s)
            got = min(c["topk"], hi - lo)
            if s >= b0 and got:
                pick = torch.randperm(hi - lo, generator=gen, device="cuda")[:got].sort()[0] + lo
                sel[u, :got] = pick.int()
                cnt[u] = got
        x["sel"], x["cnt"] = sel, cnt
    else:
        x["k"], x["v"] = _kv(gen, c, cents)
        base = _mixture(gen, _empty(1, c["hq"], DH), cents, c["n"])
        rows = base.float() + 0.15 * torch.randn(c["steps"], c["hq"], DH, generator=gen, device="cuda")
        x["q"] = rows.to(torch.bfloat16)
    return x


# ---------------------------------------------------------------- the calls


def _params(c):
    return S.params(num_q_heads=c["hq"], num_kv_heads=c["hkv"], sub_chunk=c["sub"], n_tokens=c["n"],
                    max_cluster_subchunks=c["cap"], outer_chunk=c["outer"], theta=c["theta"], block_size=c["block"],
                    top_k=c["topk"], n_sink=c["sink"], n_local=c["local"])


def _mode(c):
    return pkg.SCALE_MODE_PER_CLUSTER if c["mode"] == "cluster" else pkg.SCALE_MODE_PER_SUBCHUNK


def _paged(k, v, page, gen):
    """K and V in a shuffled pool of pages with a few spare ones."""
    n, hkv = k.shape[:2]
    used = -(-n // page)
    table = torch.randperm(used + 3, generator=gen, device="cuda")[:used]
    pool = []
    for x in (k, v):
        p = torch.zeros(used + 3, page, hkv, DH, dtype=x.dtype, device="cuda")
        full = torch.zeros(used * page, hkv, DH, dtype=x.dtype, device="cuda")
        full[:n] = x
        p[table] = full.view(used, page, hkv, DH)
        pool.append(p)
    return (*pool, table.int())


def prepare(case, seed):
    c = dict(case)
    st = _inputs(c, seed)
    st["c"], st["p"], st["mode"] = c, _params(c), _mode(c)
    p = st["p"]
    if c["kind"] == "decode":
        st["cache"] = torch.empty(S.scale_decode_cache_size(p), dtype=torch.uint8, device="cuda")
        st["ws"] = torch.empty(S.scale_decode_workspace_size(p), dtype=torch.uint8, device="cuda")
        st["out"] = _empty(c["steps"], c["hq"], DH)
        S.scale_decode_cache_init(st["cache"])
        S.scale_workspace_init(st["ws"])
        return st
    buf = st["buf"] = pkg.allocate(p, st["mode"], want_scores=c["kind"] == "select")
    st["units"] = units = _units(c)
    if c["kind"] in ("select", "attend"):
        starts = [s // c["sub"] for s, _ in units] + [-(-c["n"] // c["sub"])]
        buf.unit_start[: len(starts)] = torch.tensor(starts, dtype=torch.int32)
        buf.n_units.fill_(len(units))
        st["first"] = sum(s < c["n"] - c["span"] for s, _ in units)
    if c["kind"] == "select":
        buf.fingerprints, buf.reps = st["fp"], st.get("reps")
    if c["kind"] == "attend" and c["page"]:
        pages = _paged(st["k"], st["v"], c["page"], torch.Generator(device="cuda").manual_seed(seed))
        st["pages"] = pages
        st["kv"] = S.kv_pages(*pages, c["page"])
        del st["k"], st["v"]
    if c["kind"] == "prefill" and c["calls"] == "loop":
        chunks = [(t, min(c["n"], t + c["outer"])) for t in range(0, c["n"], c["outer"])]
        step = c["sub"] if c["mode"] == "subchunk" else c["outer"]
        st["loop"] = [((a, b), [(t, min(b, t + step)) for t in range(a, b, step)]) for a, b in chunks]
    return st


def run(state):
    c, p, mode = state["c"], state["p"], state["mode"]
    if c["kind"] == "decode":
        t0 = c["n"] - c["steps"]
        for i in range(c["steps"]):
            S.scale_decode_step(p, t0 + i, state["q"][i], state["k"], state["v"], state["cache"], state["out"][i],
                                state["ws"])
        return {"out": state["out"]}
    buf = state["buf"]
    if c["kind"] == "build":
        S.scale_build_reps(p, state["q"], state["k"], buf.reps, buf.fingerprints, buf.unit_start, buf.n_units, buf.ws)
        return {"reps": buf.reps, "fingerprints": buf.fingerprints, "unit_start": buf.unit_start,
                "n_units": buf.n_units}
    if c["kind"] == "select":
        pkg.scale.select(p, mode, c["n"] - c["span"], c["n"], state.get("k"), buf)
        u0, u1 = state["first"], len(state["units"])
        return {"sel": buf.sel_blocks[u0:u1], "count": buf.sel_count[u0:u1], "scores": buf.sel_scores[u0:u1]}
    if c["kind"] == "attend":
        b0 = c["n"] - c["span"]
        if c["page"]:
            S.scale_sparse_prefill_paged(p, mode, b0, c["n"], state["q"], state["kv"], buf.unit_start, buf.n_units,
                                         state["sel"], state["cnt"], buf.out, buf.ws)
        else:
            S.scale_sparse_prefill(p, mode, b0, c["n"], state["q"], state["k"], state["v"], buf.unit_start,
                                   buf.n_units, state["sel"], state["cnt"], buf.out, buf.ws)
        return {"out": buf.out[b0:]}
    q, k, v = state["q"], state["k"], state["v"]
    if c["calls"] == "whole":
        pkg.run_path(p, mode, q, k, v, buf)
    else:
        for (a, b), units in state["loop"]:
            S.scale_build_reps_range(p, a, b, q, k, buf.reps, buf.fingerprints, buf.unit_start, buf.n_units, buf.ws)
            for ua, ub in units:
                pkg.scale.select(p, mode, ua, ub, k, buf)
                S.scale_sparse_prefill(p, mode, ua, ub, q, k, v, buf.unit_start, buf.n_units, buf.sel_blocks,
                                       buf.sel_count, buf.out, buf.ws)
    u = len(state["units"])
    return {"out": buf.out, "unit_start": buf.unit_start, "n_units": buf.n_units, "sel": buf.sel_blocks[:u],
            "count": buf.sel_count[:u]}


# ---------------------------------------------------------------- what a pass cannot do without


def _distant(c, s):
    """Keys below the window that a unit starting at s attends to, with a full selection inside [sink, W)."""
    w = max(0, s - c["local"])
    lo, hi = _candidates(c, s)
    return min(c["sink"], w) + min(max(0, w - c["sink"]), c["block"] * min(c["topk"], hi - lo))


def work(case):
    c = case
    row_q, row_kv = c["hq"] * DH * 2, c["hkv"] * DH * 2
    if c["kind"] == "decode":
        t = c["n"] - 1
        cand = max(0, max(0, t - c["local"]) - c["sink"])
        keys = min(t + 1, c["sink"] + min(c["topk"], cand) + c["local"] + 1)
        return {"bytes": cand * row_kv + c["steps"] * (2 * keys * row_kv + 2 * row_q),
                "flops": 2.0 * DH * c["hq"] * (cand + c["steps"] * 2 * keys)}
    nb = -(-c["n"] // c["block"])
    m = -(-c["n"] // c["sub"])
    if c["kind"] == "build":
        return {"bytes": c["n"] * (row_q + row_kv) + 4 * DH * (c["hkv"] * nb + c["hq"] * m),
                "flops": float(c["n"] * (c["hq"] + c["hkv"]) * DH)}
    units = [u for u in _units(c) if u[0] >= c["n"] - c.get("span", c["n"])]
    score = sum(hi - lo for lo, hi in (_candidates(c, s) for s, _ in units))
    if c["kind"] == "select":
        top = max(_candidates(c, s)[1] for s, _ in units)
        per_block = row_kv if c["block"] == 1 else 2 * row_kv
        return {"bytes": top * per_block + 4 * len(units) * (c["hq"] * DH + c["topk"] + nb),
                "flops": 2.0 * DH * c["hq"] * score}
    pairs, rows, first = 0, 0, c["n"]
    for s, e in units:
        w = max(0, s - c["local"])
        pairs += (e - s) * _distant(c, s) + (e - s) * (s - w) + (e - s) * (e - s + 1) // 2
        rows += e - s
        first = min(first, w)
    flops = 4.0 * DH * c["hq"] * pairs
    if c["kind"] == "attend":
        keys = min(c["n"], c["n"] - first + sum(_distant(c, s) for s, _ in units))
        return {"bytes": 2 * rows * row_q + 2 * keys * row_kv, "flops": flops}
    return {"bytes": 2 * rows * (row_q + row_kv), "flops": flops + 2.0 * DH * c["hq"] * score}


def tolerance(case):
    # About four times the distance from exact(), in these cases and in drawn ones.
    kind = case["kind"]
    if kind == "build":  # fp32 means of bf16 values: the order of the additions (2.4e-8 measured)
        return {"rel": 2e-7, "max": 2e-6, "differ": 0.005}
    if kind == "select":  # fp32 logits of up to some tens in the exponent (1.5e-7); ties may swap list entries
        return {"rel": 1e-6, "max": 5e-5, "differ": 0.01}
    # outputs rounded to bf16, from probabilities rounded to bf16 except in decode (1.7e-3 to 2.4e-3)
    return {"rel": 0.01, "max": 0.1, "differ": 0.01}


# ---------------------------------------------------------------- the same in 64 bits


def _score64(c, fp, keys, s):
    """Soft-vote scores of a unit's candidates: fp [hq, 128], keys [hkv, blocks, 128]."""
    lo, hi = _candidates(c, s)
    g = c["hq"] // c["hkv"]
    score = torch.zeros(hi - lo, dtype=torch.float64, device="cuda")
    for j in range(c["hkv"] if hi > lo else 0):
        z = fp[j * g:(j + 1) * g].double() @ keys[j, lo:hi].double().T
        score += torch.softmax(z, dim=-1).sum(0)
    return score


def _pick64(c, score, s):
    lo, _ = _candidates(c, s)
    order = torch.sort(score, descending=True, stable=True)[1][: c["topk"]]
    return order.sort()[0] + lo


def _distant64(c, blocks, s):
    """The keys of the sinks and of the picked blocks below the window, each once."""
    w = max(0, s - c["local"])
    t = (blocks[:, None] * c["block"] + torch.arange(c["block"], device="cuda")).flatten()
    t = t[(t >= c["sink"]) & (t < w)]
    return torch.cat([torch.arange(min(c["sink"], w), device="cuda"), t])


def _attend64(c, q, k, v, out, s, e, keys):
    """out[s:e] (rows of q from `s`) over the distant keys and the causal window of the unit [s, e)."""
    g, w = c["hq"] // c["hkv"], max(0, s - c["local"])
    for a in range(s, e, 512):
        b = min(e, a + 512)
        idx = torch.cat([keys, torch.arange(w, b, device="cuda")])
        pos = torch.cat([torch.zeros_like(keys) - 1, torch.arange(w, b, device="cuda")])
        dead = pos[None, :] > torch.arange(a, b, device="cuda")[:, None]
        for j in range(c["hkv"]):
            qq = q[a:b, j * g:(j + 1) * g].double().transpose(0, 1)
            z = (qq @ k[idx, j].double().T) / math.sqrt(DH)
            z.masked_fill_(dead, -math.inf)
            out[a:b, j * g:(j + 1) * g] = (torch.softmax(z, dim=-1) @ v[idx, j].double()).transpose(0, 1)


def exact(case, seed):
    c = dict(case)
    if work(c)["flops"] > 8e12 or (c["kind"] == "select" and c["block"] == 1 and len(_units(c)) * c["n"] > 2e8):
        return None
    x = _inputs(c, seed)
    if c["kind"] == "decode":
        out = torch.empty(c["steps"], c["hq"], DH, dtype=torch.float64, device="cuda")
        t0 = c["n"] - c["steps"]
        picks = _pick64(c, _score64(c, x["q"][0], x["k"].transpose(0, 1), t0), t0)
        for i in range(c["steps"]):
            t = t0 + i
            keys = _distant64(c, picks, t)
            _attend64(c, _Row(x["q"][i], t), x["k"], x["v"], _Row(out[i], t), t, t + 1, keys)
        return {"out": out}
    if c["kind"] in ("build", "prefill"):
        m, nb = -(-c["n"] // c["sub"]), -(-c["n"] // c["block"])
        fp = torch.stack([x["q"][i * c["sub"]:(i + 1) * c["sub"]].double().mean(0) for i in range(m)])
        if c["block"] == 1:
            reps = x["k"].transpose(0, 1)
        else:
            reps = torch.stack([x["k"][i * c["block"]:(i + 1) * c["block"]].double().mean(0) for i in range(nb)], 1)
        if c["kind"] == "build":
            return {"reps": reps, "fingerprints": fp.flatten(1), "unit_start": None, "n_units": None}
    elif c["kind"] == "select":
        fp = x["fp"].view(-1, c["hq"], DH)
        reps = x["k"].transpose(0, 1) if c["block"] == 1 else x["reps"]
    units = _units(c)
    if c["kind"] == "select":
        rows = []
        for s, _ in units:
            if s >= c["n"] - c["span"]:
                lo, hi = _candidates(c, s)
                row = torch.full((-(-c["n"] // c["block"]),), math.nan, dtype=torch.float64, device="cuda")
                row[lo:hi] = _score64(c, fp[s // c["sub"]], reps, s)
                rows.append(row)
        return {"sel": None, "count": None, "scores": torch.stack(rows)}
    out = torch.empty(c["n"], c["hq"], DH, dtype=torch.float64, device="cuda")
    b0 = c["n"] - c.get("span", c["n"])
    for u, (s, e) in enumerate(units):
        if s < b0:
            continue
        if c["kind"] == "attend":
            picks = x["sel"][u, : int(x["cnt"][u])].long()
        else:
            picks = _pick64(c, _score64(c, fp[s // c["sub"]], reps, s), s)
        _attend64(c, x["q"], x["k"], x["v"], out, s, e, _distant64(c, picks, s))
    if c["kind"] == "attend":
        return {"out": out[b0:]}
    return {"out": out, "unit_start": None, "n_units": None, "sel": None, "count": None}


class _Row:
    """One token's row [heads, 128] addressed as row t of a longer tensor."""

    def __init__(self, row, t):
        self.row, self.t = row, t

    def __getitem__(self, at):
        return self.row[None][:, at[1]]

    def __setitem__(self, at, value):
        self.row[None][:, at[1]] = value
