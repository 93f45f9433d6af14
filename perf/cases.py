"""Performance cases of the framework's public calls (`paper_2607_10661_gb300.ptd`).

Every case is one pass of work that a decoding program hands to the library: a layer's tree
attention, a whole tree-verify step, a top-k over logits, the LM head with its top-k, sampling
verification, the rotary encoding with the K/V append, and the draft forest and candidate pool
update.  `listed()` holds fixed sizes, `draw()` further ones from the same ranges.  Inputs are
drawn on the GPU from the seed: Q, K, V ~ N(0, 1), logits ~ N(0, 2) with one token per row
raised by 6, trees pruned at random from a full branching tree, draft tokens that match their
parent's best token about half of the time.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

from paper_2607_10661_gb300 import ptd
from paper_2607_10661_gb300 import synthetic as syn

DEV = "cuda"
BRANCHING = (4, 3, 2, 2, 1, 1)   # 185 nodes in full: every tree of 1 .. 128 nodes is a pruning of it
MAX_BYTES = 1.2e9                # of one pass (what a drawn case may read and write)
MAX_FLOPS = 2.7e11


def listed():
    return [
        # the smallest whole step: a small fp32 model (parity runs, draft models), latency only
        {"name": "step_tiny_f32", "kind": "step", "dtype": "f32", "batch": 1, "layers": 1, "hq": 8, "hkv": 8, "d": 64,
         "ctx": 256, "nodes": 15, "page": 0, "vocab": 1000, "k": 2},
        # one layer early in a chat: a short prompt and a small tree, ragged sizes
        {"name": "attn_short", "kind": "attn", "dtype": "bf16", "batch": 1, "layers": 1, "hq": 32, "hkv": 8, "d": 128,
         "ctx": 611, "nodes": 13, "page": 0},
        # one layer of a 7B MHA model, as an engine that runs layer by layer calls it
        {"name": "attn_mha", "kind": "attn", "dtype": "bf16", "batch": 1, "layers": 1, "hq": 32, "hkv": 32, "d": 128,
         "ctx": 2048, "nodes": 31, "page": 0},
        # one layer over a long document with a wide tree: tensor-core bound
        {"name": "attn_long", "kind": "attn", "dtype": "bf16", "batch": 1, "layers": 1, "hq": 64, "hkv": 8, "d": 128,
         "ctx": 32768, "nodes": 128, "page": 0},
        # one layer of a GQA model kept in fp32 (evaluation without rounding)
        {"name": "attn_f32", "kind": "attn", "dtype": "f32", "batch": 1, "layers": 1, "hq": 32, "hkv": 8, "d": 128,
         "ctx": 2048, "nodes": 63, "page": 0},
        # the largest: the whole step over every layer of an 8B GQA model
        {"name": "step_gqa_32_layers", "kind": "step", "dtype": "bf16", "batch": 1, "layers": 32, "hq": 32, "hkv": 8,
         "d": 128, "ctx": 8192, "nodes": 63, "page": 0, "vocab": 128256, "k": 4},
        # batched serving: eight ragged sequences over 16-token pages
        {"name": "step_batched_paged", "kind": "step", "dtype": "bf16", "batch": 8, "layers": 1, "hq": 32, "hkv": 8,
         "d": 128, "ctx": 4096, "nodes": 64, "page": 16, "vocab": 128256, "k": 4},
        # top-k of fp32 logits (heads that accumulate in and return fp32)
        {"name": "topk_f32", "kind": "topk", "dtype": "f32", "rows": 63, "vocab": 128256, "k": 4},
        # the LM head of an 8B model fused with its top-k
        {"name": "lm_head", "kind": "lm_head", "rows": 63, "vocab": 128256, "d_model": 4096, "k": 4},
        # sampling verification of a served batch
        {"name": "sampling", "kind": "sampling", "dtype": "bf16", "batch": 8, "nodes": 48, "vocab": 128256,
         "temperature": 0.8},
        # rotary encoding and K/V append of a tree in all layers
        {"name": "rope_append", "kind": "rope", "dtype": "bf16", "batch": 1, "layers": 32, "hq": 32, "hkv": 8, "d": 128,
         "ctx": 1500, "nodes": 63, "page": 0},
        # the draft forest's update and the candidate pool's merge and retrieval after a step
        {"name": "forest_pool", "kind": "forest", "nodes": 60, "expand": 2, "width": 4, "max_depth": 6,
         "capacity": 128, "pool": 65536},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _attention_sizes(rng, dtype):
    heads = rng.choice([(32, 32), (32, 8), (64, 8), (16, 2), (28, 4), (40, 8)])
    paged = rng.random() < 0.4
    case = {"dtype": dtype, "batch": 1 if rng.random() < 0.5 else _log(rng, 2, 16), "layers": 1 if rng.random() < 0.6 else _log(rng, 2, 32),
            "hq": heads[0], "hkv": heads[1], "d": 128, "ctx": _log(rng, 96, 32768), "nodes": _log(rng, 1, 128),
            "page": rng.choice([16, 32, 64, 128]) if paged else 0}
    if dtype == "f32":
        hq, hkv = rng.choice([(8, 8), (16, 16), (32, 8)])
        case.update(hq=hq, hkv=hkv, d=rng.choice([32, 64, 128]), ctx=_log(rng, 64, 4096), batch=rng.choice([1, 1, 2, 3]),
                    layers=rng.choice([1, 1, 2]))
    return case


def draw(rng: random.Random):
    """One more case of the same ranges (sizes spread over their logarithm), no costlier than the largest listed."""
    kinds = ["attn", "attn", "attn_f32", "step", "step", "topk", "lm_head", "sampling", "rope", "forest"]
    kind = rng.choice(kinds)
    while True:
        if kind in ("attn", "attn_f32"):
            case = {"kind": "attn", **_attention_sizes(rng, "f32" if kind == "attn_f32" else "bf16")}
        elif kind == "step":
            case = {"kind": "step", **_attention_sizes(rng, "f32" if rng.random() < 0.2 else "bf16"),
                    "vocab": rng.choice([1000, 32000, 128256, 152064]), "k": rng.randint(1, 8)}
        elif kind == "topk":
            case = {"kind": "topk", "dtype": rng.choice(["bf16", "f32"]), "rows": _log(rng, 1, 512),
                    "vocab": rng.choice([32000, 50257, 128256, 152064, _log(rng, 1000, 150000)]), "k": rng.randint(1, 16)}
        elif kind == "lm_head":
            case = {"kind": "lm_head", "rows": _log(rng, 1, 128), "vocab": rng.choice([32000, 50257, 128256, 152064]),
                    "d_model": 64 * rng.randint(16, 80), "k": rng.randint(1, 8)}
        elif kind == "sampling":
            case = {"kind": "sampling", "dtype": rng.choice(["bf16", "f32"]), "batch": _log(rng, 1, 16),
                    "nodes": _log(rng, 2, 128), "vocab": rng.choice([32000, 50257, 128256, 152064]),
                    "temperature": round(rng.uniform(0.4, 1.3), 3)}
        elif kind == "rope":
            case = {"kind": "rope", **_attention_sizes(rng, rng.choice(["bf16", "bf16", "f32"]))}
            case["ctx"] = min(case["ctx"], 4096)
        else:
            case = {"kind": "forest", "nodes": rng.randint(8, 120), "expand": rng.randint(1, 4), "width": rng.randint(2, 6),
                    "max_depth": rng.randint(3, 8), "capacity": 128, "pool": 2 ** rng.randint(16, 19)}
        w = work(case)
        if w["bytes"] <= MAX_BYTES and w["flops"] <= MAX_FLOPS and _resident(case) <= 1.5e9:
            return case


# ------------------------------------------------------------------------------- inputs
def _torch_dtype(name):
    return torch.bfloat16 if name == "bf16" else torch.float32


def _shape(case):
    """Tree sizes and contexts of the case's sequences (the batch is ragged: 1/4 .. all of both)."""
    g = np.random.default_rng([case["nodes"], case.get("ctx", 0), case["batch"]])
    B = case["batch"]
    if B == 1:
        return [case["nodes"]], [case.get("ctx", 0)]
    T = [case["nodes"]] + [int(g.integers(max(1, case["nodes"] // 4), case["nodes"] + 1)) for _ in range(B - 1)]
    C = [case.get("ctx", 0)] + [int(g.integers(case.get("ctx", 0) // 4, case.get("ctx", 0) + 1)) for _ in range(B - 1)]
    return T, C


def _resident(case):
    """Bytes of the K/V cache that the case's buffers hold (rectangular where the cache is)."""
    if "ctx" not in case:
        return 0
    es = 2 if case["dtype"] == "bf16" else 4
    T, C = _shape(case)
    slots = sum(t + c for t, c in zip(T, C)) if case["page"] else case["batch"] * max(t + c for t, c in zip(T, C))
    return 2 * case["layers"] * slots * case["hkv"] * case["d"] * es


def _logits(gen, rows, vocab, dtype):
    x = torch.randn((rows, vocab), generator=gen, device=DEV, dtype=torch.float32).mul_(2.0)
    at = torch.randint(0, vocab, (rows,), generator=gen, device=DEV)
    x[torch.arange(rows, device=DEV), at] += 6.0
    return x.to(_torch_dtype(dtype))


class _Trees:
    """A batch of random trees on the device, with their host arrays."""

    def __init__(self, case, seed):
        self.T, self.C = _shape(case)
        g = np.random.default_rng([seed, 1])
        self.parents = [syn.pruned_tree(BRANCHING, t, g) for t in self.T]
        self.off = np.concatenate([[0], np.cumsum(self.T)]).astype(np.int32)
        i32 = dict(dtype=torch.int32, device=DEV)
        self.dev = (torch.tensor(self.off, **i32), torch.tensor(np.concatenate(self.parents), **i32),
                    torch.tensor(self.C, **i32))
        self.n = int(self.off[-1])
        self.tree = ptd.Tree(*self.dev, max_nodes=max(self.T), max_ctx=max(self.C))

    def tokens(self, logits, seed, p_match=0.5):
        """Draft tokens: a child matches its parent's best token with p_match (one sibling at most)."""
        best = logits.float().argmax(dim=1).cpu().numpy()
        vocab = logits.shape[1]
        g = np.random.default_rng([seed, 2])
        tok = g.integers(0, vocab, size=self.n)
        for b, par in enumerate(self.parents):
            matched = set()
            for c in range(1, len(par)):
                p = int(par[c])
                if p not in matched and g.random() < p_match:
                    matched.add(p)
                    tok[self.off[b] + c] = best[self.off[b] + p]
        return torch.tensor(tok, dtype=torch.int32, device=DEV)


def _cache(case, trees, gen, seed):
    L, hkv, d, dt = case["layers"], case["hkv"], case["d"], _torch_dtype(case["dtype"])
    slots = [t + c for t, c in zip(trees.T, trees.C)]
    table = None
    if case["page"]:
        ps = case["page"]
        need = [-(-s // ps) for s in slots]
        pages = sum(need) + 3
        perm = np.random.default_rng([seed, 3]).permutation(pages)
        table = np.zeros((len(slots), max(need)), np.int32)
        at = 0
        for b, n in enumerate(need):
            table[b, :n] = perm[at:at + n]
            at += n
        table = torch.tensor(table, device=DEV)
        shape = (L, pages, ps, hkv, d)
    else:
        shape = (L, len(slots), max(slots), hkv, d)
    k = torch.randn(shape, generator=gen, device=DEV, dtype=dt)
    v = torch.randn(shape, generator=gen, device=DEV, dtype=dt)
    return ptd.KVCache(k, v, hkv, d, case["page"], table)


def prepare(case, seed):
    gen = torch.Generator(device=DEV).manual_seed(seed)
    i32 = dict(dtype=torch.int32, device=DEV)
    s = {"case": case, "status": torch.zeros(1, **i32)}
    kind = case["kind"]
    if kind in ("attn", "step", "rope", "sampling"):
        trees = s["trees"] = _Trees(case, seed)
    if kind in ("attn", "step", "rope"):
        dt = _torch_dtype(case["dtype"])
        s["cache"] = _cache(case, trees, gen, seed)
        s["q"] = torch.randn((case["layers"], trees.n, case["hq"], case["d"]), generator=gen, device=DEV, dtype=dt)
    if kind == "attn":
        s["out"] = torch.empty_like(s["q"])
        n = ptd.attention_workspace_size(trees.tree, s["cache"], case["hq"])
        s["ws"] = torch.empty(n, dtype=torch.uint8, device=DEV) if n else None
    elif kind == "step":
        logits = _logits(gen, trees.n, case["vocab"], case["dtype"])
        B, k = case["batch"], case["k"]
        n = ptd.step_workspace_size(trees.tree, s["cache"], case["hq"])
        s["bufs"] = ptd.StepBuffers(
            s["q"], case["hq"], torch.empty_like(s["q"]), logits, k, trees.tokens(logits, seed),
            torch.zeros((trees.n, k), **i32), torch.zeros((trees.n, k), device=DEV), torch.zeros((B, max(trees.T)), **i32),
            torch.zeros(B, **i32), torch.zeros(B, **i32), torch.zeros(B, **i32), s["status"],
            torch.empty(max(n, 16), dtype=torch.uint8, device=DEV))
    elif kind == "topk":
        s["logits"] = _logits(gen, case["rows"], case["vocab"], case["dtype"])
        s["idx"] = torch.zeros((case["rows"], case["k"]), **i32)
        s["val"] = torch.zeros((case["rows"], case["k"]), device=DEV)
    elif kind == "lm_head":
        rows, vocab, dm, k = case["rows"], case["vocab"], case["d_model"], case["k"]
        s["hidden"] = torch.randn((rows, dm), generator=gen, device=DEV, dtype=torch.bfloat16)
        s["weight"] = torch.randn((vocab, dm), generator=gen, device=DEV, dtype=torch.bfloat16).mul_(dm ** -0.5)
        s["idx"], s["val"] = torch.zeros((rows, k), **i32), torch.zeros((rows, k), device=DEV)
        s["ws"] = torch.empty(ptd.lm_head_workspace_size(rows, vocab), dtype=torch.uint8, device=DEV)
    elif kind == "sampling":
        s["logits"] = _logits(gen, trees.n, case["vocab"], case["dtype"])
        s["tokens"] = trees.tokens(s["logits"], seed)
        s["u"] = torch.rand(trees.n, generator=gen, device=DEV)
        s["ub"] = torch.rand(case["batch"], generator=gen, device=DEV)
        s["outs"] = (torch.zeros((case["batch"], max(trees.T)), **i32), torch.zeros(case["batch"], **i32),
                     torch.zeros(case["batch"], **i32))
    elif kind == "rope":
        kv = (case["layers"], trees.n, case["hkv"], case["d"])
        s["k"] = torch.randn(kv, generator=gen, device=DEV, dtype=dt)
        s["v"] = torch.randn(kv, generator=gen, device=DEV, dtype=dt)
        s["pos"] = torch.zeros(trees.n, **i32)
    elif kind == "forest":
        n, cap = case["nodes"], case["capacity"]
        g = np.random.default_rng([seed, 4])
        pool = s["pool"] = ptd.CandidatePool(case["pool"], DEV)
        s["step"] = 0

        def forest():
            par = syn.pruned_tree(BRANCHING, n, g)
            return torch.tensor(par.reshape(1, -1), **i32), torch.tensor(g.integers(0, 32000, (1, n)), **i32)

        s["count"] = torch.full((1,), n, **i32)
        for _ in range(16):   # what earlier steps left in the pool
            par, tok = forest()
            pool.merge(s["step"], s["count"], par, tok, s["status"])
            s["step"] += 1
        s["par"], s["tok"] = forest()
        s["drafts"] = torch.tensor(g.integers(0, 32000, (n, 4)), **i32)
        s["new"] = (torch.zeros(1, **i32), torch.zeros((1, cap), **i32), torch.zeros((1, cap), **i32),
                    torch.zeros((1, cap), **i32), torch.zeros((1, n), **i32))
        s["root"] = s["tok"][0, :1].clone()
        s["got"] = (torch.zeros(1, **i32), torch.zeros(64, **i32), torch.zeros(64, **i32))
    return s


# ------------------------------------------------------------------------------- one pass
def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "attn":
        ptd.tree_attention(s["trees"].tree, s["cache"], s["q"], s["out"], case["hq"], s["status"], workspace=s["ws"])
        return {"out": s["out"], "status": s["status"]}
    if kind == "step":
        b = s["bufs"]
        ptd.tree_verify_step(s["trees"].tree, s["cache"], b)
        return {"attn": b.attn_out, "idx": b.topk_idx, "val": b.topk_val, "accepted": b.accepted, "len": b.accept_len,
                "bonus": b.bonus, "ctx": b.new_ctx, "status": b.dev_status, "k": s["cache"].k, "v": s["cache"].v}
    if kind == "topk":
        ptd.topk_draft(s["logits"], case["k"], s["idx"], s["val"])
        return {"idx": s["idx"], "val": s["val"]}
    if kind == "lm_head":
        ptd.lm_head_topk(s["hidden"], s["weight"], case["k"], s["idx"], s["val"], s["ws"], s["status"])
        return {"idx": s["idx"], "val": s["val"], "status": s["status"]}
    if kind == "sampling":
        acc, length, bonus = s["outs"]
        ptd.verify_sampling(s["trees"].tree, s["tokens"], s["logits"], case["temperature"], s["u"], s["ub"], acc, length,
                            bonus, s["status"])
        return {"accepted": acc, "len": length, "bonus": bonus, "status": s["status"]}
    if kind == "rope":
        ptd.tree_rope_append(s["trees"].tree, s["cache"], 0, s["q"], case["hq"], s["k"], s["v"], 500000.0, s["status"],
                             positions_out=s["pos"])
        return {"q": s["q"], "pos": s["pos"], "k": s["cache"].k, "v": s["cache"].v, "status": s["status"]}
    count, par, tok, depth, old = s["new"]
    ptd.draft_tree_update(s["count"], s["par"], s["tok"], s["drafts"], case["expand"], case["width"], case["max_depth"],
                          case["capacity"], count, par, tok, depth, old, s["status"])
    s["pool"].merge(s["step"], count, par, tok, s["status"])
    s["step"] += 1
    s["pool"].retrieve(s["root"], 4, 6, 64, *s["got"])
    return {"count": count, "parents": par, "tokens": tok, "depths": depth, "old_to_new": old, "got": list(s["got"]),
            "status": s["status"]}


# ------------------------------------------------------------------------------- what it takes
def work(case):
    kind = case["kind"]
    es = 2 if case.get("dtype", "bf16") == "bf16" else 4
    if kind == "topk":
        return {"bytes": case["rows"] * (case["vocab"] * es + case["k"] * 8), "flops": 0}
    if kind == "lm_head":
        rows, vocab, dm = case["rows"], case["vocab"], case["d_model"]
        return {"bytes": (vocab + rows) * dm * 2 + rows * case["k"] * 8, "flops": 2.0 * rows * vocab * dm}
    if kind == "forest":
        n, cap = case["nodes"], case["capacity"]
        return {"bytes": 4 * (n * (2 + case["expand"] + 1) + 3 * cap + 2 * 64) + 24 * cap, "flops": 0}
    T, C = _shape(case)
    n = sum(T)
    if kind == "sampling":   # one visited row per tree at least
        return {"bytes": case["batch"] * case["vocab"] * es + n * 16, "flops": 0}
    L, hq, hkv, d = case["layers"], case["hq"], case["hkv"], case["d"]
    if kind == "rope":
        return {"bytes": 2 * L * n * (hq + 2 * hkv) * d * es + n * 8, "flops": 3.0 * L * n * (hq + hkv) * d}
    bytes_ = L * es * d * (2 * hkv * sum(t + c for t, c in zip(T, C)) + 2 * hq * n)
    flops = 4.0 * L * hq * d * sum(t * (t + c) for t, c in zip(T, C))
    if kind == "step":
        bytes_ += n * (case["vocab"] * es + case["k"] * 8 + 8)
    return {"bytes": bytes_, "flops": flops}


def tolerance(case):
    kind = case["kind"]
    if kind in ("topk", "sampling", "forest"):
        return "exact"   # selections and decisions: the same bits
    # about four times the distance from exact() that the calls show
    if kind == "lm_head":   # fp32 sums of bf16 products (4.1e-6); near ties may swap places
        return {"rel": 1.6e-5, "max": 2e-4, "differ": 0.01}
    if kind == "rope":   # one rounding of each rotated value (1.7e-3); repeated passes turn q again
        return {"rel": 7e-3, "max": 0.1} if case["dtype"] == "bf16" else {"rel": 2e-6, "max": 2e-5}
    # bf16: probabilities and outputs are rounded to bf16 (2.3e-3); fp32: fp32 sums (4.8e-7)
    return {"rel": 9e-3, "max": 0.15} if case["dtype"] == "bf16" else {"rel": 2e-6, "max": 3e-5}


# ------------------------------------------------------------------------------- in 64 bits
def _slot_rows(s, b, n):
    """Cache rows (flattened over the dimensions before the heads) of sequence b's first n slots."""
    cache, ps = s["cache"], s["case"]["page"]
    slot = torch.arange(n, device=DEV)
    if ps:
        return cache.block_table[b].long()[slot // ps] * ps + slot % ps
    return b * cache.k.shape[2] + slot


def _exact_attention(s):
    case, trees = s["case"], s["trees"]
    L, hq, hkv, d = case["layers"], case["hq"], case["hkv"], case["d"]
    out = torch.zeros((L, trees.n, hq, d), dtype=torch.float64, device=DEV)
    for b, par in enumerate(trees.parents):
        T, C, n0 = trees.T[b], trees.C[b], int(trees.off[b])
        see = np.zeros((T, C + T), bool)
        see[:, :C] = True
        for i in range(T):
            if i:
                see[i, C:] = see[par[i], C:]
            see[i, C + i] = True
        hide = ~torch.from_numpy(see).to(DEV)
        rows = _slot_rows(s, b, C + T)
        for layer in range(L):
            k = s["cache"].k[layer].reshape(-1, hkv, d)[rows].double()
            v = s["cache"].v[layer].reshape(-1, hkv, d)[rows].double()
            q = s["q"][layer, n0:n0 + T].double()
            for h in range(hq):
                p = (q[:, h] @ k[:, h // (hq // hkv)].T) * d ** -0.5
                p = torch.softmax(p.masked_fill_(hide, -math.inf), dim=1)
                out[layer, n0:n0 + T, h] = p @ v[:, h // (hq // hkv)]
    return out


def exact(case, seed):
    kind = case["kind"]
    if kind in ("sampling", "forest") or work(case)["flops"] > 4e11:
        return None
    s = prepare(case, seed)
    if kind == "topk":
        return {"idx": None, "val": torch.topk(s["logits"].double(), case["k"], dim=1).values}
    if kind == "lm_head":
        x = s["hidden"].double()
        best = [torch.topk(x @ w.double().T, min(case["k"], w.shape[0]), dim=1).values for w in s["weight"].split(8192)]
        return {"idx": None, "val": torch.topk(torch.cat(best, 1), case["k"], dim=1).values, "status": None}
    if kind == "rope":
        trees = s["trees"]
        d, half = case["d"], case["d"] // 2
        freq = 500000.0 ** (-2.0 * torch.arange(half, dtype=torch.float64, device=DEV) / d)
        k_all, v_all = (x.double() for x in (s["cache"].k, s["cache"].v))
        q, k, v = (s[x].double() for x in ("q", "k", "v"))
        for b, par in enumerate(trees.parents):
            T, C, n0 = trees.T[b], trees.C[b], int(trees.off[b])
            depth = np.zeros(T)
            for i in range(1, T):
                depth[i] = depth[par[i]] + 1
            a = torch.from_numpy(C + depth).to(DEV)[:, None] * freq
            cos, sin = a.cos()[None, :, None], a.sin()[None, :, None]
            for x in (q, k):
                lo, hi = x[:, n0:n0 + T, :, :half].clone(), x[:, n0:n0 + T, :, half:].clone()
                x[:, n0:n0 + T, :, :half] = lo * cos - hi * sin
                x[:, n0:n0 + T, :, half:] = lo * sin + hi * cos
            rows = _slot_rows(s, b, C + T)[C:]
            for all_, x in ((k_all, k), (v_all, v)):
                all_.view(case["layers"], -1, case["hkv"], d)[:, rows] = x[:, n0:n0 + T]
        return {"q": q, "pos": None, "k": k_all, "v": v_all, "status": None}
    attn = _exact_attention(s)
    if kind == "attn":
        return {"out": attn, "status": None}
    val = torch.topk(s["bufs"].logits.double(), case["k"], dim=1).values
    return {"attn": attn, "idx": None, "val": val, "accepted": None, "len": None, "bonus": None, "ctx": None,
            "status": None, "k": None, "v": None}
