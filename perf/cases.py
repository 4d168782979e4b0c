"""What a user of this framework has it do, as measurable cases.

Five kinds of work, each through the public entry points of ``paper_2604_03260_b200.binding`` and in the order a program calls
them:

* ``prefill``   one attention layer over a prompt: ``focus_assign`` (queries, keys), ``focus_build_tiles`` in the layout the
                library chooses, ``focus_attn_fwd``.
* ``decode``    one generation step of a layer: the new token's groups (``focus_assign`` on its query and key vectors), its key
                mask appended to the cached ones, ``focus_decode_step`` over the cache.
* ``route``     the router in the paper's own form: ``focus_assign_hidden`` from hidden states to the masks of a layer.
* ``train``     the training-time forward: ``focus_router_scores``, ``focus_sinkhorn``, ``focus_gate_attn_fwd``.
* ``sinkhorn``  the normalisation and its derivative as a training step of the router runs them: ``focus_sinkhorn``, then
                ``focus_sinkhorn_bwd``.

The listed sizes are the workloads of ``paper_2604_03260_b200.inputs`` (head counts, dimensions, groups, windows) at the lengths
the paper's context sweep runs over; the 1M-token one is left out because a pass takes seconds.
"""
import math
from dataclasses import replace

import torch

from paper_2604_03260_b200 import binding as fb
from paper_2604_03260_b200 import inputs as fi

TAU, ITERS, LAMBDA, D_G = 0.1, 10, 10.0, 16

#: head counts and dimension (query heads, KV heads, head dimension, softcap) of the workloads of inputs.py
HEADS = {"gpt2": (12, 12, 64, 0.0), "llama": (32, 8, 128, 0.0), "gemma": (16, 8, 256, 50.0)}


def _prefill(name, heads, n, K, topk, window, batch=1, draw="iid"):
    Hq, Hkv, D, cap = HEADS[heads]
    return {"name": name, "kind": "prefill", "Hq": Hq, "Hkv": Hkv, "D": D, "softcap": cap, "n": n, "K": K, "topk": topk,
            "window": window, "batch": batch, "draw": draw}


def _decode(name, heads, n, K, topk, window, batch=1):
    return dict(_prefill(name, heads, n, K, topk, window, batch), kind="decode")


def listed():
    return [
        # the smallest prompt of the repository: every launch is a few microseconds long
        _prefill("prefill-gpt2-1k", "gpt2", 1024, 4, 2, 64),
        # serving: a few prompts of one odd length in a batch, top-1 groups
        _prefill("prefill-batch3-3001", "llama", 3001, 4, 1, 512, batch=3),
        # an ordinary prompt, top-2 of 4 groups, too short for a sorted layout
        _prefill("prefill-llama-8k", "llama", 8192, 4, 2, 512),
        # many groups with skewed, clustered memberships: the layout with a separate window pass
        _prefill("prefill-mistral-32k", "llama", 32768, 8, 2, 1024, draw="clustered"),
        # head dimension 256 with logit softcap, top-1: the class-sorted layout where most pairs fall away
        _prefill("prefill-gemma-64k", "gemma", 65536, 4, 1, 4096),
        # the long prompt the repository quotes its rate on
        _prefill("prefill-llama-128k", "llama", 131072, 4, 2, 2048),
        # generation, one sequence with a short, odd cache: latency
        _decode("decode-llama-2k", "llama", 2049, 4, 2, 512),
        # generation, a batch of eight sequences
        _decode("decode-batch8-16k", "llama", 16385, 4, 2, 2048, batch=8),
        # generation at the end of a long context
        _decode("decode-llama-128k", "llama", 131072, 4, 2, 2048),
        # the router on the hidden states of an 8B-sized model
        {"name": "route-32k-4096", "kind": "route", "Hq": 32, "Hkv": 8, "D": 128, "n": 32768, "K": 4, "topk": 2, "d_model": 4096, "batch": 1},
        # training-time forward of one layer
        {"name": "train-8k", "kind": "train", "Hq": 32, "Hkv": 8, "D": 128, "n": 8192, "K": 8, "window": 1024, "d_model": 4096, "batch": 1},
        # the router's part of a training step: assignments and their derivative
        {"name": "sinkhorn-128k", "kind": "sinkhorn", "n": 131072, "K": 8, "batch": 1},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: the kinds in the proportion of the listed ones, lengths and caches over their whole range."""
    kind = rng.choice(["prefill"] * 6 + ["decode"] * 3 + ["route", "train", "sinkhorn"])
    K, topk = rng.choice([(4, 1), (4, 2), (8, 1), (8, 2)])
    if kind in ("prefill", "decode"):
        heads = rng.choice(["gpt2", "llama", "llama", "gemma"])
        window = rng.choice([64, 256, 512, 1024, 2048, 4096])
        if kind == "decode":
            n = _log_int(rng, 500, 131072)
            batch = min(rng.randint(1, 16), max(1, 131072 // n))
            return {k: v for k, v in _decode("", heads, n, K, topk, window, batch).items() if k != "name"}
        n = _log_int(rng, 500, 80000)
        batch = min(rng.randint(1, 4), max(1, 16000 // n))
        c = _prefill("", heads, n, K, topk, window, batch, rng.choice(["iid", "iid", "clustered", "runs"]))
        return {k: v for k, v in c.items() if k != "name"}
    if kind == "route":
        return {"kind": kind, "Hq": 32, "Hkv": 8, "D": 128, "n": _log_int(rng, 300, 131072), "K": K, "topk": topk,
                "d_model": rng.choice([768, 3584, 4096]), "batch": 1}
    if kind == "train":
        Hq, Hkv, D, _ = HEADS[rng.choice(["gpt2", "llama", "gemma"])]
        return {"kind": kind, "Hq": Hq, "Hkv": Hkv, "D": D, "n": _log_int(rng, 500, 32768), "K": K, "window": rng.choice([64, 512, 1024, 2048]),
                "d_model": Hq * D, "batch": 1}
    n = _log_int(rng, 1000, 262144)
    return {"kind": kind, "n": n, "K": K, "batch": min(rng.randint(1, 4), max(1, 65536 // n))}


def _inputs(case, seed):
    """Q [batch, Hq, n, D], K and V [batch, Hkv, n, D] bf16, centroids [Hkv, K, D] fp32 (one set for the batch)"""
    wl = fi.Workload("case", case["Hq"], case["Hkv"], case["D"], case["n"], case["K"], case.get("topk", 1), case.get("window", 0),
                     clustered=case.get("draw") == "clustered", runs=512.0 if case.get("draw") == "runs" else 0.0, flip=0.001)
    parts = [fi.make_inputs(replace(wl, seed=seed * 16 + b), "cuda") for b in range(case["batch"])]
    if len(parts) == 1:
        return tuple(x[None] for x in parts[0][:3]) + (parts[0][3],)
    return tuple(torch.stack([p[i] for p in parts]) for i in range(3)) + (parts[0][3],)


def _padded(x, ld):
    out = torch.zeros(x.shape[:-1] + (ld,), dtype=torch.float32, device="cuda")
    out[..., :x.shape[-1]] = x
    return out


def prepare(case, seed):
    kind, n, K, B = case["kind"], case["n"], case["K"], case["batch"]
    i32 = lambda *s: torch.empty(s, dtype=torch.int32, device="cuda")
    f32 = lambda *s: torch.empty(s, dtype=torch.float32, device="cuda")
    s = {"kind": kind, "near": torch.zeros(1, dtype=torch.int64, device="cuda"), "status": torch.zeros(4, dtype=torch.int32, device="cuda")}
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    randn = lambda *shape: torch.randn(shape, generator=gen, device="cuda")
    if kind == "sinkhorn":
        ld = fb.focus_soft_ld(K)
        s["shape"] = fb.make_shape(1, 1, n, 128, K, 1, 0, batch=B)
        s["scores"] = _padded(0.3 * randn(B, n, K), ld)
        s["dg"] = _padded(randn(B, n, K), ld)
        s["g"], s["ds"] = f32(B, n, ld), f32(B, n, ld)
        s["ws"] = torch.empty(fb.focus_sinkhorn_workspace_bytes(s["shape"], ITERS), dtype=torch.uint8, device="cuda")
        s["ws_bwd"] = torch.empty(fb.focus_sinkhorn_bwd_workspace_bytes(s["shape"], ITERS), dtype=torch.uint8, device="cuda")
        return s
    Hq, Hkv, D = case["Hq"], case["Hkv"], case["D"]
    s["Hq"], s["Hkv"] = Hq, Hkv
    shape = fb.make_shape(Hq, Hkv, n, D, K, case.get("topk", 1), case.get("window", 0), 0.0, case.get("softcap", 0.0), batch=B)
    s["shape"] = shape
    if kind in ("route", "train"):
        d = case["d_model"]
        s["h"] = randn(B, n, d).to(torch.bfloat16)
        s["Wg"], s["C"] = randn(d, D_G) / d ** 0.5, randn(K, D_G)
        s["folded"] = f32(K, d)
        if kind == "route":
            s["bias"] = 0.3 * randn(K)
            s["mq"], s["mk"] = i32(B * Hq, n), i32(B * Hkv, n)
            return s
        s["C"] *= 0.2
        ld = fb.focus_soft_ld(K)
        s["scores"], s["g"] = f32(B, n, ld), f32(B, n, ld)
        s["ws"] = torch.empty(fb.focus_sinkhorn_workspace_bytes(shape, ITERS), dtype=torch.uint8, device="cuda")
    s["q"], s["k"], s["v"], centroids = _inputs(case, seed)
    if kind == "train":
        s["o"], s["lse"] = torch.empty_like(s["q"]), f32(B * Hq, n)
        return s
    s["centroids"] = centroids
    if kind == "decode":
        s["q"] = s["q"][:, :, -1:, :].contiguous()
        s["one"] = fb.make_shape(Hq, Hkv, 1, D, K, case["topk"], case["window"], batch=B)
        s["k_new"] = s["k"][:, :, -1:, :]
        s["mk"] = i32(B * Hkv, n)
        fb.focus_assign(shape, s["k"], Hkv, centroids, s["mk"], s["near"])
        s["mq_new"], s["mk_new"] = i32(B * Hq, 1), i32(B * Hkv, 1)
        s["o"], s["lse"] = torch.empty((B, Hq, D), dtype=torch.bfloat16, device="cuda"), f32(B * Hq)
        s["ws"] = torch.empty(fb.focus_decode_workspace_bytes(shape), dtype=torch.uint8, device="cuda")
        return s
    s["layout"] = fb.focus_tiles_layout_of(shape, fb.FOCUS_LAYOUT_AUTO).layout
    s["ws"] = fb.alloc_workspace(shape, s["layout"])
    s["mq"], s["mk"] = i32(B * Hq, n), i32(B * Hkv, n)
    s["o"], s["lse"] = torch.empty_like(s["q"]), f32(B * Hq, n)
    return s


def run(s):
    kind, shape = s["kind"], s["shape"]
    if kind == "prefill":
        fb.focus_assign(shape, s["q"], s["Hq"], s["centroids"], s["mq"], s["near"])
        fb.focus_assign(shape, s["k"], s["Hkv"], s["centroids"], s["mk"], s["near"])
        fb.focus_build_tiles(shape, s["mq"], s["mk"], s["layout"], s["ws"])
        fb.focus_attn_fwd(shape, s["q"], s["k"], s["v"], s["mq"], s["mk"], s["ws"], s["layout"], s["o"], s["lse"], s["status"])
        return {"o": s["o"], "lse": s["lse"], "mq": s["mq"], "mk": s["mk"], "status": s["status"]}
    if kind == "decode":
        fb.focus_assign(s["one"], s["q"], s["Hq"], s["centroids"], s["mq_new"], s["near"])
        fb.focus_assign(s["one"], s["k_new"], s["Hkv"], s["centroids"], s["mk_new"], s["near"])
        s["mk"][:, -1:].copy_(s["mk_new"])
        fb.focus_decode_step(shape, s["q"][:, :, 0], s["k"], s["v"], s["mq_new"], s["mk"], s["o"], s["lse"], s["ws"])
        return {"o": s["o"], "lse": s["lse"], "mq_new": s["mq_new"], "mk": s["mk"]}
    if kind == "route":
        fb.focus_assign_hidden(shape, s["h"], s["Wg"], s["C"], s["bias"], s["folded"], s["mq"], s["mk"], s["near"])
        return {"mq": s["mq"], "mk": s["mk"], "folded": s["folded"]}
    if kind == "train":
        fb.focus_router_scores(shape, s["h"], s["Wg"], s["C"], s["folded"], s["scores"])
        fb.focus_sinkhorn(shape, s["scores"], TAU, ITERS, s["ws"], s["g"])
        fb.focus_gate_attn_fwd(shape, s["q"], s["k"], s["v"], s["g"], LAMBDA, s["o"], s["lse"], s["status"])
        return {"o": s["o"], "lse": s["lse"], "g": s["g"], "scores": s["scores"], "status": s["status"]}
    fb.focus_sinkhorn(shape, s["scores"], TAU, ITERS, s["ws"], s["g"])
    fb.focus_sinkhorn_bwd(shape, s["scores"], TAU, ITERS, s["ws_bwd"], s["dg"], s["ds"])
    return {"g": s["g"], "ds": s["ds"]}


def work(case):
    kind, n, K, B = case["kind"], case["n"], case["K"], case["batch"]
    if kind == "sinkhorn":
        # scores read, assignments written; scores and dg read, dS written.  Per iteration and entry: an exponential, an
        # addition and a multiplication forward, twice that backward
        return {"bytes": 5 * 4.0 * B * n * K, "flops": 9.0 * ITERS * B * n * K}
    Hq, Hkv, D = case["Hq"], case["Hkv"], case["D"]
    if kind == "route":
        d = case["d_model"]
        return {"bytes": B * n * (2.0 * d + 4 * (Hq + Hkv)), "flops": 2.0 * B * n * d * K}
    if kind == "train":
        d = case["d_model"]
        io = B * n * (2.0 * d + 2 * 4 * K + 2 * D * (2 * Hq + 2 * Hkv) + 4 * Hq)
        return {"bytes": io, "flops": B * (2.0 * n * d * K + 4.0 * D * Hq * n * (n + 1) / 2)}
    # the share of distant pairs that meet in a group when memberships are uniform (the clustered and run-structured draws are
    # within a tenth of it)
    share = 1.0 - math.comb(K - case["topk"], case["topk"]) / math.comb(K, case["topk"])
    w = case["window"]
    if kind == "decode":
        local = min(n, w + 1)
        # a key is read when one of the query heads of its KV head attends it
        read = local + (1.0 - (1.0 - share) ** (Hq // Hkv)) * (n - local)
        return {"bytes": B * (Hkv * (4.0 * D * read + 4 * n) + 4.0 * D * Hq), "flops": 4.0 * D * B * Hq * (local + share * (n - local))}
    far = max(0, n - 1 - w)
    far = far * (far + 1) / 2
    pairs = n * (n + 1) / 2 - (1.0 - share) * far
    return {"bytes": B * n * (2.0 * D * (2 * Hq + 2 * Hkv) + 4 * Hq + 4 * (Hq + Hkv)), "flops": 4.0 * D * B * Hq * pairs}


def tolerance(case):
    """About four times what the path differs by from the same computation in fp64."""
    if case["kind"] == "route":
        # masks are whole numbers (two scores closer than their fp32 rounding may swap); the folded router is a sum of 16 fp32 products
        return {"rel": 1e-6, "max": 1e-5, "differ": 1e-5}
    if case["kind"] == "sinkhorn":
        return {"rel": 8e-6, "max": 1e-3}
    # probabilities and outputs are bf16 (seen: rel 2e-3, max 0.04); masks as above
    return {"rel": 1e-2, "max": 0.15, "differ": 1e-5}


# ---- the same outputs in 64 bits, by plain torch

def _sinkhorn64(scores):
    """log-domain iteration over [batch, n, K] fp64"""
    x = scores / TAU
    for _ in range(ITERS):
        x = x - torch.logsumexp(x, dim=1, keepdim=True)
        x = x - torch.logsumexp(x, dim=2, keepdim=True)
    return torch.exp(x)


def _members64(x, centroids, topk):
    """0/1 membership [batch, H, n, K] of the vectors x [batch, H, n, D]: the topk groups of largest cosine"""
    c = centroids.double()
    c = c / c.norm(dim=-1, keepdim=True)
    out = torch.zeros(x.shape[:3] + (c.shape[1],), dtype=torch.float32, device=x.device)
    group = x.shape[1] // c.shape[0]
    for b in range(x.shape[0]):
        for h in range(x.shape[1]):
            v = x[b, h].double()
            cos = (v @ c[h // group].T) / v.norm(dim=-1, keepdim=True)
            out[b, h].scatter_(1, cos.topk(topk, dim=1).indices, 1.0)
    return out


def _attend64(q, k, v, first, cap, window, share=None, gate=None):
    """O [n, D], lse [n] of the rows of q, at positions first.., over their causal keys; `share` = memberships of rows and keys
    (a distant pair without a common group is left out), `gate` = soft assignments (a distant pair's logit is scaled)"""
    o, lse = torch.empty(q.shape, dtype=torch.float64, device=q.device), torch.empty(q.shape[0], dtype=torch.float64, device=q.device)
    k, v = k.double(), v.double()
    for r in range(0, q.shape[0], 1024):
        rows = slice(r, min(r + 1024, q.shape[0]))
        i = torch.arange(first + rows.start, first + rows.stop, device=q.device)[:, None]
        m = first + rows.stop
        j = torch.arange(m, device=q.device)[None]
        s = (q[rows].double() @ k[:m].T) / q.shape[-1] ** 0.5
        if cap:
            s = cap * torch.tanh(s / cap)
        if gate is not None:
            s = torch.where(i - j > window, s * torch.sigmoid(LAMBDA * (gate[0][rows] @ gate[1][:m].T)), s)
        if share is not None:
            s.masked_fill_((i - j > window) & ((share[0][rows] @ share[1][:m].T) < 0.5), -math.inf)
        s.masked_fill_(j > i, -math.inf)
        lse[rows] = torch.logsumexp(s, dim=1)
        o[rows] = torch.exp(s - lse[rows, None]) @ v[:m]
    return o, lse


def exact(case, seed):
    kind, n, K, B = case["kind"], case["n"], case["K"], case["batch"]
    Hq = case.get("Hq", 1)
    if kind in ("prefill", "train") and float(B) * Hq * n * n > 1.5e11:
        return None                                # longer than a check should take
    s = prepare(case, seed)
    if kind == "sinkhorn":
        x = s["scores"][..., :K].double().requires_grad_()
        g = _sinkhorn64(x)
        ds, = torch.autograd.grad(g, x, s["dg"][..., :K].double())
        pad = (0, s["scores"].shape[-1] - K)
        return {"g": torch.nn.functional.pad(g.detach(), pad), "ds": torch.nn.functional.pad(ds, pad)}
    if kind == "route":
        return {"mq": None, "mk": None, "folded": s["C"].double() @ s["Wg"].double().T}
    G, w = Hq // case["Hkv"], case["window"]
    q, k, v = s["q"], s["k"], s["v"]
    o, lse = torch.empty(q.shape, dtype=torch.float64, device="cuda"), torch.empty(q.shape[:3], dtype=torch.float64, device="cuda")
    if kind == "train":
        folded = s["C"].double() @ s["Wg"].double().T
        scores = torch.stack([torch.cat([part.double() @ folded.T for part in h.split(16384)]) for h in s["h"]])
        g = _sinkhorn64(scores)
    else:
        mq, mk = _members64(q, s["centroids"], case["topk"]), _members64(k, s["centroids"], case["topk"])
    for b in range(B):
        for h in range(Hq):
            pair = {"gate": (g[b], g[b])} if kind == "train" else {"share": (mq[b, h], mk[b, h // G])}
            o[b, h], lse[b, h] = _attend64(q[b, h], k[b, h // G], v[b, h // G], n - q.shape[2], case["softcap"] if kind != "train" else 0.0, w, **pair)
    if kind == "train":
        pad = (0, s["g"].shape[-1] - K)
        return {"o": o, "lse": lse.view(B * Hq, n), "g": torch.nn.functional.pad(g, pad), "scores": torch.nn.functional.pad(scores, pad), "status": None}
    if kind == "decode":
        return {"o": o[:, :, 0], "lse": lse.view(B * Hq), "mq_new": None, "mk": None}
    return {"o": o, "lse": lse.view(B * Hq, n), "mq": None, "mk": None, "status": None}
