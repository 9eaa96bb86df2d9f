"""The work that a user of this library has it do, as cases that can be timed and compared.

A case is one call (or one serving step of calls) through the public entry
points of ``binding``: the chain and tree draft-and-verify steps, verify
attention, the acceptance step, the drafter's sampler and the semantic router.
Inputs are the seeded serving-shaped tensors of ``workloads``, with the seed
in place of the workload's cell number.
"""
from __future__ import annotations

import math

import torch

from paper_2607_20507_gb300 import binding
from paper_2607_20507_gb300 import workloads as W

DEVICE = "cuda:0"
D = 128


# --------------------------------------------------------------------------
# the cases
# --------------------------------------------------------------------------
def _attn(batch, rows, hq, hkv, page, ctx, lo, hi):
    """Attention geometry: ctx "const" (lo tokens), "uniform" [lo, hi] or "lognormal" (median 2048, clipped)."""
    return dict(batch=batch, rows=rows, hq=hq, hkv=hkv, page=page, ctx=ctx, lo=lo, hi=hi)


def _logits(vocab, dtype, sigma, temperature):
    return dict(vocab=vocab, dtype=dtype, sigma=sigma, temperature=temperature)


def listed():
    return [
        # one interactive request, the smallest step a server runs: latency and launches
        dict(name="step-b1", op="step", **_attn(1, 5, 32, 8, 16, "const", 512, 512),
             **_logits(32000, "f32", 1.0, 1.0)),
        # a lightly loaded server's whole step, sampled
        dict(name="step-b8", op="step", **_attn(8, 6, 32, 8, 16, "uniform", 1024, 4096),
             **_logits(128256, "bf16", 0.5, 0.7)),
        # the same load with a 34-node candidate tree in place of the chain
        dict(name="tree-step-b8", op="tree_step", tree="3,2,2,1", **_attn(8, 34, 32, 8, 16, "uniform", 1024, 4096),
             **_logits(128256, "bf16", 0.5, 0.7)),
        # parallel serving: ragged contexts, seven query heads per KV head
        dict(name="attn-b64-ragged", op="attn", **_attn(64, 5, 28, 4, 16, "lognormal", 512, 8192)),
        # a full server with long contexts: the largest call
        dict(name="attn-b256-long", op="attn", **_attn(256, 9, 64, 8, 32, "uniform", 2048, 16384)),
        # short drafts: few query rows per KV head
        dict(name="attn-b64-k2", op="attn", **_attn(64, 3, 32, 8, 16, "const", 4096, 4096)),
        # acceptance of the two serving loads above
        dict(name="accept-b64", op="accept", batch=64, rows=5, **_logits(151936, "bf16", 1.0, 1.0)),
        dict(name="accept-b256", op="accept", batch=256, rows=9, **_logits(128256, "bf16", 0.7, 0.8)),
        # a vocabulary with one added token: rows that start at odd addresses
        dict(name="accept-b32-odd", op="accept", batch=32, rows=4, **_logits(32001, "bf16", 0.5, 1.0)),
        # deterministic decoding
        dict(name="accept-b8-greedy", op="accept", batch=8, rows=6, **_logits(128256, "bf16", 0.5, 0.0)),
        # one position of the drafter for a full server
        dict(name="sample-b256", op="sample", batch=256, **_logits(128256, "bf16", 0.0, 0.8)),
        # a burst of requests matched against the group index
        dict(name="route-b1024", op="route", batch=1024, groups=16384, dim=384),
    ]


_TREES = ("2,2,1", "4,2,1", "3,2,2,1", "2,2,2,2", "1,1,1,1,1,1", "4,4,2", "8,2,1", "6,1,1,1,1")
_HEADS = ((32, 8), (28, 4), (64, 8), (16, 4), (32, 32), (40, 8))


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _draw_vocab(rng):
    return rng.choice(W.SWEEP_VOCABS) if rng.random() < 0.3 else _log_int(rng, 8000, 256000)


def _draw_logits(rng):
    t = 0.0 if rng.random() < 0.2 else round(rng.uniform(0.5, 1.2), 3)
    return _logits(_draw_vocab(rng), "f32" if rng.random() < 0.25 else "bf16",
                   rng.choice((0.1, 0.5, 0.7, 1.0, 2.0)), t)


def _draw_attn(rng, rows_of, max_rows):
    while True:
        hq, hkv = rng.choice(_HEADS)
        rows, batch = rows_of(rng), _log_int(rng, 1, 256)
        lo = _log_int(rng, 128, 8192)
        hi = _log_int(rng, lo, 16384)
        # at most the keys of the largest listed case, and the query rows a call takes
        if rows * (hq // hkv) <= max_rows and batch * hkv * (lo + hi) / 2 <= 256 * 8 * 9000 and lo > rows:
            return _attn(batch, rows, hq, hkv, rng.choice((16, 16, 32, 64)), "uniform", lo, hi)


def draw(rng):
    op = rng.choice(("step", "tree_step", "attn", "attn", "accept", "accept", "accept", "sample", "route"))
    chain = lambda r: 1 + _log_int(r, 1, 16)  # noqa: E731
    if op == "attn":
        return dict(op=op, **_draw_attn(rng, chain, 144))
    if op == "step":
        while True:
            c = dict(op=op, **_draw_attn(rng, chain, 144), **_draw_logits(rng))
            if c["batch"] * c["rows"] * c["vocab"] <= 256 * 9 * 128256:
                return c
    if op == "tree_step":
        tree = rng.choice(_TREES)
        n = len(W.tree_parents([int(x) for x in tree.split(",")]))
        while True:
            c = dict(op=op, tree=tree, **_draw_attn(rng, lambda r: n, 1024), **_draw_logits(rng))
            if c["batch"] * n * c["vocab"] <= 1 << 28:
                return c
    if op == "accept":
        while True:
            c = dict(op=op, batch=_log_int(rng, 1, 512), rows=chain(rng), **_draw_logits(rng))
            if c["batch"] * c["rows"] * c["vocab"] <= 256 * 9 * 128256:
                return c
    if op == "sample":
        return dict(op=op, batch=_log_int(rng, 1, 512), **_draw_logits(rng))
    return dict(op=op, batch=_log_int(rng, 1, 4096), groups=_log_int(rng, 100, 32768),
                dim=rng.choice((384, 384, 256, 128)))


# --------------------------------------------------------------------------
# inputs
# --------------------------------------------------------------------------
def _workload(case, seed):
    ctx = {"const": ("const", case.get("lo", 64)), "uniform": ("uniform", case.get("lo"), case.get("hi")),
           "lognormal": ("lognormal", 2048, 0.6, case.get("lo"), case.get("hi"))}[case.get("ctx", "const")]
    kw = dict(batch=case["batch"], vocab=case.get("vocab", 32000), logit_dtype=case.get("dtype", "bf16"),
              draft_sigma=case.get("sigma", 1.0), temperatures=(case.get("temperature", 1.0),),
              n_q_heads=case.get("hq", 8), n_kv_heads=case.get("hkv", 8), head_dim=D, ctx=ctx,
              page_size=case.get("page", 16), cell=seed)
    if "tree" in case:
        return W.TreeWorkload(wid=31, name="case", branching=tuple(int(x) for x in case["tree"].split(",")), **kw)
    return W.Workload(wid=30, name="case", n_draft=case.get("rows", 1) - 1,
                      contiguous=case["batch"] == 1, **kw)


def _new_rows(case, w, seed):
    """The K and V rows of the verify positions, as the target's layer has just produced them."""
    shape = (case["batch"], case["rows"], case["hkv"], D)
    g = torch.Generator(device=DEVICE).manual_seed(5_000_000 + seed)
    return [torch.randn(shape, generator=g, device=DEVICE).to(torch.bfloat16) for _ in range(2)]


def _fixed_pool(a, case):
    """The pools of a server have a fixed number of pages, whatever the contexts: room for every request's longest."""
    pages = case["batch"] * -(-case["hi"] // case["page"])
    for p in ("k_pages", "v_pages"):
        pool = torch.zeros((pages, *a[p].shape[1:]), dtype=a[p].dtype, device=DEVICE)
        pool[:a[p].shape[0]] = a[p]
        a[p] = pool
    return a


def prepare(case, seed):
    op = case["op"]
    if op == "route":
        inp = W.route_inputs(W.RouteWorkload(30, "case", case["batch"], case["groups"], case["dim"]), DEVICE, seed=seed)
        # the group index changes slowly: its norms are kept beside it
        return dict(case=case, inv_norms=binding.cs_route_norms(inp["centroids"]), **inp)
    w, s = _workload(case, seed), dict(case=case)
    if op in ("attn", "step"):
        s["attn"] = W.attention_inputs(w, DEVICE)
    if op == "tree_step":
        s["attn"] = W.tree_attention_inputs(w, DEVICE)
        s["acc"] = W.tree_accept_inputs(w, case["temperature"], DEVICE)
    if op in ("accept", "step"):
        s["acc"] = W.accept_inputs(w, case["temperature"], DEVICE)
    if op in ("step", "tree_step"):
        _fixed_pool(s["attn"], case)
        s["new_k"], s["new_v"] = _new_rows(case, w, seed)
    if op == "sample":
        g = torch.Generator(device=DEVICE).manual_seed(seed)
        dt = torch.float32 if case["dtype"] == "f32" else torch.bfloat16
        z = torch.randn((case["batch"], case["vocab"]), generator=g, device=DEVICE) * 3.0
        s["logits"] = z.to(dt)
        s["uniforms"] = torch.rand((case["batch"],), generator=g, device=DEVICE)
    return s


# --------------------------------------------------------------------------
# one pass
# --------------------------------------------------------------------------
def run(state):
    case = state["case"]
    op = case["op"]
    if op == "route":
        group, best, score = binding.cs_route(state["emb"], state["centroids"], state["inv_norms"], W.ROUTE_TAU)
        return dict(group=group, best=best, score=score)
    if op == "sample":
        return dict(tokens=binding.cs_sample(state["logits"], state["uniforms"], case["temperature"]))
    out = {}
    a = state.get("attn")
    if op in ("step", "tree_step"):
        binding.cs_kv_append(state["new_k"], state["new_v"], a["k_pages"], a["v_pages"], a["page_table"],
                             a["ctx_lens"])
    if op in ("attn", "step"):
        out["out"] = binding.cs_verify_attention(a["q"], a["k_pages"], a["v_pages"], a["page_table"], a["ctx_lens"],
                                                 case["rows"] - 1)
    elif op == "tree_step":
        out["out"] = binding.cs_tree_verify_attention(a["q"], a["k_pages"], a["v_pages"], a["page_table"],
                                                      a["ctx_lens"], a["parents"])
    if op == "attn":
        return out
    c, T = state["acc"], case["temperature"]
    draft = c["draft"] if T > 0 else None
    if op == "tree_step":
        out["tokens"], out["path"], out["n"] = binding.cs_tree_accept(c["target"], draft, c["parents"],
                                                                      c["node_tokens"], c["uniforms"], T)
    else:
        out["tokens"], out["n"] = binding.cs_spec_accept(c["target"], draft, c["draft_tokens"], c["uniforms"], T)
    if op == "accept":
        return out
    # the next step's context lengths (the scheduler keeps this step's)
    out["ctx_lens"] = a["ctx_lens"].clone()
    if op == "tree_step":
        binding.cs_kv_commit_tree(a["k_pages"], a["v_pages"], a["page_table"], out["ctx_lens"], out["path"], out["n"])
    else:
        binding.cs_kv_commit(out["ctx_lens"], out["n"], case["rows"] - 1)
    out["k_pages"], out["v_pages"] = a["k_pages"], a["v_pages"]
    return out


# --------------------------------------------------------------------------
# what a pass cannot do without
# --------------------------------------------------------------------------
def _mean_ctx(case):
    if case["ctx"] == "lognormal":
        return 2048 * math.exp(0.18)
    return (case["lo"] + case["hi"]) / 2


def _accept_rate(case):
    """Chance that one drafted token is accepted: logits that differ by N(0, s^2) at the temperature overlap
    by 2 Phi(-s / 2) (the arg max of a greedy call agrees about as often as at T = 1)."""
    return math.erfc(case["sigma"] / (case["temperature"] or 1.0) / (2 * math.sqrt(2)))


def work(case):
    op, B = case["op"], case["batch"]
    if op == "route":
        n, d = case["groups"], case["dim"]
        return dict(bytes=2 * d * (B + n) + 4 * n + 12 * B, flops=2 * B * n * d)
    nbytes = flops = 0
    if op in ("attn", "step", "tree_step"):
        L, rows, hq, hkv = _mean_ctx(case), case["rows"], case["hq"], case["hkv"]
        nbytes += B * L * hkv * D * 4 + 2 * B * rows * hq * D * 2 + 4 * B * math.ceil(L / case["page"])
        flops += 4 * B * rows * hq * D * L
        if op != "attn":
            nbytes += 2 * 2 * B * rows * hkv * D * 2   # the appended rows, read and written
    if op == "attn":
        return dict(bytes=nbytes, flops=flops)
    V, s = case["vocab"], 4 if case["dtype"] == "f32" else 2
    # The rule reads a request's rows up to its first rejection: per
    # position one target row and, sampling, one draft row.
    if op == "sample":
        rows = 1.0
    else:
        a = _accept_rate(case)
        depth = len(case["tree"].split(",")) if "tree" in case else case["rows"] - 1
        reach = [a ** i for i in range(depth + 1)]   # chance that the walk comes to depth i
        rows = sum(reach) + (sum(reach[:-1]) if case["temperature"] > 0 else 0.0)
    nbytes += B * rows * V * s
    flops += 4 * B * rows * V
    return dict(bytes=nbytes, flops=flops)


# --------------------------------------------------------------------------
# the results
# --------------------------------------------------------------------------
def tolerance(case):
    op = case["op"]
    if op == "route":
        # fp32 sums of 384 bf16 products (about 3e-7 off 64 bits); a near-tie may pick the other of two groups
        return dict(rel=2e-6, max=1e-5, differ=0.005)
    # token ids: a uniform that falls within rounding of a CDF edge may take the neighbouring id
    differ = 0.0 if case.get("temperature") == 0.0 else 0.01
    if op in ("accept", "sample"):
        return dict(rel=0.0, differ=differ)
    # bf16 outputs of fp32 sums: about 1.7e-3 off 64 bits, half an ulp (2^-9) at most for each value
    return dict(rel=6e-3, max=2e-2, differ=differ)


def _attention_exact(a, case, ancestors=None):
    """Attention of one request after another in 64 bits: q [B, R, Hq, D] over the paged K and V."""
    q, out = a["q"], torch.empty(a["q"].shape, dtype=torch.float64, device=DEVICE)
    R, hq, hkv = case["rows"], case["hq"], case["hkv"]
    ps = a["k_pages"].shape[2]
    for b, L in enumerate(a["ctx_lens"].tolist()):
        pages = a["page_table"][b, :-(-L // ps)].long()
        k, v = (a[p][pages].permute(1, 0, 2, 3).reshape(hkv, -1, D)[:, :L].double() for p in ("k_pages", "v_pages"))
        seen = torch.ones((R, L), dtype=torch.bool, device=DEVICE)
        seen[:, L - R:] = torch.ones((R, R), dtype=torch.bool, device=DEVICE).tril() if ancestors is None else ancestors
        x = q[b].double().permute(1, 0, 2).reshape(hkv, hq // hkv * R, D)
        s = torch.einsum("hrd,hld->hrl", x, k) / math.sqrt(D)
        s.masked_fill_(~seen.repeat(hq // hkv, 1)[None], -math.inf)
        o = torch.einsum("hrl,hld->hrd", torch.softmax(s, dim=-1), v)
        out[b] = o.reshape(hq, R, D).permute(1, 0, 2)
    return out


def exact(case, seed):
    op = case["op"]
    if op in ("accept", "sample"):
        return None   # token ids and counts
    s = prepare(case, seed)
    if op == "route":
        e, c = s["emb"].double(), s["centroids"].double()
        cos = (e / e.norm(dim=1, keepdim=True)) @ (c / c.norm(dim=1, keepdim=True)).T
        return dict(group=None, best=None, score=cos.max(dim=1).values)
    a = s["attn"]
    if op in ("step", "tree_step"):   # the appended rows take their slots first
        R, ps = case["rows"], a["k_pages"].shape[2]
        pos = a["ctx_lens"][:, None].long() - R + torch.arange(R, device=DEVICE)[None]
        page = torch.gather(a["page_table"].long(), 1, pos // ps)
        for pool, new in (("k_pages", "new_k"), ("v_pages", "new_v")):
            a[pool][page, :, pos % ps] = s[new]
    anc = None
    if op == "tree_step":
        par = a["parents"][0].tolist()
        anc = torch.eye(len(par), dtype=torch.bool, device=DEVICE)
        for c in range(1, len(par)):
            anc[c] |= anc[par[c]]
    out = dict(out=_attention_exact(a, case, anc))
    if op == "step":
        out.update(tokens=None, n=None, ctx_lens=None, k_pages=None, v_pages=None)
    elif op == "tree_step":
        out.update(tokens=None, path=None, n=None, ctx_lens=None, k_pages=None, v_pages=None)
    return out
