"""What the PLD+ library is timed on: decode steps, generation loops, drafting, verification
and head identification, each through the public entry points of the Python binding.

Contexts are text-like: token ids follow Zipf's law (a few ids are most of a text, as in any
language or code), and an output copies spans of its prompt, which is what PLD+ drafts from.
So x_t, the token looked up, is sometimes a word seen once before and sometimes one that
occurs thousands of times.  Hidden rows are N(0, 1) with copied positions close to their
sources, attention rows softmax-like with mass on the copy source, logits N(0, 1) with the
next token of the ground truth holding most of the probability.  Lengths are ragged.
"""
import math

import numpy as np
import torch

import paper_2412_01447_gb300 as pk

CAND_CAP = 1024          # candidate list capacity per sequence, as in the benchmark
COPY_NOISE = 0.1         # a copied position's hidden row against its source's


def listed():
    return [
        # one user, a short prompt, fp32 artifacts and logits: latency and launches
        dict(name="step_b1_ctx512_f32", op="step", calls="fused", B=1, ctx=512, V=32000, K=10, logits="f32",
             d=4096, h="f32", R=0, layout="key", n_sel=0, agg="max", ngram=3),
        # a small batch through the separate calls, hidden ranking
        dict(name="step_b8_ctx4k", op="step", calls="separate", B=8, ctx=4096, V=32000, K=10, logits="bf16",
             d=4096, h="bf16", R=0, layout="key", n_sel=0, agg="max", ngram=3),
        # a mid-size serving batch, one-launch drafting, a wider model
        dict(name="step_b64_ctx16k", op="step", calls="fused", B=64, ctx=16384, V=32000, K=16, logits="bf16",
             d=5120, h="bf16", R=0, layout="key", n_sel=0, agg="max", ngram=3),
        # attention ranking on 32 selected heads of 128, rows as the attention wrote them
        dict(name="step_b32_ctx8k_attn", op="step", calls="separate", B=32, ctx=8192, V=128256, K=10, logits="bf16",
             d=0, h="bf16", R=128, layout="head", n_sel=32, agg="max", ngram=3),
        # Eq. 1 as printed (unigram match): hundreds of candidates a sequence, both rankings
        dict(name="step_b16_ctx32k_eq1", op="step", calls="separate", B=16, ctx=32768, V=32000, K=10, logits="bf16",
             d=4096, h="bf16", R=128, layout="key", n_sel=0, agg="max", ngram=1),
        # drafting of the benchmark's batch in one launch, scanning the contexts, both rankings
        dict(name="draft_b128_ctx32k", op="draft", calls="fused", B=128, ctx=32768, V=128256, K=12, logits="bf16",
             d=4096, h="bf16", R=128, layout="key", n_sel=0, agg="max", ngram=3),
        # two users with a whole book each
        dict(name="draft_b2_ctx128k", op="draft", calls="fused", B=2, ctx=131072, V=128256, K=12, logits="bf16",
             d=4096, h="bf16", R=0, layout="key", n_sel=0, agg="max", ngram=3),
        # the benchmark's batch from prefill on: token index, first draft, 8 steps that verify
        # greedily and draft again, both rankings
        dict(name="generate_b128_ctx32k", op="generate", mode="greedy", B=128, ctx=32768, V=128256, K=12,
             logits="bf16", d=4096, h="bf16", R=128, layout="key", n_sel=0, agg="max", ngram=3, steps=8),
        # the same with sampling at T = 1, a smaller batch
        dict(name="generate_b16_ctx8k_sampled", op="generate", mode="sample", B=16, ctx=8192, V=128256, K=10,
             logits="bf16", d=4096, h="bf16", R=0, layout="key", n_sel=0, agg="max", ngram=3, steps=8),
        # verification of the benchmark's batch: the logits are the bytes of a decode step
        dict(name="verify_b128_v128256", op="verify", mode="greedy", B=128, V=128256, K=12, logits="bf16"),
        # a vocabulary with one added token: rows that are not a whole number of 16 bytes
        dict(name="verify_b64_v32001", op="verify", mode="greedy", B=64, V=32001, K=10, logits="bf16"),
        # picking the induction heads of a 32-layer, 32-head model, offline
        dict(name="identify_b32_r1024_ctx4k", op="identify", B=32, ctx=4096, V=32000, R=1024, top=32, logits="bf16"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["step", "step", "step", "draft", "generate", "verify", "verify", "identify"])
    logits = rng.choice(["bf16", "bf16", "f32"])
    V = _log(rng, 2000, 160000)
    if rng.random() < 0.6:
        V = (V + 63) // 64 * 64
    K = rng.randint(3, 20)
    if op == "verify":
        B = _log(rng, 1, 192)
        while B * (K + 1) * V * 4 > 400e6:
            B = max(1, B // 2)
        return dict(op=op, mode=rng.choice(["greedy", "sample"]), B=B, V=V, K=K, logits=logits)
    if op == "identify":
        ctx, R = _log(rng, 400, 32768), rng.choice([32, 72, 128, 256, 1000, 1024])
        B = max(1, min(_log(rng, 1, 128), int(500e6 / (ctx * R * 4))))
        return dict(op=op, B=B, ctx=ctx, V=V, R=R, top=min(32, R), logits=logits)
    calls = "fused" if op != "step" else rng.choice(["fused", "separate"])
    B, ctx = _log(rng, 1, 128), _log(rng, 300, 65536)
    h = rng.choice(["bf16", "bf16", "f32"])
    kinds = rng.choice(["hidden", "attention", "both"])
    d = 0 if kinds == "attention" else rng.choice([64, 512, 1000, 2048, 4096, 5120, 8192])
    if d and calls == "separate" and rng.random() < 0.25:
        d -= 3                                                  # rows the fused call does not take
    R = 0 if kinds == "hidden" else rng.choice([8, 20, 32, 128, 144])
    while B * ctx * (4 * d + 4 * R) > 12e9:
        B, ctx = max(1, B // 2), max(300, ctx * 3 // 4)
    while B * (K + 1) * V * 4 > 200e6:
        B = max(1, B // 2)
    case = dict(op=op, B=B, ctx=ctx, V=V, K=K, logits=logits, d=d, h=h, R=R, layout=rng.choice(["key", "head"]),
                n_sel=rng.choice([0, R // 4]), agg=rng.choice(["max", "max", "sum"]), ngram=rng.choice([1, 2, 3, 3, 4]))
    if op == "generate":
        case["mode"], case["steps"] = rng.choice(["greedy", "sample"]), rng.randint(2, 6)
        while B * V * 64 > 1.2e9:
            B = max(1, B // 2)
        case["B"] = B
    else:
        case["calls"] = calls
    return case


# ----------------------------------------------------------------------------
# inputs
# ----------------------------------------------------------------------------
def _dtype(name):
    return {"f32": torch.float32, "bf16": torch.bfloat16}[name]


def _zipf(V):
    p = 1.0 / (np.arange(V) + 2.7)                              # Zipf-Mandelbrot
    return p / p.sum()


def _stream(case, gen, total):
    """Tokens [B, total] (int64) and, for copied output positions, their source (else -1).
    The first five eighths are prompt; after it segments of 2 to 32 tokens are copies of
    prompt spans with probability 0.8, else fresh text."""
    B, P, dev = case["B"], max(64, case["ctx"] * 5 // 8), "cuda"
    cdf = torch.from_numpy(np.cumsum(_zipf(case["V"]))).to(dev)
    names = torch.randperm(case["V"], generator=gen, device=dev)
    tok = torch.empty((B, total), dtype=torch.int64, device=dev)
    for b in range(B):
        u = torch.rand(total, generator=gen, device=dev, dtype=torch.float64)
        tok[b] = names[torch.searchsorted(cdf, u).clamp(max=case["V"] - 1)]
    n_seg = (total - P) // 2 + 2
    lens = torch.randint(2, 33, (B, n_seg), generator=gen, device=dev)
    ends = lens.cumsum(1)
    pos = torch.arange(total - P, device=dev).expand(B, -1).contiguous()
    seg = torch.searchsorted(ends, pos, right=True)
    start = (ends - lens).gather(1, seg)
    s0 = (torch.rand((B, n_seg), generator=gen, device=dev) * (P - 34)).long() + 1
    copied = (torch.rand((B, n_seg), generator=gen, device=dev) < 0.8).gather(1, seg)
    src = torch.full((B, total), -1, dtype=torch.int64, device=dev)
    src[:, P:] = torch.where(copied, s0.gather(1, seg) + pos - start, torch.full_like(seg, -1))
    tok = torch.where(src >= 0, tok.gather(1, src.clamp(min=0)), tok)
    return tok, src


def _lengths(case, gen):
    lo = case["ctx"] - case["ctx"] // 4
    return torch.randint(lo, case["ctx"] + 1, (case["B"],), generator=gen, device="cuda").to(torch.int32)


def _hidden(case, src, rows, gen):
    B, d = case["B"], case["d"]
    H = torch.empty((B, rows, d), dtype=_dtype(case["h"]), device="cuda")
    for b in range(B):
        H[b].normal_(generator=gen)
        p = torch.nonzero(src[b, 1:rows] >= 0)[:, 0] + 1
        noise = torch.empty((p.numel(), d), dtype=torch.float32, device="cuda").normal_(generator=gen)
        H[b, p - 1] = (H[b, src[b, p] - 1].float() + COPY_NOISE * noise).to(H.dtype)
    return H


def _attention(case, L, src, keys, gen):
    """[B, R, keys] probabilities of query t-1; a quarter of the heads look at x_t's source."""
    B, R = case["B"], case["R"]
    shape = (B, keys, R) if case["layout"] == "key" else (B, R, keys)
    A = torch.empty(shape, dtype=_dtype(case["h"]), device="cuda")
    s = src.gather(1, (L.long() - 1)[:, None])[:, 0]
    for b in range(B):
        x = torch.empty(shape[1:], dtype=torch.float32, device="cuda").normal_(generator=gen).exp_()
        if s[b] >= 0:
            (x if case["layout"] == "key" else x.t())[s[b], ::4] *= math.exp(6.0)
        A[b] = (x / (keys * math.exp(0.5))).to(A.dtype)
    return A.transpose(1, 2) if case["layout"] == "key" else A


def _plant(case, targets, gen):
    """Logits [B, K+1, V]: N(0, 1), the target with most of the probability."""
    shape = (case["B"], case["K"] + 1, case["V"])
    x = torch.empty(shape, dtype=_dtype(case["logits"]), device="cuda").normal_(generator=gen)
    return x.scatter_(2, targets[..., None], math.log(case["V"]) + 2.5)


def _next_tokens(tok, L, K):
    at = L.long()[:, None] + torch.arange(K + 1, device="cuda")[None]
    return tok.gather(1, at.clamp(max=tok.shape[1] - 1))


def _ints(*shape):
    return torch.full(shape, -1, dtype=torch.int32, device="cuda")


def _zeros(n):
    return torch.zeros(n, dtype=torch.uint8, device="cuda")


def prepare(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    s = {"case": case, **{"identify": _prepare_identify, "verify": _prepare_verify}.get(case["op"], _prepare_context)(case, gen)}
    if case["op"] == "generate":
        _prepare_loop(case, s, gen)
    return s


def _prepare_verify(case, gen):
    B, K, V = case["B"], case["K"], case["V"]
    draft = torch.randint(0, V, (B, K), generator=gen, device="cuda")
    draft_len = torch.randint(max(1, K - 2), K + 1, (B,), generator=gen, device="cuda")
    accept = torch.randint(0, K + 1, (B,), generator=gen, device="cuda")
    targets = torch.randint(0, V, (B, K + 1), generator=gen, device="cuda")
    keep = torch.arange(K, device="cuda")[None] < accept[:, None]
    targets[:, :K] = torch.where(keep, draft, targets[:, :K])
    s = dict(logits=_plant(case, targets, gen), draft=draft.to(torch.int32), draft_len=draft_len.to(torch.int32),
             tokens=_ints(B, K + 1), accept=_ints(B), next=_ints(B))
    if case["mode"] == "sample":
        s["u"] = torch.rand((B, K + 1), generator=gen, device="cuda")
        s["ws"] = _zeros(pk.pldp_verify_sample_workspace_size(B, K, V, s["logits"].dtype))
    else:
        s["ws"] = _zeros(pk.pldp_verify_workspace_size(B, K, V))
    return s


def _prepare_identify(case, gen):
    B, R, ctx = case["B"], case["R"], case["ctx"]
    tok, src = _stream(case, gen, ctx)
    L = _lengths(case, gen)
    return dict(ids=tok.to(torch.int32), pos=L - 1, counts=_ints(R), r_star=_ints(B), rows=_ints(case["top"]),
                A=_attention(dict(case, h=case["logits"], layout="head"), L, src, (ctx + 7) // 8 * 8, gen))


def _prepare_context(case, gen):
    B, K = case["B"], case["K"]
    cap = (case["ctx"] + (K + 1) * case.get("steps", 1) + 7) // 8 * 8
    tok, src = _stream(case, gen, cap + K + 1)
    L = _lengths(case, gen)
    ids = tok[:, :cap].to(torch.int32).contiguous()
    ids[torch.arange(cap, device="cuda")[None] >= L[:, None]] = 0
    s = dict(tok=tok, ids=ids, len0=L, seq_len=L.clone(), cand=_ints(B, CAND_CAP), count=_ints(B), match=_ints(B),
             draft=_ints(B, K), draft_len=_ints(B), accept=_ints(B), next=_ints(B), keep=_ints(B), H=None, A=None)
    if case["d"]:
        s["H"] = _hidden(case, src, cap, gen)
        s.update(best_h=_ints(B), score_h=torch.zeros((B, CAND_CAP), device="cuda"), top_h=torch.zeros(B, device="cuda"))
    if case["R"]:
        s["A"] = _attention(case, L, src, cap, gen)
        s.update(best_a=_ints(B), score_a=torch.zeros((B, CAND_CAP), device="cuda"), top_a=torch.zeros(B, device="cuda"))
    s["sel"] = (torch.randperm(case["R"], generator=gen, device="cuda")[:case["n_sel"]].to(torch.int32)
                if case["R"] and case["n_sel"] else None)
    if case["op"] == "step":
        s["logits"] = _plant(case, _next_tokens(tok, L, K), gen)
        s["ws"] = _zeros(pk.pldp_verify_workspace_size(B, K, case["V"]))
    if case.get("calls") == "fused":
        s["draft_ws"] = _zeros(pk.pldp_draft_workspace_size(B))
    return s


def _prepare_loop(case, s, gen):
    """The index's memory and each step's logits: the loop run once, the logits of each step
    following the ground truth from where the step before left the contexts."""
    B, K, V = case["B"], case["K"], case["V"]
    s["index"] = torch.empty(pk.pldp_index_size(B, V), dtype=torch.uint8, device="cuda")
    if case["mode"] == "sample":
        s["u"] = [torch.rand((B, K + 1), generator=gen, device="cuda") for _ in range(case["steps"])]
        s["ws"] = _zeros(pk.pldp_verify_sample_draft_workspace_size(B, K, V, _dtype(case["logits"])))
    else:
        s["ws"] = _zeros(pk.pldp_verify_workspace_size(B, K, V))
    s["logits"] = []
    _begin(s)
    for i in range(case["steps"]):
        s["logits"].append(_plant(case, _next_tokens(s["tok"], s["seq_len"], K), gen))
        _advance(s, i)


# ----------------------------------------------------------------------------
# a pass
# ----------------------------------------------------------------------------
def _rankings(s, scores=True):
    """The ranking arguments of the fused calls."""
    case, kw = s["case"], {}
    if case["d"]:
        kw.update(H=s["H"], best_h=s["best_h"])
        if scores:
            kw.update(h_scores=s["score_h"], best_h_score=s["top_h"])
    if case["R"]:
        kw.update(A=s["A"], best_a=s["best_a"], row_idx=s["sel"], agg=_agg(case))
        if scores:
            kw.update(a_scores=s["score_a"], best_a_score=s["top_a"])
    kw["draft_from"] = "hidden" if case["d"] else "attention"
    return kw


def _agg(case):
    return pk.PLDP_AGG_SUM if case["agg"] == "sum" else pk.PLDP_AGG_MAX


def _draft(s):
    case, ids, L = s["case"], s["ids"], s["seq_len"]
    if case["calls"] == "fused":
        pk.pldp_draft_step(ids, L, 1, case["ngram"], s["cand"], s["count"], s["match"], case["K"], s["draft"],
                           s["draft_len"], s["draft_ws"], **_rankings(s))
        return
    pk.pldp_find_candidates(ids, L, 1, case["ngram"], s["cand"], s["count"], s["match"])
    if case["d"]:
        pk.pldp_rank_hidden(s["H"], L, s["cand"], s["count"], s["best_h"], scores=s["score_h"], best_score=s["top_h"])
    if case["R"]:
        pk.pldp_rank_attention(s["A"], L, s["cand"], s["count"], s["best_a"], row_idx=s["sel"], agg=_agg(case),
                               scores=s["score_a"], best_score=s["top_a"])
    pk.pldp_extract_draft(ids, L, s["best_h"] if case["d"] else s["best_a"], s["draft"], s["draft_len"])


def _begin(s):
    """Prefill: the contexts as the prompts left them, their index and the first draft."""
    case = s["case"]
    s["seq_len"].copy_(s["len0"])
    pk.pldp_index_build(s["ids"], s["seq_len"], case["V"], s["index"])
    pk.pldp_draft_step(s["ids"], s["seq_len"], 1, case["ngram"], s["cand"], s["count"], s["match"], case["K"],
                       s["draft"], s["draft_len"], None, index=s["index"], V=case["V"], **_rankings(s, scores=False))


def _advance(s, i):
    """One decode step: this step's draft verified, the next one made."""
    case = s["case"]
    args = (s["ids"], s["seq_len"], 1, case["ngram"], s["cand"], s["count"], s["match"], s["draft"], s["draft_len"],
            s["index"])
    if case["mode"] == "sample":
        pk.pldp_verify_sample_draft(s["logits"][i], s["u"][i], s["draft"], s["draft_len"], s["accept"], s["next"],
                                    s["ws"], *args, kv_keep_len=s["keep"], **_rankings(s, scores=False))
    else:
        pk.pldp_verify_greedy_draft(s["logits"][i], s["draft"], s["draft_len"], s["accept"], s["next"], s["ws"], *args,
                                    kv_keep_len=s["keep"], **_rankings(s, scores=False))


def run(s):
    case = s["case"]
    if case["op"] == "verify":
        if case["mode"] == "sample":
            pk.pldp_verify_sample(s["logits"], s["u"], s["draft"], s["draft_len"], s["accept"], s["next"], s["ws"],
                                  sampled=s["tokens"])
        else:
            pk.pldp_verify_greedy(s["logits"], s["draft"], s["draft_len"], s["accept"], s["next"], s["ws"],
                                  argmax=s["tokens"])
        return [s["tokens"], s["accept"], s["next"]]
    if case["op"] == "identify":
        s["counts"].zero_()
        pk.pldp_identify_heads(s["ids"], s["pos"], s["A"], s["counts"], r_star=s["r_star"])
        pk.pldp_top_heads(s["counts"], case["top"], s["rows"])
        return [s["counts"], s["r_star"], s["rows"]]
    if case["op"] == "generate":
        _begin(s)
        for i in range(case["steps"]):
            _advance(s, i)
        return {k: s[k] for k in ("ids", "seq_len", "draft", "draft_len", "accept", "next", "keep", "count", "match")}
    if case["op"] == "step":
        s["seq_len"].copy_(s["len0"])                          # a request taken up again where its prompt ended
    _draft(s)
    names = ["cand", "count", "match", "draft", "draft_len"]
    if case["op"] == "step":
        pk.pldp_verify_greedy(s["logits"], s["draft"], s["draft_len"], s["accept"], s["next"], s["ws"], ids=s["ids"],
                              seq_len=s["seq_len"], kv_keep_len=s["keep"])
        names += ["ids", "seq_len", "accept", "next", "keep"]
    names += [k for k in ("best_h", "score_h", "top_h", "best_a", "score_a", "top_a") if k in s]
    return {k: s[k] for k in names}


# ----------------------------------------------------------------------------
# what a pass cannot do without, and what its results may differ by
# ----------------------------------------------------------------------------
def _expected_candidates(case):
    """Candidates per sequence: the occurrences of a Zipf token for the unigram match (listed
    up to the capacity), about two for longer suffixes of copied text."""
    if case["ngram"] > 1:
        return 2.0
    p = _zipf(case["V"])
    return float((p * np.minimum(CAND_CAP, 0.875 * case["ctx"] * p)).sum())


def work(case):
    es = 2 if case["logits"] == "bf16" else 4
    if case["op"] == "identify":
        p = 0.875 * case["ctx"]
        return {"bytes": case["B"] * p * (case["R"] * es + 4) + 4 * case["R"], "flops": case["B"] * p * case["R"]}
    B, K, V = case["B"], case["K"], case["V"]
    verify = B * (K + 1) * V * es
    if case["op"] == "verify":
        return {"bytes": verify, "flops": verify / es * (1 if case["mode"] == "greedy" else 3)}
    hs = 2 if case["h"] == "bf16" else 4
    n = _expected_candidates(case)
    rank = B * ((n + 1) * case["d"] * hs + n * (case["n_sel"] or case["R"]) * hs + n * 8 + K * 4)
    flops = B * n * (6 * case["d"] + case["R"])
    scan = B * 0.875 * case["ctx"] * 4
    if case["op"] == "draft":
        return {"bytes": scan + rank, "flops": flops}
    if case["op"] == "step":
        return {"bytes": scan + rank + verify, "flops": flops + verify / es}
    steps = case["steps"]
    return {"bytes": 2 * scan + (steps + 1) * rank + steps * verify, "flops": (steps + 1) * flops + steps * verify / es}


def tolerance(case):
    # Scores are cosines and attention sums added up in 32 bits (attention maxima are exact);
    # against 64 bits they measure up to 1.5e-7, more where a single cosine near 0 is all there
    # is to compare, and in another order as much again.  Drawn tokens may differ where a
    # uniform lies within rounding of a boundary.
    if case["op"] in ("step", "draft"):
        return {"rel": 2e-6, "max": 1e-5}
    return {"differ": 0.002} if case.get("mode") == "sample" else "exact"


def exact(case, seed):
    """The scores in 64 bits, from the definitions; whole-number outputs have no such value."""
    if case["op"] not in ("step", "draft"):
        return None
    s = prepare(dict(case), seed)
    out = {k: None for k in ("cand", "count", "match", "draft", "draft_len")}
    if case["op"] == "step":
        out.update({k: None for k in ("ids", "seq_len", "accept", "next", "keep")})
    for k in ("best_h", "score_h", "top_h", "best_a", "score_a", "top_a"):
        if k in s:
            out[k] = None if k.startswith("best") else torch.zeros_like(s[k], dtype=torch.float64)
    for b in range(case["B"]):
        t = int(s["len0"][b]) - 1
        x = s["ids"][b, :t + 1]
        same = x[:t] == x[t]
        found = torch.nonzero(same)[:, 0]
        for n in range(1, case["ngram"]):
            longer = found[(found >= n)]
            longer = longer[x[longer - n] == x[t - n]]
            if not longer.numel():
                break
            found = longer
        j = found[:CAND_CAP]
        if case["d"]:
            q = s["H"][b, t - 1].double()
            row = s["H"][b, (j - 1).clamp(min=0)].double()
            c = (row @ q) / (row.norm(dim=1) * q.norm())
            out["score_h"][b, :j.numel()] = torch.where(j > 0, c, torch.full_like(c, -math.inf))
            out["top_h"][b] = out["score_h"][b, :j.numel()].max() if j.numel() else -math.inf
        if case["R"]:
            a = s["A"][b, :, j].double()
            a = a if s["sel"] is None else a[s["sel"].long()]
            c = a.sum(0) if case["agg"] == "sum" else a.amax(0)
            out["score_a"][b, :j.numel()] = c
            out["top_a"][b] = c.max() if j.numel() else -math.inf
    return out
