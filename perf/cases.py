"""Performance cases of the ranking path: what a serving process asks of the library, request by request, and the offline
pass over its corpus, through the public wrapper (`binding.Lime`).

A case of kind "rank" is one batch of requests through the online path: ragged offsets, history lookup, (optionally) the
links contextualised per user, the stacked XOR layers, then the scores of every user's candidates.  A case of kind
"offline" is the candidate -> link precompute over a corpus, which a deployment repeats whenever item embeddings change.

Fields of a "rank" case: the model (`dtype`, `d`, `H`, `ell`, `layers`, `phi`); the batch (`B` users with `n_min` .. `n_max`
history items and `c_min` .. `c_max` candidates each); the corpus (`V` rows, history ids Zipf(`zipf`)); how candidates
arrive, `cands`: "dense" (their embeddings and cached weights as streams), "ids" (a fixed number of ids per user into the
corpus caches) or "lists" (ids, lists of differing length); `head`: hidden widths of the interaction network, "" for the dot
product; `d_c`: context features per user for the contextualised links, 0 for the shared links; `raw`: the history is
looked up as stored and normalised by the first layer instead of by the lookup.
"""
import math

import numpy as np
import torch

from paper_2510_18239_b200 import binding

ES = {"f32": 4, "bf16": 2}

# the models: those of the named workloads, and those of the paper's table of hyper-parameters (three XOR layers)
BASE = dict(dtype="bf16", d=128, H=4, ell=32, layers=2, V=1_000_000, zipf=1.1)
LONG = dict(dtype="bf16", d=128, H=4, ell=64, layers=4, V=1_000_000, zipf=1.1)
PROD = dict(dtype="bf16", d=256, H=8, ell=64, layers=4, V=4_000_000, zipf=1.05)
TINY = dict(dtype="f32", d=64, H=2, ell=8, layers=1, V=768, zipf=0.0)
FP32 = dict(dtype="f32", d=64, H=2, ell=8, layers=2, V=200_000, zipf=1.1)
PUBLIC = dict(dtype="bf16", d=32, H=4, ell=16, layers=3, V=200_000, zipf=1.1)
INDUSTRIAL = dict(dtype="bf16", d=256, H=4, ell=32, layers=3, V=1_000_000, zipf=1.1)


def rank(model, B, n, c, cands, phi="softmax", head="", d_c=0, raw=False, **name):
    (n_min, n_max), (c_min, c_max) = n, c
    return dict(name, kind="rank", **model, phi=phi, B=B, n_min=n_min, n_max=n_max, c_min=c_min, c_max=c_max, cands=cands,
                head=head, d_c=d_c, raw=raw)


def offline(dtype, d, ell, M, **name):
    return dict(name, kind="offline", dtype=dtype, d=d, ell=ell, M=M)


def listed():
    return [
        # one request of one user, ranked on arrival: the latency of the whole chain of small launches
        rank(BASE, 1, (187, 187), (333, 333), "ids", name="one_request"),
        # the smallest named workload: fp32 storage, a handful of short histories
        rank(TINY, 4, (64, 64), (128, 128), "dense", name="tiny_fp32"),
        # the benchmark's workload, the ordinary batch of a ranking server
        rank(BASE, 256, (512, 512), (2048, 2048), "dense", name="bf16_baseline"),
        # the far end of the candidate sweep: ranking straight after a very wide retrieval
        rank(BASE, 64, (1024, 1024), (32768, 32768), "dense", name="candidate_sweep_32768"),
        # the far end of the history sweep: lifelong histories, four layers
        rank(LONG, 32, (32768, 32768), (1024, 1024), "ids", name="long_history_32768"),
        # the production-shaped batch, candidates by id from the caches of a 4M-item corpus
        rank(PROD, 1024, (1024, 4096), (8192, 8192), "ids", name="production_ragged"),
        # what retrieval hands over in earnest: lists of differing length, ragged histories (some users have none yet)
        rank(BASE, 100, (0, 1000), (20, 1500), "lists", raw=True, name="ragged_lists"),
        # links contextualised per user (Eq. 2) and the SiLU form of the attention
        rank(BASE, 128, (50, 700), (1024, 1024), "ids", phi="silu", d_c=32, name="contextual_silu"),
        # the paper's industrial model (d = 256, 32 links, histories to 1024) with its 96-wide interaction network
        rank(INDUSTRIAL, 64, (100, 1024), (500, 500), "ids", head="96", name="industrial_head"),
        # the paper's public-dataset model (d = 32, 16 links, histories to 256) with its three-layer interaction network
        rank(PUBLIC, 128, (10, 256), (200, 200), "ids", head="512,128,64", name="public_head"),
        # fp32 storage in an ordinary batch (exact scores wanted, e.g. for calibration or replay)
        rank(FP32, 64, (50, 1000), (1000, 1000), "ids", name="fp32_batch"),
        # the offline pass over a corpus of a million items
        offline("bf16", 128, 32, 1_000_000, name="offline_corpus"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw(rng):
    kind = rng.choice(["request", "batch", "batch", "wide", "long", "prod", "lists", "context", "industrial", "public", "fp32", "offline"])
    base = dict(rng.choice([BASE, LONG]), layers=rng.randint(1, 4))
    if kind == "request":
        n, c = _log(rng, 1, 2000), _log(rng, 1, 4000)
        return rank(base, rng.randint(1, 3), (n, n), (c, c), "ids")
    if kind == "batch":
        n, c = _log(rng, 16, 1500), _log(rng, 16, 4000)
        return rank(base, _log(rng, 4, 400), (rng.choice([0, n // 4, n]), n), (c, c), rng.choice(["dense", "ids"]),
                    phi=rng.choice(["softmax", "softmax", "softmax", "silu"]), raw=rng.random() < 0.25)
    if kind == "wide":
        n, c = _log(rng, 100, 2000), _log(rng, 4000, 32768)
        return rank(base, _log(rng, 1, 64), (n, n), (c, c), rng.choice(["dense", "ids"]))
    if kind == "long":
        n = _log(rng, 3000, 32768)
        return rank(dict(LONG, layers=rng.randint(2, 4)), _log(rng, 1, 32), (rng.choice([n // 2, n]), n), (1024, 1024), "ids")
    if kind == "prod":
        n = _log(rng, 64, 4096)
        return rank(PROD, _log(rng, 8, 900), (n // 4, n), (_log(rng, 100, 8192),) * 2, rng.choice(["dense", "ids"]))
    if kind == "lists":
        n, c = _log(rng, 16, 1500), _log(rng, 30, 4000)
        return rank(base, _log(rng, 4, 256), (0, n), (rng.randint(0, c // 2), c), "lists", raw=rng.random() < 0.5)
    if kind == "context":
        n, c = _log(rng, 16, 1500), _log(rng, 16, 4000)
        return rank(base, _log(rng, 4, 256), (n // 8, n), (c, c), rng.choice(["dense", "ids"]), phi=rng.choice(["softmax", "silu"]),
                    d_c=8 * rng.randint(1, 8))
    if kind == "industrial":
        n, c = _log(rng, 16, 1024), _log(rng, 16, 1500)
        return rank(INDUSTRIAL, _log(rng, 1, 64), (n // 8, n), (c, c), rng.choice(["dense", "ids"]), head=rng.choice(["", "96"]))
    if kind == "public":
        n, c = _log(rng, 8, 256), _log(rng, 8, 300)
        return rank(PUBLIC, _log(rng, 1, 200), (n // 8, n), (c, c), rng.choice(["dense", "ids"]), head=rng.choice(["", "512,128,64"]))
    if kind == "fp32":
        n, c = _log(rng, 8, 1000), _log(rng, 8, 2000)
        return rank(dict(FP32, layers=rng.randint(1, 3)), _log(rng, 1, 80), (n // 8, n), (c, c), rng.choice(["dense", "ids"]))
    dtype, d, ell = rng.choice([("bf16", 128, 32), ("bf16", 128, 64), ("bf16", 256, 64), ("bf16", 32, 16), ("f32", 64, 8)])
    return offline(dtype, d, ell, _log(rng, 1000, 2_000_000))


def draw(rng):
    most = max(_cost(c) for c in listed())
    while True:
        case = _draw(rng)
        if _cost(case) <= most:
            return case


# ---------------------------------------------------------------------------------------------------- inputs
class _Draws:
    """Seeded inputs, made on the GPU."""

    def __init__(self, seed, dtype):
        self.g = torch.Generator("cuda").manual_seed(seed)
        self.dtype = {"f32": torch.float32, "bf16": torch.bfloat16}[dtype]

    def normal(self, *shape, std=1.0, dtype=None):
        return (torch.randn(shape, generator=self.g, device="cuda", dtype=torch.float32) * std).to(dtype or self.dtype)

    def ints(self, lo, hi, n):
        return torch.randint(lo, hi + 1, (n,), generator=self.g, device="cuda", dtype=torch.int32)

    def lengths(self, lo, hi, n):
        """Uniform on [lo, hi], in pairs around the middle: the same total for every seed."""
        half = self.ints(lo, hi, n // 2)
        both = torch.cat([half, lo + hi - half, half.new_full((n % 2,), (lo + hi) // 2)])
        return both[torch.randperm(n, generator=self.g, device="cuda")]

    def zipf(self, n, V, s):
        """P(rank k) ~ k^-s, ranks scattered over the table's rows."""
        cdf = torch.arange(1, V + 1, device="cuda", dtype=torch.float64).pow_(-s).cumsum_(0)
        u = torch.rand(n, generator=self.g, device="cuda", dtype=torch.float64) * cdf[-1]
        rows = torch.randperm(V, generator=self.g, device="cuda")
        return rows[torch.searchsorted(cdf, u).clamp_(max=V - 1)].to(torch.int32)

    def ffn(self, *widths):
        return [(self.normal(a, b, std=a ** -0.5), self.normal(b, std=0.1, dtype=torch.float32)) for a, b in zip(widths, widths[1:])]


def prepare(case, seed):
    c, r = case, _Draws(seed, case["dtype"])
    d, ell = c["d"], c["ell"]
    dtype = binding.LIME_F32 if c["dtype"] == "f32" else binding.LIME_BF16
    if c["kind"] == "offline":
        lime = binding.Lime(d, 1 if d <= 128 else d // 128, ell, 1, dtype=dtype, gated_mlp=False)
        lime.set_weights(r.normal(ell, d), [{}])
        return dict(kind="offline", lime=lime, items=r.normal(c["M"], d, std=0.02))
    tiny = c["zipf"] == 0.0
    lime = binding.Lime(d, c["H"], ell, c["layers"], dtype=dtype,
                        phi=binding.LIME_PHI_SILU if c["phi"] == "silu" else binding.LIME_PHI_SOFTMAX)
    weights = [{k: r.normal(d, d, std=d ** -0.5) for k in ("Wq", "Wk", "Wv", "Wg", "Wu", "Wo")} for _ in range(c["layers"])]
    lime.set_weights(r.normal(ell, d, std=d ** -0.5 if tiny else 1.0), weights)
    s = dict(kind="rank", lime=lime, B=c["B"], cands=c["cands"], head=bool(c["head"]), raw=c["raw"], user_ctx=None, C=0,
             lengths=r.lengths(c["n_min"], c["n_max"], c["B"]))
    s["table"] = r.normal(c["V"], d, std=d ** -0.5 if tiny else 0.02)
    tokens = int(s["lengths"].sum())
    if tiny:                        # every row of the table is used once
        s["hist_ids"] = torch.randperm(c["V"], generator=r.g, device="cuda")[:tokens].to(torch.int32)
    else:
        s["hist_ids"] = r.zipf(tokens, c["V"], c["zipf"])
    if c["d_c"]:
        lime.set_context_mlp(c["d_c"], r.ffn(d + c["d_c"], d, d))
        s["user_ctx"] = r.normal(c["B"], c["d_c"])
    if c["head"]:
        lime.set_head(r.ffn(2 * d, *(int(w) for w in c["head"].split(",")), 1))
    if c["cands"] == "lists":
        s["cand_lengths"] = r.lengths(c["c_min"], c["c_max"], c["B"])
        total = int(s["cand_lengths"].sum())
    else:
        s["C"], total = c["c_max"], c["B"] * c["c_max"]
    ids = r.ints(0, c["V"] - 1, total)
    if c["cands"] == "dense":
        s["emb"] = s["table"][ids.long()]
        s["w"] = lime.precompute_candidate_links(s["emb"])
        s["ids"] = None
    else:
        s["emb"] = s["table"]
        s["w"] = lime.precompute_candidate_links(s["table"])
        s["ids"] = ids
    return s


def run(state):
    s, lime = state, state["lime"]
    if s["kind"] == "offline":
        return lime.precompute_candidate_links(s["items"])
    off = lime.lengths_to_offsets(s["lengths"])
    link_ctx = None if s["user_ctx"] is None else lime.contextualize_links(s["user_ctx"])
    if s["raw"]:
        link_states = lime.encode_user(lime.gather_history(s["table"], s["hist_ids"]), off, link_ctx)
    else:
        link_states = lime.encode_user_normalized(lime.gather_history_normalized(s["table"], s["hist_ids"]), off, link_ctx)
    cand_off = lime.lengths_to_offsets(s["cand_lengths"]) if s["cands"] == "lists" else None
    score = lime.score_candidates_head if s["head"] else lime.score_candidates
    logits = score(link_states, s["w"], s["emb"], C=s["C"], cand_off=cand_off, cand_ids=s["ids"])
    return {"link_states": link_states, "logits": logits}


# ---------------------------------------------------------------------------------------------------- work
def _distinct(n, V, s):
    """Expected number of distinct rows among n Zipf(s) ids over V rows."""
    p = np.arange(1, V + 1, dtype=np.float64) ** -s
    return float(-np.expm1(-n * (p / p.sum())).sum())


def work(case):
    c, es, d, ell = case, ES[case["dtype"]], case["d"], case["ell"]
    if c["kind"] == "offline":
        return {"bytes": c["M"] * es * (d + ell), "flops": 2.0 * c["M"] * d * ell}
    B, H, n = c["B"], c["H"], c["layers"]
    N, M = B * (c["n_min"] + c["n_max"]) / 2, B * (c["c_min"] + c["c_max"]) / 2
    # history: ids and each table row once; then 4 bytes of length and the link states per user
    rows = N if c["zipf"] == 0.0 else _distinct(N, c["V"], c["zipf"])
    size = 4 * N + es * d * rows + B * (4 + es * ell * d)
    # candidates: embedding and cached weights of each distinct one, the id where there is one, the logit
    distinct = M if c["cands"] == "dense" else c["V"] * -math.expm1(-M / c["V"])
    size += distinct * es * (d + ell) + M * (4 if c["cands"] == "dense" else 8)
    # XOR layers, links <- history: the history projected to keys and values, or those projections folded into the link
    # side (whichever is less work); the same choice for the history's queries and for its values through the GatedMLP
    flops = n * N * min(4 * ell * d + 4 * d * d, 4 * H * ell * d)
    update = min(2 * d * d + 2 * ell * d, 2 * H * ell * d) + min(2 * ell * d + 4 * d * d, 4 * H * ell * d) + 2 * d * d
    flops += (n - 1) * N * update
    # link rows: query, key, value, GatedMLP (the first layer's projections of shared links need no request)
    flops += B * ell * (n * 6 * d * d + (n if c["d_c"] else n - 1) * 6 * d * d)
    if c["d_c"]:
        flops += 2.0 * B * (c["d_c"] * d + ell * d * d)
    # scores: the mix of the link states and the dot product, or the network on the mix and the candidate
    if c["head"]:
        widths = [int(w) for w in c["head"].split(",")] + [1]
        flops += M * (2 * (ell + d) * widths[0] + sum(2 * a * b for a, b in zip(widths, widths[1:]))) + B * 2 * ell * d * widths[0]
    else:
        flops += M * 2 * (ell * d + d)
    return {"bytes": float(size), "flops": float(flops)}


def _cost(case):
    """Rough size of a case in bytes, at about 50 operations a byte; CUDA-core shapes count their operations in full."""
    w = work(case)
    slow = case["dtype"] == "f32" or case["d"] == 32
    return max(w["bytes"], w["flops"] / (5 if slow else 50))


def tolerance(case):
    if case["dtype"] == "f32":
        return {"rel": 1e-5}
    if case["kind"] == "offline":
        return {"rel": 5e-3}
    # every layer rounds its rows, operands, probabilities and GatedMLP product to bf16 once each
    return {"rel": 2e-2}
