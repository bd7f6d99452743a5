"""Performance cases of the MLA decode step: what is timed, on which inputs, against which values.

Each case is one call (or the few calls that always go together) through the
public binding ``paper_2607_27269_gb300.abi``, on synthetic inputs of the five
draft-layer shapes of ``paper_2607_27269_gb300.workloads``:

  step      one decode step of the converted layer (``DecodeStep``): append of
            the new entries, absorption, attention, combine, projections;
  attn      the attention core alone (``decode_attn`` + ``combine``);
  project   hidden states into the cache and the queries (``project_append``);
  out_proj  W_UV and W_O on the attention's output (``out_proj``);
  accept    acceptance statistics of draft against target logits;
  gqa       decode attention of the original GQA layer (``GqaStep``).

Sequence lengths are the evenly spaced quantiles of U[kv_lo, kv_hi] in a seeded
order, so that a case costs the same for every seed.  Everything else is drawn
on the GPU from the seed.  ``exact`` evaluates the same formulas in fp64 with
plain torch.
"""
from __future__ import annotations

import math

import torch

from paper_2607_27269_gb300 import abi

PAGE = 64

# Layer shapes: the four shapes of the workloads (a tiny layer, then the
# Qwen2.5-0.5B, Llama-3.2-1B and Llama-3.2-3B drafts).
LAYERS = {
    "tiny": dict(H=8, G=8, d_nope=64, d_rope=32, d_v=64, rank=128, hidden=0),
    "qwen05b": dict(H=14, G=2, d_nope=64, d_rope=64, d_v=64, rank=256, hidden=896),
    "llama1b": dict(H=32, G=8, d_nope=64, d_rope=64, d_v=64, rank=512, hidden=2048),
    "llama3b": dict(H=24, G=8, d_nope=128, d_rope=64, d_v=128, rank=512, hidden=3072),
}


def listed():
    return [
        # The smallest call: one proposal step of a tiny draft layer, one sequence; launches and latency are all.
        dict(name="step_tiny_b1", kind="step", layer="tiny", batch=1, q_len=1, kv_lo=256, kv_hi=256, paged=False,
             graph=True),
        # A proposal step of a small batch of equal lengths in a serving loop (replayed as a CUDA graph).
        dict(name="step_qwen_b16", kind="step", layer="qwen05b", batch=16, q_len=1, kv_lo=2048, kv_hi=2048,
             paged=False, graph=True),
        # The catch-up step of a big ragged paged batch: five new entries a sequence, everything included.
        dict(name="step_paged_b128", kind="step", layer="llama1b", batch=128, q_len=5, kv_lo=133, kv_hi=8197,
             paged=True, graph=False),
        # The attention core on a speculative chunk (gamma + 1 = 5 queries), contiguous equal lengths.
        dict(name="attn_chunk_b32", kind="attn", layer="llama1b", batch=32, q_len=5, kv_lo=4096, kv_hi=4096,
             paged=False),
        # The attention core on a few long documents, one query each.
        dict(name="attn_long_b8", kind="attn", layer="llama3b", batch=8, q_len=1, kv_lo=16384, kv_hi=32768,
             paged=False),
        # The attention core at a proposal (one query) of an odd-sized ragged paged batch.
        dict(name="attn_propose_b61", kind="attn", layer="llama1b", batch=61, q_len=1, kv_lo=133, kv_hi=8197,
             paged=True),
        # The projection of a catch-up chunk's hidden states: many rows.
        dict(name="project_b128_q5", kind="project", layer="llama1b", batch=128, n_new=5),
        # W_UV and W_O of a speculative chunk.
        dict(name="out_proj_b32_q5", kind="out_proj", layer="llama1b", batch=32, q_len=5),
        # Verification statistics of a big batch's chunk, bf16 logits.
        dict(name="accept_bf16_r640", kind="accept", rows=640, vocab=128256, dtype="bf16"),
        # The same for eight sequences' chunks with fp32 logits over the larger vocabulary.
        dict(name="accept_f32_r40", kind="accept", rows=40, vocab=151936, dtype="f32"),
        # The original layer beside the converted one: the big ragged paged batch ...
        dict(name="gqa_paged_b128", kind="gqa", layer="llama1b", batch=128, q_len=5, kv_lo=133, kv_hi=8197,
             paged=True),
        # ... and the long documents (head width 128).
        dict(name="gqa_long_b8", kind="gqa", layer="llama3b", batch=8, q_len=1, kv_lo=16384, kv_hi=32768,
             paged=False),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "step", "attn", "attn", "gqa", "gqa", "accept", "project", "out_proj"])
    if kind == "accept":
        dtype = rng.choice(["bf16", "bf16", "f32"])
        vocab = rng.choice([32000, 50257, 128256, 151936, rng.randrange(1000, 160000)])
        most = min(640, 640 * 128256 * 2 // (vocab * (4 if dtype == "f32" else 2)))
        return dict(kind=kind, rows=_log_int(rng, 2, most), vocab=vocab, dtype=dtype)
    layer = rng.choice(["qwen05b", "llama1b", "llama1b", "llama3b"] + (["tiny"] if kind in ("step", "attn") else []))
    if kind in ("project", "out_proj"):
        batch = _log_int(rng, 1, 128)
        n = rng.randrange(1, 9)
        while batch * n > 640:
            n -= 1
        return dict(kind=kind, layer=layer, batch=batch, **({"n_new": n} if kind == "project" else {"q_len": n}))
    q_len = rng.choice([1, 1, 1, 2, 3, 4, 5, 6, 8])
    batch = _log_int(rng, 1, 128)
    # tokens of cache in all: up to the big batch's, fewer where more query rows or wider entries meet them
    L = LAYERS[layer]
    width = (L["rank"] + L["d_rope"]) / 576 if kind != "gqa" else L["G"] * L["d_v"] / 512
    most = 520000 / max(width, 0.5) / max(1.0, q_len * L["H"] / 160)
    hi = _log_int(rng, 100, min(32768, most / batch if most / batch > 200 else 200))
    lo = rng.choice([hi, rng.randrange(q_len, hi + 1), max(q_len, hi // 8)])
    case = dict(kind=kind, layer=layer, batch=batch, q_len=q_len, kv_lo=lo, kv_hi=hi, paged=rng.random() < 0.5)
    if kind == "step":
        case["graph"] = rng.random() < 0.5
    return case


# ---------------------------------------------------------------- inputs

def _lengths(case):
    B, lo, hi = case["batch"], case["kv_lo"], case["kv_hi"]
    return [lo + int((hi - lo) * (2 * i + 1) / (2 * B)) if hi > lo else lo for i in range(B)]


class _Draw:
    """Seeded bf16 tensors on the GPU."""

    def __init__(self, seed):
        self.gen = torch.Generator(device="cuda")
        self.gen.manual_seed(seed)
        self.host = torch.Generator(device="cpu")
        self.host.manual_seed(seed + 1)

    def normal(self, *shape, std=1.0, dtype=torch.bfloat16):
        t = torch.empty(*shape, dtype=dtype, device="cuda")
        return t.normal_(0.0, std, generator=self.gen)

    def lengths(self, case):
        kv = torch.tensor(_lengths(case), dtype=torch.int32)
        return kv[torch.randperm(kv.numel(), generator=self.host)]

    def tables(self, tokens):
        """Shuffled block table of units with these token counts, and the pool's pages."""
        pages = [(t + PAGE - 1) // PAGE for t in tokens]
        perm = torch.randperm(sum(pages), generator=self.host).to(torch.int32)
        bt = torch.full((len(pages), max(pages)), -1, dtype=torch.int32)
        at = 0
        for b, n in enumerate(pages):
            bt[b, :n] = perm[at:at + n]
            at += n
        return bt.cuda(), sum(pages)


def _dims(L):
    return abi.Dims(L["H"], L["G"], L["d_nope"], L["d_rope"], L["d_v"], L["rank"], L["hidden"],
                    1.0 / math.sqrt(L["d_nope"] + L["d_rope"]), 0, 10000.0)


def _gqa_dims(L):
    return abi.GqaDims(L["H"], L["G"], L["d_v"], 1.0 / math.sqrt(L["d_v"]), 0, 10000.0)


def _cache(d, kv, paged, units, first, second):
    """Cache over ``units`` units a sequence; first / second: widths of c_kv and k_rope."""
    tokens = [int(t) for t in kv for _ in range(units)]
    if paged:
        bt, pages = d.tables(tokens)
        return abi.Cache(d.normal(pages, PAGE, first), d.normal(pages, PAGE, second), bt.shape[1] * PAGE, bt, PAGE,
                         pages)
    cap = max(tokens)
    return abi.Cache(d.normal(len(tokens), cap, first), d.normal(len(tokens), cap, second), cap)


def _inputs(case, seed):
    """The case's tensors (a dict), the same ones for prepare and exact."""
    d = _Draw(seed)
    kind = case["kind"]
    s = dict(kind=kind, case=case)
    if kind == "accept":
        stride = (case["vocab"] + 7) // 8 * 8
        dt = torch.bfloat16 if case["dtype"] == "bf16" else torch.float32
        target = torch.empty(case["rows"], stride, dtype=torch.float32, device="cuda").normal_(0.0, 3.0,
                                                                                               generator=d.gen)
        draft = target + torch.empty_like(target).normal_(0.0, 1.0, generator=d.gen)
        s["draft"], s["target"] = (t.to(dt)[:, :case["vocab"]] for t in (draft, target))
        return s
    L = LAYERS[case["layer"]]
    H, G, r, dr = L["H"], L["G"], L["rank"], L["d_rope"]
    B = case["batch"]
    if kind == "project":
        n, D = case["n_new"], L["hidden"]
        cap = n + 251
        s["cache"] = abi.Cache(d.normal(B, cap, r), d.normal(B, cap, dr), cap)
        s["start"] = torch.randint(0, cap - n + 1, (B,), generator=d.host).to(torch.int32).cuda()
        s["h"] = d.normal(B, n, D)
        s["w_dkv"], s["w_kr"] = d.normal(r, D, std=D ** -0.5), d.normal(dr, D, std=D ** -0.5)
        s["w_q"] = d.normal(H * (L["d_nope"] + dr), D, std=D ** -0.5)
        return s
    q = case["q_len"]
    if kind == "out_proj":
        # a softmax average of unit-variance rows: small values
        s["o_lat"] = d.normal(B, q, H, r, std=0.1, dtype=torch.float32)
        s["w_uv"] = d.normal(G, L["d_v"], r, std=r ** -0.5)
        s["w_o"] = d.normal(L["hidden"], H * L["d_v"], std=(H * L["d_v"]) ** -0.5)
        return s
    kv = d.lengths(case)
    s["kv"] = kv.cuda()
    s["lens"] = [int(t) for t in kv]
    if kind == "gqa":
        dk = L["d_v"]
        s["cache"] = _cache(d, kv, case["paged"], G, dk, dk)
        s["q"] = d.normal(B, q, H, dk)
        return s
    s["cache"] = _cache(d, kv, case["paged"], 1, r, dr)
    if kind == "attn":
        # an absorbed query: W_UK^T q_nope has variance d_nope / rank
        s["q_abs"] = torch.cat([d.normal(B, q, H, r, std=math.sqrt(L["d_nope"] / r)), d.normal(B, q, H, dr)], -1)
        return s
    s["w_uk"], s["w_uv"] = d.normal(G, L["d_nope"], r, std=r ** -0.5), d.normal(G, L["d_v"], r, std=r ** -0.5)
    s["w_o"] = d.normal(L["hidden"], H * L["d_v"], std=(H * L["d_v"]) ** -0.5) if L["hidden"] else None
    s["q_nope"], s["q_pe"] = d.normal(B, q, H, L["d_nope"]), d.normal(B, q, H, dr)
    s["c_new"], s["kr_new"] = d.normal(B, q, r), d.normal(B, q, dr)
    s["start"] = (kv - q).to(torch.int32).cuda()
    return s


def prepare(case, seed):
    s = _inputs(case, seed)
    kind = s["kind"]
    if kind == "accept":
        rows = case["rows"]
        s["out"] = (torch.empty(rows, dtype=torch.float32, device="cuda"),
                    *(torch.empty(rows, dtype=torch.int32, device="cuda") for _ in range(3)))
        return s
    L = LAYERS[case["layer"]]
    B = case["batch"]
    if kind == "gqa":
        s["step"] = abi.GqaStep(_gqa_dims(L), s["cache"], B, case["q_len"], max(s["lens"]))
        return s
    s["dims"] = dims = _dims(L)
    if kind == "step":
        s["step"] = abi.DecodeStep(dims, s["cache"], B, case["q_len"], max(s["lens"]), graph=case["graph"])
    elif kind == "attn":
        q = case["q_len"]
        s["max_kv"] = max(s["lens"])
        ob, lb, s["splits"] = abi.workspace_size(dims, B, q, s["max_kv"])
        s["o_part"] = torch.empty(ob // 4, dtype=torch.float32, device="cuda")
        s["lse_part"] = torch.empty(lb // 4, dtype=torch.float32, device="cuda")
        s["o_lat"] = torch.empty(B, q, L["H"], L["rank"], dtype=torch.float32, device="cuda")
        s["lse"] = torch.empty(B, q, L["H"], dtype=torch.float32, device="cuda")
    elif kind == "project":
        n = case["n_new"]
        s["q_nope"] = torch.empty(B, n, L["H"], L["d_nope"], dtype=torch.bfloat16, device="cuda")
        s["q_pe"] = torch.empty(B, n, L["H"], L["d_rope"], dtype=torch.bfloat16, device="cuda")
    else:
        q = case["q_len"]
        s["o"] = torch.empty(B, q, L["H"], L["d_v"], dtype=torch.bfloat16, device="cuda")
        s["out"] = torch.empty(B, q, L["hidden"], dtype=torch.bfloat16, device="cuda")
    return s


def run(s):
    kind = s["kind"]
    if kind == "step":
        out = s["step"](s["q_nope"], s["q_pe"], s["kv"], s["w_uk"], s["w_uv"], s["w_o"], c_new=s["c_new"],
                        kr_new=s["kr_new"], start_pos=s["start"])
        return {"out": out, "lse": s["step"].lse, "c_kv": s["cache"].c_kv, "k_rope": s["cache"].k_rope}
    if kind == "attn":
        B, q = s["q_abs"].shape[:2]
        abi.decode_attn(s["dims"], s["cache"], s["kv"], s["max_kv"], s["q_abs"], s["o_part"], s["lse_part"],
                        s["splits"])
        abi.combine(s["dims"], B, q, s["kv"], s["max_kv"], s["o_part"], s["lse_part"], s["o_lat"], s["lse"],
                    s["splits"])
        return {"o_lat": s["o_lat"], "lse": s["lse"]}
    if kind == "project":
        abi.project_append(s["dims"], s["cache"], s["h"], s["w_dkv"], s["w_kr"], s["w_q"], s["start"], s["q_nope"],
                           s["q_pe"])
        return {"q_nope": s["q_nope"], "q_pe": s["q_pe"], "c_kv": s["cache"].c_kv, "k_rope": s["cache"].k_rope}
    if kind == "out_proj":
        abi.out_proj(s["dims"], s["o_lat"], s["w_uv"], s["w_o"], s["o"], s["out"])
        return {"o": s["o"], "out": s["out"]}
    if kind == "accept":
        alpha, am_d, am_t, greedy = abi.acceptance_stats(s["draft"], s["target"], *s["out"])
        return {"alpha": alpha, "argmax_draft": am_d, "argmax_target": am_t, "greedy": greedy}
    o = s["step"](s["q"], s["kv"])
    return {"o": o, "lse": s["step"].lse}


# ---------------------------------------------------------------- what a pass cannot do without

def _visible(case):
    """Sum over sequences and queries of the keys each query sees."""
    q = case["q_len"]
    return sum(sum(t - q + i + 1 for i in range(q)) for t in _lengths(case))


def work(case):
    kind = case["kind"]
    if kind == "accept":
        n = case["rows"] * case["vocab"]
        return {"bytes": 2 * n * (2 if case["dtype"] == "bf16" else 4) + 16 * case["rows"], "flops": 8 * n}
    L = LAYERS[case["layer"]]
    H, G, r, dr, dn, dv, D = (L[k] for k in ("H", "G", "rank", "d_rope", "d_nope", "d_v", "hidden"))
    B = case["batch"]
    if kind == "project":
        rows, cols = B * case["n_new"], r + dr + H * (dn + dr)
        return {"bytes": 2 * (cols * D + rows * D + rows * cols), "flops": 2 * rows * cols * D}
    rows = B * case["q_len"]
    uv = 2 * rows * H * dv * r
    wo = 2 * rows * H * dv * D
    if kind == "out_proj":
        return {"bytes": 4 * rows * H * r + 2 * G * dv * r + 2 * D * H * dv + 2 * rows * (H * dv + D),
                "flops": uv + wo}
    tokens = sum(_lengths(case))
    if kind == "gqa":
        return {"bytes": tokens * G * 2 * dv * 2 + rows * H * (2 * dv + 4 * dv + 4),
                "flops": 4 * H * dv * _visible(case)}
    core = H * (2 * (r + dr) + 2 * r) * _visible(case)
    cache = 2 * tokens * (r + dr)
    if kind == "attn":
        return {"bytes": cache + rows * H * (2 * (r + dr) + 4 * r + 4), "flops": core}
    # a step: the cache, the new entries in and out, queries, weights, result
    weights = 2 * (G * dn * r + G * dv * r + D * H * dv)
    new = rows * (2 * H * (dn + dr) + 4 * (r + dr) + 4 * H + 2 * (D or H * dv))
    return {"bytes": cache + weights + new, "flops": core + 2 * rows * H * dn * r + uv + wo}


def tolerance(case):
    """Four times the largest distance from ``exact`` measured on the GPU (bf16 operands, fp32 sums)."""
    return {
        "step": {"rel": 1.4e-2},      # bf16 absorbed queries, weights P, o and out: 3.5e-3
        "attn": {"rel": 5e-3},        # bf16 weights P: 1.2e-3
        "project": {"rel": 7e-3},     # one bf16 rounding of each result: 1.7e-3
        "out_proj": {"rel": 1.2e-2},  # o rounded to bf16 before W_O, out after it: 2.9e-3
        "accept": {"rel": 1.5e-6},    # fp32 sums: 3.5e-7; the argmaxes are decided on the logits, without slack
        "gqa": {"rel": 1e-2},         # bf16 rotated queries and weights P: 2.4e-3
    }[case["kind"]]


# ---------------------------------------------------------------- the same values in 64 bits

def _rope(x, pos):
    """Rotate-half RoPE, base 10000, of x [..., d] at positions broadcast over the leading axes."""
    h = x.shape[-1] // 2
    theta = 10000.0 ** (-torch.arange(h, dtype=torch.float64, device=x.device) / h)
    ang = pos.double()[..., None] * theta
    c, s = torch.cos(ang), torch.sin(ang)
    a, b = x[..., :h], x[..., h:]
    return torch.cat([a * c - b * s, b * c + a * s], -1)


def _rows(cache, unit, n):
    """Where tokens 0 .. n - 1 of a unit live: (block, slot) index tensors."""
    t = torch.arange(n, device="cuda")
    if cache.block_table is None:
        return torch.full_like(t, unit), t
    return cache.block_table[unit].long()[t // PAGE], t % PAGE


def _attend(scores, q_len, n):
    """Causal softmax of scores [q_len, heads, n] and its log-sum-exp."""
    i = torch.arange(q_len, device="cuda")[:, None, None]
    scores = scores.masked_fill(torch.arange(n, device="cuda") > n - q_len + i, -math.inf)
    return torch.softmax(scores, -1), torch.logsumexp(scores, -1)


def _exact_core(q_abs, cache, lens, r, scale):
    """Absorbed attention of fp64 queries over a bf16 cache (plus fp64 caches, where given as such)."""
    B, q = q_abs.shape[:2]
    o, lse = [], []
    for b in range(B):
        blk, slot = _rows(cache, b, lens[b])
        c, k = cache.c_kv[blk, slot].double(), cache.k_rope[blk, slot].double()
        sc = torch.cat([c, k], -1) @ q_abs[b].reshape(-1, q_abs.shape[-1]).T * scale  # [n, q H]
        p, l = _attend(sc.T.reshape(q, -1, lens[b]), q, lens[b])
        o.append(p @ c)
        lse.append(l)
    return torch.stack(o), torch.stack(lse)


def exact(case, seed):
    s = _inputs(case, seed)
    kind = s["kind"]
    if kind == "accept":
        d, t = s["draft"], s["target"]
        alpha = torch.stack([torch.minimum(torch.softmax(a.double(), 0), torch.softmax(b.double(), 0)).sum()
                             for a, b in zip(d, t)])

        def first_max(x):  # the lowest index among equal maxima
            y = torch.arange(x.shape[1], device="cuda").expand_as(x)
            return torch.where(x == x.amax(1, keepdim=True), y, x.shape[1]).amin(1)

        am_d, am_t = first_max(d), first_max(t)
        return {"alpha": alpha, "argmax_draft": am_d, "argmax_target": am_t, "greedy": (am_d == am_t).long()}
    L = LAYERS[case["layer"]]
    H, G, r, dr, dn, dv = (L[k] for k in ("H", "G", "rank", "d_rope", "d_nope", "d_v"))
    B = case["batch"]
    if kind == "project":
        n = case["n_new"]
        h = s["h"].double()
        pos = s["start"].long()[:, None] + torch.arange(n, device="cuda")
        at = (torch.arange(B, device="cuda")[:, None].expand(B, n), pos)
        c_kv, k_rope = s["cache"].c_kv.double(), s["cache"].k_rope.double()
        c_kv[at] = h @ s["w_dkv"].double().T
        k_rope[at] = _rope(h @ s["w_kr"].double().T, pos)
        qq = (h @ s["w_q"].double().T).reshape(B, n, H, dn + dr)
        return {"q_nope": qq[..., :dn], "q_pe": qq[..., dn:], "c_kv": c_kv, "k_rope": k_rope}
    q = case["q_len"]
    scale = 1.0 / math.sqrt(dn + dr)

    def up(o_lat):
        w = s["w_uv"].double()[torch.arange(H, device="cuda") // (H // G)]  # [H, d_v, r]
        o = torch.einsum("bqhr,hvr->bqhv", o_lat, w)
        return o, None if s["w_o"] is None else o.reshape(B, q, H * dv) @ s["w_o"].double().T

    if kind == "out_proj":
        o, out = up(s["o_lat"].double())
        return {"o": o, "out": out}
    pos = s["kv"].long()[:, None] - q + torch.arange(q, device="cuda")  # [B, q]
    if kind == "gqa":
        qr = _rope(s["q"].double(), pos[..., None]).reshape(B, q, G, H // G, dv)
        o = torch.empty(B, q, G, H // G, dv, dtype=torch.float64, device="cuda")
        lse = torch.empty(B, q, G, H // G, dtype=torch.float64, device="cuda")
        for b, n in enumerate(s["lens"]):
            at = [_rows(s["cache"], b * G + g, n) for g in range(G)]
            blk, slot = (torch.stack([a[j] for a in at]) for j in (0, 1))
            k, v = s["cache"].k_rope[blk, slot].double(), s["cache"].c_kv[blk, slot].double()  # [G, n, d]
            x = qr[b].transpose(0, 1).reshape(G, -1, dv)  # [G, q hpg, d]
            sc = (x @ k.transpose(1, 2) / math.sqrt(dv)).reshape(G, q, -1, n).transpose(0, 1).reshape(q, -1, n)
            p, l = _attend(sc, q, n)
            p = p.reshape(q, G, -1, n).transpose(0, 1).reshape(G, -1, n)
            o[b] = (p @ v).reshape(G, q, -1, dv).transpose(0, 1)
            lse[b] = l.reshape(q, G, -1)
        return {"o": o.reshape(B, q, H, dv), "lse": lse.reshape(B, q, H)}
    if kind == "attn":
        o, lse = _exact_core(s["q_abs"].double(), s["cache"], s["lens"], r, scale)
        return {"o_lat": o, "lse": lse}
    cache = s["cache"]
    c_kv, k_rope = cache.c_kv.double(), cache.k_rope.double()
    for b, n in enumerate(s["lens"]):
        blk, slot = _rows(cache, b, n)
        c_kv[blk[n - q:], slot[n - q:]] = s["c_new"][b].double()
        k_rope[blk[n - q:], slot[n - q:]] = _rope(s["kr_new"][b].double(), pos[b])
    cache = abi.Cache(c_kv, k_rope, cache.capacity, cache.block_table, cache.page_size, cache.num_pages)
    w_uk = s["w_uk"].double()[torch.arange(H, device="cuda") // (H // G)]  # [H, d_nope, r]
    q_lat = torch.einsum("bqhd,hdr->bqhr", s["q_nope"].double(), w_uk)
    q_abs = torch.cat([q_lat, _rope(s["q_pe"].double(), pos[..., None])], -1)
    o_lat, lse = _exact_core(q_abs, cache, s["lens"], r, scale)
    o, out = up(o_lat)
    return {"out": o if out is None else out, "lse": lse, "c_kv": c_kv, "k_rope": k_rope}
