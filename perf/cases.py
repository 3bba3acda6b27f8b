"""What is timed when this library's speed is followed from one version to the next: calls of its public entry points
over the range of shapes they are used on.

The eviction pass is timed in its parts, scoring (`madakv_score`, `madakv_score_lse`) apart from what follows it
(`madakv_allocate`, `madakv_select`, `madakv_compact`), because the parts after scoring are discontinuous in the
scores: one token more or less in one head moves every later segment of the ragged cache. With the scores as inputs
their results are exact; the scores themselves are compared as the floating-point sums they are.

Inputs follow the recipe of the package's synthetic workloads (interleaved visual and text spans, N(0, 1) queries, keys
and values, visual keys shifted per head, a few strongly attended keys per modality), drawn on the GPU from the seed.
"""
import math

import numpy as np
import torch

from paper_2506_15724_b200 import binding as mk

DTYPES = {"bf16": torch.bfloat16, "f32": torch.float32}


def _case(name, kind, dtype, B, L, Hq, Hkv, d, n, **kw):
    c = dict(name=name, kind=kind, dtype=dtype, B=B, L=L, Hq=Hq, Hkv=Hkv, d=d, n=n)
    c.update(kw)
    return c


def listed():
    return [
        # --- scoring after prefill, all layers in one call
        # a prompt of 128 images on a grouped-query model: the largest single prompt
        _case("score_long", "score", "bf16", 1, 32, 32, 8, 128, 131072, w=64, ragged=0.0),
        # several images on a dense-attention model, the ordinary prompt
        _case("score_llava", "score", "bf16", 1, 32, 32, 32, 128, 8192, w=32, ragged=0.0),
        # a serving batch whose prompts have different lengths, 7 query heads per KV head
        _case("score_batched", "score", "bf16", 8, 28, 28, 4, 128, 16384, w=32, ragged=0.5),
        # a long prompt on the dense-attention model (see _scorable on its length)
        _case("score_dense_long", "score", "bf16", 1, 32, 32, 32, 128, 20480, w=32, ragged=0.0),
        # the smallest call: one fp32 layer of a short prompt (development and checking against fp32)
        _case("score_f32_small", "score", "f32", 1, 1, 4, 4, 64, 512, w=8, ragged=0.0),
        # scoring one layer at a time, right after that layer's prefill, with the log-sum-exps the prefill kept
        _case("score_layers", "score_layers", "bf16", 1, 28, 28, 4, 128, 32768, w=32, ragged=0.0),
        # --- budgets, selection and compaction on given scores
        _case("evict_long", "evict", "bf16", 1, 32, 32, 8, 128, 131072, w=64, ragged=0.0, budget=4096, theta=0.218545,
              hcc=mk.HCC_PAPER, mpa=1, pool=1, keep=0),
        _case("evict_llava", "evict", "bf16", 1, 32, 32, 32, 128, 8192, w=32, ragged=0.0, budget=1638, theta=0.471452,
              hcc=mk.HCC_PAPER, mpa=1, pool=1, keep=0),
        # a layer at a time, the budget state carried from layer to layer
        _case("evict_layers", "evict_layers", "bf16", 1, 28, 28, 4, 128, 32768, w=32, ragged=0.0, budget=2048,
              theta=0.324026, hcc=mk.HCC_PAPER, mpa=1, pool=1, keep=0),
        # --- decode steps that append a token each, on a ragged compressed cache
        # dense attention, all layers in one call
        _case("decode_llava", "decode", "bf16", 1, 32, 32, 32, 128, 8192, rows=1638, spread=0.3, steps=4),
        # a serving batch, 7 query heads per KV head
        _case("decode_batched", "decode", "bf16", 8, 28, 28, 4, 128, 16384, rows=2512, spread=0.6, steps=4),
        # a model's own order: one call per layer, few segments each
        _case("decode_layers", "decode_layers", "bf16", 1, 32, 32, 8, 128, 131072, rows=2952, spread=0.4, steps=2),
    ]


def _log_int(rng, lo, hi):
    """An integer of [lo, hi], uniform in its logarithm, odd or even as it falls."""
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    """One more case of the same ranges. No drawn case has more cache bytes or window logits than `score_long`; fp32
    shapes and windows beyond 256 rows per KV head, which cost far more arithmetic, stay at a sixteenth of that."""
    kind = rng.choice(["score", "score", "score", "score_layers", "evict", "evict", "evict_layers", "decode", "decode",
                       "decode_layers"])
    dtype = "f32" if rng.random() < 0.12 else "bf16"
    Hq, Hkv = rng.choice([(4, 4), (32, 32), (40, 40), (28, 4), (28, 4), (32, 8), (32, 8), (8, 2), (16, 8)])
    d = 64 if rng.random() < 0.15 else 128
    w = rng.choice([8, 16, 24, 32, 32, 32, 48, 64, 64])
    n = _log_int(rng, 384, 131072)
    B = rng.choice([1, 1, 1, 2, 3, 5, 8])
    L = rng.choice([1, 2, 5, 28, 32, 40])
    small = dtype == "f32" or (Hq // Hkv) * w > 256
    elems = 32 * 8 * 131072 * 128 // (16 if small else 1)  # elements of K
    logits = 32 * 8 * 131072 * 256 // (16 if small else 1)
    while B * L * Hkv * n * d > elems or B * L * Hq * w * n > logits:
        if B > 1:
            B = (B + 1) // 2
        elif L > 1:
            L = (L + 1) // 2
        else:
            n = n * 2 // 3
    ragged = 0.0 if B == 1 else round(rng.uniform(0.0, 0.8), 2)
    if kind == "score":
        n, ragged = _scorable(dtype, Hq // Hkv * w, n, ragged)
    c = _case("", kind, dtype, B, L, Hq, Hkv, d, n)
    del c["name"]
    if kind.startswith("decode"):
        c.update(rows=max(16, int(n * math.exp(rng.uniform(math.log(0.02), math.log(0.6))))),
                 spread=round(rng.uniform(0.0, 0.8), 2), steps=rng.choice([1, 2, 4]))
        while c["steps"] > 1 and c["steps"] * B * L * Hkv * c["rows"] * d > 1.5 * elems:
            c["steps"] //= 2
        return c
    c.update(w=w, ragged=ragged)
    if kind.startswith("evict"):
        share = math.exp(rng.uniform(math.log(0.03), math.log(0.6)))
        c.update(budget=max(16, int(n * share)), theta=round(_mass_share(share, (Hq // Hkv) * w), 6),
                 hcc=rng.choice([mk.HCC_PAPER, mk.HCC_PAPER, mk.HCC_OFF, mk.HCC_LITERAL, mk.HCC_DEMAND]),
                 mpa=0 if rng.random() < 0.15 else 1, pool=rng.choice([1, 1, 1, 1, 7]),
                 keep=1 if rng.random() < 0.2 else 0)
    return c


def _scorable(dtype, rows, n, ragged):
    """bf16 prompts with up to 64 window rows per KV head and more tokens than stay on chip (16384 for up to 32 rows,
    8192 beyond) come as whole stretches of 1024 tokens: the version this file was written with runs into the bound of
    its waits on some other lengths, so there is nothing to compare with there."""
    if dtype == "bf16" and rows <= 64 and n > (16384 if rows <= 32 else 8192):
        return n // 1024 * 1024, 0.0
    return n, ragged


def _mass_share(share, rows):
    """Share of the attention mass that the largest `share` of the keys hold, for sums of `rows` log-normal weights:
    the threshold of Eq. 9 at which the demand is about the budget."""
    sigma = math.sqrt(math.log(1.0 + (math.e - 1.0) / rows))
    lo, hi = -8.0, 8.0
    for _ in range(60):
        mid = 0.5 * (lo + hi)
        lo, hi = (mid, hi) if 0.5 * math.erfc(-mid / math.sqrt(2.0)) < share else (lo, mid)
    return 0.5 * math.erfc(-(lo + sigma) / math.sqrt(2.0))


# ------------------------------------------------------------------------------------------------- inputs
def _lengths(case):
    """Prompt lengths of the batch: the first is n, the others fall towards (1 - ragged) * n."""
    B, n = case["B"], case["n"]
    return [max(2 * case["w"], n - int(case["ragged"] * n * b / B) - (1 if b else 0)) for b in range(B)]


def _mask(case, rng):
    """Interleaved text and visual spans, text at the end of every prompt."""
    B, n = case["B"], case["n"]
    mask = np.zeros((B, n), np.uint8)
    for b, length in enumerate(_lengths(case)):
        pos, share = 0, rng.uniform(0.3, 0.9) if B > 1 else 0.7
        unit = max(8, min(768, length // 12))
        while pos < length - case["w"]:
            pos += int(rng.randint(1, max(2, int(2 * unit * (1 - share)))))
            end = pos + int(rng.randint(unit // 2, max(unit // 2 + 1, int(2 * unit * share))))
            mask[b, pos:min(end, length - case["w"])] = 1
            pos = end
    return torch.from_numpy(mask).cuda()


def _normal(gen, shape, dtype):
    """N(0, 1) in the case's type, made in pieces (the fp32 image of the largest caches would not be small)."""
    out = torch.empty(shape, dtype=dtype, device="cuda")
    flat = out.view(-1)
    step = 1 << 28
    for a in range(0, flat.numel(), step):
        part = flat[a:a + step]
        part.copy_(torch.randn(part.numel(), generator=gen, device="cuda", dtype=torch.float32))
    return out


def _prompt(case, seed, want_v):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    rng = np.random.RandomState(seed % (1 << 31))
    B, L, Hq, Hkv, d, n, w = (case[x] for x in ("B", "L", "Hq", "Hkv", "d", "n", "w"))
    dtype = DTYPES[case["dtype"]]
    mask = _mask(case, rng)
    q = _normal(gen, (B, L, Hq, w, d), dtype)
    k = _normal(gen, (B, L, Hkv, n, d), dtype)
    v = _normal(gen, (B, L, Hkv, n, d), dtype) if want_v else None
    beta = 0.5 * torch.randn((L, Hkv, 1, d), generator=gen, device="cuda")
    qbar = q.float().view(B, L, Hkv, -1, d).mean(dim=3, keepdim=True)
    boost = 4.0 * math.sqrt(d) * qbar / (qbar * qbar).sum(-1, keepdim=True)
    for b, length in enumerate(_lengths(case)):
        vis = mask[b].view(1, n, 1).to(dtype)
        strong = torch.from_numpy(rng.choice(length - w, size=min(32, (length - w) // 4), replace=False)).cuda()
        for l in range(L):
            k[b, l] += vis * beta[l].to(dtype)
            k[b, l, :, strong] += boost[b, l].to(dtype)
    return dict(q=q, k=k, v=v, mask=mask, seq_len=torch.tensor(_lengths(case), dtype=torch.int32, device="cuda"))


def _attention_of_window(case, inp):
    """Scores [B, L, Hkv, n] and row log-sum-exps [B, L, Hq, w] of the prompt's last w queries, by plain fp32 torch."""
    B, L, Hq, Hkv, d, n, w = (case[x] for x in ("B", "L", "Hq", "Hkv", "d", "n", "w"))
    psi = torch.zeros((B, L, Hkv, n), device="cuda")
    lse = torch.empty((B, L, Hq, w), device="cuda")
    row = torch.arange(w, device="cuda").repeat(Hq // Hkv).view(-1, 1)
    for b, length in enumerate(_lengths(case)):
        seen = torch.arange(length - w, length, device="cuda").view(1, -1) <= length - w + row
        for l in range(L):
            s = (inp["q"][b, l].float().view(Hkv, -1, d) / math.sqrt(d)) @ inp["k"][b, l, :, :length].float().mT
            s[:, :, length - w:].masked_fill_(~seen, -math.inf)
            z = torch.logsumexp(s, dim=2, keepdim=True)
            lse[b, l] = z.view(Hq, w)
            psi[b, l, :, :length] = s.sub_(z).exp_().sum(dim=1)
    return psi, lse


def _config(case, **kw):
    args = dict(window=case.get("w", 32), max_new_tokens=16)
    if "budget" in case:
        args.update(theta=case["theta"], hcc_mode=case["hcc"], mpa=case["mpa"], pool_kernel=case["pool"],
                    keep_window=case["keep"])
    args.update(kw)
    L = args.pop("L", case["L"])
    return mk.make_config(DTYPES[case["dtype"]], case["B"], L, case["Hq"], case["Hkv"], case["d"], case["n"], **args)


def _segments(case):
    """Rows kept by every (sequence, layer, KV head): around case["rows"], uneven from head to head."""
    units = case["B"] * case["L"] * case["Hkv"]
    u = np.arange(units, dtype=np.float64)
    frac = (u + 1) * 0.6180339887498949 % 1.0
    rows = np.floor(case["rows"] * (1.0 + case["spread"] * (2.0 * frac - 1.0))).astype(np.int64)
    return np.clip(rows, 1, case["n"])


def prepare(case, seed):
    kind, B, L, Hq, Hkv, d, n = (case[x] for x in ("kind", "B", "L", "Hq", "Hkv", "d", "n"))
    dtype = DTYPES[case["dtype"]]
    s = dict(kind=kind, layers=range(L))
    if kind.startswith("decode"):
        # the ragged cache as compaction leaves it, with room behind every segment for the tokens to come
        gen = torch.Generator(device="cuda").manual_seed(seed)
        cfg = _config(case)
        rows = _segments(case)
        off = np.concatenate([[0], np.cumsum(rows + cfg.max_new_tokens)])
        T = case["steps"]
        s.update(cfg=cfg, steps=range(T), ws=mk.new_workspace(cfg),
                 seg_off=torch.from_numpy(off).cuda(), rows=torch.from_numpy(rows.astype(np.int32)).cuda(),
                 kept_len=torch.zeros(len(rows), dtype=torch.int32, device="cuda"),
                 k_c=_normal(gen, (int(off[-1]), d), dtype), v_c=_normal(gen, (int(off[-1]), d), dtype),
                 q=_normal(gen, (T, B, L, Hq, d), dtype), k_new=_normal(gen, (T, B, L, Hkv, d), dtype),
                 v_new=_normal(gen, (T, B, L, Hkv, d), dtype),
                 out=torch.zeros((T, B, L, Hq, d), dtype=dtype, device="cuda"),
                 lse=torch.zeros((T, B, L, Hq), device="cuda"))
        return s
    inp = _prompt(case, seed, want_v=kind.startswith("evict"))
    s.update(inp)
    if kind == "score":
        s.update(cfg=_config(case), lse=torch.zeros((B, L, Hq, case["w"]), device="cuda"),
                 psi=torch.zeros((B, L, Hkv, n), device="cuda"))
        s["ws"] = mk.new_workspace(s["cfg"])
        return s
    if kind == "score_layers":
        _, lse = _attention_of_window(case, inp)
        s.update(cfg=_config(case, L=1), lse=lse.transpose(0, 1).contiguous(),  # [L, B, Hq, w]
                 psi=[torch.zeros((B, Hkv, n), device="cuda") for _ in range(L)])
        s["ws"] = mk.new_workspace(s["cfg"])
        return s
    psi, _ = _attention_of_window(case, inp)
    s.update(cfg=_config(case), budget=torch.full((B,), case["budget"], dtype=torch.int32, device="cuda"))
    slack = min(n, 2 * case["budget"] + 2 * case["w"]) + s["cfg"].max_new_tokens
    if kind == "evict":
        s["buf"] = mk.EvictionBuffers(s["cfg"], B * L * Hkv * slack)
        s["buf"].psi.copy_(psi)
        return s
    # layer by layer: every layer has its own ragged cache; the per-layer arrays lie behind one another, but for the
    # scores, whose rows may have any length and whose base is aligned
    z = lambda *shape, dtype=torch.int32: torch.zeros(shape, dtype=dtype, device="cuda")  # noqa: E731
    cap = B * Hkv * min(slack * 2, n + s["cfg"].max_new_tokens)
    s.update(one=_config(case, L=1), ws=mk.new_workspace(s["cfg"]), psi=[psi[:, l].clone() for l in range(L)],
             mass=z(L, B, Hkv, 2, dtype=torch.float64), pref=z(L, B, Hkv, 2, dtype=torch.float64),
             demand=z(L, B, Hkv, 2), budgets=z(L, B, Hkv, 2), phi=z(B, L, dtype=torch.float64),
             kept_len=z(L, B * Hkv), seg_off=z(L, B * Hkv + 1, dtype=torch.int64), kept_idx=z(L, cap),
             k_c=z(L, cap, d, dtype=dtype), v_c=z(L, cap, d, dtype=dtype))
    return s


# ------------------------------------------------------------------------------------------------- one pass
def run(s):
    kind = s["kind"]
    if kind == "score":
        mk.madakv_score(s["cfg"], s["q"], s["k"], s["seq_len"], s["lse"], s["psi"], s["ws"])
        return {"psi": s["psi"], "lse": s["lse"]}
    if kind == "score_layers":
        for l in s["layers"]:
            mk.madakv_score_lse(s["cfg"], s["q"][:, l:l + 1], s["k"][:, l:l + 1], s["seq_len"], s["lse"][l],
                                s["psi"][l], s["ws"])
        return {"psi": s["psi"]}
    if kind == "evict":
        b, c = s["buf"], s["cfg"]
        mk.madakv_allocate(c, b.psi, s["mask"], s["seq_len"], s["budget"], b.mass, b.pref, b.demand, b.phi, b.budgets,
                           b.ws)
        mk.madakv_select(c, b.psi, s["mask"], s["seq_len"], b.budgets, b.kept_len, b.seg_off, b.kept_idx, b.ws)
        mk.madakv_compact(c, s["k"], s["v"], b.kept_idx, b.seg_off, b.kept_len, b.k_c, b.v_c, b.ws)
        return {"mass": b.mass, "pref": b.pref, "demand": b.demand, "phi": b.phi, "budgets": b.budgets,
                "kept_len": b.kept_len, "seg_off": b.seg_off, "kept_idx": b.kept_idx, "k_c": b.k_c, "v_c": b.v_c}
    if kind == "evict_layers":
        c, one = s["cfg"], s["one"]
        for l in s["layers"]:
            mk.madakv_allocate_layer(c, l, s["psi"][l], s["mask"], s["seq_len"], s["budget"], s["mass"][l],
                                     s["pref"][l], s["demand"][l], s["phi"], s["budgets"][l], s["ws"])
            mk.madakv_select(one, s["psi"][l], s["mask"], s["seq_len"], s["budgets"][l], s["kept_len"][l],
                             s["seg_off"][l], s["kept_idx"][l], s["ws"])
            mk.madakv_compact(one, s["k"][:, l:l + 1], s["v"][:, l:l + 1], s["kept_idx"][l], s["seg_off"][l],
                              s["kept_len"][l], s["k_c"][l], s["v_c"][l], s["ws"])
        return {x: s[x] for x in ("mass", "pref", "demand", "phi", "budgets", "kept_len", "seg_off", "kept_idx", "k_c",
                                  "v_c")}
    # decode: the cache starts a pass as the eviction left it, then every step appends a token and attends
    s["kept_len"].copy_(s["rows"])
    for t in s["steps"]:
        for l in ((-1,) if kind == "decode" else s["layers"]):
            mk.madakv_decode_attn(s["cfg"], l, s["q"][t], s["k_new"][t], s["v_new"][t], s["k_c"], s["v_c"],
                                  s["seg_off"], s["kept_len"], s["out"][t], s["lse"][t], s["ws"])
    return {x: s[x] for x in ("out", "lse", "kept_len", "k_c", "v_c")}


# ------------------------------------------------------------------------------------------------- cost, tolerance
def work(case):
    L, Hq, Hkv, d, n = (case[x] for x in ("L", "Hq", "Hkv", "d", "n"))
    e = 2 if case["dtype"] == "bf16" else 4
    if case["kind"].startswith("decode"):
        T, rows = case["steps"], _segments(case)
        per_step = rows.sum() + len(rows) * (T + 1) / 2.0  # rows attended: a step more per step before it
        heads = case["B"] * L * Hq
        return {"bytes": float(T * (2 * per_step * d * e + 2 * heads * d * e + heads * 4 + 4 * len(rows) * d * e)),
                "flops": float(T * per_step * (Hq // Hkv) * d * 4)}
    w, tokens = case["w"], sum(_lengths(case))
    if case["kind"].startswith("score"):
        return {"bytes": float(L * Hkv * (tokens * d * e + case["B"] * n * 4) + case["B"] * L * Hq * w * (d * e + 4)),
                "flops": float(2 * L * Hq * w * tokens * d)}
    kept = sum(min(t, max(case["budget"], w if case["keep"] else 0)) for t in _lengths(case))
    # scores and mask once, kept rows of K and V read and written, positions written; an addition and a comparison each
    return {"bytes": float(L * Hkv * (tokens * 4 + kept * (4 * d * e + 4)) + tokens), "flops": float(2 * L * Hkv * tokens)}


def tolerance(case):
    if case["kind"].startswith("evict"):
        return "exact"
    # about four times the distance from the same sums in 64 bits, over the listed and two dozen drawn shapes
    if case["kind"].startswith("score"):
        return {"rel": 4e-6, "max": 1.2e-5}  # fp32 logits, their exponentials, sums of up to a hundred thousand terms
    if case["dtype"] == "bf16":
        return {"rel": 8e-3, "max": 3.5e-2}  # results rounded to bf16, weights too before the contraction with V
    return {"rel": 1.5e-6, "max": 5e-6}
