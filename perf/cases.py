"""Timed cases of the carve library: what a user of it has it do, through its public entry points.

A case is a dict of plain values; its "call" says which entry points one pass goes through:

  carve   `tc_carve`: scores, selection and gather of a batch of images at prefill.
          rank_cap > 0 is the caller's bound on the numerical rank, 0 the solve without one.
  host    `tc_carve_host`: the same from and to pinned host memory.
  staged  `tc_score`, `tc_prune`, `tc_merge`, `tc_compact`: the stages one by one, for callers that
          look at the scores or change the lists between them.
  probe   `tc_probe`: the layer-2 attention output and probe rows from queries, keys and values.
  resume  `tc_reassemble`, `tc_rope_tables`: the sequence the later layers run on and its tables.

The inputs are synthetic with the structure the path meets: an attention output of known numerical
rank plus noise, softmaxed attention rows, Gaussian hidden states, keys and values.  The tokens come
in three tiers, as patches of an image do: a few that carry much information, near copies of some of
those with less of it, and a background; that also keeps the scores at the two cuts and the
similarities at the merge cut apart by far more than float32 rounding, so that every correct
implementation selects the same tokens.
"""
from __future__ import annotations

import math

import torch

from paper_2503_10501_b200 import binding as tcb
from paper_2503_10501_b200 import inputs

TORCH_DTYPE = {"f16": torch.float16, "bf16": torch.bfloat16, "f32": torch.float32}
BYTES = {"f16": 2, "bf16": 2, "f32": 4}
RANK_TOL = 2e-3
NOISE = 0.01


def _carve(name, call="carve", cfg=None, **kw):
    """A carve-like case with the shapes of one of the package's own configurations."""
    c = {"name": name, "call": call, "kv_cache": True, "sim": "O", "weighted": False}
    if cfg is not None:
        g = inputs.CONFIGS[cfg]
        c.update(batch=g.batch, tokens=g.n_tokens, width=g.d_model, heads=g.n_heads, head_dim=g.head_dim,
                 query=g.n_query, keep=g.keep, rank=g.rank, rank_cap=g.rank_cap, dtype=g.dtype, tau=g.tau)
    c.update(kw)
    return c


def listed():
    return [
        # one chat request with one image: the latency a user waits for before the first token
        _carve("carve_1_f16", cfg="cfg2_llava7b_f16", batch=1),
        # the same in float32 (a caller that runs the early layers in full precision)
        _carve("carve_1_f32", cfg="cfg1_single_f32"),
        # a serving batch at the two model widths of the package's configurations
        _carve("carve_16_f16", cfg="cfg2_llava7b_f16"),
        _carve("carve_16_wide_f16", cfg="cfg3_llava13b_f16"),
        # a full batch: offline processing of many images
        _carve("carve_64_f16", cfg="cfg5_sweep_f16"),
        # high-resolution images cut into tiles: five times the tokens, a larger rank
        _carve("carve_4_tiles_f16", cfg="cfg4_anyres_f16"),
        # no bound on the rank is known: the singular value decomposition as the paper states it
        _carve("carve_2_full_f16", cfg="cfg2_llava7b_f16", batch=2, rank_cap=0),
        # a model of other sizes: odd token count (27 x 27 patches), bfloat16, a rank bound that is
        # no multiple of a tile, matching on the keys and the score-weighted merge
        _carve("carve_6_odd_bf16", batch=6, tokens=729, width=3072, heads=24, head_dim=128, query=40, keep=150,
               rank=150, rank_cap=180, dtype="bf16", tau=2.0, sim="meanK", weighted=True),
        # tensors that live in pinned host memory, results back there
        _carve("host_8_f16", call="host", cfg="cfg2_llava7b_f16", batch=8),
        # stage by stage, every score and list handed to the caller
        _carve("staged_8_f16", call="staged", cfg="cfg5_sweep_f16", batch=8, query=64, keep=192),
        # the layer-2 attention the carve starts from, a batch of prompts around the images
        {"name": "probe_16_f16", "call": "probe", "batch": 16, "tokens": 576, "heads": 32, "n_sys": 35, "n_text": 64,
         "query": 64, "dtype": "f16"},
        # one request's sequence after the compression
        {"name": "resume_1_f16", "call": "resume", "batch": 1, "tokens": 576, "width": 4096, "keep": 128, "n_sys": 35,
         "n_text": 64, "head_dim": 128, "dtype": "f16"},
    ]


def _log_int(rng, lo, hi, step=1):
    v = math.exp(rng.uniform(math.log(lo), math.log(hi + 0.999)))
    return min(hi, max(lo, int(v) // step * step))


def draw(rng):
    call = rng.choices(["carve", "full", "host", "staged", "probe", "resume"], [60, 8, 6, 10, 9, 7])[0]
    dtype = rng.choices(["f16", "bf16", "f32"], [60, 25, 15])[0]
    if call == "probe":
        c = {"call": "probe", "tokens": _log_int(rng, 144, 2880), "heads": rng.choice([16, 24, 32, 40]),
             "n_sys": rng.randint(1, 100), "n_text": _log_int(rng, 8, 256), "dtype": rng.choice(["f16", "f16", "bf16"])}
        c["query"] = rng.choice([c["n_text"], max(1, c["n_text"] // 2)])
        most = 64 * 32 * 700 ** 2 // (c["heads"] * (c["tokens"] + c["n_sys"] + c["n_text"]) ** 2)
        c["batch"] = _log_int(rng, 1, max(1, min(64, most)))
        return c
    if call == "resume":
        n = _log_int(rng, 144, 2880)
        return {"call": "resume", "batch": _log_int(rng, 1, 64), "tokens": n, "width": 128 * rng.randint(8, 40),
                "keep": max(8, int(n * rng.uniform(0.08, 0.35))), "n_sys": rng.randint(0, 100),
                "n_text": _log_int(rng, 1, 512), "head_dim": rng.choice([64, 96, 128]), "dtype": dtype}
    full = call == "full"
    n = _log_int(rng, 96, 576) if full else _log_int(rng, 260, 2880)
    heads = rng.randint(8, 40)
    rank = _log_int(rng, 48, 144) if full else _log_int(rng, 64, max(64, min(400, n // 4)))
    rank = min(rank, n // 2)
    cap = 0 if full else min(n - 4, rank + 16 + rng.randint(0, max(8, rank // 2)))
    c = {"call": "carve" if full else call, "tokens": n, "width": 128 * heads, "heads": heads, "head_dim": 128,
         "query": _log_int(rng, 16, 512), "keep": max(8, int(n * rng.uniform(0.08, 0.35))), "rank": rank,
         "rank_cap": cap, "dtype": dtype, "tau": round(rng.uniform(1.0, 2.5), 2), "kv_cache": rng.random() < 0.9,
         "sim": "O", "weighted": rng.random() < 0.2}
    if call == "carve" and not full:
        c["sim"] = rng.choices(["O", "X", "meanK"], [80, 10, 10])[0]
    if c["sim"] == "meanK":
        c["kv_cache"] = True
    # no dearer than the largest of the listed cases: its bytes, and the work of its decompositions
    most = min(1.2e9 / (work(dict(c, batch=1))["bytes"]), 4 * 736 ** 3 / max(cap, 1) ** 3, 2 if full else 64)
    c["batch"] = _log_int(rng, 1, max(1, min(8 if call == "host" else 64, int(most))))
    return c


def _counts(c):
    m = min(c["keep"] // 2, c["tokens"] - c["keep"])
    p = c["keep"] + m
    return m, p, p // 2, p - p // 2   # merged, survivors, Set A, Set B


def _params(c):
    return tcb.Params(batch=c["batch"], n_tokens=c["tokens"], d_model=c["width"], n_heads=c["heads"],
                      head_dim=c["head_dim"], n_query=c["query"], keep=c["keep"], rank_tol=RANK_TOL, dtype=c["dtype"],
                      rank_cap=c["rank_cap"], sim_source=c["sim"], weighted_merge=c["weighted"])


def _orthonormal(m):
    """Columns of m [..., n, r] made orthonormal (two Cholesky passes in double precision)."""
    m = m.double()
    for _ in range(2):
        r = torch.linalg.cholesky(m.mT @ m, upper=True)
        m = torch.linalg.solve_triangular(r, m, upper=True, left=False)
    return m


def _tiers(c, g):
    """Per image a random order of its tokens: Set A, Set B (near copies of Set A tokens first), background."""
    return torch.rand(c["batch"], c["tokens"], generator=g, device="cuda").argsort(dim=1)


def _near_copies(t, order, c, dim_tokens, src):
    """Overwrites the first M tokens of Set B with near copies of Set A tokens (cosine 0.99)."""
    m, _, na, _ = _counts(c)
    for b in range(c["batch"]):
        rows = t[b].transpose(0, dim_tokens - 1) if dim_tokens > 1 else t[b]
        dst, frm = order[b, na:na + m], order[b, :na][src[b]]
        rows[dst] = 0.99 * rows[frm] + 0.14 * rows[dst]


def _attention_output(c, order, src, g):
    """O = U diag(s) W + noise with orthonormal U, W: s geometric from 1 to 0.01, and the rows of U
    scaled so that the information scores of the three tiers lie apart."""
    B, n, d, r = c["batch"], c["tokens"], c["width"], c["rank"]
    m, p, na, nb = _counts(c)
    u = torch.randn(B, n, r, generator=g, device="cuda", dtype=torch.float32)
    _near_copies(u, order, c, 1, src)
    rank_of = torch.empty_like(order).scatter_(1, order, torch.arange(n, device="cuda").expand(B, n))
    level = torch.rand(B, n, generator=g, device="cuda", dtype=torch.float32)
    tier = torch.where(rank_of < na, 1.6 + 0.6 * level, torch.where(rank_of < p, 0.95 + 0.3 * level, 0.35 + 0.35 * level))
    s = torch.logspace(0, -2, r, device="cuda", dtype=torch.float64)
    u = _orthonormal(u)
    for _ in range(3):
        score = (u.abs() * s).sum(-1)
        u = _orthonormal(u * (tier / score).unsqueeze(-1))
    w = _orthonormal(torch.randn(B, d, r, generator=g, device="cuda", dtype=torch.float32))
    o = ((u * (s * math.sqrt(n * d))).float() @ w.float().mT)
    o += NOISE * torch.randn(B, n, d, generator=g, device="cuda", dtype=torch.float32)
    return o.to(TORCH_DTYPE[c["dtype"]])


def _normal(g, dtype, *shape):
    """N(0, 1) of the storage type, an image at a time (the float32 draws of a large batch are big)."""
    return torch.stack([torch.randn(shape[1:], generator=g, device="cuda", dtype=torch.float32).to(dtype)
                        for _ in range(shape[0])])


def prepare(case, seed):
    c = dict(case)
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    dt = TORCH_DTYPE[c["dtype"]]
    B, n = c["batch"], c["tokens"]
    if c["call"] == "probe":
        L, H = c["n_sys"] + n + c["n_text"], c["heads"]
        p = tcb.Params(batch=B, n_tokens=n, d_model=H * 128, n_heads=H, head_dim=128, n_query=c["query"],
                       keep=max(1, n // 5), dtype=c["dtype"])
        return {"c": c, "p": p, "q": _normal(g, dt, B, H, L, 128), "k": _normal(g, dt, B, H, L, 128),
                "v": _normal(g, dt, B, H, L, 128)}
    if c["call"] == "resume":
        L, d = c["n_sys"] + n + c["n_text"], c["width"]
        p = tcb.Params(batch=B, n_tokens=n, d_model=d, n_heads=max(1, d // 128), head_dim=128, n_query=1, keep=c["keep"],
                       dtype=c["dtype"])
        kept = torch.rand(B, n, generator=g, device="cuda").argsort(dim=1)[:, :c["keep"]].sort(dim=1).values
        return {"c": c, "p": p, "h": _normal(g, dt, B, L, d), "x": _normal(g, dt, B, c["keep"], d),
                "kept": kept.to(torch.int32).contiguous()}
    m, _, na, _ = _counts(c)
    order = _tiers(c, g)
    src = torch.randint(0, na, (B, m), generator=g, device="cuda")
    st = {"c": c, "p": _params(c), "O": _attention_output(c, order, src, g)}
    rows = []
    for _ in range(B):
        z = torch.randn(c["heads"], c["query"], n, generator=g, device="cuda", dtype=torch.float32)
        rows.append(torch.softmax(c["tau"] * z, dim=-1).to(dt))
    st["A"] = torch.stack(rows)
    st["X"] = _normal(g, dt, B, n, c["width"])
    st["K"] = st["V"] = None
    if c["kv_cache"]:
        st["K"] = _normal(g, dt, B, c["heads"], n, c["head_dim"])
        st["V"] = _normal(g, dt, B, c["heads"], n, c["head_dim"])
    if c["sim"] == "X":
        _near_copies(st["X"], order, c, 1, src)
    if c["sim"] == "meanK":
        _near_copies(st["K"], order, c, 2, src)
    if c["call"] == "host":
        for k in ("O", "A", "X", "K", "V"):
            if st[k] is not None:
                st[k] = st[k].cpu().pin_memory()
        pin = lambda t: None if t is None else torch.empty(t, dtype=dt, pin_memory=True)  # noqa: E731
        kv = (B, c["heads"], c["keep"], c["head_dim"]) if c["kv_cache"] else None
        st["out"] = (pin((B, c["keep"], c["width"])), pin(kv), pin(kv),
                     torch.empty(B, c["keep"], dtype=torch.int32, pin_memory=True),
                     torch.empty(B, dtype=torch.int32, pin_memory=True))
    st["ws"] = tcb.workspace(st["p"], host=c["call"] == "host")
    return st


def run(s):
    c, p = s["c"], s["p"]
    if c["call"] == "carve":
        return tcb.tc_carve(p, s["O"], s["A"], s["X"], s["K"], s["V"], ws=s["ws"])
    if c["call"] == "host":
        return tcb.tc_carve_host(p, s["O"], s["A"], s["X"], s["K"], s["V"], s["out"], s["ws"])
    if c["call"] == "staged":
        sc = tcb.tc_score(p, s["O"], s["A"], s["ws"])
        a, b = tcb.tc_prune(p, sc["E"], s["ws"])
        src, dst, kept = tcb.tc_merge(p, s["O"], a, b, s["ws"])
        if c["weighted"]:
            x, k, v = tcb.tc_compact_weighted(p, s["X"], s["K"], s["V"], kept, src, dst, sc["E"], s["ws"])
        else:
            x, k, v = tcb.tc_compact(p, s["X"], s["K"], s["V"], kept, src, dst, s["ws"])
        return sc, a, b, src, dst, kept, x, k, v
    if c["call"] == "probe":
        return tcb.tc_probe(p, c["n_sys"], c["n_text"], c["n_sys"] + c["tokens"] + c["n_text"] - c["query"],
                            s["q"], s["k"], s["v"])
    h, pos = tcb.tc_reassemble(p, c["n_sys"], c["n_text"], s["h"], s["x"], s["kept"])
    cos, sin = tcb.tc_rope_tables(pos, c["head_dim"])
    return h, pos, cos, sin


def work(case):
    c = case
    B, n, e = c["batch"], c["tokens"], BYTES[c["dtype"]]
    if c["call"] == "probe":
        # queries of the visual and probe rows, all keys and values once; O and A written.  Scores
        # and products with V over what a causal row sees, the probe rows' scores.
        H, L, T = c["heads"], c["n_sys"] + n + c["n_text"], c["query"]
        seen = sum(range(c["n_sys"] + 1, c["n_sys"] + n + 1))
        probe = sum(range(L - T + 1, L + 1))
        return {"bytes": B * H * e * (128 * (n + T + 2 * L + n) + T * n), "flops": B * H * 2 * 128 * (2 * seen + probe)}
    if c["call"] == "resume":
        rows = c["n_sys"] + c["keep"] + c["n_text"]
        return {"bytes": B * (2 * rows * c["width"] * e + rows * (4 + 4 * c["head_dim"])), "flops": B * rows * c["head_dim"]}
    # O and A once, the survivors' rows of X, K and V, the kept rows written; the symmetric Gram
    # matrix, one product with a basis of the rank, and the eigenvectors of its projection
    m, p, _, _ = _counts(c)
    d, H, r = c["width"], c["heads"], c["rank"]
    per_row = d * e + (2 * H * c["head_dim"] * e if c["kv_cache"] else 0)
    read = (n * d * e if c["call"] != "host" else 0) + H * c["query"] * n * e + p * per_row + c["keep"] * per_row
    if c["call"] == "host":
        read += n * d * e
    return {"bytes": B * read, "flops": B * (n * n * d + 2 * n * n * r + 4 * r ** 3 // 3 + 2 * n * r * r)}


def tolerance(case):
    """Lists and copied rows are the same whatever the rounding of the scores (see the module text);
    merged rows are one rounding of a float32 mean; the scores and singular values of a staged call
    come from a float32 Gram matrix; probabilities are rounded to the storage type before they
    multiply V in the probe."""
    eps = {"f16": 2.0 ** -11, "bf16": 2.0 ** -8, "f32": 1e-5}[case["dtype"]]
    if case["call"] == "probe":
        return {"rel": 4 * eps}
    if case["call"] == "resume":
        return {"rel": 1e-6}
    if case["call"] == "staged":
        return {"rel": max(eps, 2e-4)}
    return {"rel": max(eps, 5e-5) if case["weighted"] else eps}   # (the weights are those scores)
