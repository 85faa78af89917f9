"""Timed cases of the attribution path, through the public entry points.

Six kinds of call, as a program that attributes a model's behaviour makes them:

  collect  one batch of captured activations and output gradients -> projected
           gradients -> unit-norm fp16 store rows (bergson_project_grads, then
           bergson_build_store or _build_store_blocks)
  tokens   per-token scores of one batch against query rows
  search   exact top-k / bottom-k of queries against a store, in one call or
           chunk by chunk (bergson_score_topk_update)
  grads    on-the-fly scores of a batch of projected rows, no store
  apply    Fisher-preconditioned rows of a batch
  fisher   the one-time Fisher fit and its inverse square root

Layer shapes are the workloads of paper_2606_11660_gb300.workloads.  Stores
that live in host memory run at the host link's rate and are not timed here.
"""
from __future__ import annotations

import math
import random

import torch

import paper_2606_11660_gb300 as bg
from paper_2606_11660_gb300 import workloads as wl

DEV = "cuda"
KINDS = {"gaussian": bg.BERGSON_PROJ_GAUSSIAN, "rademacher": bg.BERGSON_PROJ_RADEMACHER,
         "uniform": bg.BERGSON_PROJ_UNIFORM}
MAX_COLLECT_BYTES = 19.4e9          # the largest batch: 48 modules, 32 x 2048 tokens
MAX_SEARCH_FLOPS = 2 * 4e6 * 8192 * 1024
MAX_SEARCH_BYTES = 4e6 * 8192 * 2
EXACT_FLOPS = 1e13                  # what 64-bit arithmetic does in some ten seconds


def listed():
    return [
        # One small linear layer and a handful of short examples: a unit-size
        # call (a toy model, a debugging session), where launches are all there is.
        dict(name="collect_tiny", op="collect", family="tiny", blocks=1, B=8, T=32, pad=0,
             k_in=16, k_out=16, kind="gaussian", moments=True, bias=False, per_module=False),
        # The last, ragged batch of a fine-tuning set: few short examples of
        # odd length, weight and bias gradients, Rademacher projections and
        # per-module unit norms.
        dict(name="collect_short", op="collect", family="pythia160m", blocks=2, B=7, T=333, pad=90,
             k_in=32, k_out=16, kind="rademacher", moments=False, bias=True, per_module=True),
        # A whole Pythia-160M-shaped model at the paper's sequence scale, one call per batch.
        dict(name="collect_160m", op="collect", family="pythia160m", blocks=12, B=32, T=2048,
             pad=409, k_in=16, k_out=16, kind="gaussian", moments=False, bias=False,
             per_module=False),
        # Larger models are collected a transformer block at a time, as their
        # activations come: Adafactor moments and k = 32 here, ...
        dict(name="collect_1b4_block", op="collect", family="pythia1b4", blocks=1, B=16, T=2048,
             pad=0, k_in=32, k_out=32, kind="gaussian", moments=True, bias=False,
             per_module=False),
        # ... and wide layers, two of which read one input, here.
        dict(name="collect_8b_block", op="collect", family="llama8b", blocks=1, B=8, T=4096, pad=0,
             k_in=16, k_out=16, kind="gaussian", moments=False, bias=False, per_module=False),
        # Which tokens of eight documents drive each of 64 query behaviours.
        dict(name="tokens_160m", op="tokens", family="pythia160m", blocks=12, B=8, T=2048, pad=409,
             k_in=16, k_out=16, kind="gaussian", moments=False, queries=64),
        # Interactive lookups against a small store.
        dict(name="search_small", op="search", N=20_011, K=3072, Q=3, topk=10, least=False,
             chunks=1),
        # An evaluation set against a fine-tuning store (K of the 48-module
        # model): the least influential rows.
        dict(name="search_mid", op="search", N=250_007, K=12_288, Q=100, topk=100, least=True,
             chunks=1),
        # A thousand queries against a pre-training store that fills HBM to a quarter.
        dict(name="search_batch", op="search", N=4_000_000, K=8192, Q=1024, topk=100, least=False,
             chunks=1),
        # Streaming attribution without a store, per training batch ...
        dict(name="grads_1024", op="grads", B=32, Q=1024, K=12_288, unit=True),
        # ... and the Fisher preconditioner applied to each batch.
        dict(name="apply_12288", op="apply", B=32, K=12_288),
        # Fitting that preconditioner on a model of 12 modules.
        dict(name="fisher_3072", op="fisher", n=1024, K=3072, damping=0.1, power="inv_sqrt",
             tol=1e-5),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["collect", "collect", "tokens", "search", "search", "grads", "apply",
                     "fisher"])
    if op in ("collect", "tokens"):
        family = rng.choice(["tiny", "pythia160m", "pythia160m", "pythia1b4", "llama8b"])
        while True:
            c = dict(op=op, family=family,
                     blocks=_log(rng, 1, 12) if family == "pythia160m" else 1,
                     B=_log(rng, 1, 32), T=_log(rng, 16, 4096), pad=0,
                     k_in=rng.choice([16, 16, 16, 32, 64]), k_out=16,
                     kind=rng.choice(["gaussian", "gaussian", "rademacher", "uniform"]),
                     moments=rng.random() < 0.4)
            c["pad"] = rng.choice([0, c["T"] // 5, c["T"] // 2])
            c["k_out"] = c["k_in"] if rng.random() < 0.7 else rng.choice([16, 32, 64])
            if op == "collect":
                c.update(bias=rng.random() < 0.25, per_module=rng.random() < 0.25)
            else:
                c["queries"] = _log(rng, 1, 256)
            w = work(c)
            # (k_in, k_out) = (64, 64) with hundreds of queries is all products:
            # keep a drawn case within the largest listed one's time
            if w["bytes"] <= MAX_COLLECT_BYTES and w["flops"] <= 2e12:
                return c
    if op == "search":
        while True:
            c = dict(op=op, N=_log(rng, 500, 4_000_000), K=8 * _log(rng, 32, 1536),
                     Q=_log(rng, 1, 1024), topk=_log(rng, 1, 500), least=rng.random() < 0.3,
                     chunks=rng.choice([1, 1, 1, 3]))
            c["topk"] = min(c["topk"], c["N"])
            w = work(c)
            if w["bytes"] <= MAX_SEARCH_BYTES and w["flops"] <= MAX_SEARCH_FLOPS:
                return c
    if op == "grads":
        return dict(op=op, B=_log(rng, 1, 200), Q=_log(rng, 1, 8192), K=4 * _log(rng, 64, 3072),
                    unit=rng.random() < 0.7)
    if op == "apply":
        return dict(op=op, B=_log(rng, 1, 200), K=4 * _log(rng, 64, 3072))
    return dict(op=op, n=_log(rng, 64, 4096), K=4 * _log(rng, 64, 1024),
                damping=rng.choice([0.1, 0.03]), power=rng.choice(["inv_sqrt", "inv_sqrt", "inv"]),
                tol=1e-5)


# ------------------------------------------------------------------ inputs

def _gen(seed):
    return wl.generator(seed, DEV)


def _modules(c):
    w = wl.COLLECT_WORKLOADS[c["family"]]
    return [s for b in range(c["blocks"]) for s in w.block_modules(b)]


def _lengths(c):
    """Tokens of each example (right padding up to `pad`): fixed by the case, not the seed."""
    r = random.Random("%d %d %d" % (c["B"], c["T"], c["pad"]))
    return [c["T"] - r.randint(0, c["pad"]) for _ in range(c["B"])]


def _mask(c):
    if c["pad"] == 0:
        return None
    n = torch.tensor(_lengths(c), device=DEV)
    return (torch.arange(c["T"], device=DEV)[None, :] < n[:, None]).to(torch.uint8)


def _module_tensors(c, seed):
    """(A, G, r, c) per module: activations ~ N(0,1)/sqrt(d), bf16, moments ~ U(0.5, 2)."""
    g = _gen(seed)
    out = []
    for s in _modules(c):
        def rows(d):
            x = torch.randn((c["B"], c["T"], d), generator=g, device=DEV, dtype=torch.bfloat16)
            return x.mul_(d ** -0.5)
        A = out[-1][0] if s.shares_input else rows(s.d_in)
        G = rows(s.d_out)
        r = ci = None
        if c["moments"]:
            r = torch.rand((s.d_out,), generator=g, device=DEV) * 1.5 + 0.5
            ci = torch.rand((s.d_in,), generator=g, device=DEV) * 1.5 + 0.5
        out.append((A, G, r, ci))
    return out


def _columns(c):
    """(weight block offsets with the end, bias offsets, row length)."""
    n, kk, ko = len(_modules(c)), c["k_in"] * c["k_out"], c["k_out"]
    w = [i * kk for i in range(n + 1)]
    bias = [n * kk + i * ko for i in range(n)] if c.get("bias") else [None] * n
    return w, bias, n * kk + (n * ko if c.get("bias") else 0)


def _layers(c, tensors, seed):
    w, bias, _ = _columns(c)
    layers = []
    for i, (A, G, r, ci) in enumerate(tensors):
        s_in, s_out = bg.bergson_module_seeds(seed, i)
        layers.append(bg.Layer(A, G, c["k_in"], c["k_out"], s_in, s_out, r, ci, w[i],
                               proj_kind=KINDS[c["kind"]], bias_col_offset=bias[i]))
    return layers


def _token_queries(c, seed):
    _, _, K = _columns(c)
    return torch.randn((c["queries"], K), generator=_gen(seed + 7_000_003), device=DEV)


def _store_and_queries(c, seed):
    """Unit rows scattered around 64 topics (documents in no order), queries from the same topics."""
    g = _gen(seed)
    N, K = c["N"], c["K"]
    topics = torch.randn((64, K), generator=g, device=DEV) * 0.25
    store = torch.empty((N, K), dtype=torch.float16, device=DEV)
    step = max(1, (1 << 29) // K)
    for r0 in range(0, N, step):
        n = min(step, N - r0)
        x = torch.randn((n, K), generator=g, device=DEV)
        x += topics[torch.randint(0, 64, (n,), generator=g, device=DEV)]
        x *= 1.0 / torch.linalg.vector_norm(x, dim=1, keepdim=True)
        store[r0:r0 + n] = x
    q = torch.randn((c["Q"], K), generator=g, device=DEV)
    q += topics[torch.randint(0, 64, (c["Q"],), generator=g, device=DEV)]
    return store, q


def _rows(n, K, seed):
    """Projected gradient rows: a common direction and noise."""
    g = _gen(seed)
    return torch.randn((n, K), generator=g, device=DEV) + \
        0.1 * torch.randn((1, K), generator=g, device=DEV)


def _preconditioner(K, seed):
    """A symmetric K x K matrix like a damped R^-1/2: a multiple of I less a low-rank part."""
    x = _rows(min(K, 256), K, seed + 1_000_003)
    M = x.T @ x
    M *= -1.0 / (4 * K)
    M.diagonal().add_(3.0)
    return M


def prepare(case, seed):
    c, op = case, case["op"]
    s = {"case": c}
    if op in ("collect", "tokens"):
        s["layers"] = _layers(c, _module_tensors(c, seed), seed)
        s["mask"] = _mask(c)
        w, _, K = _columns(c)
        if op == "collect":
            s["blocks"] = w + ([K] if c["bias"] else [])
            s["K"] = K
            s["ws"] = bg.workspace_tensor(
                bg.bergson_project_grads_workspace(s["layers"], c["B"], c["T"]))
            s["proj"] = torch.empty((c["B"], K), device=DEV)
            s["store"] = torch.empty((c["B"], K), dtype=torch.float16, device=DEV)
        else:
            s["queries"] = _token_queries(c, seed)
            s["ws"] = bg.workspace_tensor(bg.bergson_token_scores_workspace(
                s["layers"], c["B"], c["T"], c["queries"]))
            s["out"] = torch.empty((c["queries"], c["B"], c["T"]), device=DEV)
    elif op == "search":
        s["store"], s["queries"] = _store_and_queries(c, seed)
        s["ws"] = bg.workspace_tensor(
            bg.bergson_score_topk_workspace(c["N"], c["K"], c["Q"], c["topk"]))
        s["scores"] = torch.empty((c["Q"], c["topk"]), device=DEV)
        s["idx"] = torch.empty((c["Q"], c["topk"]), dtype=torch.int64, device=DEV)
        n = -(-c["N"] // c["chunks"])
        s["chunks"] = [(r0, min(n, c["N"] - r0)) for r0 in range(0, c["N"], n)]
    elif op == "grads":
        s["x"], s["y"] = _rows(c["B"], c["K"], seed), _rows(c["Q"], c["K"], seed + 5_000_011)
        s["ws"] = bg.workspace_tensor(bg.bergson_score_grads_workspace(c["B"], c["K"], c["Q"]))
        s["out"] = torch.empty((c["B"], c["Q"]), device=DEV)
    elif op == "apply":
        s["x"], s["M"] = _rows(c["B"], c["K"], seed), _preconditioner(c["K"], seed)
        s["ws"] = bg.workspace_tensor(bg.bergson_score_grads_workspace(c["B"], c["K"], c["K"]))
        s["out"] = torch.empty((c["B"], c["K"]), device=DEV)
    else:
        K = c["K"]
        s["x"] = _rows(c["n"], K, seed)
        s["R"], s["M"] = torch.empty((K, K), device=DEV), torch.empty((K, K), device=DEV)
        s["fit_ws"] = bg.workspace_tensor(bg.bergson_fisher_fit_workspace(c["n"], K))
        s["ws"] = bg.workspace_tensor(bg.bergson_fisher_preconditioner_workspace(K))
    return s


# --------------------------------------------------------------------- run

def run(s):
    c = s["case"]
    op = c["op"]
    if op == "collect":
        B, K = c["B"], s["K"]
        bg.bergson_project_grads(s["layers"], B, c["T"], s["mask"], s["proj"], s["ws"])
        if c["per_module"]:
            bg.bergson_build_store_blocks(s["proj"], B, K, s["blocks"], s["store"], 0)
        else:
            bg.bergson_build_store(s["proj"], B, K, True, s["store"], 0)
        return {"proj": s["proj"], "store": s["store"]}
    if op == "tokens":
        bg.bergson_token_scores(s["layers"], c["B"], c["T"], s["mask"], s["queries"], s["out"],
                                s["ws"])
        return {"scores": s["out"]}
    if op == "search":
        if c["chunks"] == 1:
            fn = bg.bergson_score_bottomk if c["least"] else bg.bergson_score_topk
            fn(s["store"], c["N"], c["K"], s["queries"], c["topk"], s["scores"], s["idx"], s["ws"])
        else:
            for i, (r0, n) in enumerate(s["chunks"]):
                bg.bergson_score_topk_update(s["store"][r0:], n, c["K"], r0, s["queries"],
                                             c["topk"], i == 0, s["scores"], s["idx"], s["ws"],
                                             least=c["least"])
        return {"scores": s["scores"], "idx": s["idx"]}
    if op == "grads":
        bg.bergson_score_grads(s["x"], c["B"], c["K"], s["y"], c["unit"], s["out"], s["ws"])
        return {"scores": s["out"]}
    if op == "apply":
        bg.bergson_precondition_rows(s["x"], c["B"], c["K"], s["M"], s["out"], s["ws"])
        return {"rows": s["out"]}
    power = bg.BERGSON_FISHER_INV if c["power"] == "inv" else bg.BERGSON_FISHER_INV_SQRT
    bg.bergson_fisher_fit(s["x"], c["n"], c["K"], s["R"], s["fit_ws"])
    bg.bergson_fisher_preconditioner_tol(s["R"], None, c["K"], 1.0, c["damping"], power, 40,
                                         c["tol"], s["M"], s["ws"])
    return {"R": s["R"], "M": s["M"]}


def work(case):
    c, op = case, case["op"]
    if op in ("collect", "tokens"):
        valid = sum(_lengths(c))
        mods = _modules(c)
        d_read = sum((0 if m.shares_input else m.d_in) + m.d_out for m in mods)
        flops = 2 * valid * sum(m.d_in * c["k_in"] + m.d_out * c["k_out"] for m in mods)
        _, _, K = _columns(c)
        if op == "collect":
            return {"bytes": 2 * valid * d_read + c["B"] * K * (4 + 2),
                    "flops": flops + 2 * valid * len(mods) * c["k_in"] * c["k_out"]}
        q = c["queries"]
        return {"bytes": 2 * valid * d_read + 4 * q * K + 4 * q * c["B"] * c["T"],
                "flops": flops + 2 * valid * len(mods) * q * (c["k_in"] * c["k_out"] +
                                                              min(c["k_in"], c["k_out"]))}
    if op == "search":
        return {"bytes": 2 * c["N"] * c["K"] + c["Q"] * (4 * c["K"] + 12 * c["topk"]),
                "flops": 2 * c["N"] * c["K"] * c["Q"]}
    if op == "grads":
        return {"bytes": 4 * ((c["B"] + c["Q"]) * c["K"] + c["B"] * c["Q"]),
                "flops": 2 * c["B"] * c["Q"] * c["K"]}
    if op == "apply":
        return {"bytes": 4 * (c["K"] ** 2 + 2 * c["B"] * c["K"]), "flops": 2 * c["B"] * c["K"] ** 2}
    # the Gram matrix (one triangle), and an iteration of three symmetric
    # products per step, some twelve steps for these condition numbers
    return {"bytes": 4 * (c["n"] * c["K"] + 2 * c["K"] ** 2),
            "flops": c["n"] * c["K"] ** 2 + 12 * 3 * c["K"] ** 3}


def tolerance(case):
    """About four times the error measured against exact() on the case's own inputs."""
    op = case["op"]
    if op == "collect":
        # fp32 rows 1e-6 .. 2e-5 off; their fp16 copies may round the other way (one ulp, 1e-3)
        return {"rel": 1e-4, "max": 2e-3}
    if op == "tokens":
        return {"rel": 2e-5, "max": 1e-3}
    if op == "search":
        # sums of thousands of fp16 products in the tensor cores' fp32 (truncating) adders, 4e-5 ..
        # 6e-5 off with the queries' fp16 rounding; rows with near-equal scores may change places
        return {"rel": 1e-4, "max": 1e-3, "differ": 0.01}
    if op in ("grads", "apply"):
        return {"rel": 4e-6, "max": 1e-4}
    # M is off by what the iteration leaves (its residual stops at 1e-5), up to 8e-5
    return {"rel": 4e-4, "max": 2e-2}


# ------------------------------------------------- the same in 64 bits, plain torch

def _i64(v):
    return v - (1 << 64) if v >= (1 << 63) else v


def _shr(x, n):
    return (x >> n) & ((1 << (64 - n)) - 1)


def _mix(x):
    """The SplitMix64 finaliser on int64 tensors (wrapping)."""
    x = (x ^ _shr(x, 30)) * _i64(0xBF58476D1CE4E5B9)
    x = (x ^ _shr(x, 27)) * _i64(0x94D049BB133111EB)
    return x ^ _shr(x, 31)


def _projection(seed, d, k, kind):
    """P [d, k] as the public header defines it, in fp64."""
    e = torch.arange(d * k, device=DEV, dtype=torch.int64)
    seed = _i64(seed)
    if kind == "gaussian":
        p = _shr(e, 1)
        h1, h2 = _mix(_mix(2 * p) ^ seed), _mix(_mix(2 * p + 1) ^ seed)
        u1 = (_shr(h1, 11) + 1).double() * 2.0 ** -53
        u2 = _shr(h2, 11).double() * 2.0 ** -53
        rad, ang = torch.sqrt(-2.0 * torch.log(u1)), 2.0 * math.pi * u2
        z = torch.where(e % 2 == 0, rad * torch.cos(ang), rad * torch.sin(ang))
    else:
        h = _mix(_mix(e) ^ seed)
        if kind == "rademacher":
            z = torch.where(h < 0, 1.0, -1.0).double()
        else:
            z = math.sqrt(3.0) * ((2 * _shr(h, 40) + 1).double() * 2.0 ** -24 - 1.0)
    return (z / math.sqrt(k)).float().double().reshape(d, k)


def _token_projections(c, seed):
    """Per module: (a~ [B, T, k_in], g~ [B, T, k_out]) in fp64, masked tokens zero."""
    mask = _mask(c)
    for i, (A, G, r, ci) in enumerate(_module_tensors(c, seed)):
        seeds = bg.bergson_module_seeds(seed, i)
        out = []
        for x, k, sd, m in ((A, c["k_in"], seeds[0], ci), (G, c["k_out"], seeds[1], r)):
            P = _projection(sd, x.shape[-1], k, c["kind"])
            if m is not None:
                P = P / m.double().sqrt()[:, None]
            y = torch.stack([xb.double() @ P for xb in x])
            out.append(y if mask is None else y * (mask != 0)[:, :, None])
        yield out


def exact(case, seed):
    c, op = case, case["op"]
    if op == "collect":
        w, bias, K = _columns(c)
        proj = torch.zeros((c["B"], K), dtype=torch.float64, device=DEV)
        for i, (a, g) in enumerate(_token_projections(c, seed)):
            proj[:, w[i]:w[i + 1]] = torch.bmm(g.transpose(1, 2), a).reshape(c["B"], -1)
            if bias[i] is not None:
                proj[:, bias[i]:bias[i] + c["k_out"]] = g.sum(1)
        ends = (w + ([K] if c["bias"] else [])) if c["per_module"] else [0, K]
        store = torch.empty_like(proj)
        for o0, o1 in zip(ends[:-1], ends[1:]):
            x = proj[:, o0:o1]
            n = torch.linalg.vector_norm(x, dim=1, keepdim=True)
            store[:, o0:o1] = x / torch.where(n > 0, n, 1.0)
        return {"proj": proj, "store": store}
    if op == "tokens":
        q = _token_queries(c, seed).double()
        w, _, _ = _columns(c)
        out = torch.zeros((c["queries"], c["B"], c["T"]), dtype=torch.float64, device=DEV)
        for i, (a, g) in enumerate(_token_projections(c, seed)):
            for j in range(c["queries"]):
                block = q[j, w[i]:w[i + 1]].reshape(c["k_out"], c["k_in"])
                out[j] += ((g @ block) * a).sum(-1)
        return {"scores": out}
    if op == "search":
        if work(c)["flops"] > EXACT_FLOPS:
            return None
        store, queries = _store_and_queries(c, seed)
        q = queries.double()
        q = q / torch.linalg.vector_norm(q, dim=1, keepdim=True)
        best = None
        for r0 in range(0, c["N"], 1 << 16):
            sc = q @ store[r0:r0 + (1 << 16)].double().T
            sc = sc if best is None else torch.cat([best, sc], 1)
            best = sc.topk(min(c["topk"], sc.shape[1]), dim=1, largest=not c["least"]).values
        return {"scores": best, "idx": None}
    if op == "grads":
        x = _rows(c["B"], c["K"], seed).double()
        y = _rows(c["Q"], c["K"], seed + 5_000_011).double()
        if c["unit"]:
            x = x / torch.linalg.vector_norm(x, dim=1, keepdim=True)
            y = y / torch.linalg.vector_norm(y, dim=1, keepdim=True)
        return {"scores": x @ y.T}
    if op == "apply":
        return {"rows": _rows(c["B"], c["K"], seed).double() @ _preconditioner(c["K"], seed).double()}
    x = _rows(c["n"], c["K"], seed).double()
    R = x.T @ x / c["n"]
    D = R.clone()
    D.diagonal().add_(c["damping"] * float(R.trace()) / c["K"])
    lam, V = torch.linalg.eigh(D)
    M = (V * lam.pow(-1.0 if c["power"] == "inv" else -0.5)) @ V.T
    return {"R": R, "M": M}
