"""Workloads by which the speed of the attribution path is measured.

Each case is work that a user of the library has it do through its public entry
points: projecting per-example gradients of one linear layer (the bulk of every
job), preconditioning queries, scoring and ranking, exact similarities with
norms and cosine, token-level scores, EK-FAC, and one whole small pass. Sizes
are those of the repository's own workloads (a 256 x 256 fp32 layer, a
Llama-style 1B block, a Llama-3-8B-shaped stack, large-model layers) and of its
tests, or lie in the ranges between them.

A case is a dict of plain values; ``kind`` names the path. ``listed()`` gives
the fixed cases, ``draw(rng)`` one more of the same ranges, ``prepare`` the
device buffers and inputs that a user's program holds before the call, ``run``
one pass, ``work`` the bytes and operations that no implementation can do
without, ``exact`` the outputs in 64 bits by plain torch.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2609_38767_gb300 as tda

SEED = 0          # projection seed: fixed for gradients that are to be compared
LAYER = 3         # layer index of the single-layer cases
MASKED = 0.01     # share of padded (zero) tokens
BF16, F32 = "bf16", "f32"


# ------------------------------------------------------------------------ cases
def listed():
    return [
        # The smallest job: one 256 x 256 fp32 layer, 64 train and 8 query examples of 32 tokens,
        # fp64 preconditioner state, all steps from the factors to the ranking. Launches and latency.
        dict(name="pass_256_fp32", kind="pass", d_in=256, d_out=256, T=32, k=16, N=64, n_q=8, topk=10),
        # MLP-up linear of the Llama-style 1B block: a part of the resident training set.
        dict(name="project_1b_up_k32", kind="project", dtype=BF16, d_in=2048, d_out=8192, T=512, k_in=32, k_out=32,
             N=128, ws=False),
        # Gate linear of the Llama-3-8B-shaped stack, one 256-example chunk: the largest launch of a job.
        dict(name="project_8b_gate_k64", kind="project", dtype=BF16, d_in=4096, d_out=14336, T=1024, k_in=64,
             k_out=64, N=256, ws=False),
        # Grouped-query k/v linear of the large-model layers, with the optional workspace.
        dict(name="project_large_kv_k128", kind="project", dtype=BF16, d_in=12288, d_out=1536, T=2048, k_in=128,
             k_out=128, N=32, ws=True),
        # Ragged everything: token count, widths that no tile divides, different projection sizes per side.
        dict(name="project_ragged_bf16", kind="project", dtype=BF16, d_in=1000, d_out=2056, T=130, k_in=32, k_out=48,
             N=96, ws=False),
        # fp32 factors (a model trained in fp32): attention linear of the 1B block.
        dict(name="project_1b_q_fp32", kind="project", dtype=F32, d_in=2048, d_out=2048, T=512, k_in=32, k_out=32,
             N=64, ws=False),
        # Curvature fit, factorisation and query solves of the seven linears of the 1B block.
        dict(name="precondition_1b", kind="precondition", D=1024, layers=7, N=4096, n_q=64),
        # The same for a layer's seven linears of the 8B stack: one step's share of the query side.
        dict(name="precondition_8b", kind="precondition", D=4096, layers=7, N=8192, n_q=256),
        # Query x train scores over the features of the 1B block's seven linears, for the stack's 8192 train
        # examples and 256 queries, and the ranking of a finished score matrix.
        dict(name="score_topk_7168", kind="score", D=7168, N=8192, n_q=256, topk=100),
        # Cosine of unprojected gradients (similarities and both sides' norms), sequences of 50 tokens.
        dict(name="cosine_exact_t50", kind="cosine", dtype=BF16, d_in=2048, d_out=2048, T=50, N=512, n_q=16),
        # Token-level scores of a few training examples against preconditioned queries (8B attention linear).
        dict(name="token_scores_8b_k64", kind="tokens", dtype=BF16, d_in=4096, d_out=4096, T=1024, k_in=64, k_out=64,
             N=16, n_q=16),
        # EK-FAC over the attention and MLP linears of the 1B block, a part of its training set.
        dict(name="ekfac_1b", kind="ekfac", widths="2048x2048,2048x8192,8192x2048", T=512, k=32, N=256, n_q=64),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _width(rng, lo, hi):
    w = _log(rng, lo, hi)
    return max(8, w // 8 * 8 if rng.random() < 0.5 else w // 64 * 64 or 64)


def draw(rng):
    kind = rng.choice(["pass", "project", "project", "project_odd", "project_fp32", "precondition", "precondition",
                       "score", "cosine", "tokens", "ekfac"])
    if kind == "pass":
        N = _log(rng, 16, 256)
        return dict(kind="pass", d_in=_width(rng, 64, 512), d_out=_width(rng, 64, 512), T=_log(rng, 4, 64),
                    k=rng.choice([8, 12, 16]), N=N, n_q=rng.randint(1, 16), topk=min(10, N))
    if kind == "project":
        k = rng.choice([16, 32, 64, 128])
        d_in, d_out, T = _width(rng, 256, 12288), _width(rng, 256, 14336), _log(rng, 8, 2048)
        most = 6e9 / (2.0 * T * (d_in + d_out))
        return dict(kind="project", dtype=BF16, d_in=d_in, d_out=d_out, T=T, k_in=k, k_out=k,
                    N=max(1, min(_log(rng, 4, 4096), int(most))), ws=rng.random() < 0.5)
    if kind in ("project_odd", "project_fp32"):
        ks = [8, 16, 24, 32, 48, 64]
        k_in, k_out = rng.choice(ks), rng.choice(ks)
        if kind == "project_fp32" and rng.random() < 0.7:
            k_in = k_out = rng.choice([16, 32, 64])
        d_in, d_out, T = _width(rng, 128, 4096), _width(rng, 128, 4096), _log(rng, 8, 1024)
        most = 4e8 / (4.0 * T * (d_in + d_out))
        return dict(kind="project", dtype=BF16 if kind == "project_odd" else F32, d_in=d_in, d_out=d_out, T=T,
                    k_in=k_in, k_out=k_out, N=max(1, min(_log(rng, 4, 512), int(most))), ws=False)
    if kind == "precondition":
        D = rng.choice([256, 576, 1024, 1600, 2304, 4096])
        return dict(kind="precondition", D=D, layers=rng.randint(1, 7), N=D * 2 + rng.randint(0, min(D, 2048)),
                    n_q=_log(rng, 4, 256))
    if kind == "score":
        return dict(kind="score", D=rng.choice([256, 576, 1024]) * rng.randint(1, 7), N=_log(rng, 200, 8192),
                    n_q=_log(rng, 4, 256), topk=100)
    if kind == "cosine":
        return dict(kind="cosine", dtype=BF16, d_in=_width(rng, 256, 4096), d_out=_width(rng, 256, 4096),
                    T=_log(rng, 5, 64), N=_log(rng, 32, 512), n_q=rng.randint(1, 16))
    if kind == "tokens":
        k = rng.choice([16, 32, 64])
        return dict(kind="tokens", dtype=BF16, d_in=_width(rng, 256, 4096), d_out=_width(rng, 256, 4096),
                    T=_log(rng, 64, 1024), k_in=k, k_out=k, N=_log(rng, 1, 16), n_q=_log(rng, 1, 64))
    w = [(_width(rng, 256, 4096), _width(rng, 256, 4096)) for _ in range(rng.randint(1, 3))]
    return dict(kind="ekfac", widths=",".join("%dx%d" % p for p in w), T=_log(rng, 32, 512),
                k=rng.choice([16, 32, 64]), N=_log(rng, 64, 256), n_q=_log(rng, 4, 64))


# ----------------------------------------------------------------------- inputs
def _gen(seed, stream):
    g = torch.Generator(device="cuda")
    g.manual_seed((seed * 1000003 + stream) % (1 << 62))
    return g


def _factors(seed, stream, N, T, d_in, d_out, dtype):
    """Activations ~ N(0, 1) and output gradients ~ N(0, 1e-3) of N examples, padded tokens zero in both."""
    td = torch.bfloat16 if dtype == BF16 else torch.float32
    g = _gen(seed, stream)
    A = torch.randn((N, T, d_in), generator=g, device="cuda", dtype=td)
    B = torch.randn((N, T, d_out), generator=g, device="cuda", dtype=td).mul_(math.sqrt(1e-3))
    pad = torch.rand((N, T), generator=g, device="cuda") < MASKED
    A[pad] = 0
    B[pad] = 0
    return A, B


def _features(seed, stream, N, D):
    """Feature rows with a different scale for each feature."""
    g = _gen(seed, stream)
    x = torch.randn((N, D), generator=g, device="cuda")
    return x.mul_(torch.rand(D, generator=g, device="cuda").mul_(1.5).add_(0.5))


def _bytes(n):
    return torch.empty(max(int(n), 256), dtype=torch.uint8, device="cuda")


def _code(c):
    return tda.TDA_BF16 if c.get("dtype") == BF16 else tda.TDA_F32


def _widths(c):
    return [tuple(int(x) for x in p.split("x")) for p in c["widths"].split(",")]


def prepare(case, seed):
    c, kind = dict(case), case["kind"]
    s = {"case": c}
    f = dict(device="cuda", dtype=torch.float32)
    if kind == "pass":
        D = c["k"] * c["k"]
        s["A"], s["B"] = _factors(seed, 1, c["N"], c["T"], c["d_in"], c["d_out"], F32)
        s["Aq"], s["Bq"] = _factors(seed, 2, c["n_q"], c["T"], c["d_in"], c["d_out"], F32)
        s["L"] = tda.LayerDesc(c["d_in"], c["d_out"], c["T"], c["k"], c["k"], seed=SEED, layer=LAYER)
        s["phi"], s["q"] = torch.empty((c["N"], D), **f), torch.empty((c["n_q"], D), **f)
        s["qhat"] = torch.empty((c["n_q"], D), device="cuda", dtype=torch.float64)
        s["state"] = _bytes(tda.tda_precondition_state_bytes(D, tda.TDA_F64))
        s["S"] = torch.empty((c["n_q"], c["N"]), **f)
        s["idx"] = torch.empty((c["n_q"], c["topk"]), device="cuda", dtype=torch.int32)
        s["val"] = torch.empty((c["n_q"], c["topk"]), **f)
    elif kind == "project":
        s["A"], s["B"] = _factors(seed, 1, c["N"], c["T"], c["d_in"], c["d_out"], c["dtype"])
        s["L"] = tda.LayerDesc(c["d_in"], c["d_out"], c["T"], c["k_in"], c["k_out"], seed=SEED, layer=LAYER)
        s["phi"] = torch.empty((c["N"], c["k_in"] * c["k_out"]), **f)
        n = tda.tda_workspace_size(tda.TDA_OP_PROJECT, s["L"], _code(c), c["N"], 0, tda.TDA_ROUTE_FACTORED)
        s["ws"], s["wsb"] = (_bytes(n), n) if c["ws"] and n else (None, 0)
    elif kind == "precondition":
        w = c["layers"] * c["D"]
        s["phi"] = _features(seed, 1, c["N"], w)
        s["q"] = _features(seed, 2, c["n_q"], w)
        s["qhat"] = torch.empty((c["n_q"], w), **f)
        s["state"] = _bytes(c["layers"] * tda.tda_precondition_state_bytes(c["D"], tda.TDA_F32))
    elif kind == "score":
        s["phi"] = _features(seed, 1, c["N"], c["D"])
        s["qhat"] = _features(seed, 2, c["n_q"], c["D"])
        s["S"] = torch.empty((c["n_q"], c["N"]), **f)
        s["done"] = torch.randn((c["n_q"], c["N"]), generator=_gen(seed, 3), **f)  # another job's scores
        s["idx"] = torch.empty((c["n_q"], c["topk"]), device="cuda", dtype=torch.int32)
        s["val"] = torch.empty((c["n_q"], c["topk"]), **f)
    elif kind == "cosine":
        s["A"], s["B"] = _factors(seed, 1, c["N"], c["T"], c["d_in"], c["d_out"], c["dtype"])
        s["Aq"], s["Bq"] = _factors(seed, 2, c["n_q"], c["T"], c["d_in"], c["d_out"], c["dtype"])
        s["L"] = L = tda.LayerDesc(c["d_in"], c["d_out"], c["T"], 1, 1, seed=SEED, layer=LAYER)
        s["S"] = torch.empty((c["n_q"], c["N"]), **f)
        s["nq"], s["nt"] = torch.empty(c["n_q"], **f), torch.empty(c["N"], **f)
        n = max(tda.tda_workspace_size(tda.TDA_OP_SIMILARITY_EXACT, L, _code(c), c["n_q"], c["N"]),
                tda.tda_workspace_size(tda.TDA_OP_NORM_EXACT, L, _code(c), c["N"], 0))
        s["wsb"] = max(256, min(8 * n, n + (1 << 30)))  # several train gradients at once where one is formed
        s["ws"] = _bytes(s["wsb"])
    elif kind == "tokens":
        D = c["k_in"] * c["k_out"]
        s["A"], s["B"] = _factors(seed, 1, c["N"], c["T"], c["d_in"], c["d_out"], c["dtype"])
        s["L"] = tda.LayerDesc(c["d_in"], c["d_out"], c["T"], c["k_in"], c["k_out"], seed=SEED, layer=LAYER)
        s["R"] = _features(seed, 2, c["n_q"], D)
        s["out"] = torch.empty((c["n_q"], c["N"] * c["T"]), **f)
        s["wsb"] = tda.tda_token_scores_workspace_size(s["L"]) * c["N"] + (4 << 20)
        s["ws"] = _bytes(s["wsb"])
    else:  # ekfac
        k, ws = c["k"], _widths(c)
        w = len(ws) * k * k
        s["layers"] = [tda.LayerDesc(a, b, c["T"], k, k, seed=SEED, layer=i) for i, (a, b) in enumerate(ws)]
        s["f"] = [_factors(seed, 10 + i, c["N"], c["T"], a, b, BF16) for i, (a, b) in enumerate(ws)]
        s["q"] = _features(seed, 2, c["n_q"], w)
        s["phi"], s["qhat"] = torch.empty((c["N"], w), **f), torch.empty((c["n_q"], w), **f)
        s["per"] = tda.tda_kfac_state_bytes(k, k)
        s["state"] = _bytes(len(ws) * s["per"])
        s["wsb"] = max(tda.tda_kfac_workspace_size(L, tda.TDA_BF16) for L in s["layers"])
        s["ws"] = _bytes(s["wsb"])
    return s


# ------------------------------------------------------------------------- pass
def run(s):
    c, kind = s["case"], s["case"]["kind"]
    if kind == "pass":
        L, N, n_q, D, f64 = s["L"], c["N"], c["n_q"], c["k"] * c["k"], tda.TDA_F64
        tda.tda_project(L, tda.TDA_F32, s["A"], s["B"], N, s["phi"], D, tda.TDA_ROUTE_FACTORED)
        tda.tda_project(L, tda.TDA_F32, s["Aq"], s["Bq"], n_q, s["q"], D, tda.TDA_ROUTE_FACTORED)
        tda.tda_precondition(tda.TDA_PC_RESET, 1, D, f64, s["state"])
        tda.tda_precondition(tda.TDA_PC_FIT_ACCUM, 1, D, f64, s["state"], phi=s["phi"], n=N, ld_phi=D)
        tda.tda_precondition(tda.TDA_PC_FACTOR, 1, D, f64, s["state"], n_total=N, lambda_abs=1e-3)
        tda.tda_precondition(tda.TDA_PC_APPLY, 1, D, f64, s["state"], q=s["q"], n_q=n_q, ld_q=D, qhat=s["qhat"],
                             ld_qhat=D)
        tda.tda_score(s["qhat"], f64, n_q, D, s["phi"], N, D, D, s["S"], N)
        tda.tda_topk(s["S"], n_q, N, N, c["topk"], s["idx"], s["val"])
        return {k: s[k] for k in ("phi", "q", "qhat", "S", "idx", "val")}
    if kind == "project":
        tda.tda_project(s["L"], _code(c), s["A"], s["B"], c["N"], s["phi"], c["k_in"] * c["k_out"],
                        tda.TDA_ROUTE_FACTORED, s["ws"], s["wsb"])
        return {"phi": s["phi"]}
    if kind == "precondition":
        nl, D, w, f32 = c["layers"], c["D"], c["layers"] * c["D"], tda.TDA_F32
        tda.tda_precondition(tda.TDA_PC_RESET, nl, D, f32, s["state"])
        tda.tda_precondition(tda.TDA_PC_FIT_ACCUM, nl, D, f32, s["state"], phi=s["phi"], n=c["N"], ld_phi=w)
        tda.tda_precondition(tda.TDA_PC_FACTOR_APPLY, nl, D, f32, s["state"], n_total=c["N"],
                             lambda_rel_mean_eig=1e-2, q=s["q"], n_q=c["n_q"], ld_q=w, qhat=s["qhat"], ld_qhat=w)
        return {"qhat": s["qhat"]}
    if kind == "score":
        D, N, n_q = c["D"], c["N"], c["n_q"]
        tda.tda_score(s["qhat"], tda.TDA_F32, n_q, D, s["phi"], N, D, D, s["S"], N)
        tda.tda_topk(s["done"], n_q, N, N, c["topk"], s["idx"], s["val"])
        return {k: s[k] for k in ("S", "idx", "val")}
    if kind == "cosine":
        L, N, n_q, dt = s["L"], c["N"], c["n_q"], _code(c)
        tda.tda_similarity_exact(L, dt, s["Aq"], s["Bq"], n_q, s["A"], s["B"], N, s["S"], N, ws=s["ws"],
                                 ws_bytes=s["wsb"])
        tda.tda_norms(tda.TDA_OP_NORM_EXACT, L, dt, s["Aq"], s["Bq"], n_q, s["nq"], ws=s["ws"], ws_bytes=s["wsb"])
        tda.tda_norms(tda.TDA_OP_NORM_EXACT, L, dt, s["A"], s["B"], N, s["nt"], ws=s["ws"], ws_bytes=s["wsb"])
        tda.tda_cosine(s["S"], n_q, N, N, s["nq"], s["nt"])
        return {k: s[k] for k in ("S", "nq", "nt")}
    if kind == "tokens":
        n = c["N"] * c["T"]
        tda.tda_token_scores(s["L"], _code(c), s["A"], s["B"], c["N"], s["R"], c["n_q"], c["k_in"] * c["k_out"],
                             s["out"], n, 0.0, s["ws"], s["wsb"])
        return {"out": s["out"]}
    k, nl = c["k"], len(s["layers"])
    w = nl * k * k
    tda.tda_kfac_reset(k, k, s["state"], n_layers=nl)
    for i, L in enumerate(s["layers"]):
        tda.tda_project_kfac(L, tda.TDA_BF16, s["f"][i][0], s["f"][i][1], c["N"], s["phi"][:, i * k * k:], w,
                             s["state"][i * s["per"]:(i + 1) * s["per"]], s["ws"], s["wsb"])
    tda.tda_kfac_eigen(k, k, s["state"], n_layers=nl)
    tda.tda_kfac_accumulate_eigenvalues(k, k, s["state"], s["phi"], c["N"], w, s["ws"], s["wsb"], n_layers=nl)
    tda.tda_kfac_apply(tda.TDA_EKFAC, k, k, s["state"], 0.0, 0.1, s["q"], c["n_q"], w, s["qhat"], w, n_layers=nl)
    return {"phi": s["phi"], "qhat": s["qhat"]}


# ------------------------------------------------------------------------- work
def _project_work(N, T, d_in, d_out, k_in, k_out, el):
    return (N * (T * (d_in + d_out) * el + 4.0 * k_in * k_out),
            2.0 * N * T * (d_in * k_in + d_out * k_out + k_in * k_out))


def work(case):
    c, kind = case, case["kind"]
    if kind == "project":
        b, f = _project_work(c["N"], c["T"], c["d_in"], c["d_out"], c["k_in"], c["k_out"],
                             2 if c["dtype"] == BF16 else 4)
    elif kind == "pass":
        D, N, n_q = c["k"] ** 2, c["N"], c["n_q"]
        b, f = _project_work(N + n_q, c["T"], c["d_in"], c["d_out"], c["k"], c["k"], 4)
        b += 8.0 * n_q * D + 4.0 * n_q * N + 8.0 * n_q * c["topk"]
        f += N * D * D + D ** 3 / 3.0 + 2.0 * D * D * n_q + 2.0 * n_q * N * D
    elif kind == "precondition":
        D, N, n_q, nl = c["D"], c["N"], c["n_q"], c["layers"]
        b = 4.0 * nl * D * (N + 2 * n_q)
        f = nl * (float(N) * D * D + D ** 3 / 3.0 + 2.0 * D * D * n_q)
    elif kind == "score":
        b = 4.0 * (c["D"] * (c["N"] + c["n_q"]) + 2 * c["n_q"] * c["N"]) + 8.0 * c["n_q"] * c["topk"]
        f = 2.0 * c["D"] * c["N"] * c["n_q"]
    elif kind == "cosine":
        # the cheaper of the two evaluations of <DW_q, DW_i>, and of each norm
        n, T, d, dd = c["N"] + c["n_q"], c["T"], c["d_in"] + c["d_out"], c["d_in"] * c["d_out"]
        pairs = c["N"] * c["n_q"]
        b = 2.0 * n * T * d + 4.0 * (pairs + n)
        f = min(2.0 * pairs * T * T * d, 2.0 * n * T * dd + 2.0 * pairs * dd) + min(2.0 * n * T * T * d / 2, 2.0 * n * T * dd)
    elif kind == "tokens":
        b, f = _project_work(c["N"], c["T"], c["d_in"], c["d_out"], c["k_in"], c["k_out"], 2)
        b += 4.0 * c["n_q"] * (c["k_in"] * c["k_out"] + c["N"] * c["T"]) - 4.0 * c["N"] * c["k_in"] * c["k_out"]
        f += 2.0 * c["n_q"] * c["N"] * c["T"] * c["k_in"] * c["k_out"]
    else:
        k, N, n_q = c["k"], c["N"], c["n_q"]
        b = f = 0.0
        for d_in, d_out in _widths(c):
            pb, pf = _project_work(N, c["T"], d_in, d_out, k, k, 2)
            b += pb + 8.0 * n_q * k * k
            f += pf + 2.0 * N * c["T"] * k * k + 4.0 * (N + 2 * n_q) * k ** 3
    return {"bytes": b, "flops": f}


# ------------------------------------------------------------------------ exact
_M64 = (1 << 64) - 1
_G = 0x9E3779B97F4A7C15


def _mix(z):
    z &= _M64
    z = ((z ^ (z >> 30)) * 0xBF58476D1CE4E5B9) & _M64
    z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & _M64
    return z ^ (z >> 31)


def _signs(layer, side, d, k):
    """The d x k Rademacher map of one side in fp64 (+1 / -1), from its published definition."""
    key = _mix(_mix(SEED + _G * (layer + 1)) + _G * (side + 1))
    groups = (d + 63) // 64
    n = (np.arange(k, dtype=np.uint64)[:, None] << np.uint64(32)) | np.arange(groups, dtype=np.uint64)[None, :]
    with np.errstate(over="ignore"):
        z = np.uint64(key) + np.uint64(_G) * (n + np.uint64(1))
        z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
    z = z ^ (z >> np.uint64(31))
    bits = (z[:, :, None] >> np.arange(64, dtype=np.uint64)) & np.uint64(1)
    s = 1.0 - 2.0 * bits.reshape(k, groups * 64)[:, :d].astype(np.float64)
    return torch.from_numpy(np.ascontiguousarray(s.T)).cuda()


def _project64(A, B, k_in, k_out, layer):
    """Phi (N x k_out*k_in) and the projected factors' covariance sums, in fp64."""
    Si = _signs(layer, 0, A.shape[2], k_in) / math.sqrt(k_in)
    So = _signs(layer, 1, B.shape[2], k_out) / math.sqrt(k_out)
    phi = torch.empty((A.shape[0], k_out * k_in), device="cuda", dtype=torch.float64)
    ca = torch.zeros((k_in, k_in), device="cuda", dtype=torch.float64)
    cg = torch.zeros((k_out, k_out), device="cuda", dtype=torch.float64)
    step = max(1, int(2e8 // (A.shape[1] * max(A.shape[2], B.shape[2]))))
    for i in range(0, A.shape[0], step):
        a, b = A[i:i + step].double() @ Si, B[i:i + step].double() @ So
        phi[i:i + step] = (b.transpose(1, 2) @ a).flatten(1)
        ca += a.flatten(0, 1).T @ a.flatten(0, 1)
        cg += b.flatten(0, 1).T @ b.flatten(0, 1)
    return phi, ca, cg


def _solve64(phi, q, lam_abs, lam_rel):
    F = phi.T @ phi / phi.shape[0]
    lam = lam_abs + lam_rel * F.diagonal().mean()
    F.diagonal().add_(lam)
    return torch.cholesky_solve(q.T, torch.linalg.cholesky(F)).T.contiguous()


def _dw64(A, B):
    return (B.double().transpose(1, 2) @ A.double()).flatten(1)


def exact(case, seed):
    s = prepare(case, seed)
    c, kind = case, case["kind"]
    if kind == "pass":
        phi = _project64(s["A"], s["B"], c["k"], c["k"], LAYER)[0]
        q = _project64(s["Aq"], s["Bq"], c["k"], c["k"], LAYER)[0]
        qhat = _solve64(phi, q, 1e-3, 0.0)
        S = qhat @ phi.T
        return {"phi": phi, "q": q, "qhat": qhat, "S": S, "idx": None, "val": S.topk(c["topk"]).values}
    if kind == "project":
        return {"phi": _project64(s["A"], s["B"], c["k_in"], c["k_out"], LAYER)[0]}
    if kind == "precondition":
        D = c["D"]
        out = [_solve64(s["phi"][:, l * D:(l + 1) * D].double(), s["q"][:, l * D:(l + 1) * D].double(), 0.0, 1e-2)
               for l in range(c["layers"])]
        return {"qhat": torch.cat(out, 1)}
    if kind == "score":
        S = torch.empty((c["n_q"], c["N"]), device="cuda", dtype=torch.float64)
        q = s["qhat"].double()
        for i in range(0, c["N"], 1024):
            S[:, i:i + 1024] = q @ s["phi"][i:i + 1024].double().T
        return {"S": S, "idx": None, "val": None}
    if kind == "cosine":
        S = torch.empty((c["n_q"], c["N"]), device="cuda", dtype=torch.float64)
        nt = torch.empty(c["N"], device="cuda", dtype=torch.float64)
        gq = _dw64(s["Aq"], s["Bq"])
        nq = (gq * gq).sum(1)
        step = max(1, int(4e8 // (c["d_in"] * c["d_out"])))
        for i in range(0, c["N"], step):
            g = _dw64(s["A"][i:i + step], s["B"][i:i + step])
            nt[i:i + step] = (g * g).sum(1)
            S[:, i:i + step] = gq @ g.T
        return {"S": S / (nq[:, None] * nt[None, :]).sqrt(), "nq": nq, "nt": nt}
    if kind == "tokens":
        a = s["A"].double() @ (_signs(LAYER, 0, c["d_in"], c["k_in"]) / math.sqrt(c["k_in"]))
        b = s["B"].double() @ (_signs(LAYER, 1, c["d_out"], c["k_out"]) / math.sqrt(c["k_out"]))
        R = s["R"].double().reshape(c["n_q"], c["k_out"], c["k_in"])
        out = torch.empty((c["n_q"], c["N"] * c["T"]), device="cuda", dtype=torch.float64)
        for j in range(c["n_q"]):
            out[j] = ((a @ R[j].T) * b).sum(2).flatten()
        return {"out": out}
    k, phis, qhats = c["k"], [], []
    for i, (A, B) in enumerate(s["f"]):
        phi, ca, cg = _project64(A, B, k, k, i)
        Ua, Ug = torch.linalg.eigh(ca)[1], torch.linalg.eigh(cg)[1]
        rot = lambda x: Ug.T @ x.reshape(-1, k, k) @ Ua  # noqa: E731
        lam = (rot(phi) ** 2).mean(0)
        q = rot(s["q"][:, i * k * k:(i + 1) * k * k].double()) / (lam + 0.1 * lam.mean())
        phis.append(phi)
        qhats.append((Ug @ q @ Ua.T).flatten(1))
    return {"phi": torch.cat(phis, 1), "qhat": torch.cat(qhats, 1)}
