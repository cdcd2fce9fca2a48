"""Timed cases of the library: what a program that uses it calls, over the sizes it meets.

Each case is one public call of ``paper_2608_01528_gb300.gramspace`` (``panel`` chains several, as
one step of a reasoning program does) on inputs that already sit on the GPU, with the basis built
beforehand as a program keeps it.  ``listed`` names the cases, ``draw`` gives more of the same
kinds, ``prepare`` / ``run`` make the inputs and one pass, ``work`` counts the bytes and
operations a pass cannot do without, ``exact`` is the same result in 64 bits, ``tolerance`` how
far two correct implementations at the same precision may lie apart.
"""
import math

import numpy as np
import torch

from paper_2608_01528_gb300 import gramspace as gs

ATTRIBUTES = (5, 6, 10, 9)  # sizes of the four attribute codebooks of a reasoning problem
PANELS = 16                 # panels per problem


def listed():
    return [
        # a batch of attribute lookups on Gram-loc queries against one global codebook of 40
        # attribute values: the smallest call, latency counts
        {"name": "lookup", "kind": "lookup", "N": 1024, "M": 40, "D": 1024, "dep": 0, "mode": "raw", "scores": False},
        # one step of a reasoning program on 128 problems of 16 panels: score all attributes, pick each
        # attribute's value, vectorize the rule's probabilities, reconstruct and bind with the role
        {"name": "panel", "kind": "panel", "problems": 128, "D": 1024, "L": 256},
        # the same lookups from full-dimensional vectors, 40 values at dimension 8192 (latency against dimension)
        {"name": "score_lookup", "kind": "score", "N": 1024, "M": 40, "D": 8192, "dep": 0, "mode": "cosine",
         "scores": False},
        # an ordinary serving batch, probabilities over the codebook returned
        {"name": "score_batch", "kind": "score", "N": 4096, "M": 256, "D": 8192, "dep": 0, "mode": "softmax",
         "scores": True},
        # the large-batch scoring of the benchmark: best entry and its score
        {"name": "score_large", "kind": "score", "N": 65536, "M": 256, "D": 8192, "dep": 0, "mode": "raw",
         "scores": False},
        # a wide codebook with dependent (bundled) entries, more basis vectors than one tile holds
        {"name": "score_wide", "kind": "score", "N": 16384, "M": 1024, "D": 10000, "dep": 102, "mode": "cosine",
         "scores": False},
        # attribute probabilities to Gram-loc, in the 16-bit form that attention reads
        {"name": "vectorize", "kind": "vectorize", "N": 65536, "M": 512, "D": 4096, "dtype": "bf16"},
        # decoding Gram-loc rows to full vectors before component-wise operators
        {"name": "reconstruct", "kind": "reconstruct", "N": 16384, "M": 922, "D": 10000, "dtype": "f32"},
        # decoding followed by unbinding, one partner per row
        {"name": "unbind", "kind": "bind", "N": 8192, "M": 512, "D": 4096, "L": 256, "op": "unbind", "partners": True},
        # attention probabilities between compressed vectors, 64 sequences of 1024
        {"name": "attention", "kind": "attention", "B": 64, "Lq": 1024, "Lk": 1024, "r": 512, "dtype": "bf16",
         "softmax": True},
        # long sequences of an odd length
        {"name": "attention_long", "kind": "attention", "B": 8, "Lq": 2900, "Lk": 2900, "r": 384, "dtype": "bf16",
         "softmax": True},
        # factoring a codebook when a program starts, or its codebook changes
        {"name": "build", "kind": "build", "M": 512, "D": 4096, "dep": 37},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _near(rng, n, step):
    """n as it is, or rounded to a multiple of step: odd sizes and even ones."""
    return n if rng.random() < 0.5 else max(step, n // step * step)


def _f(v):
    return float(v)


def draw(rng):
    kind = rng.choice(["lookup", "panel", "score", "score", "vectorize", "reconstruct", "bind", "attention", "build"])
    if kind == "panel":
        return {"kind": kind, "problems": _log(rng, 4, 2048), "D": 256 * rng.randint(2, 16),
                "L": rng.choice([64, 128, 256])}
    if kind == "attention":
        while True:
            c = {"kind": kind, "B": _log(rng, 1, 256), "Lq": _near(rng, _log(rng, 32, 4096), 32),
                 "Lk": _near(rng, _log(rng, 32, 4096), 32), "r": 8 * rng.randint(2, 64),
                 "dtype": rng.choice(["bf16", "bf16", "bf16", "f32"]), "softmax": rng.random() < 0.75}
            w = work(c)
            if w["bytes"] <= 5e8 and w["flops"] <= 7e10:
                return c
    if kind == "build":
        D = _near(rng, _log(rng, 256, 8192), 64)
        M = _log(rng, 16, min(512, D, math.isqrt((1 << 30) // D)))
        return {"kind": kind, "M": M, "D": D, "dep": rng.randint(0, M // 8)}
    if kind == "lookup":
        M = _log(rng, 8, 512)
        return {"kind": kind, "N": _near(rng, _log(rng, 64, 65536), 64), "M": M, "D": max(512, M),
                "dep": rng.randint(0, M // 10), "mode": rng.choice(["raw", "cosine", "softmax"]),
                "scores": rng.random() < 0.5}
    if kind == "vectorize":
        M = _log(rng, 8, 1024)
        N = min(_log(rng, 128, 131072), (1 << 25) // M)
        return {"kind": kind, "N": _near(rng, N, 64), "M": M, "D": max(1024, M),
                "dtype": rng.choice(["bf16", "bf16", "f32"])}
    while True:
        N, D = _near(rng, _log(rng, 128, 65536), 64), _near(rng, _log(rng, 256, 16384), 64)
        M = _log(rng, 8, min(1024, D))
        if kind == "score":
            c = {"kind": kind, "N": N, "M": M, "D": D, "dep": rng.randint(0, M // 10),
                 "mode": rng.choice(["raw", "cosine", "softmax"]), "scores": rng.random() < 0.4}
            if N * D <= 1 << 29 and work(c)["flops"] <= 3.2e11:
                return c
        elif kind == "reconstruct":
            c = {"kind": kind, "N": N, "M": M, "D": D, "dtype": rng.choice(["f32", "f32", "f32", "bf16"])}
            if work(c)["bytes"] <= 7e8 and work(c)["flops"] <= (3e11 if c["dtype"] == "f32" else 5e10):
                return c
        else:
            L = rng.choice([64, 128, 256, 256, 512, 1024])
            D = max(1, D // L) * L
            c = {"kind": "bind", "N": N, "M": min(M, D), "D": D, "L": L, "op": rng.choice(["bind", "unbind"]),
                 "partners": rng.random() < 0.7}
            if work(c)["bytes"] <= 1.2e9 and work(c)["flops"] <= 1.5e11:
                return c


# --------------------------------------------------------------------------- inputs
def _gen(seed, stream):
    g = torch.Generator(device="cuda")
    g.manual_seed((int(seed) * 1000003 + stream) & 0x7FFFFFFF)
    return g


def _codebook(seed, M, D, dep=0, stream=0):
    """M x D: bipolar atoms, `dep` of them bundles (a +- b) / sqrt(2) of two others, rows shuffled."""
    g = _gen(seed, stream)
    C = (torch.randint(0, 2, (M, D), generator=g, device="cuda", dtype=torch.int8) * 2 - 1).float()
    if dep:
        ind = M - dep
        a = torch.randint(0, ind, (dep,), generator=g, device="cuda")
        b = (a + torch.randint(1, ind, (dep,), generator=g, device="cuda")) % ind
        C[ind:] = (C[a] + C[b] * (torch.randint(0, 2, (dep, 1), generator=g, device="cuda") * 2 - 1)) * math.sqrt(0.5)
        C = C[torch.randperm(M, generator=g, device="cuda")].contiguous()
    return C


def _queries(seed, C, N, sigma):
    """Random codewords plus noise: what a perception front end hands to the scoring."""
    g = _gen(seed, 7)
    X = torch.randn((N, C.shape[1]), generator=g, device="cuda")
    X.mul_(sigma)
    lab = torch.randint(0, C.shape[0], (N,), generator=g, device="cuda")
    for i in range(0, N, 8192):
        X[i:i + 8192] += C[lab[i:i + 8192]]
    return X


def _probs(seed, N, M, stream=9):
    return torch.softmax(2.0 * torch.randn((N, M), generator=_gen(seed, stream), device="cuda"), dim=1)


def _rank(case):
    return case["M"] - case.get("dep", 0)


def _scale(case):
    """Softmax temperature: the matching codeword's logit is about 8, the others' near 0."""
    return 8.0 / case["D"] if case["mode"] == "softmax" else 1.0


def _attn_scale(case):
    return 1.0 / math.sqrt(case["r"])


def _offsets():
    return [0] + [int(v) for v in np.cumsum(ATTRIBUTES)]


def _attn_inputs(case, seed):
    dt = torch.bfloat16 if case["dtype"] == "bf16" else torch.float32
    g = _gen(seed, 3)
    q = torch.randn((case["B"], case["Lq"], case["r"]), generator=g, device="cuda")
    k = torch.randn((case["B"], case["Lk"], case["r"]), generator=g, device="cuda")
    return q.to(dt), k.to(dt)


def _inputs(case, seed):
    """The case's tensors, without any handle of the library."""
    kind = case["kind"]
    if kind == "attention":
        q, k = _attn_inputs(case, seed)
        return {"q": q, "k": k}
    if kind == "panel":
        N, D, off = case["problems"] * PANELS, case["D"], _offsets()
        C = torch.cat([_codebook(seed, m, D, stream=20 + i) for i, m in enumerate(ATTRIBUTES)])
        g = _gen(seed, 5)
        X = torch.randn((N, D), generator=g, device="cuda") * 0.5
        for i, m in enumerate(ATTRIBUTES):  # a panel is the bundle of its attribute values
            X += C[off[i] + torch.randint(0, m, (N,), generator=g, device="cuda")]
        P = torch.cat([_probs(seed, N, m, 30 + i) for i, m in enumerate(ATTRIBUTES)], dim=1)
        role = torch.randn((1, D), generator=g, device="cuda") / math.sqrt(case["L"])
        return {"C": C, "X": X, "P": P, "role": role}
    C = _codebook(seed, case["M"], case["D"], case.get("dep", 0))
    out = {"C": C}
    if kind == "score":
        out["X"] = _queries(seed, C, case["N"], 1.0)
    elif kind == "vectorize":
        out["P"] = _probs(seed, case["N"], case["M"])
    elif kind in ("reconstruct", "bind"):
        T = torch.randn((case["N"], case["M"]), generator=_gen(seed, 11), device="cuda")
        out["T"] = T.bfloat16() if case.get("dtype") == "bf16" else T
        if kind == "bind":
            n = case["N"] if case["partners"] else 1
            out["Y"] = torch.randn((n, case["D"]), generator=_gen(seed, 13), device="cuda") / math.sqrt(case["L"])
    elif kind == "lookup":
        # Gram-loc queries: a codeword's coordinates (computed here, so that they do not depend on
        # the library's last bits) plus noise
        g = _gen(seed, 17)
        lab = torch.randint(0, case["M"], (case["N"],), generator=g, device="cuda")
        noise = torch.randn((case["N"], _rank(case)), generator=g, device="cuda") * 0.5
        out["Y"] = _gram_schmidt(C)[1].float()[lab] + noise
    return out


def prepare(case, seed):
    kind = case["kind"]
    s = _inputs(case, seed)
    s["case"] = case
    if kind == "panel":
        s["basis"] = gs.build_basis_grouped(s.pop("C"), _offsets())
    elif kind not in ("attention", "build"):
        s["basis"] = gs.build_basis(s.pop("C"))
    return s


# --------------------------------------------------------------------------- one pass
def run(state):
    c = state["case"]
    kind = c["kind"]
    if kind == "lookup":
        return gs.similarity_coeffs(state["basis"], state["Y"], mode=c["mode"], scale=_scale(c), want_S=c["scores"])
    if kind == "score":
        return gs.project_similarity(state["basis"], state["X"], mode=c["mode"], scale=_scale(c), want_S=c["scores"])
    if kind == "panel":
        b = state["basis"]
        s = gs.project_similarity(b, state["X"], want_S=True, want_argmax=False, want_maxval=False)
        g = gs.group_argmax(s["S"], _offsets())
        v = gs.prob_vectorize(b, state["P"])
        z = gs.reconstruct_bind(b, v, state["role"], c["L"])
        return {"S": s["S"], "argmax": g["argmax"], "maxval": g["maxval"], "V": v, "Z": z}
    if kind == "vectorize":
        return gs.prob_vectorize(state["basis"], state["P"],
                                 dtype=torch.bfloat16 if c["dtype"] == "bf16" else torch.float32)
    if kind == "reconstruct":
        return gs.reconstruct(state["basis"], state["T"])
    if kind == "bind":
        return gs.reconstruct_bind(state["basis"], state["T"], state["Y"], c["L"], op=c["op"])
    if kind == "attention":
        return gs.attention_scores(state["q"], state["k"], _attn_scale(c), apply_softmax=c["softmax"])
    b = gs.build_basis(state["C"])  # the factors, as a program saves them
    return {"Q": b.Q.clone(), "R": b.R.clone(), "cnorm": b.cnorm.clone()}


# --------------------------------------------------------------------------- work
def work(case):
    kind = case["kind"]
    if kind == "attention":
        B, Lq, Lk, r = (_f(case[k]) for k in ("B", "Lq", "Lk", "r"))
        e = 2 if case["dtype"] == "bf16" else 4
        return {"bytes": B * (e * r * (Lq + Lk) + 4 * Lq * Lk), "flops": 2 * B * Lq * Lk * r}
    if kind == "panel":
        N, D, M, G = _f(case["problems"] * PANELS), _f(case["D"]), _f(sum(ATTRIBUTES)), len(ATTRIBUTES)
        return {"bytes": 4 * (2 * N * D + 3 * N * M + 2 * M * D + D) + 8 * N * G, "flops": 2 * N * M * (2 * D + 2 * M)}
    M, D, r = _f(case["M"]), _f(case["D"]), _f(_rank(case))
    if kind == "build":  # two projection passes per row, each the dots with the rows before and their subtraction
        return {"bytes": 4 * (M * D + r * D + M * r + M), "flops": 4 * M * r * D}
    N = _f(case["N"])
    out = 8 * N + (4 * N * M if case.get("scores") else 0)
    if kind == "lookup":
        return {"bytes": 4 * N * r + 4 * M * r + out, "flops": 2 * N * M * r}
    if kind == "score":
        return {"bytes": 4 * N * D + 2 * r * D + 4 * M * r + out, "flops": 2 * N * r * (D + M)}
    e = 2 if case.get("dtype") == "bf16" else 4
    if kind == "vectorize":
        return {"bytes": 4 * N * M + 4 * M * r + e * N * r, "flops": 2 * N * M * r}
    rec = {"bytes": e * N * r + 2 * r * D + 4 * N * D, "flops": 2 * N * r * D}
    if kind == "bind":  # and the block transforms: three of L log L per block
        rec["bytes"] += 4 * D * (N if case["partners"] else 1)
        rec["flops"] += 3 * 2.5 * N * D * math.log2(case["L"])
    return rec


# --------------------------------------------------------------------------- tolerance
# About four times the error against 64 bits that each precision was seen to have over the ranges of
# draw(): F32 for sums of 32-bit products, HALF_SCORE / HALF_ROWS where the call documents one fp16
# rounding of its operands (large, aligned calls), SPLIT where it documents 16-bit pairs.
F32 = {"rel": 4e-6, "max": 1e-4}
SPLIT = {"rel": 4e-5, "max": 1e-3}
HALF_SCORE = {"rel": 2.5e-4, "max": 1.2e-3}
HALF_ROWS = {"rel": 1.5e-3, "max": 9e-3}


def tolerance(case):
    kind = case["kind"]
    if kind == "score":
        return HALF_SCORE if case["N"] * case["D"] >= 1 << 24 and case["D"] % 4 == 0 else F32
    if kind == "panel":
        return HALF_SCORE if case["problems"] * PANELS * case["D"] >= 1 << 24 else F32
    if kind in ("reconstruct", "bind"):
        large = case["N"] >= 512 and 2 * case["N"] * case["M"] * case["D"] >= 2e9 and case["D"] >= 1024
        return HALF_ROWS if large and case["M"] % 4 == 0 and case.get("dtype") != "bf16" else F32
    if kind == "vectorize":  # 16-bit outputs, or 32-bit ones from 16-bit pairs
        return {"rel": 7e-3, "max": 1.6e-2} if case["dtype"] == "bf16" else SPLIT
    if kind == "lookup":
        return SPLIT
    if kind == "attention":
        return {"rel": 4e-6, "max": 2e-5}
    return {"rel": 2e-7, "max": 1e-6}  # build: 64-bit sums, results rounded to 32 bits


# --------------------------------------------------------------------------- 64 bits
def _gram_schmidt(C, tol=1e-6):
    """Q (r x D), R (M x r) of C = R Q in row order, two projection passes per row, in 64 bits."""
    C = C.double()
    M, D = C.shape
    Q = torch.zeros((min(M, D), D), dtype=torch.float64, device=C.device)
    R = torch.zeros((M, min(M, D)), dtype=torch.float64, device=C.device)
    k = 0
    for i in range(M):
        v = C[i]
        for _ in range(2):
            t = Q[:k] @ v
            v = v - t @ Q[:k]
            R[i, :k] += t
        n = float(v.norm())
        if k < D and n > tol * float(C[i].norm()):
            Q[k] = v / n
            R[i, k] = n
            k += 1
    return Q[:k].clone(), R[:, :k].clone()


def _bind64(X, Y, L, op):
    N, D = X.shape
    fx, fy = torch.fft.rfft(X.view(N, D // L, L)), torch.fft.rfft(Y.double().view(-1, D // L, L))
    return torch.fft.irfft(fx * (fy if op == "bind" else fy.conj()), n=L).reshape(N, D)


def _rows(N, D):
    return max(256, (1 << 27) // max(1, D))


def _scores(case, S, xnorm, cnorm):
    """The outputs of a scoring call from its plain scores S = <x, c>."""
    S = S * _scale(case)
    if case["mode"] == "cosine":
        S = S / (xnorm[:, None] * cnorm[None, :])
    elif case["mode"] == "softmax":
        S = torch.softmax(S, dim=1)
    v, i = S.max(dim=1)
    return ({"S": S} if case["scores"] else {}), i.int(), v


def _score64(case, rows, C):
    parts = []
    for i in range(0, rows.shape[0], _rows(*rows.shape)):
        x = rows[i:i + _rows(*rows.shape)].double()
        parts.append(_scores(case, x @ C.T, x.norm(dim=1), C.norm(dim=1)))
    out = {"argmax": torch.cat([p[1] for p in parts]), "maxval": torch.cat([p[2] for p in parts])}
    if case["scores"]:
        out["S"] = torch.cat([p[0]["S"] for p in parts])
    return out


def exact(case, seed):
    kind = case["kind"]
    t = _inputs(case, seed)
    if kind == "attention":
        parts = []
        for q, k in zip(t["q"], t["k"]):
            a = (q.double() @ k.double().T) * _attn_scale(case)
            parts.append(torch.softmax(a, dim=1) if case["softmax"] else a)
        return torch.stack(parts)
    if kind == "panel":
        off = _offsets()
        C = t["C"].double()
        S = t["X"].double() @ C.T
        best = [S[:, a:b].max(dim=1) for a, b in zip(off, off[1:])]
        R = torch.block_diag(*[_gram_schmidt(C[a:b])[1] for a, b in zip(off, off[1:])])
        P = t["P"].double()
        return {"S": S, "argmax": torch.stack([b.indices for b in best], 1).int(),
                "maxval": torch.stack([b.values for b in best], 1), "V": P @ R,
                "Z": _bind64(P @ C, t["role"], case["L"], "bind")}
    if kind == "score":
        return _score64(case, t["X"], t["C"].double())
    Q, R = _gram_schmidt(t["C"])
    if kind == "build":
        return {"Q": Q, "R": R, "cnorm": t["C"].double().norm(dim=1)}
    if kind == "lookup":
        return _score64(case, t["Y"], R)
    if kind == "vectorize":
        return t["P"].double() @ R
    X = t["T"].double() @ Q
    return X if kind == "reconstruct" else _bind64(X, t["Y"], case["L"], case["op"])
