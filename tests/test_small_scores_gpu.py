"""The CUDA-core scoring kernels of small calls (k_ps_small: r <= 32; k_scores with a K-split projection or
given Gram-loc rows: r <= 64), against 64-bit scores, at the edges of their tiles: one query to a few blocks,
D below, at and past a chunk of 128, rows off 16-byte boundaries, codebooks past one staged chunk, every
mode and output.  |error| <= (D + r) 2^-24 sum of magnitudes bounds any order of the fp32 sums."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def setup(N, D, M, r, seed):
    rng = np.random.default_rng(seed)
    C = torch.from_numpy((rng.integers(0, 2, size=(r, D)) * 2 - 1).astype(np.float32)).cuda()
    if M > r:  # dependent entries: sums of two
        i, j = rng.integers(0, r, size=(2, M - r))
        C = torch.cat([C, C[torch.from_numpy(i).cuda()] * 0.5 + C[torch.from_numpy(j).cuda()] * 0.75])
    X = torch.from_numpy(rng.standard_normal((N, D)).astype(np.float32)).cuda() + C[torch.arange(N, device="cuda") % M]
    return C, X


def check(out, X, C, mode, scale, tol):
    S = scale * (X.double() @ C.double().T)
    mag = abs(scale) * (X.double().norm(dim=1)[:, None] * C.double().norm(dim=1)[None, :])
    if mode == "cosine":
        S, mag = S / (mag / abs(scale)), torch.ones_like(S)
    err = tol * mag
    if mode == "softmax":
        S, err = torch.softmax(S, 1), (2 * tol * mag.max() + 1e-5).expand_as(S)
    best = S.max(1).values
    if "S" in out:
        assert bool(((out["S"].double() - S).abs() <= err).all())
    pick = S.gather(1, out["argmax"].long()[:, None])[:, 0]
    assert bool((best - pick <= 2 * err.amax(1)).all())
    assert bool(((out["maxval"].double() - best).abs() <= err.amax(1)).all())


@pytest.mark.parametrize("N,D,M,r", [(1, 1, 1, 1), (3, 127, 9, 8), (4, 128, 20, 9), (5, 516, 40, 17), (607, 1024, 30, 30),
                                     (609, 130, 32, 32), (2100, 1001, 700, 31), (1, 9000, 33, 33), (64, 515, 64, 64),
                                     (65, 4096, 63, 63), (1000, 2047, 3000, 50), (1024, 8192, 40, 40)])
@pytest.mark.parametrize("mode", ["raw", "cosine", "softmax"])
def test_project_similarity(gs, N, D, M, r, mode):
    r = min(r, D)
    C, X = setup(N, D, M, r, [N, D, M])
    b = gs.build_basis(C)
    scale = 4.0 / D if mode == "softmax" else -1.5 if mode == "raw" else 1.0
    tol = (D + b.r) * 2.0 ** -24
    out = gs.project_similarity(b, X, mode=mode, scale=scale, path="simt", want_S=True, want_Y=True)
    few = gs.project_similarity(b, X, mode=mode, scale=scale, path="simt")
    gs.stream_status()
    check(out, X, C, mode, scale, tol + 1e-6)
    assert torch.equal(few["argmax"], out["argmax"]) and torch.equal(few["maxval"], out["maxval"])
    Y = X.double() @ b.Q.double().T
    assert bool(((out["Y"].double() - Y).abs() <= tol * X.double().norm(dim=1)[:, None] + 1e-30).all())


# 64 coordinates: 173 codewords fit a staged chunk, one more takes the product and the row pass; rows x codewords
# at and past 2^19
@pytest.mark.parametrize("N,M,r", [(300, 173, 64), (300, 174, 64), (8192, 64, 64), (8193, 64, 64)])
@pytest.mark.parametrize("mode", ["raw", "cosine", "softmax"])
def test_route_edges(gs, N, M, r, mode):
    C, X = setup(N, 515, M, r, [N, M])
    b = gs.build_basis(C)
    scale = 4.0 / 515 if mode == "softmax" else 1.0
    out = gs.project_similarity(b, X, mode=mode, scale=scale, path="simt", want_S=True)
    few = gs.project_similarity(b, X, mode=mode, scale=scale, path="simt")
    gs.stream_status()
    check(out, X, C, mode, scale, (515 + b.r) * 2.0 ** -24 + 1e-6)
    assert torch.equal(few["argmax"], out["argmax"]) and torch.equal(few["maxval"], out["maxval"])


# up to 32 coordinates: 65 codewords go through the ring, 768 (16 queries, 32 coordinates) to 1,408 (4, 8) fill it
@pytest.mark.parametrize("N,M,r", [(5, 65, 8), (100, 1409, 8), (601, 65, 16), (1000, 3000, 12), (2433, 768, 32), (2450, 769, 30),
                                   (1, 5000, 32)])
@pytest.mark.parametrize("mode", ["raw", "cosine", "softmax"])
def test_more_codewords_than_kept(gs, N, M, r, mode):
    C, X = setup(N, 261, M, r, [N, M])
    b = gs.build_basis(C)
    scale = 4.0 / 261 if mode == "softmax" else 1.0
    out = gs.project_similarity(b, X, mode=mode, scale=scale, path="simt", want_S=True)
    few = gs.project_similarity(b, X, mode=mode, scale=scale, path="simt")
    gs.stream_status()
    check(out, X, C, mode, scale, (261 + b.r) * 2.0 ** -24 + 1e-6)
    assert torch.equal(few["argmax"], out["argmax"]) and torch.equal(few["maxval"], out["maxval"])


@pytest.mark.parametrize("N,M,r", [(1, 1, 1), (8, 5, 4), (9, 33, 7), (1300, 40, 40), (10000, 1024, 61), (300, 2500, 64)])
@pytest.mark.parametrize("mode", ["raw", "cosine", "softmax"])
def test_similarity_coeffs(gs, N, M, r, mode):
    C, _ = setup(1, 256, M, r, [N, M])
    b = gs.build_basis(C)
    Y = torch.randn((N, b.r + 3), generator=torch.Generator(device="cuda").manual_seed(N), device="cuda")[:, :b.r]
    scale = 0.05 if mode == "softmax" else 1.0
    out = gs.similarity_coeffs(b, Y, mode=mode, scale=scale, path="simt", want_S=True)
    few = gs.similarity_coeffs(b, Y, mode=mode, scale=scale, path="simt")
    gs.stream_status()
    check(out, Y, b.R, mode, scale, b.r * 2.0 ** -24 + 1e-6)
    assert torch.equal(few["argmax"], out["argmax"]) and torch.equal(few["maxval"], out["maxval"])


# k_ps_small, k_scores on the projection's parts, the product and the row pass; k_scores on given rows
@pytest.mark.parametrize("M,r", [(25, 20), (60, 50), (400, 50)])
@pytest.mark.parametrize("given", [False, True])
@pytest.mark.parametrize("mode", ["raw", "cosine", "softmax"])
def test_not_finite(gs, M, r, given, mode):
    """Rows with a NaN or an infinity have NaN and infinities where the products, in the same form but in 64
    bits, have them; a NaN never wins (entry 0 when nothing else does), and no other row notices."""
    C, X = setup(40, 300, M, r, 3)
    b = gs.build_basis(C)
    Q, R = b.Q.double(), b.R.double()
    if given:
        X = (X.double() @ Q.T).float()
    bad = [7, 9, 11]
    X[bad, 13] = torch.tensor([float("nan"), float("inf"), -float("inf")], device="cuda")
    if given:
        out = gs.similarity_coeffs(b, X, mode=mode, scale=0.01, path="simt", want_S=True)
    else:
        out = gs.project_similarity(b, X, mode=mode, scale=0.01, path="simt", want_S=True)
    gs.stream_status()
    Y = X.double() if given else X.double() @ Q.T
    S = 0.01 * (Y @ R.T)
    if mode == "cosine":
        den = X.double().norm(dim=1)[:, None] * C.double().norm(dim=1)[None, :]
        S = torch.where(den > 0, S / den, torch.zeros_like(S))
    best = torch.where(torch.isnan(S), torch.full_like(S, -float("inf")), S).max(1)
    index = torch.where(best.values > -float("inf"), best.indices, torch.zeros_like(best.indices))
    if mode == "softmax":
        S = torch.softmax(S, 1)
    for f in (torch.isnan, torch.isposinf, torch.isneginf):
        assert torch.equal(f(out["S"]), f(S))
    assert torch.equal(out["argmax"][bad].long(), index[bad])
    good = [i for i in range(40) if i not in bad]
    err = (320 * 2.0 ** -24 + 1e-6) * (0.01 * Y[good].norm(dim=1).max() * R.norm(dim=1).max() if mode == "raw" else 1.0)
    assert bool(((out["S"][good].double() - S[good]).abs() <= 8 * err).all())
