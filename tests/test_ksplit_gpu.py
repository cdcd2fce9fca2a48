"""The fused project + similarity with a tile's K range shared by a cluster of 2, 4 or 8 CTAs (batches
with few 128-row tiles), against the 64-bit scores: every mode and output, ragged rows, K-blocks that
the cluster cannot share evenly, narrow bases, rows that need the range redo, repeated calls."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

TOL = 1e-4  # |S - S*| <= 1e-4 ||x|| ||c||, the documented bound


def setup(M, D, N, seed):
    rng = np.random.default_rng(seed)
    C = torch.from_numpy((rng.integers(0, 2, size=(M, D)) * 2 - 1).astype(np.float32)).cuda()
    lab = torch.from_numpy(rng.integers(0, M, size=N)).cuda()
    X = C[lab] + torch.from_numpy(rng.standard_normal((N, D)).astype(np.float32)).cuda()
    return C, X, lab


# tiles of 128 rows: 1 and 16 (clusters of 8), 17 to 38 (4), 39 to 76 (2), 77 (no split)
@pytest.mark.parametrize("N,D,M", [(1, 1024, 256), (77, 2500, 40), (128, 16388, 256), (2047, 8200, 100), (2049, 8192, 256),
                                   (4865, 4460, 17), (4096, 4096, 256), (5000, 4100, 130), (9728, 4228, 250),
                                   (9729, 4228, 256)])
@pytest.mark.parametrize("mode", ["raw", "cosine", "softmax"])
def test_every_output(gs, N, D, M, mode):
    C, X, lab = setup(M, D, N, [N, D])
    b = gs.build_basis(C)
    scale = 8.0 / D if mode == "softmax" else 1.0
    out = gs.project_similarity(b, X, mode=mode, scale=scale, path="tensor", want_S=True, want_Y=True)
    few = gs.project_similarity(b, X, mode=mode, scale=scale, path="tensor")
    gs.stream_status()
    Xd, Cd = X.double(), C.double()
    S = Xd @ Cd.T
    mag = Xd.norm(dim=1)[:, None] * Cd.norm(dim=1)[None, :]
    if mode == "raw":
        tol = TOL * mag
    elif mode == "cosine":
        S, tol = S / mag, TOL
    else:  # d softmax <= max |d logit| (and the exponentials' fp32 rounding)
        S, tol = torch.softmax(scale * S, 1), 2 * TOL * scale * mag.max() + 1e-5
    assert bool(((out["S"].double() - S).abs() <= tol).all())
    assert torch.equal(out["argmax"].long(), lab) and torch.equal(few["argmax"], out["argmax"])
    assert torch.equal(few["maxval"], out["maxval"])
    Y = Xd @ b.Q.double().T
    assert bool(((out["Y"].double() - Y).abs() <= TOL * Xd.norm(dim=1)[:, None]).all())


@pytest.mark.parametrize("N", [300, 4096, 7000])
@pytest.mark.parametrize("rows", ["one", "all"])
def test_range_redo(gs, N, rows):
    """Rows far below and above fp16's range have their tile computed again, cluster-wide."""
    C, X, lab = setup(200, 4160, N, [N, 5])
    f = torch.ones((N, 1), device="cuda")
    if rows == "all":
        f[::2], f[1::2] = 1e-7, 1e6
    else:
        f[N // 2] = 1e6
    X = (X * f).contiguous()
    b = gs.build_basis(C)
    S = X.double() @ C.double().T
    for _ in range(3):
        out = gs.project_similarity(b, X, path="tensor", want_S=True)
        gs.stream_status()
        tol = TOL * X.double().norm(dim=1)[:, None] * C.double().norm(dim=1)[None, :]
        assert bool(((out["S"].double() - S).abs() <= tol).all())
        assert torch.equal(out["argmax"].long(), lab)


def test_repeated_calls_agree(gs):
    C, X, lab = setup(256, 8192, 4096, 9)
    b = gs.build_basis(C)
    first = gs.project_similarity(b, X, want_S=True)
    for _ in range(10):
        out = gs.project_similarity(b, X, want_S=True)
        assert torch.equal(out["S"], first["S"])
    gs.stream_status()


@pytest.mark.parametrize("N", [5000, 12000])  # a shared K range, and none
@pytest.mark.parametrize("mode", ["raw", "cosine", "softmax"])
def test_unaligned_score_rows(gs, N, mode):
    C, X, lab = setup(60, 4096, N, [N, 4])
    b = gs.build_basis(C)
    scale = 8 / 4096 if mode == "softmax" else 1.0
    buf = torch.full((N, 61), -7.0, device="cuda")
    out = gs.project_similarity(b, X, mode=mode, scale=scale, path="tensor", want_S=True, out={"S": buf[:, :60]})
    gs.stream_status()
    S = X.double() @ C.double().T
    mag = X.double().norm(dim=1)[:, None] * C.double().norm(dim=1)[None, :]
    if mode == "raw":
        tol = TOL * mag
    elif mode == "cosine":
        S, tol = S / mag, TOL
    else:
        S, tol = torch.softmax(scale * S, 1), 2 * TOL * scale * mag.max() + 1e-5
    assert bool(((out["S"].double() - S).abs() <= tol).all())
    assert torch.equal(out["argmax"].long(), lab)
    assert bool((buf[:, 60] == -7.0).all())  # nothing between the rows


# clusters of 8, 4 and 2, no split: more codewords than the basis has rows, so that the scores of a row
# take more shared memory than its coefficients
@pytest.mark.parametrize("N", [500, 3000, 6000, 20000])
def test_zero_and_nan_rows(gs, N):
    """A zero query ties everywhere: the first entry wins.  A NaN query wins nowhere: entry 0, the lowest value."""
    rng = np.random.default_rng(N)
    B = torch.from_numpy((rng.integers(0, 2, size=(20, 4160)) * 2 - 1).astype(np.float32)).cuda()
    mix = torch.from_numpy(rng.integers(-1, 2, size=(250, 20)).astype(np.float32)).cuda()
    mix[:20] = torch.eye(20)
    C = mix @ B  # small whole numbers: exact in fp32
    X = torch.from_numpy(rng.standard_normal((N, 4160)).astype(np.float32)).cuda()
    zero, nan = [0, 129, N - 1], [1, 131, N - 2]
    X[zero] = 0
    X[nan, 7] = float("nan")
    b = gs.build_basis(C)
    assert b.r == 20
    out = gs.project_similarity(b, X, path="tensor", want_S=True)
    gs.stream_status()
    assert bool((out["argmax"][zero + nan] == 0).all()) and bool((out["maxval"][zero] == 0).all())
    assert bool((out["maxval"][nan] == torch.finfo(torch.float32).min).all())
    keep = torch.ones(N, dtype=torch.bool, device="cuda")
    keep[nan] = False
    S = X[keep].double() @ C.double().T
    tol = TOL * X[keep].double().norm(dim=1)[:, None] * C.double().norm(dim=1)[None, :]
    assert bool(((out["S"][keep].double() - S).abs() <= tol).all())
    assert torch.equal(out["S"][keep].argmax(1), out["argmax"][keep].long())


@pytest.mark.parametrize("N", [500, 3000, 6000, 20000])
@pytest.mark.parametrize("used", [40, 130])
def test_codewords_that_use_part_of_the_basis(gs, N, used):
    """A basis of 256 rows kept for a codebook of which only the first `used` entries are left: the scores are
    there before the last columns of Y are, which are outputs all the same."""
    C, X, _ = setup(256, 4160, N, [N, used])
    full = gs.build_basis(C)
    left = torch.arange(256, device="cuda") % used
    b = gs.import_basis(full.Q, full.R[left].contiguous())
    assert b.r == 256
    Xd, Cd = X.double(), C[left].double()
    S, Y = Xd @ Cd.T, Xd @ full.Q.double().T
    tol_s = TOL * Xd.norm(dim=1)[:, None] * Cd.norm(dim=1)[None, :]
    for _ in range(5):
        out = gs.project_similarity(b, X, path="tensor", want_S=True, want_Y=True)
        gs.stream_status()
        assert bool(((out["S"].double() - S).abs() <= tol_s).all())
        assert bool(((out["Y"].double() - Y).abs() <= TOL * Xd.norm(dim=1)[:, None]).all())
