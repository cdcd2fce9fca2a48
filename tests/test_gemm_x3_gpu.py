"""The fp32-accurate GEMM on the tensor cores (operands in three bf16 parts), through the calls that
take it: large reconstructions and vectorizations whose rows are not 16-byte aligned, bf16 T, short
rows, fp32 attention.  Element-wise against the 64-bit product:

    |error| <= (12 + ceil(K / 128)) 2^-23 sum_k |a_k| |b_k|

a bound from the kernel's arithmetic: at most 8 accumulation steps per 128 terms, each losing at
most 2^-23 of the sum of magnitudes; the small products' steps, 2^-8 of that and 6 times as many; the
products left out, below 2^-23; one fp32 addition per 128 terms.
"""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def bound(K, mag):
    return (12 + -(-K // 128)) * 2.0 ** -23 * mag + 1e-30


def bipolar(rng, M, D):
    return torch.from_numpy((rng.integers(0, 2, size=(M, D)) * 2 - 1).astype(np.float32)).cuda()


# (N, r, D): ragged row and column tiles, K a whole number of K-blocks, one past, one short, one and
# several accumulation chunks, rows starting on 4-, 8- and 16-byte boundaries
SHAPES = [(2049, 161, 8200), (1500, 255, 5001), (777, 130, 9001), (2048, 511, 1999), (1300, 513, 2050),
          (1025, 922, 3000), (1100, 1031, 1500), (2000, 320, 900)]


@pytest.mark.parametrize("N,r,D", SHAPES)
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
def test_reconstruct_against_64_bits(gs, N, r, D, dtype):
    rng = np.random.default_rng([N, r, D])
    b = gs.build_basis(bipolar(rng, r, D))
    T = torch.from_numpy(rng.standard_normal((N, b.r)).astype(np.float32)).cuda()
    T[N // 2] *= 1e20  # rows of other magnitudes
    T[N // 3] *= 1e-20
    T = T.to(dtype)
    X = gs.reconstruct(b, T)
    gs.stream_status()
    ref = T.double() @ b.Q.double()
    if dtype == torch.float32 and b.r % 4 == 0 and D >= 1024:
        tol = 1e-4 * T.double().norm(dim=1, keepdim=True)  # the fp16 path's documented bound
    else:
        tol = bound(b.r, T.double().abs() @ b.Q.double().abs())
    assert bool(((X.double() - ref).abs() <= tol).all())


@pytest.mark.parametrize("N,M", [(4001, 333), (9000, 517), (2500, 1030)])
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
def test_vectorize_unaligned(gs, N, M, dtype):
    rng = np.random.default_rng([N, M])
    b = gs.build_basis(bipolar(rng, M, 1536))
    P = torch.softmax(torch.from_numpy(2 * rng.standard_normal((N, M)).astype(np.float32)).cuda(), 1)
    base = torch.zeros(N * M + 1, device="cuda")
    Pu = base[1:].view(N, M).copy_(P)  # rows off every vector boundary
    V = gs.prob_vectorize(b, Pu, dtype=dtype)
    gs.stream_status()
    ref = P.double() @ b.R.double()
    tol = bound(M, P.double() @ b.R.double().abs())
    if dtype == torch.bfloat16:
        tol = tol + 2.0 ** -8 * ref.abs()
    assert bool(((V.double() - ref).abs() <= tol).all())


def test_attention_fp32_batched(gs):
    g = torch.Generator(device="cuda").manual_seed(3)
    q = torch.randn((5, 391, 130), generator=g, device="cuda")
    k = torch.randn((5, 1517, 130), generator=g, device="cuda")
    A = gs.attention_scores(q, k, 0.5, apply_softmax=False)
    gs.stream_status()
    ref = 0.5 * (q.double() @ k.double().transpose(1, 2))
    tol = 0.5 * bound(130, q.double().abs() @ k.double().abs().transpose(1, 2))
    assert bool(((A.double() - ref).abs() <= tol).all())


def test_scores_of_odd_dimension(gs):
    """D % 4 != 0: the projection and the scores both take the general path."""
    rng = np.random.default_rng(8)
    C = bipolar(rng, 300, 2501)
    b = gs.build_basis(C)
    X = C[torch.arange(7000, device="cuda") % 300] + torch.randn((7000, 2501), device="cuda")
    out = gs.project_similarity(b, X, mode="cosine", want_S=True)
    gs.stream_status()
    ref = (X.double() @ C.double().T) / (X.double().norm(dim=1)[:, None] * C.double().norm(dim=1)[None, :])
    assert float((out["S"].double() - ref).abs().max()) <= 2e-5
    assert torch.equal(out["argmax"].long(), ref.argmax(1))


@pytest.mark.parametrize("bad", [float("inf"), -float("inf"), float("nan"), 3.4e38])
def test_not_finite_as_on_the_cuda_cores(gs, bad):
    """Rows with an infinity, a NaN or a value beyond bf16's range: the same infinities and NaN in the
    same places as the CUDA-core path, every other output within the bound."""
    rng = np.random.default_rng(5)
    b = gs.build_basis(bipolar(rng, 131, 9003))
    T = torch.from_numpy(rng.standard_normal((1100, b.r)).astype(np.float32)).cuda()
    T[7, 3] = bad
    T[1099, 130] = bad
    X, S = gs.reconstruct(b, T), gs.reconstruct(b, T, path="simt")
    gs.stream_status()
    for f in (torch.isnan, torch.isposinf, torch.isneginf):
        assert torch.equal(f(X), f(S))
    rows = [i for i in range(1100) if i not in (7, 1099)]
    ref = T.double() @ b.Q.double()
    assert bool(((X.double() - ref).abs() <= bound(b.r, T.double().abs() @ b.Q.double().abs()))[rows].all())


# few output tiles over a deep K: chunks of K to partial products, the last one shorter; rows on and off
# 16-byte boundaries, odd K
@pytest.mark.parametrize("N,D,M", [(130, 8191, 300), (1000, 4100, 500), (257, 15999, 700), (640, 2048, 900), (1, 32768, 512)])
def test_split_k(gs, N, D, M):
    rng = np.random.default_rng([N, D])
    C = torch.from_numpy((rng.integers(0, 2, size=(M, D)) * 2 - 1).astype(np.float32)).cuda()
    lab = torch.from_numpy(rng.integers(0, M, size=N)).cuda()
    X = C[lab] + torch.from_numpy(rng.standard_normal((N, D)).astype(np.float32)).cuda()
    if N > 8:
        X[3, D - 1], X[4, 0] = float("inf"), float("nan")
    b = gs.build_basis(C)
    out = gs.project_similarity(b, X, want_S=True, want_Y=True)
    ref = gs.project_similarity(b, X, want_Y=True, path="simt")
    again = gs.project_similarity(b, X, want_Y=True)
    gs.stream_status()
    fin = torch.isfinite(ref["Y"])
    assert torch.equal(torch.isfinite(out["Y"]), fin) and torch.equal(again["Y"][fin], out["Y"][fin])
    ok = torch.isfinite(X).all(1)
    Xd = X[ok].double()
    Y = Xd @ b.Q.double().T
    # six bf16 products of the three-way split leave 2^-24 of |x||q|, the fp32 sums of 128 terms a few more
    assert bool(((out["Y"][ok].double() - Y).abs() <= 1e-6 * Xd.norm(dim=1)[:, None]).all())
    assert torch.equal(out["argmax"][ok].long(), lab[ok])


@pytest.mark.parametrize("e", [-108, -115, -122, -130])
def test_small_operands(gs, e):
    """Operands down to fp32's subnormals lose nothing: the bound holds with no absolute slack but fp32's own
    rounding of subnormal sums, 2^-149 a term, twice."""
    def close(X, ref, K, mag):
        assert bool(((X.double() - ref).abs() <= (12 + -(-K // 128)) * 2.0 ** -23 * mag + K * 2.0 ** -148).all())

    rng = np.random.default_rng(-e)
    b = gs.build_basis(bipolar(rng, 161, 8200))
    T = (torch.from_numpy(rng.standard_normal((2049, 161))).cuda() * 2.0 ** e).float()
    close(gs.reconstruct(b, T), T.double() @ b.Q.double(), 161, T.double().abs() @ b.Q.double().abs())
    q = (torch.from_numpy(rng.standard_normal((5, 391, 130))).cuda() * 2.0 ** e).float()
    k = (torch.from_numpy(rng.standard_normal((5, 1517, 130))).cuda() * 2.0 ** 40).float()
    for x, y in ((q, k), (k, q)):
        A = gs.attention_scores(x, y, 1.0, apply_softmax=False)
        xt, yt = x.double(), y.double().transpose(1, 2)
        close(A, xt @ yt, 130, xt.abs() @ yt.abs())
    gs.stream_status()


def test_large_operands(gs):
    """Beyond 2^120 the parts' factors overflow: the plain fp32 dot product instead."""
    rng = np.random.default_rng(6)
    b = gs.build_basis(bipolar(rng, 161, 8200))
    T = torch.from_numpy(rng.standard_normal((2049, 161)).astype(np.float32)).cuda()
    T[5] *= 1e36
    T[700:900] *= 3e35
    X = gs.reconstruct(b, T)
    gs.stream_status()
    ref = T.double() @ b.Q.double()
    # (161 terms in order: 161 x 2^-24)
    assert bool(((X.double() - ref).abs() <= bound(161, T.double().abs() @ b.Q.double().abs()) * (161 / 14)).all())


@pytest.mark.parametrize("bad", [float("inf"), float("nan")])
def test_not_finite_past_the_end_of_a_codeword(gs, bad):
    """Entry i's coordinates end at i + 1: a bad coordinate past it is not multiplied by the zeros there, tile
    by tile of 64 entries as on the CUDA cores."""
    rng = np.random.default_rng(7)
    b = gs.build_basis(bipolar(rng, 333, 2000))
    Y = torch.from_numpy(rng.standard_normal((4000, b.r)).astype(np.float32)).cuda()
    Y[17, 140] = bad
    Y[3999, 332] = bad
    for mode in ("raw", "cosine"):
        out = gs.similarity_coeffs(b, Y, mode=mode, want_S=True)
        ref = gs.similarity_coeffs(b, Y, mode=mode, want_S=True, path="simt")
        gs.stream_status()
        assert bool(torch.isfinite(ref["S"][17, :128]).all())
        for f in (torch.isnan, torch.isposinf, torch.isneginf):
            assert torch.equal(f(out["S"]), f(ref["S"]))
        fin = torch.isfinite(ref["S"])
        top = (Y[:17].norm(dim=1).max() * b.cnorm.max()) if mode == "raw" else 1.0
        assert bool(((out["S"] - ref["S"])[fin].abs() <= 1e-4 * top).all())


# the CUDA-core GEMM's tiles of 64 and of 128 rows, its last ones ragged; rows that 16-byte loads may take and not
@pytest.mark.parametrize("B,Lq,Lk,r", [(64, 37, 70, 33), (200, 64, 129, 64), (40, 113, 500, 17), (40, 128, 500, 20),
                                       (30, 129, 501, 48), (1, 2500, 1100, 15), (1, 1, 1, 1)])
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
def test_cuda_core_tiles(gs, B, Lq, Lk, r, dtype):
    g = torch.Generator(device="cuda").manual_seed(B + Lq)
    q = torch.randn((B, Lq, r), generator=g, device="cuda").to(dtype)
    k = torch.randn((B, Lk, r), generator=g, device="cuda").to(dtype)
    A = gs.attention_scores(q, k, 0.5, apply_softmax=False, path="simt")
    gs.stream_status()
    qd, kd = q.double(), k.double().transpose(1, 2)
    assert bool(((A.double() - 0.5 * (qd @ kd)).abs() <= r * 2.0 ** -24 * (qd.abs() @ kd.abs()) + 1e-30).all())


@pytest.mark.parametrize("M,N", [(33, 700), (64, 700), (130, 65), (260, 20000)])
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
def test_cuda_core_columns(gs, M, N, dtype):
    """The same for a second operand that is read by columns."""
    rng = np.random.default_rng([M, N])
    b = gs.build_basis(bipolar(rng, M, 333))
    T = torch.from_numpy(rng.standard_normal((N, b.r)).astype(np.float32)).cuda().to(dtype)
    X = gs.reconstruct(b, T, path="simt")
    gs.stream_status()
    Td, Q = T.double(), b.Q.double()
    assert bool(((X.double() - Td @ Q).abs() <= b.r * 2.0 ** -24 * (Td.abs() @ Q.abs())).all())
