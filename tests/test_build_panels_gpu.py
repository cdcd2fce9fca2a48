"""The panel factorisation of the basis build (Cholesky QR of 16 rows, with the row-by-row kernel for
the panels whose rank decisions the pivots cannot settle), against a row-by-row Gram-Schmidt in 64
bits.  Q and R are held in fp32: 2^-23 of the entry's own size covers their rounding, and the factors
themselves agree to 64-bit accuracy times the conditioning of the accepted rows (below 1e5 here)."""
import concurrent.futures as cf

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def reference(C, tol):
    C = C.double()
    Q, rows = [], []
    for c in C:
        v, t = c.clone(), torch.zeros(len(Q), dtype=torch.float64, device=c.device)
        for _ in range(2):
            for j, q in enumerate(Q):
                h = torch.dot(q, v)
                t[j] += h
                v = v - h * q
        n = float(v.norm())
        if len(Q) < C.shape[1] and n > tol * float(c.norm()):
            Q.append(v / n)
            t = torch.cat([t, torch.tensor([n], dtype=torch.float64, device=c.device)])
        rows.append(t)
    r = len(Q)
    R = torch.stack([torch.cat([t, torch.zeros(r - len(t), dtype=torch.float64, device=C.device)]) for t in rows])
    return (torch.stack(Q) if r else C.new_zeros((0, C.shape[1]))), R


def codebook(M, D, seed=1):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return (torch.randint(0, 2, (M, D), generator=g, device="cuda") * 2 - 1).float()


def check(gs, C, tol=1e-6):
    b = gs.build_basis(C, rank_tol=tol)
    gs.stream_status()
    Q, R = reference(C, tol)
    assert b.r == Q.shape[0]
    if b.r:
        assert float((b.Q.double() - Q).abs().max()) <= 1e-7
        assert float((b.R.double() - R).abs().max()) <= 1e-7 * float(R.abs().max())
        assert float((b.Q.double() @ b.Q.double().T - torch.eye(b.r, device="cuda")).abs().max()) <= 1e-6


@pytest.mark.parametrize("M,D", [(1, 1), (16, 16), (17, 33), (33, 20), (48, 131), (40, 1216), (35, 4867), (20, 14600)])
def test_panel_and_slice_edges(gs, M, D):
    check(gs, codebook(M, D))


def test_dependent_rows_in_and_across_panels(gs):
    C = codebook(50, 300)
    C[3] = C[1]                   # duplicates and sums within a panel,
    C[15] = C[2] + C[14]
    C[16] = C[0]                  # across panels,
    C[20] = 0                     # zero rows,
    C[32:] = C[:18]               # a whole dependent panel
    check(gs, C)
    check(gs, C, tol=1e-9)        # too tight for the pivots to settle: row by row


def test_nearly_dependent_rows(gs):
    C = codebook(40, 300)
    C[5] = C[4] + 1e-3 * C[6]     # accepted, below the pivots' certain range: row by row
    C[30] = C[29] + 1e-7 * C[31]  # dependent at 1e-6
    check(gs, C)


@pytest.mark.parametrize("scale", [1e-25, 1e18])
def test_scale(gs, scale):
    C = codebook(40, 500)
    a, b = gs.build_basis(C), gs.build_basis(C * scale)
    gs.stream_status()
    assert a.r == b.r
    assert float((a.Q - b.Q).abs().max()) <= 1e-7


@pytest.mark.parametrize("rows", [3, 4])
@pytest.mark.parametrize("tol", [1e-6, 1e-9])
def test_rows_close_to_what_earlier_ones_left_over(gs, rows, tol):
    """a, a + e b, b + d c, and a, a + e b, b + f c, c + d g, all exact in fp32: every row is off the span of
    those before it by more than three times the tolerance, but the last pivot's noise in a Gram matrix,
    2^-53 (2 / e)^2 of the row or 2^-53 (4 / (e f))^2, is above d^2."""
    def exact(rng, bits):
        return rng.integers(-2 ** bits, 2 ** bits + 1, 300) / 2.0 ** bits

    for seed in range(100):
        rng = np.random.default_rng([seed, rows])
        e, f = 2.0 ** -rng.integers(7, 10), 2.0 ** -rng.integers(4, 8)
        d = 2.0 ** -18 * rng.integers(1, 4)
        a, b, c, g = exact(rng, 9), exact(rng, 9), exact(rng, 3 if rows == 3 else 9), exact(rng, 3)
        if rows == 4:
            e = 2.0 ** -rng.integers(4, 8)
        C = np.stack([a, a + e * b, b + d * c] if rows == 3 else [a, a + e * b, b + f * c, c + d * g])
        C = torch.from_numpy(C.astype(np.float32)).cuda()
        b = gs.build_basis(C, rank_tol=tol)
        assert b.r == rows, (seed, e, f, d)
        Q, R = b.Q.double(), b.R.double()
        # fp32 factors: 2^-24 of each of two factors per term
        assert bool(((C.double() - R @ Q).abs() <= 2.0 ** -22 * (R.abs() @ Q.abs())).all()), seed
    gs.stream_status()


def test_builds_from_two_threads(gs):
    """Codebooks of short and of long rows, whose kernels need different amounts of shared memory, at once."""
    def build(D):
        with torch.cuda.stream(torch.cuda.Stream()):
            C = codebook(100, D)
            return [gs.build_basis(C).r for _ in range(25)]

    with cf.ThreadPoolExecutor(2) as ex:
        for ranks in ex.map(build, [512, 14600]):
            assert ranks == [100] * 25
    gs.stream_status()
