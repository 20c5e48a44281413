"""The mixed contraction at the edges of its 128-column tiles (one CTA per SM): one tile and its
remainder, several, one and two row tiles, rows that are and are not multiples of 16 bytes, the last
chunk of the samples shorter than the others.

Against a QR solve, J = 9 L rows, cond(M) <= 4: the contraction truncates at most 3 J / 8 FP32 sums
(J <= 2304), 1e-4 of M and B, times cond(M): 4e-4. X read in place (a strided mode of a dense sweep)
against X transposed first: the same products in the same order."""

import pytest
import torch

from paper_2010_08581_gb300 import inputs
from paper_2010_08581_gb300 import trals as T

pytestmark = pytest.mark.gpu

DEV = "cuda:0"


def _randn(*s, seed):
    return torch.randn(s, generator=torch.Generator().manual_seed(seed), dtype=torch.float64)


@pytest.mark.parametrize("Rl,Rr,I", [(5, 5, 103), (8, 8, 65), (10, 10, 28), (10, 10, 29), (10, 10, 500),
                                     (10, 10, 501), (11, 11, 300), (8, 16, 129), (10, 13, 125),
                                     (12, 12, 500), (16, 16, 1), (16, 16, 1025)])
def test_solve_matches_qr(Rl, Rr, I):
    L = Rl * Rr
    J = min(9 * L + 7, 2304)
    A, Y = _randn(J, L, seed=L).float(), _randn(J, I, seed=I).float()
    Q, R = torch.linalg.qr(A.double())
    ref = torch.linalg.solve_triangular(R, Q.T @ Y.double(), upper=True).T.reshape(I, Rr, Rl).transpose(1, 2)
    out = torch.empty((I, Rl, Rr), dtype=torch.float64, device=DEV)
    ctx = T.Context(0)
    try:
        T.tr_solve(ctx, A.to(DEV), Y.to(DEV), Rl, Rr, T.TR_PREC_MIXED, out)
        T.tr_status_sync(ctx)
    finally:
        ctx.close()
    assert (out.cpu() - ref).norm() <= 4e-4 * ref.norm()


@pytest.mark.parametrize("dims,ranks", [((40, 30, 251), (10, 10, 10)), ((41, 31, 250), (10, 11, 10)),
                                        ((33, 200, 64), (8, 8, 8)), ((20, 150, 120), (14, 12, 11))])
def test_x_in_place_equals_transposed_x(dims, ranks):
    X, _ = inputs.tr_plus_noise(dims, ranks, seed=31, rel_noise=1e-2)
    init = [inputs.slice_major(c).to(DEV) for c in inputs.random_cores(dims, ranks, 32)]
    got = []
    for x in (X, X.double()):
        got.append(T.empty_cores(dims, ranks))
        ctx = T.Context(0)
        try:
            T.tr_als(ctx, x.to(DEV), ranks, 1, 0, T.TR_PREC_MIXED, got[-1], init_cores=init)
        finally:
            ctx.close()
    for u, v in zip(*got):
        assert torch.equal(u, v)
