"""FP64 leverage scores of tall cores through an FP32 inverse (L >= 88, I >= L), and the
mixed LS step's blocked factor for L > 160: block edges, one row above square, columns of very
different lengths (the FP32 factorisation gives up: the FP64 one runs), scales outside FP32's
range, dependent columns.

The scores come from the Gram matrix: eps cond(A)^2 times a modest factor, 64 L."""

import pytest
import torch

from paper_2010_08581_gb300 import trals as T

pytestmark = pytest.mark.gpu

DEV = "cuda:0"
EPS = 2.2e-16


def _randn(*s, seed):
    return torch.randn(s, generator=torch.Generator().manual_seed(seed), dtype=torch.float64)


def _scores(A):
    U, S, _ = torch.linalg.svd(A, full_matrices=False)
    U = U[:, S > 1e-9 * S[0]]
    p = (U * U).sum(1)
    return p / p.sum(), float(S[0] / S[S > 1e-9 * S[0]][-1])


def _leverage(ctx, A, Rl, Rr):
    p = torch.empty(A.shape[0], dtype=torch.float64, device=DEV)
    cdf = torch.empty_like(p)
    T.tr_leverage(ctx, A.reshape(A.shape[0], Rl, Rr).contiguous().to(DEV), p, cdf)
    T.tr_status_sync(ctx)
    assert torch.allclose(torch.cumsum(p, 0), cdf, rtol=0, atol=1e-12)
    return p.cpu()


@pytest.mark.parametrize("Rl,Rr", [(4, 12), (7, 7), (8, 8), (10, 10), (8, 16), (10, 13), (11, 12), (10, 16),
                                   (12, 16), (14, 14), (15, 15), (16, 16)])
def test_scores_match_svd(Rl, Rr):
    L = Rl * Rr
    ctx = T.Context(0)
    try:
        for I in (L, L + 1, 2 * L + 31, 4001):
            A = _randn(I, L, seed=I + L)
            ref, cond = _scores(A)
            got = _leverage(ctx, A, Rl, Rr)
            assert ((got - ref).abs() <= 64 * L * EPS * cond ** 2 * ref).all()
    finally:
        ctx.close()


@pytest.mark.parametrize("Rl,Rr", [(6, 8), (10, 10), (16, 16)])
def test_scores_outside_fp32(Rl, Rr):
    """Powers of two: the scores do not change, whichever form computes them."""
    L, I = Rl * Rr, 3 * Rl * Rr + 5
    A = _randn(I, L, seed=L)
    ref, cond = _scores(A)
    ctx = T.Context(0)
    try:
        for d in (torch.tensor(2.0 ** 80), torch.tensor(2.0 ** -80),
                  torch.pow(torch.tensor(2.0, dtype=torch.float64), -torch.arange(L, dtype=torch.float64) % 12)):
            got = _leverage(ctx, A * d, Rl, Rr)
            assert ((got - ref).abs() <= 64 * L * EPS * cond ** 2 * ref).all()
        A[:, 5] = A[:, 0] + A[:, 7]
        ref, cond = _scores(A)
        got = _leverage(ctx, A, Rl, Rr)
        assert ((got - ref).abs() <= 64 * L * EPS * cond ** 2 * ref).all()
    finally:
        ctx.close()


@pytest.mark.parametrize("Rl,Rr", [(10, 13), (12, 16), (16, 16)])
def test_mixed_solve_of_a_singular_matrix_is_refused(Rl, Rr):
    L = Rl * Rr
    A = _randn(4 * L, L, seed=L).float()
    A[:, L - 2] = A[:, 3]
    out = torch.empty((9, Rl, Rr), dtype=torch.float64, device=DEV)
    ctx = T.Context(0)
    try:
        with pytest.raises(T.TrError) as e:
            T.tr_solve(ctx, A.to(DEV), _randn(4 * L, 9, seed=1).float().to(DEV), Rl, Rr, T.TR_PREC_MIXED, out)
            T.tr_status_sync(ctx)
        assert e.value.status == T.TR_ERR_SINGULAR
    finally:
        ctx.close()
