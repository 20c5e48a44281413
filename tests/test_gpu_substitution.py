"""The blocked substitutions (LS solve and FP64 leverage rows) at the edges of their panels (16
columns in FP64, 32 in FP32), of the row groups (32, 64, 128, 256 rows) and of the vectors per CTA
(4, 8 from 8 per SM on).

Well-conditioned problems, J = 9 L rows: cond(M) <= 4. FP64 solves to 1e-11. Mixed: the
contraction truncates at most 3 J / 8 FP32 sums (J <= 2304), 1e-4 of M and B, times cond(M):
4e-4. Leverage scores from the FP64 Gram matrix to 1e-11."""

import pytest
import torch

from paper_2010_08581_gb300 import trals as T

pytestmark = pytest.mark.gpu

DEV = "cuda:0"
RANKS = [(1, 1), (3, 5), (4, 4), (1, 16), (2, 9), (3, 11), (8, 8), (5, 13), (8, 16), (13, 10), (10, 16),
         (7, 15), (15, 15), (16, 16)]


def _randn(*s, seed):
    return torch.randn(s, generator=torch.Generator().manual_seed(seed), dtype=torch.float64)


@pytest.mark.parametrize("Rl,Rr", RANKS)
@pytest.mark.parametrize("prec,dt,tol", [(T.TR_PREC_FP64, torch.float64, 1e-11),
                                         (T.TR_PREC_MIXED, torch.float32, 4e-4)])
def test_solve_matches_qr(Rl, Rr, prec, dt, tol):
    L = Rl * Rr
    J = max(9 * L, 40)
    A = _randn(J, L, seed=L)
    Q, R = torch.linalg.qr(A.to(dt).double())
    ctx = T.Context(0)
    try:
        for I in (1, 5, 8 * torch.cuda.get_device_properties(0).multi_processor_count + 3):
            Y = _randn(J, I, seed=I).to(dt)
            Z = torch.linalg.solve_triangular(R, Q.T @ Y.double(), upper=True)
            ref = Z.T.reshape(I, Rr, Rl).transpose(1, 2)
            out = torch.empty((I, Rl, Rr), dtype=torch.float64, device=DEV)
            T.tr_solve(ctx, A.to(dt).to(DEV), Y.to(DEV), Rl, Rr, prec, out)
            T.tr_status_sync(ctx)
            assert (out.cpu() - ref).norm() <= tol * ref.norm()
    finally:
        ctx.close()


@pytest.mark.parametrize("Rl,Rr", RANKS)
def test_leverage_rows_match_qr(Rl, Rr):
    L = Rl * Rr
    ctx = T.Context(0)
    try:
        for I in (9 * L, 9 * L + 5, 1300 + 9 * L):
            core = _randn(I, Rl, Rr, seed=I)
            Q, _ = torch.linalg.qr(core.transpose(1, 2).reshape(I, L))
            p = (Q * Q).sum(1)
            p = p / p.sum()
            got = torch.empty(I, dtype=torch.float64, device=DEV)
            cdf = torch.empty(I, dtype=torch.float64, device=DEV)
            T.tr_leverage(ctx, core.to(DEV), got, cdf)
            T.tr_status_sync(ctx)
            assert ((got.cpu() - p).abs() <= 1e-11 * p).all()
            assert (cdf.cpu() - torch.cumsum(p, 0)).abs().max() <= 1e-11
    finally:
        ctx.close()
