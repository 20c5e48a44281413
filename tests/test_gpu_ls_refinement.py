"""The FP64 LS step for L >= 88 (an explicit inverse of the factor, then one step of refinement):
as small a residual as a factorisation leaves, for well and badly conditioned normal equations.

Whole numbers in A and Y: M = A^T A and B = A^T Y are exact, here and in the kernels. With f > 1,
ten columns form five pairs that differ by random signs, one part in f of their entries: cond(M)
is about 5.6 f^2. The residual of the refined z is the rounding of z itself, u ||M|| ||z|| with
u = 2^-53, and the rounding of r = b - M z: together below 1.5 u ||M||_2 ||z||_F (a factorisation:
0.3 to 1.6 u, the explicit inverse alone: 1.8 to 8 u, with NumPy's products)."""

import numpy as np
import pytest
import torch

from paper_2010_08581_gb300 import trals as T

pytestmark = pytest.mark.gpu

DEV = "cuda:0"
BOUND = 1.5 * 2.0 ** -53


def _problem(J, L, I, f, seed):
    rng = np.random.default_rng(seed)
    A = f * (2.0 * rng.integers(0, 2, (J, L)) - 1)
    for k in range(5 if f > 1 else 0):
        A[:, 2 * k + 1] = A[:, 2 * k] + (2.0 * rng.integers(0, 2, J) - 1)
    return A, rng.integers(-9, 10, (J, I)).astype(float)


def _residual(A, Y, core):
    I, Rl, Rr = core.shape
    z = core.transpose(0, 2, 1).reshape(I, Rl * Rr).T       # unknown a + Rl * b
    M, B = A.T @ A, A.T @ Y
    r = B.astype(np.longdouble) - M.astype(np.longdouble) @ z.astype(np.longdouble)
    return float(np.linalg.norm(r.astype(float)) / (np.linalg.norm(M, 2) * np.linalg.norm(z)))


def _solve(A, Y, Rl, Rr, noalloc):
    out = torch.empty((Y.shape[1], Rl, Rr), dtype=torch.float64, device=DEV)
    Ad, Yd = torch.from_numpy(A).to(DEV), torch.from_numpy(Y).to(DEV)
    if noalloc:
        T.tr_solve_noalloc(Ad, Yd, Rl, Rr, T.TR_PREC_FP64, out)
        torch.cuda.synchronize()
    else:
        ctx = T.Context(0)
        try:
            T.tr_solve(ctx, Ad, Yd, Rl, Rr, T.TR_PREC_FP64, out)
            T.tr_status_sync(ctx)
        finally:
            ctx.close()
    return out.cpu().numpy()


@pytest.mark.parametrize("Rl,Rr", [(8, 11), (10, 10), (12, 12), (15, 15), (16, 16)])
@pytest.mark.parametrize("f", [1, 16, 64, 128])
def test_residual_is_that_of_a_factorisation(Rl, Rr, f):
    L = Rl * Rr
    A, Y = _problem(10 * L, L, 9, f, seed=L)
    for noalloc in (False, True) if L <= 144 else (False,):      # (a fixed scratch of 16 MiB)
        assert _residual(A, Y, _solve(A, Y, Rl, Rr, noalloc)) <= BOUND


@pytest.mark.parametrize("I", [60, 200, 540])
def test_many_right_hand_sides(I):
    """Two chunks of the samples, the least scratch."""
    A, Y = _problem(127, 90, I, 1, seed=I)
    assert _residual(A, Y, _solve(A, Y, 9, 10, False)) <= BOUND
