"""The LS step's device-gated factorisations (FP64 from 88 unknowns on, mixed precision from 161 on) on
matrices that are too poor for the FP32 inverse: a pivot that FP32 cannot resolve, ||X M X^T - I|| too
large for the series, a dependent column under both rank rules, columns of very different lengths.

FP64, whole numbers in A and Y (M and B are exact): pairs of columns that differ by random signs, one
part in f of their entries, cond(M) about 6 f^2 and more with many pairs. In NumPy's FP32 the norm is
0.08 to 0.16 where the series ends at 0.01, and a pivot of 1 / f^2 is below L 2^-23 where it has to
be. The residual of a factorisation is a sum of L products of each entry: sqrt(L) 2^-53 ||M|| ||z||.
That the factorisation ran is read off its time (an SM takes 100 us at least; the gated launch 7).

Columns scaled by powers of two (down to 2^-11): every step scales exactly, so a solve is as accurate as
with the columns as they were, cond(M) <= 4: 1e-11 in FP64, 4e-4 mixed (3 J / 8 truncated FP32 sums,
J <= 2304, 1e-4 of M and B)."""

import numpy as np
import pytest
import torch

import oracle as orc
from paper_2010_08581_gb300 import trals as T

pytestmark = pytest.mark.gpu

DEV = "cuda:0"
U = 2.0 ** -53


def _pairs(J, L, I, f, pairs, seed):
    rng = np.random.default_rng(seed)
    A = f * (2.0 * rng.integers(0, 2, (J, L)) - 1)
    for k in range(pairs):
        A[:, 2 * k + 1] = A[:, 2 * k] + (2.0 * rng.integers(0, 2, J) - 1)
    return A, rng.integers(-9, 10, (J, I)).astype(float)


def _solution(core):
    return core.cpu().numpy().transpose(0, 2, 1).reshape(core.shape[0], -1).T     # unknown a + Rl * b


def _solve(A, Y, Rl, Rr, prec, drop=False, out=None):
    """(core, milliseconds of the factorisation)"""
    dt = torch.float64 if prec == T.TR_PREC_FP64 else torch.float32
    if out is None:
        out = torch.full((Y.shape[1], Rl, Rr), float("nan"), dtype=torch.float64, device=DEV)
    ctx = T.Context(0)
    try:
        if drop:
            T.tr_set_ls_rank(ctx, T.TR_LS_RANK_DROP)
        Ad, Yd = torch.from_numpy(A).to(DEV, dt), torch.from_numpy(Y).to(DEV, dt)
        T.tr_solve(ctx, Ad, Yd, Rl, Rr, prec, out)
        T.tr_status_sync(ctx)
        T.tr_profile_begin(ctx)
        T.tr_solve(ctx, Ad, Yd, Rl, Rr, prec, out)
        ms = T.tr_profile_end(ctx)["cholesky_solve"][0]
        T.tr_status_sync(ctx)
    finally:
        ctx.close()
    return out, ms


@pytest.mark.parametrize("Rl,Rr,f,pairs", [(10, 10, 160, 50), (15, 15, 128, 112), (16, 16, 128, 128),
                                           (10, 10, 400, 3), (15, 15, 240, 3), (16, 16, 240, 128)])
def test_fp64_factorisation_takes_over(Rl, Rr, f, pairs):
    L = Rl * Rr
    A, Y = _pairs(10 * L, L, 9, f, pairs, seed=L)
    out, ms = _solve(A, Y, Rl, Rr, T.TR_PREC_FP64)
    assert ms > 0.05
    M, B = A.T @ A, A.T @ Y
    cores = [out]
    if L <= 144:                                             # (a fixed scratch of 16 MiB)
        other = torch.full_like(out, float("nan"))
        info = torch.full((1,), -7, dtype=torch.int32, device=DEV)
        T.tr_solve_noalloc(torch.from_numpy(A).to(DEV), torch.from_numpy(Y).to(DEV), Rl, Rr,
                           T.TR_PREC_FP64, other, info)
        torch.cuda.synchronize()
        assert int(info) == 0 and torch.equal(other, out)
    for core in cores:
        z = _solution(core)
        r = (B.astype(np.longdouble) - M.astype(np.longdouble) @ z.astype(np.longdouble)).astype(float)
        assert np.linalg.norm(r) <= L ** 0.5 * U * np.linalg.norm(M, 2) * np.linalg.norm(z)


@pytest.mark.parametrize("Rl,Rr,prec,tol", [(10, 10, T.TR_PREC_FP64, 1e-11), (15, 15, T.TR_PREC_FP64, 1e-11),
                                            (12, 16, T.TR_PREC_MIXED, 4e-4), (16, 16, T.TR_PREC_MIXED, 4e-4)])
def test_columns_of_very_different_lengths(Rl, Rr, prec, tol):
    L = Rl * Rr
    rng = np.random.default_rng(L)
    A = rng.standard_normal((9 * L, L)).astype(np.float32).astype(np.float64)
    Y = rng.standard_normal((9 * L, 33)).astype(np.float32).astype(np.float64)
    d = 2.0 ** -(np.arange(L) % 12)
    Q, R = np.linalg.qr(A)
    ref = np.linalg.solve(R, Q.T @ Y)
    out, ms = _solve(A * d, Y, Rl, Rr, prec)
    assert ms > 0.05
    assert np.linalg.norm(_solution(out) * d[:, None] - ref) <= tol * np.linalg.norm(ref)


@pytest.mark.parametrize("Rl,Rr", [(10, 10), (15, 15), (12, 16), (16, 16)])
@pytest.mark.parametrize("prec,tol", [(T.TR_PREC_FP64, 1e-9), (T.TR_PREC_MIXED, 4e-4)])
def test_dependent_columns_under_both_rules(Rl, Rr, prec, tol):
    L = Rl * Rr
    rng = np.random.default_rng(L)
    A = rng.standard_normal((9 * L, L)).astype(np.float32).astype(np.float64)
    A[:, L // 2 + 3] = A[:, 2]
    A[:, L - 1] = 0.0
    Y = rng.standard_normal((9 * L, 17)).astype(np.float32).astype(np.float64)
    out = torch.full((17, Rl, Rr), 3.0, dtype=torch.float64, device=DEV)
    with pytest.raises(T.TrError) as e:
        _solve(A, Y, Rl, Rr, prec, out=out)
    assert e.value.status == T.TR_ERR_SINGULAR and torch.all(out == 3.0)
    if L <= 144:
        dt = torch.float64 if prec == T.TR_PREC_FP64 else torch.float32
        info = torch.zeros((1,), dtype=torch.int32, device=DEV)
        T.tr_solve_noalloc(torch.from_numpy(A).to(DEV, dt), torch.from_numpy(Y).to(DEV, dt), Rl, Rr, prec, out, info)
        torch.cuda.synchronize()
        assert int(info) > 0 and torch.all(out == 3.0)
    eps = 2.220446049250313e-16 if prec == T.TR_PREC_FP64 else 1.1920928955078125e-07
    ref, keep = orc.sampled_ls_normal_drop(A, Y, L * eps)
    assert list(np.nonzero(~keep)[0]) == [L // 2 + 3, L - 1]
    out, _ = _solve(A, Y, Rl, Rr, prec, drop=True)
    z = _solution(out)
    assert np.all(z[~keep] == 0.0)
    assert np.linalg.norm(z - ref) <= tol * np.linalg.norm(ref)
