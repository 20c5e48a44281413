"""tr_rel_error over the forms its kernels take (Sec. 5.1): row blocks of 64, 128 and 256, one
column tile and many, ragged rows and columns, left groups of one and of many modes (short last
modes included), contraction lengths up to 256, misaligned X, and a context whose budget leaves
no room for the FP32 slice tables.

FP32 X: the products are TF32 pairs with FP32 accumulation, so TR carries at most 3 K / 8 + 2
truncations of 2^-23 (K <= 256 terms) and the FP32 slice products a few more: 1.2e-5 of ||TR||.
FP64 X: sums of FP64 products, 1e-12."""

import numpy as np
import pytest
import torch

import oracle as orc
from paper_2010_08581_gb300 import inputs
from paper_2010_08581_gb300 import trals as T

pytestmark = pytest.mark.gpu

DEV = "cuda:0"


def _case(dims, ranks, dtype):
    X, cores = inputs.tr_plus_noise(dims, ranks, seed=5, rel_noise=1e-2, dtype=dtype)
    off = inputs.random_cores(dims, ranks, 6)
    return X, [c + 0.02 * e for c, e in zip(cores, off)]


def _error(ctx, X, ranks, cores):
    return T.tr_rel_error(ctx, X, ranks, [inputs.slice_major(c).to(DEV) for c in cores])


SHAPES = [((2, 2), (1, 1)), ((1, 1, 500), (2, 3, 4)), ((500, 1, 1), (2, 3, 4)),
          ((40, 30, 20), (3, 4, 2)), ((65, 3, 257), (7, 9, 11)), ((3, 200, 2, 129), (16, 15, 16, 16)),
          ((70, 60, 50), (16, 12, 14)), ((9, 8, 7, 6, 5, 4, 3, 2), (3, 4, 5, 6, 7, 8, 9, 10)),
          ((2,) * 16, (3,) * 16), ((300, 300), (16, 16)), ((100, 3, 90, 31), (5, 10, 10, 8)),
          ((60, 50, 1031), (10, 10, 10))]


@pytest.mark.parametrize("dims,ranks", SHAPES)
@pytest.mark.parametrize("dtype,tol", [(torch.float32, 1.2e-5), (torch.float64, 1e-12)])
def test_error_matches_oracle(dims, ranks, dtype, tol):
    X, cores = _case(dims, ranks, dtype)
    ctx = T.Context(0)
    try:
        got = _error(ctx, X.to(DEV), ranks, cores)
    finally:
        ctx.close()
    ref = orc.rel_error([c.numpy() for c in cores], X.double().numpy())
    assert abs(got - ref) <= tol


@pytest.mark.parametrize("shift", [1, 2, 3])
def test_error_of_a_misaligned_tensor(shift):
    dims, ranks = (33, 21, 47), (5, 6, 7)
    X, cores = _case(dims, ranks, torch.float32)
    buf = torch.zeros(X.numel() + 8, dtype=torch.float32, device=DEV)
    view = buf[shift:shift + X.numel()].view(dims)
    view.copy_(X)
    ctx = T.Context(0)
    try:
        got = _error(ctx, view, ranks, cores)
    finally:
        ctx.close()
    assert abs(got - orc.rel_error([c.numpy() for c in cores], X.double().numpy())) <= 1.2e-5


def test_error_without_room_for_the_slice_tables():
    dims, ranks = (900, 40, 130), (12, 10, 14)
    X, cores = _case(dims, ranks, torch.float32)
    Xd = X.to(DEV)
    ref = orc.rel_error([c.numpy() for c in cores], X.double().numpy())
    done = 0
    for kb in range(1024, 16384, 256):      # the smallest budgets that the call accepts
        ctx = T.Context(0, kb << 10)
        try:
            assert abs(_error(ctx, Xd, ranks, cores) - ref) <= 1.2e-5
            done += 1
        except T.TrError as e:
            assert e.status == T.TR_ERR_BUDGET
        finally:
            ctx.close()
        if done == 2:
            break
    assert done == 2


def test_error_in_the_least_room():
    """Ranks of 16 (K = 256) with a budget for FP32 right factors only: the FP64 form, W in FP32
    (5e-7 of ||TR||); one byte less is refused. FP64 X with one partial sum per 32 rows."""
    dims, ranks = (70, 13, 9, 50), (16, 16, 16, 16)
    for dtype, es, edge in ((torch.float32, 4, 64), (torch.float64, 8, 32)):
        X, cores = _case(dims, ranks, dtype)
        ref = orc.rel_error([c.numpy() for c in cores], X.double().numpy())
        cols, rows = 9 * 50, 70 * 13       # the split at 256 columns
        blocks = min((rows + edge - 1) // edge, 4 * torch.cuda.get_device_properties(0).multi_processor_count)
        need = (16 * blocks + 255) // 256 * 256 + cols * 256 * es
        ctx = T.Context(0, need)
        try:
            assert abs(_error(ctx, X.to(DEV), ranks, cores) - ref) <= 1e-6
        finally:
            ctx.close()
        ctx = T.Context(0, need - 1)
        try:
            with pytest.raises(T.TrError) as e:
                _error(ctx, X.to(DEV), ranks, cores)
            assert e.value.status == T.TR_ERR_BUDGET
        finally:
            ctx.close()


def test_served_request_in_the_least_arena():
    """A request with K = 256 in the smallest arena that admits it: the same cores as with room
    to spare, and fits within the two forms' bounds of each other (1.2e-5 + 1e-6)."""
    dims, ranks, J = (40, 30, 60), (16, 16, 16), 2560
    X, _ = inputs.tr_plus_noise(dims, (4, 4, 4), seed=21, rel_noise=1e-2)
    X = X.to(DEV)
    init = inputs.random_cores(dims, ranks, 22)

    def run(arena):
        srv = T.Server(max_slots=1, max_modes=3, max_dim=60, max_rank=16, max_samples=J, max_sweeps=2,
                       fit_tol=0.0, X_dtype=T.TR_F32, prec=T.TR_PREC_MIXED,
                       hbm_budget_bytes=1 << 30, arena_bytes=arena)
        try:
            cores = [inputs.slice_major(c).to(DEV) for c in init]
            t = srv.submit(X, ranks, J, 23, cores, init_given=True)
            for _ in range(200):
                if srv.poll(t)["done"]:
                    break
                srv.tick()
            r = srv.poll(t)
            assert r["done"]
            return r["fit_history"][:r["sweeps"]], cores
        finally:
            srv.close()

    with pytest.raises(T.TrError) as e:
        run(1 << 20)
    assert e.value.status == T.TR_ERR_BUDGET
    need = int(str(e.value).split("workspace ")[1].split(")")[0])
    with pytest.raises(T.TrError):
        run(need - 256)
    fits, cores = run(need)
    big, ref = run(64 << 20)
    assert len(fits) == len(big) == 2
    assert np.abs(np.asarray(fits) - np.asarray(big)).max() <= 1.3e-5
    for u, v in zip(cores, ref):
        assert torch.equal(u, v)
