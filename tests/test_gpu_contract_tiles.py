"""The normal-equation contractions at the edges of their tiles.

FP64 (32 x 32 tiles, those below the diagonal written by their mirror images): tr_solve of a
well-conditioned A (cond <= 4) against a QR solve; J eps cond^2 < 1e-11 at the sizes here.
Batched (tiles of 32 or 64 columns, half the rows where an instance has few unknowns): the tile
never changes a result, for L up to half a tile, a tile and beyond, J not a multiple of 16."""

import pytest
import torch

from paper_2010_08581_gb300 import inputs
from paper_2010_08581_gb300 import trals as T

pytestmark = pytest.mark.gpu

DEV = "cuda:0"


@pytest.mark.parametrize("J,Rl,Rr,I", [(1, 1, 1, 1), (40, 2, 2, 3), (300, 4, 8, 1), (333, 3, 11, 31),
                                       (2000, 5, 5, 100), (577, 8, 8, 257), (900, 9, 7, 33),
                                       (1000, 10, 10, 4), (2500, 16, 16, 40)])
def test_fp64_solve_matches_qr(J, Rl, Rr, I):
    g = torch.Generator().manual_seed(J)
    A = torch.randn((J, Rl * Rr), generator=g, dtype=torch.float64)
    Y = torch.randn((J, I), generator=g, dtype=torch.float64)
    Q, R = torch.linalg.qr(A)
    Z = torch.linalg.solve_triangular(R, Q.T @ Y, upper=True)         # L x I
    ref = Z.T.reshape(I, Rr, Rl).transpose(1, 2)
    out = torch.empty((I, Rl, Rr), dtype=torch.float64, device=DEV)
    ctx = T.Context(0)
    try:
        T.tr_solve(ctx, A.to(DEV), Y.to(DEV), Rl, Rr, T.TR_PREC_FP64, out)
        T.tr_status_sync(ctx)
    finally:
        ctx.close()
    assert (out.cpu() - ref).norm() <= 1e-11 * ref.norm()


@pytest.mark.parametrize("prec,dt", [(T.TR_PREC_MIXED, torch.float32), (T.TR_PREC_FP64, torch.float64)])
def test_batched_tile_never_changes_a_result(prec, dt):
    shapes = [((20, 18, 16), (2, 3, 2), 77), ((25, 31, 12), (4, 4, 4), 160), ((30, 41, 22), (5, 4, 8), 331),
              ((34, 70, 33), (8, 7, 9), 640), ((60, 90, 50), (11, 12, 10), 1325)]
    ref = None
    for tile in (64, 32):
        probs = []
        for i, (d, r, J) in enumerate(shapes):
            X, _ = inputs.tr_plus_noise(d, r, seed=30 + i, rel_noise=1e-2, dtype=dt)
            init = [inputs.slice_major(c).to(DEV) for c in inputs.random_cores(d, r, 40 + i)]
            probs.append(dict(X=X.to(DEV), ranks=r, J=J, seed=50 + i, cores=init, init=True))
        ctx = T.Context(0)
        try:
            T.tr_set_batched_tiles(ctx, 4, tile)
            T.tr_als_sampled_batched(ctx, probs, 2, prec)
        finally:
            ctx.close()
        got = [c for p in probs for c in p["cores"]]
        ref = ref or got
    for u, v in zip(ref, got):
        assert torch.equal(u, v)
