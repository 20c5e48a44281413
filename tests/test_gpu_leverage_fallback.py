"""The FP64 distributions' fallback behind a device flag, inside the driver's two branches: with
TRALS_LEV_TAU=0 every series is refused and the FP64 factorisation and row solves run instead, as
with TRALS_LEV_PRECOND=0, where they run alone. Both form the same Gram and the same factor, so the
cores are equal, in a graph and out of it."""

import pytest
import torch

from paper_2010_08581_gb300 import inputs
from paper_2010_08581_gb300 import trals as T

pytestmark = pytest.mark.gpu

DEV = "cuda:0"


def _cores(dims, ranks, J, sweeps, drop, prof):
    X, _ = inputs.tr_plus_noise(dims, ranks, seed=3, rel_noise=1e-2, dtype=torch.float64)
    init = [inputs.slice_major(c).to(DEV) for c in inputs.random_cores(dims, ranks, 4)]
    out = T.empty_cores(dims, ranks)
    ctx = T.Context(0)
    try:
        if drop:
            T.tr_set_ls_rank(ctx, T.TR_LS_RANK_DROP)
        if prof:
            T.tr_profile_begin(ctx)
        for _ in range(2):        # (the second call replays the first one's graph)
            T.tr_als_sampled(ctx, X.to(DEV), ranks, J, sweeps, 9, T.TR_PREC_FP64, out, init_cores=init)
        T.tr_status_sync(ctx)
    finally:
        ctx.close()
    return out


@pytest.mark.parametrize("dims,ranks,J", [((120, 130, 140), (10, 10, 10), 1500),
                                          ((260, 270, 257), (12, 13, 16), 3000)])
@pytest.mark.parametrize("drop", [False, True])
@pytest.mark.parametrize("prof", [False, True])
def test_refused_series_gives_the_factorisation_form(dims, ranks, J, drop, prof, monkeypatch):
    monkeypatch.setenv("TRALS_LEV_TAU", "0")
    a = _cores(dims, ranks, J, 2, drop, prof)
    monkeypatch.delenv("TRALS_LEV_TAU")
    monkeypatch.setenv("TRALS_LEV_PRECOND", "0")
    b = _cores(dims, ranks, J, 2, drop, prof)
    for u, v in zip(a, b):
        assert torch.isfinite(u).all() and torch.equal(u, v)
