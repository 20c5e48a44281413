"""The batched draws and Grams at their edges, against the single-problem driver in FP64 (same
draws; 1e-8 per core as in the other batched tests): one unknown, odd sizes, Grams of more
blocks than one CTA takes, wide modes, fibres longer than the entries loaded ahead, chunks of
samples that do not fill a CTA."""

import pytest
import torch

from paper_2010_08581_gb300 import inputs
from paper_2010_08581_gb300 import trals as T

pytestmark = pytest.mark.gpu

DEV = "cuda:0"
SHAPES = [((300, 20, 18), (1, 1, 1), 50), ((290, 31, 12), (3, 5, 4), 131), ((8, 40, 9, 33), (4, 4, 3, 5), 333),
          ((50, 60, 70), (11, 12, 13), 1600), ((300, 90, 100), (7, 9, 8), 700)]


@pytest.mark.parametrize("spw", [1, 4, 8])
def test_batched_matches_single_fp64(spw):
    probs, ref = [], []
    ctx = T.Context(0)
    try:
        for i, (dims, ranks, J) in enumerate(SHAPES):
            X, _ = inputs.tr_plus_noise(dims, ranks, seed=70 + i, rel_noise=1e-2, dtype=torch.float64)
            init = [inputs.slice_major(c).to(DEV) for c in inputs.random_cores(dims, ranks, 80 + i)]
            X = X.to(DEV)
            out = T.empty_cores(dims, ranks)
            T.tr_als_sampled(ctx, X, ranks, J, 1, 90 + i, T.TR_PREC_FP64, out, init_cores=init)
            ref.append(out)
            probs.append(dict(X=X, ranks=ranks, J=J, seed=90 + i, cores=[c.clone() for c in init], init=True))
        T.tr_set_batched_tiles(ctx, spw, 64)
        T.tr_als_sampled_batched(ctx, probs, 1, T.TR_PREC_FP64)
    finally:
        ctx.close()
    for p, r in zip(probs, ref):
        for u, v in zip(p["cores"], r):
            assert (u - v).norm() <= 1e-8 * v.norm()
