"""Which form a dense sweep's FP32 rows take: by runs of the fastest mode where the runs are long or few,
row by row where they are short and many (by the launches that the profile names), with equal cores
from X in FP32 and in FP64 and the oracle's final error either way."""

import numpy as np
import pytest
import torch

import oracle as orc
from paper_2010_08581_gb300 import inputs
from paper_2010_08581_gb300 import trals as T

pytestmark = pytest.mark.gpu

DEV = "cuda:0"


@pytest.mark.parametrize("dims,r,runs,rows", [((8,) * 5, 3, True, False), ((2,) * 12, 2, False, True),
                                              ((20, 20, 4, 4), 3, True, True), ((12, 10, 9, 9), 4, True, False),
                                              ((41, 37, 3, 2), 2, True, True), ((3, 3, 30, 40), 3, True, False)])
def test_form_and_error(dims, r, runs, rows):
    ranks = (r,) * len(dims)
    X, _ = inputs.tr_plus_noise(dims, ranks, seed=51, rel_noise=0.05)
    init = inputs.random_cores(dims, ranks, 52)
    got = []
    for x in (X, X.double()):
        out = T.empty_cores(dims, ranks)
        ctx = T.Context(0)
        try:
            T.tr_profile_begin(ctx)
            T.tr_als(ctx, x.to(DEV), ranks, 2, 0, T.TR_PREC_MIXED, out,
                     init_cores=[inputs.slice_major(c).to(DEV) for c in init])
            names = T.tr_profile_end(ctx)
        finally:
            ctx.close()
        assert ("dense_rows" in names, "subchain" in names) == (runs, rows)
        got.append(out)
    for u, v in zip(*got):
        assert torch.equal(u, v)
    ref = orc.rel_error(orc.tr_als(X.double().numpy(), [c.numpy() for c in init], 2), X.double().numpy())
    err = orc.rel_error([np.transpose(u.cpu().numpy(), (1, 0, 2)) for u in got[0]], X.double().numpy())
    assert abs(err - ref) < 0.01 * ref
