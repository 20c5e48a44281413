"""Which form the mixed drivers' tall distributions take outside the preconditioned one: the initial
ones, all of the column-dropping rule and those of more than 128 unknowns, by the double-float
factorisation up to 160 unknowns and by FP64 products with an FP32 inverse beyond."""

import pytest
import torch

from paper_2010_08581_gb300 import inputs
from paper_2010_08581_gb300 import trals as T

pytestmark = pytest.mark.gpu

DEV = "cuda:0"


@pytest.mark.parametrize("ranks,J,products", [((10, 10, 10), 1000, False), ((8, 11, 8), 1000, False),
                                              ((10, 16, 10), 2000, False), ((13, 13, 13), 2000, True)])
@pytest.mark.parametrize("drop", [False, True])
def test_form_of_the_mixed_distributions(ranks, J, products, drop):
    dims = (200, 190, 180)
    X, cores = inputs.tr_plus_noise(dims, ranks, seed=21, rel_noise=1e-2, dtype=torch.float32, device=DEV)
    out = T.empty_cores(dims, ranks)
    ctx = T.Context(0)
    try:
        if drop:
            T.tr_set_ls_rank(ctx, T.TR_LS_RANK_DROP)
        T.tr_profile_begin(ctx)
        T.tr_als_sampled(ctx, X, ranks, J, 2, 5, T.TR_PREC_MIXED, out,
                         init_cores=[inputs.slice_major(c).to(DEV) for c in cores])
        names = T.tr_profile_end(ctx)
        assert ("lev64_factor" in names) == products
        assert T.tr_rel_error(ctx, X, ranks, out) < 2e-2       # the noise, twice over
    finally:
        ctx.close()
