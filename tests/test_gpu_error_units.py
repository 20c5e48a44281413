"""The FP64 error's CTAs at the edges of what is resident: three, two and one per SM by the length of
the contraction (K = 9, 80, 121, 144, 256), as many units as resident CTAs, a few more (one each) and
many. Against the whole tensor in FP64: sums of n squares of entries with
n <= 3e5 and K <= 256 products each: relative rounding below (n + 256 |TR| / |TR - X|) 2^-53 < 1e-10."""

import pytest
import torch

from paper_2010_08581_gb300 import inputs
from paper_2010_08581_gb300 import trals as T

pytestmark = pytest.mark.gpu

DEV = "cuda:0"


@pytest.mark.parametrize("dims,ranks", [((100, 3, 3), (3, 3, 3)), ((120, 9, 270), (5, 16, 16)),
                                        ((7, 900, 11), (11, 11, 11)), ((7, 1000, 12), (11, 11, 11)),
                                        ((300, 490), (5, 16)), ((300, 620), (12, 12)), ((33, 1000, 9), (16, 16, 16)),
                                        ((5, 1217, 33), (8, 12, 12)), ((90, 9, 300), (12, 6, 14))])
def test_error_matches_the_whole_tensor(dims, ranks):
    X, cores = inputs.tr_plus_noise(dims, ranks, seed=41, rel_noise=1e-2, dtype=torch.float64)
    P = cores[0].permute(1, 0, 2)                       # product of slices, [index][R_last][R]
    for c in cores[1:]:
        P = torch.einsum("pab,bic->piac", P, c).reshape(-1, P.shape[1], c.shape[2])
    TR = P.diagonal(dim1=1, dim2=2).sum(1).reshape(dims)
    ref = float((TR - X).norm() / X.norm())
    ctx = T.Context(0)
    try:
        got = T.tr_rel_error(ctx, X.to(DEV), ranks, [inputs.slice_major(c).to(DEV) for c in cores])
    finally:
        ctx.close()
    assert abs(got - ref) <= 1e-10 * ref
