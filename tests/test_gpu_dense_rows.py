"""Dense TR-ALS (tr_als) at the edges of its row kernel and of the contraction that reads X in
place: runs of one row, of a part of a tile and of several tiles, cores with more entries than
the unfoldings have rows, two modes and many, strides of 1, below and above 8 and not multiples
of 32, one and several 64- or 80-column tiles.

An FP64 X on the mixed path is transposed to FP32 rows first, an FP32 X is read through its
strides: the same products in the same order, so the cores are equal. FP64 sweeps keep the
oracle's cores to 1e-8 and mixed ones its final error to 1 %, as in the other dense tests."""

import numpy as np
import pytest
import torch

import oracle as orc
from paper_2010_08581_gb300 import inputs
from paper_2010_08581_gb300 import trals as T

pytestmark = pytest.mark.gpu

DEV = "cuda:0"


def _als(X, dims, ranks, sweeps, prec, init):
    out = T.empty_cores(dims, ranks)
    ctx = T.Context(0)
    try:
        T.tr_als(ctx, X.to(DEV), ranks, sweeps, 0, prec, out,
                 init_cores=[inputs.slice_major(c).to(DEV) for c in init])
    finally:
        ctx.close()
    return out


@pytest.mark.parametrize("dims,ranks", [((300, 41), (5, 4)), ((40, 33, 8), (4, 3, 5)),
                                        ((23, 35, 37), (9, 16, 8)), ((70, 90, 31), (16, 5, 16)),
                                        ((9, 10, 11, 7), (3, 2, 4, 3)), ((18, 3, 50, 9), (6, 7, 3, 5)),
                                        ((513, 12, 65), (10, 10, 10)), ((6, 5, 4, 3, 40), (2, 2, 3, 2, 3)),
                                        ((90, 80, 100), (1, 1, 1))])
def test_x_in_place_equals_transposed_x(dims, ranks):
    X, _ = inputs.tr_plus_noise(dims, ranks, seed=11, rel_noise=1e-2)
    init = inputs.random_cores(dims, ranks, 12)
    a = _als(X, dims, ranks, 2, T.TR_PREC_MIXED, init)
    b = _als(X.double(), dims, ranks, 2, T.TR_PREC_MIXED, init)
    for u, v in zip(a, b):
        assert torch.equal(u, v)


@pytest.mark.parametrize("dims,ranks", [((90, 7), (2, 3)), ((19, 18, 17), (4, 4, 3)),
                                        ((4, 5, 3, 4, 5), (2, 2, 2, 2, 2)), ((12, 300, 1), (2, 2, 2)),
                                        ((3, 4, 600), (2, 2, 1)), ((8, 9, 7, 3), (1, 2, 3, 2)),
                                        ((40, 30, 20), (5, 1, 6))])
def test_rows_match_oracle_fp64(dims, ranks):
    X, _ = inputs.tr_plus_noise(dims, ranks, seed=13, rel_noise=1e-2, dtype=torch.float64)
    init = inputs.random_cores(dims, ranks, 14)
    ref = orc.tr_als(X.numpy(), [c.numpy() for c in init], 1)
    out = _als(X, dims, ranks, 1, T.TR_PREC_FP64, init)
    for u, r in zip(out, ref):
        g = np.transpose(u.cpu().numpy(), (1, 0, 2))
        assert np.linalg.norm(g - r) < 1e-8 * np.linalg.norm(r)


@pytest.mark.parametrize("dims,ranks", [((90, 31), (2, 3)), ((19, 18, 17), (4, 4, 3)), ((24, 33, 15), (5, 2, 6)),
                                        ((5, 6, 4, 40), (3, 2, 4, 3)), ((16, 4, 3, 5, 16), (2, 3, 2, 3, 2)),
                                        ((30, 300, 17), (2, 1, 2)), ((35, 17, 130), (10, 16, 9))])
def test_rows_by_runs_match_oracle_error(dims, ranks):
    X, _ = inputs.tr_plus_noise(dims, ranks, seed=15, rel_noise=0.05)
    init = inputs.random_cores(dims, ranks, 16)
    ref = orc.rel_error(orc.tr_als(X.double().numpy(), [c.numpy() for c in init], 3), X.double().numpy())
    out = _als(X, dims, ranks, 3, T.TR_PREC_MIXED, init)
    got = orc.rel_error([np.transpose(u.cpu().numpy(), (1, 0, 2)) for u in out], X.double().numpy())
    assert abs(got - ref) < 0.01 * ref
