"""tr_rel_error of FP32 X with K = 256 under a budget for the tensor cores' operand of W and one
partial sum per row block of 128 (the room of one CTA per row block): the tensor-core form, not the
FP64 one. Its FP32 sums do not depend on how the tiles are dealt out to the CTAs, and the FP64 sums
of those differ in their order alone: 1e-12 of the value with room to spare. The FP64 form, which
takes half the room and forms its products in FP64, differs by more than 1e-9."""

import pytest
import torch

from paper_2010_08581_gb300 import inputs
from paper_2010_08581_gb300 import trals as T

pytestmark = pytest.mark.gpu

DEV = "cuda:0"


@pytest.mark.parametrize("dims", [(70, 13, 9, 50), (160, 31, 9, 50)])
def test_partial_sums_give_way_before_the_form(dims):
    ranks = (16, 16, 16, 16)
    X, cores = inputs.tr_plus_noise(dims, ranks, seed=5, rel_noise=1e-2, dtype=torch.float32)
    off = inputs.random_cores(dims, ranks, 6)
    cores = [inputs.slice_major(c + 0.02 * e).to(DEV) for c, e in zip(cores, off)]
    X = X.to(DEV)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    rows, cols = dims[0] * dims[1], dims[2] * dims[3]      # the split at 256 columns
    operand = (cols + 127) // 128 * 8 * 32768              # tiles, chunks of 32 terms, both parts
    blocks = min((rows + 127) // 128, sms)
    plain = (16 * min((rows + 63) // 64, 4 * sms) + 255) // 256 * 256 + cols * 256 * 4
    got = []
    for budget in (0, (16 * blocks + 255) // 256 * 256 + operand, plain):
        ctx = T.Context(0, budget)
        try:
            got.append(T.tr_rel_error(ctx, X, ranks, cores))
        finally:
            ctx.close()
    assert abs(got[1] - got[0]) <= 1e-12 * got[0]
    assert abs(got[2] - got[0]) > 1e-9 * got[0]
