"""Which form a tall matrix's FP64 leverage scores take: products with the FP32 inverse where they
are the faster one (by the launches that the profile names), and the same scores from either form on
both sides of the line, to 1e-11 (eps cond(A)^2 is at most 1e-14 at these sizes)."""

import pytest
import torch

from paper_2010_08581_gb300 import trals as T

pytestmark = pytest.mark.gpu

DEV = "cuda:0"


def _randn(*s, seed):
    return torch.randn(s, generator=torch.Generator().manual_seed(seed), dtype=torch.float64)


@pytest.mark.parametrize("Rl,Rr,I,products", [
    (9, 9, 300, False), (8, 11, 300, True), (10, 10, 3200, True), (10, 10, 3201, False),
    (10, 10, 20000, False), (10, 16, 5120, True), (10, 16, 5121, False), (13, 13, 10816, True),
    (13, 13, 10817, False), (16, 16, 16384, True), (16, 16, 16385, False)])
def test_form_and_scores(Rl, Rr, I, products):
    core = _randn(I, Rl, Rr, seed=I)
    p = torch.empty(I, dtype=torch.float64, device=DEV)
    cdf = torch.empty_like(p)
    ctx = T.Context(0)
    try:
        T.tr_profile_begin(ctx)
        T.tr_leverage(ctx, core.to(DEV), p, cdf)
        names = T.tr_profile_end(ctx)
        T.tr_status_sync(ctx)
    finally:
        ctx.close()
    assert ("lev64_factor" in names) == products
    A = core.reshape(I, Rl * Rr).to(DEV)
    Q, _ = torch.linalg.qr(A)
    ref = (Q * Q).sum(1)
    ref = ref / ref.sum()
    assert ((p - ref).abs() <= 1e-11 * ref).all()
