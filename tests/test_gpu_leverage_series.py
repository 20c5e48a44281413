"""The series for (I + E)^-1/2 behind the FP64 leverage scores of tall cores with L >= 88: A = Q S V^T with
prescribed singular values, whose scores are those of Q, at cond(A)^2 for which ||E||_F lies in each of
the series' ranges (E^3, E^5, E^7; in NumPy, with an FP32 Cholesky factor, 4e-5 to 1e-4, 6e-4 to 1.3e-3 and
1.5e-3 to 7e-3).

The rounding of E is what remains: 0.01 to 0.06 of eps cond(A)^2 max(l) there, so 0.1 is the bound.
Cut after E the series is 1000 times above it and more, after E^2 5 to 50 times at the two largest cond;
what E^4 and the terms behind it add is below the rounding everywhere."""

import pytest
import torch

from paper_2010_08581_gb300 import trals as T

pytestmark = pytest.mark.gpu

DEV = "cuda:0"
EPS = 2.220446049250313e-16


@pytest.mark.parametrize("Rl,Rr", [(8, 11), (10, 10), (10, 13), (12, 16), (16, 16)])
@pytest.mark.parametrize("cond2", [1e3, 3e4, 1e5, 2e5])
def test_scores_of_an_orthogonal_factor(Rl, Rr, cond2):
    L = Rl * Rr
    I = 2 * L + 31
    g = torch.Generator().manual_seed(L)
    Q, _ = torch.linalg.qr(torch.randn((I, L), generator=g, dtype=torch.float64))
    V, _ = torch.linalg.qr(torch.randn((L, L), generator=g, dtype=torch.float64))
    s = cond2 ** (-0.5 * torch.arange(L, dtype=torch.float64) / (L - 1))
    ref = (Q * Q).sum(1)
    ref = ref / ref.sum()
    p = torch.empty(I, dtype=torch.float64, device=DEV)
    cdf = torch.empty_like(p)
    ctx = T.Context(0)
    try:
        core = ((Q * s) @ V.T).reshape(I, Rl, Rr).contiguous().to(DEV)
        T.tr_leverage(ctx, core, p, cdf)
        T.tr_status_sync(ctx)
        T.tr_profile_begin(ctx)
        T.tr_leverage(ctx, core, p, cdf)
        ms = T.tr_profile_end(ctx)
    finally:
        ctx.close()
    assert ms["lev64_factor"][1] == 1
    if L <= 160 or cond2 <= 1e5:        # (gated launch: the series ran; larger ones are near its end)
        assert ms["cholesky_leverage"][0] < 0.05
    assert (p.cpu() - ref).abs().max() <= 0.1 * EPS * cond2 * ref.max()
