"""Kernels launched while their predecessors run: calls queued one after another without a
synchronisation, on two streams, give what the same calls give one at a time, and what they give
from a captured graph (which is laid down without such launches). Equal results."""

import pytest
import torch

from paper_2010_08581_gb300 import trals as T

pytestmark = pytest.mark.gpu

DEV = "cuda:0"


def _randn(*s, seed, dt):
    return torch.randn(s, generator=torch.Generator().manual_seed(seed), dtype=torch.float64).to(dt).to(DEV)


@pytest.mark.parametrize("prec,dt", [(T.TR_PREC_MIXED, torch.float32), (T.TR_PREC_FP64, torch.float64)])
@pytest.mark.parametrize("Rl,Rr,I", [(5, 5, 40), (10, 10, 300), (12, 15, 200)])
def test_queued_and_captured_calls(prec, dt, Rl, Rr, I):
    L = Rl * Rr
    J = 6 * L
    A = [_randn(J, L, seed=s, dt=dt) for s in range(4)]
    Y = [_randn(J, I, seed=10 + s, dt=dt) for s in range(4)]
    out = [torch.zeros((I, Rl, Rr), dtype=torch.float64, device=DEV) for _ in range(4)]
    p = [torch.zeros(I, dtype=torch.float64, device=DEV) for _ in range(4)]
    cdf = [torch.zeros(I, dtype=torch.float64, device=DEV) for _ in range(4)]
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    ctxs = [T.Context(0), T.Context(0)]

    def call(s, stream=None):
        T.tr_solve(ctxs[s % 2], A[s], Y[s], Rl, Rr, prec, out[s], stream=stream)
        T.tr_leverage(ctxs[s % 2], out[s], p[s], cdf[s], stream=stream)

    try:
        for s in range(4):
            call(s)
            torch.cuda.synchronize()
        ref = [t.clone() for t in out + p + cdf]
        for t in out + p + cdf:
            t.zero_()
        torch.cuda.synchronize()
        for s in range(4):
            call(s, streams[s % 2])
        torch.cuda.synchronize()
        assert all(torch.equal(a, b) for a, b in zip(ref, out + p + cdf))
        for t in out + p + cdf:
            t.zero_()
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            call(0, torch.cuda.current_stream())
        g.replay()
        torch.cuda.synchronize()
        for k in (0, 4, 8):
            assert torch.equal(ref[k], (out + p + cdf)[k])
    finally:
        for c in ctxs:
            c.close()
