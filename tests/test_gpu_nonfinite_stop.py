"""A solve without a tolerance whose fit is not finite stops within a few iterations:
a call with a long limit takes about as long as one with a short limit, however many
iterations the GPU has queued."""
import math
import time

import pytest
import torch

from _util import ensure_built
from paper_1806_07985_gb300 import nncp

pytestmark = pytest.mark.gpu


def _seconds(solve, iters):
    best = math.inf
    for _ in range(4):
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        with pytest.raises(nncp.NNCPError, match="non-finite fit"):
            solve(iters)
        best = min(best, time.perf_counter() - t0)
    return best


def _data(dims, R):
    X = torch.rand(math.prod(dims), device="cuda")
    X[5] = float("nan")
    return X, [torch.rand(d, R, device="cuda") for d in dims]


# 8 iterations are queued when the first look finds the flag; twice that leaves room
def test_context():
    ensure_built()
    dims, R = (256, 256, 256), 16
    X, H0 = _data(dims, R)
    H = [h.clone() for h in H0]
    c = nncp.Context(dims, R)

    def solve(iters):
        for h, g in zip(H, H0):
            h.copy_(g)
        c.solve(iters, 0.0)
    try:
        c.set_tensor(X)
        c.set_factors(H)
        assert _seconds(solve, 5000) <= 2 * _seconds(solve, 8)
    finally:
        c.close()


def test_batch():
    ensure_built()
    dims, R, n = (40, 30, 20), 8, 64
    data = [_data(dims, R) for _ in range(n)]
    b = nncp.Batch([dims] * n, [R] * n, max_iters=5000)

    try:
        b.set_data([d[0] for d in data], [d[1] for d in data])
        solve = lambda iters: b.solve(iters, 0.0)  # (the tensors stay non-finite whatever the factors)
        assert _seconds(solve, 5000) <= 2 * _seconds(solve, 8)
    finally:
        b.close()
