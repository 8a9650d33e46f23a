"""MTTKRPs captured on a caller's stream behind the kernel that writes their tensor.
The producer is a float32 MTTKRP whose work is cut over the GPU: its last kernel,
the sum of the partial tiles, lets its successor start at once, so a successor that
read its tensor before waiting would read the previous replay's.  Replays with new
contents give the bits of the same calls made one after another."""
import math

import pytest
import torch

from _util import ensure_built
from paper_1806_07985_gb300 import nncp

pytestmark = pytest.mark.gpu

P_DIMS, P_R = (2048, 40, 33), 64  # the producer: M_1 (2048 x 64) is the consumer's tensor
DIMS, R = (64, 64, 32), 20


def _rand(*shape, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return torch.rand(*shape, generator=g, device="cuda")


def _check(make_consumer, outs):
    """make_consumer(X, stream) -> a function that queues calls writing `outs`."""
    ensure_built()
    stream = torch.cuda.Stream()
    src = torch.empty(math.prod(P_DIMS), device="cuda")
    PH = [_rand(d, P_R, seed=10 + n) for n, d in enumerate(P_DIMS)]
    X = torch.zeros(P_DIMS[0], P_R, device="cuda")
    consume, close = make_consumer(X.view(-1), stream)
    try:
        def calls():
            nncp.nncp_mttkrp_noalloc(P_DIMS, P_R, src, PH, 1, X, stream=stream)
            consume()
        expected, data = [], [_rand(src.numel(), seed=100 + t) for t in range(4)]
        torch.cuda.synchronize()
        for d in data:  # each call finished before the next
            src.copy_(d)
            torch.cuda.synchronize()
            nncp.nncp_mttkrp_noalloc(P_DIMS, P_R, src, PH, 1, X, stream=stream)
            torch.cuda.synchronize()
            consume()
            torch.cuda.synchronize()
            expected.append([o.clone() for o in outs])
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            calls()
        for _ in range(5):
            for d, exp in zip(data, expected):
                src.copy_(d)
                torch.cuda.synchronize()
                graph.replay()
                torch.cuda.synchronize()
                for o, e in zip(outs, exp):
                    assert torch.equal(o, e)
    finally:
        close()


@pytest.mark.parametrize("mode", [1, 2, 3])
def test_noalloc(mode):
    M = torch.empty(DIMS[mode - 1], R, device="cuda")
    H = [_rand(d, R, seed=n) for n, d in enumerate(DIMS)]

    def make(X, stream):
        return (lambda: nncp.nncp_mttkrp_noalloc(DIMS, R, X, H, mode, M, stream=stream)), (lambda: None)
    _check(make, [M])


def _context(precision, call, outs):
    def make(X, stream):
        c = nncp.Context(DIMS, R, precision=precision, root_split=1, stream=stream)
        c.set_tensor(X)
        c.set_factors([_rand(d, R, seed=n) for n, d in enumerate(DIMS)])
        return (lambda: call(c)), c.close
    _check(make, outs)


@pytest.mark.parametrize("side", [0, 1])
def test_partial_fp32(side):
    T = torch.empty(DIMS[0] if side == 0 else DIMS[1] * DIMS[2], R, device="cuda")
    _context("fp32_simt", lambda c: c.partial_mttkrp(side, T), [T])


@pytest.mark.parametrize("tree", [0, 1])
def test_context_mttkrp_fp32(tree):
    Ms = [torch.empty(d, R, device="cuda") for d in DIMS]
    _context("fp32_simt", lambda c: [c.mttkrp(n + 1, tree, M) for n, M in enumerate(Ms)], Ms)


@pytest.mark.parametrize("side", [0, 1])
@pytest.mark.parametrize("precision", ["tf32", "split_bf16x3"])
def test_partial_tensor_cores(precision, side):
    T = torch.empty(DIMS[0] if side == 0 else DIMS[1] * DIMS[2], R, device="cuda")
    _context(precision, lambda c: c.partial_mttkrp(side, T), [T])


@pytest.mark.parametrize("side", [0, 1])
def test_partial_bf16(side):
    T = torch.empty(DIMS[0] if side == 0 else DIMS[1] * DIMS[2], R, device="cuda")

    def make(X, stream):
        Xb = torch.empty(X.numel(), dtype=torch.bfloat16, device="cuda")
        c = nncp.Context(DIMS, R, precision="bf16_stored", root_split=1, stream=stream)
        c.set_tensor(Xb)
        c.set_factors([_rand(d, R, seed=n) for n, d in enumerate(DIMS)])

        def consume():
            nncp.nncp_tensor_to_bf16(X, Xb, stream=stream)
            c.partial_mttkrp(side, T)
        return consume, c.close
    _check(make, [T])
