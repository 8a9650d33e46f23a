"""The float32 MTTKRP kernel at the edges of its tiles, steps and work split, against
the float64 definition.  Sums are of nonnegative terms in chains of at most about
a thousand float32 additions per partial: sqrt(1024) 2^-24 = 1.9e-6 relative."""
import math

import numpy as np
import pytest
import torch

from _util import ensure_built, rel_fro
from paper_1806_07985_gb300 import nncp

pytestmark = pytest.mark.gpu
TOL = 2e-6

CASES = [
    # tile edges of the outputs (32 .. 256 rows) and ends of the contraction in a step
    ((31, 33), 8), ((32, 4, 8), 9), ((33, 3, 11), 7), ((255, 31), 16), ((256, 129), 17), ((257, 7, 9), 5),
    # fastest contracted mode shorter than, equal to and longer than a step; unit modes
    ((1, 2, 3, 40), 6), ((2, 5, 31, 3), 12), ((3, 32, 2, 5), 4), ((5, 1, 33, 2), 3), ((36, 1, 1, 34), 20),
    # every alignment of the contiguous index
    ((64, 20, 12), 8), ((65, 21, 13), 8), ((66, 22, 14), 10), ((67, 23, 15), 11),
    # ranks around the groups of eight, the highest, and one whose factor rows are taken in blocks
    ((40, 30, 9), 1), ((40, 30, 9), 31), ((40, 30, 9), 33), ((28, 30, 17), 64), ((28, 30, 17), 65),
    ((60, 44, 7), 127), ((60, 44, 7), 128), ((1, 2, 3, 2, 5, 2, 3, 4), 128), ((2, 3, 2, 1, 7, 2, 3, 5), 97),
    # many tiles (a cut last wave, runs over two tiles) and few tiles with a long contraction
    ((40003, 9), 12), ((70, 700, 11), 24), ((12, 64, 900), 33), ((9, 20000), 100), ((30011, 5, 3), 3),
]


def _reference(x, dims, H, n):
    N, L, Q = len(dims), math.prod(dims[:n]), math.prod(dims[n + 1:])

    def krp(fs):
        k = np.ones((1, H[0].shape[1]))
        for f in fs:
            k = (f[:, None, :] * k[None, :, :]).reshape(-1, k.shape[1])
        return k
    T = x.reshape(Q * dims[n], L) @ krp(H[:n])
    return (T.reshape(Q, dims[n], -1) * krp(H[n + 1:N])[:, None, :]).sum(0)


@pytest.mark.parametrize("dims,R", CASES)
def test_every_mode_and_both_root_branches(dims, R):
    ensure_built()
    rng = np.random.default_rng(sum(dims) * 131 + R)
    x = rng.random(math.prod(dims)).astype(np.float32)
    H = [rng.random((d, R)).astype(np.float32) for d in dims]
    X64, H64 = x.astype(np.float64), [h.astype(np.float64) for h in H]
    X, Hd = torch.from_numpy(x).cuda(), [torch.from_numpy(h).cuda() for h in H]
    refs = [_reference(X64, dims, H64, n) for n in range(len(dims))]
    for n, ref in enumerate(refs):
        if dims[n] * R > 1 << 20:
            continue
        M = torch.full((dims[n], R), float("nan"), device="cuda")
        nncp.nncp_mttkrp_noalloc(dims, R, X, Hd, n + 1, M)
        torch.cuda.synchronize()
        assert rel_fro(M.cpu().numpy(), ref) <= TOL, n
    for split in range(1, len(dims)):
        c = nncp.Context(dims, R, root_split=split)
        try:
            c.set_tensor(X)
            c.set_factors(Hd)
            for n, ref in enumerate(refs):
                for tree in (0, 1):
                    M = torch.full((dims[n], R), float("nan"), device="cuda")
                    c.mttkrp(n + 1, tree, M)
                    torch.cuda.synchronize()
                    assert rel_fro(M.cpu().numpy(), ref) <= TOL, (split, n, tree)
        finally:
            c.close()


def test_unaligned_output_and_bits_repeat():
    # an output that is not 16-byte aligned takes the scalar stores; the same bits
    dims, R = (70, 33, 9), 12
    g = torch.Generator(device="cuda")
    g.manual_seed(3)
    X = torch.rand(math.prod(dims), generator=g, device="cuda")
    H = [torch.rand(d, R, generator=g, device="cuda") for d in dims]
    torch.cuda.synchronize()
    c = nncp.Context(dims, R, root_split=1)
    try:
        c.set_tensor(X)
        c.set_factors(H)
        for n in range(3):
            a, b = torch.empty(dims[n], R, device="cuda"), torch.empty(dims[n] * R + 1, device="cuda")
            c.mttkrp(n + 1, 0, a)
            c.mttkrp(n + 1, 0, b[1:].view(dims[n], R))
            torch.cuda.synchronize()
            assert torch.equal(a.reshape(-1), b[1:])
    finally:
        c.close()


# Runs of at most a few hundred additions, many of them: their roundings average out, and
# what is left is the result's own rounding (2^-24 / sqrt(3) over uniform mantissas) and a
# handful of additions in pairs, each level's errors sqrt(2) smaller: below 2^-24 together.
@pytest.mark.parametrize("dims,R,n", [
    ((301, 257, 199), 20, 0), ((10, 52, 880), 4, 0), ((130, 77, 65, 12), 20, 3), ((227, 154, 50), 4, 2)])
def test_sums_of_many_runs(dims, R, n):
    ensure_built()
    rng = np.random.default_rng(17)
    x = rng.random(math.prod(dims)).astype(np.float32)
    H = [rng.random((d, R)).astype(np.float32) for d in dims]
    ref = _reference(x.astype(np.float64), dims, [h.astype(np.float64) for h in H], n)
    M = torch.empty(dims[n], R, device="cuda")
    nncp.nncp_mttkrp_noalloc(dims, R, torch.from_numpy(x).cuda(), [torch.from_numpy(h).cuda() for h in H], n + 1, M)
    torch.cuda.synchronize()
    assert rel_fro(M.cpu().numpy(), ref) <= 2.0 ** -24


# A chain of n float32 additions of nonnegative terms of one size is off by at most
# 2^-24 sqrt(n) / 3 of its sum (rms; each addition rounds by up to 2^-24 / sqrt(3) of a partial
# sum).  A run of up to 32 steps is added in segments of 160 elements, a longer one in
# segments of 320, and the segments one after the other; then come the result's own rounding
# and the pairs above.
@pytest.mark.parametrize("dims,R,split,seg", [
    ((300, 256, 200), 20, 1, 160), ((301, 257, 199), 20, 1, 160), ((33, 23, 120, 82), 93, 2, 160),
    ((521, 110, 111), 85, 1, 160), ((1140, 130, 162), 35, 1, 320)])
def test_long_runs_in_segments(dims, R, split, seg):
    ensure_built()
    rng = np.random.default_rng(23)
    x = rng.random(math.prod(dims)).astype(np.float32)
    H = [rng.random((d, R)).astype(np.float32) for d in dims]
    L = math.prod(dims[:split])
    k = np.ones((1, R))
    for h in H[:split]:
        k = (h.astype(np.float64)[:, None] * k).reshape(-1, R)
    ref = x.astype(np.float64).reshape(-1, L) @ k
    c = nncp.Context(dims, R, root_split=split)
    try:
        c.set_tensor(torch.from_numpy(x).cuda())
        c.set_factors([torch.from_numpy(h).cuda() for h in H])
        T = torch.full(ref.shape, float("nan"), device="cuda", dtype=torch.float32)
        c.partial_mttkrp(1, T)
        torch.cuda.synchronize()
    finally:
        c.close()
    segs = [min(seg, L - a) for a in range(0, L, seg)]
    bound = 2.0 ** -24 / 3 * math.sqrt(sum(n ** 3 for n in segs) / L ** 2 + len(segs) + 3)
    assert rel_fro(T.cpu().numpy(), ref) <= bound
