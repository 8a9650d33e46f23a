"""||X||^2 where the squares leave float32's range within the few loads that are added
in float32 pairs, and the elements past the last 16-byte load, against float64.
Bound: four squares are added in float32 (4 x 2^-24), the rest in 48 bits or more."""
import math

import numpy as np
import pytest
import torch

import oracle
from _util import ensure_built
from paper_1806_07985_gb300 import nncp, synth

pytestmark = pytest.mark.gpu


def _alpha(x, dims):
    ensure_built()
    r = nncp.ParRank(dims, (1,) * len(dims), (0,) * len(dims), 2)
    try:
        return r.alpha_local(torch.from_numpy(x).cuda())
    finally:
        r.close()


# one load per thread, a few, and whole groups of eight; every remainder by four
@pytest.mark.parametrize("dims", [(3, 1, 1), (41, 17, 29), (101, 99, 131), (173, 173, 174), (177, 173, 175)])
@pytest.mark.parametrize("scale", [1.0, 6e18])
def test_alpha(dims, scale):
    x = (np.random.default_rng(7).random(math.prod(dims)) * 0.5 + 0.5).astype(np.float32) * np.float32(scale)
    ref = float(np.sum(x.astype(np.float64) ** 2))
    assert abs(_alpha(x, dims) - ref) <= 4 * 2.0 ** -24 * ref


def test_last_elements_in_float64():
    x = np.array([1 / 3, 2 / 7, 5 / 11], dtype=np.float32)
    ref = float(np.sum(x.astype(np.float64) ** 2))
    assert abs(_alpha(x, (3, 1, 1)) - ref) <= 4 * 2.0 ** -53 * ref


def _sparse(dims, runs):
    # one thread's loads large, of both signs: their squares' sum is 3.9e38, of which a
    # nonnegative model holds little
    x = np.zeros(math.prod(dims), dtype=np.float32)
    sign = 1.0
    for lo, n in runs:
        x[lo:lo + n] = 3.5e18 * sign * np.where(np.arange(n) % 2, -1.0, 1.0)
        sign = -sign
    return x


def test_solve_of_a_bf16_tensor():
    ensure_built()
    dims, R = (256, 160, 128), 2
    x = _sparse(dims, [(k * 8 * 4 * 152 * 256, 8) for k in range(4)])
    Xb = torch.from_numpy(x).to(torch.bfloat16).cuda()
    x = Xb.double().cpu().numpy()
    H0 = synth.init_factors(dims, R, seed=3)
    ref = oracle.nncp_hals(x, dims, [h.astype(np.float64) for h in H0], max_iters=2, use_dimtree=True, s=1)
    c = nncp.Context(dims, R, precision="bf16_stored", root_split=1)
    try:
        c.set_tensor(Xb)
        c.set_factors([torch.from_numpy(h.copy()).cuda() for h in H0])
        lam, k, fit = c.solve(2, 0.0)
    finally:
        c.close()
    assert k == 2 and abs(fit - ref["fits"][-1]) <= 1e-4


def test_solve_of_a_batch():
    ensure_built()
    dims, R = (64, 40, 24), 2
    x = _sparse(dims, [(1024 * q, 4) for q in range(8)])
    H0 = synth.init_factors(dims, R, seed=3)
    ref = oracle.nncp_hals(x.astype(np.float64), dims, [h.astype(np.float64) for h in H0], max_iters=2,
                           use_dimtree=True, s=1)
    b = nncp.Batch([dims], [R], max_iters=2)
    try:
        b.set_data([torch.from_numpy(x).cuda()], [[torch.from_numpy(h.copy()).cuda() for h in H0]])
        iters, fits, _ = b.solve(2, 0.0)
    finally:
        b.close()
    assert iters[0] == 2 and abs(fits[0] - ref["fits"][-1]) <= 1e-4
