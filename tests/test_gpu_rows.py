"""Mode updates past the one-cluster sizes (long modes, ranks above 64) and the solve's
initialisation, against the float64 oracle: one outer iteration, so that the
comparison is of the kernels' own arithmetic (float32 rows: 1e-4 leaves three
orders of magnitude over the 2^-24 rounding for the sweep's dependent columns)."""
import numpy as np
import pytest
import torch

import oracle
from _util import rel_fro
from paper_1806_07985_gb300 import nncp, synth

pytestmark = pytest.mark.gpu

# rows per block 64, blocks at most 304 (19,456 rows in one pass); four columns per lane and
# 16 (past rank 64: 64) per register chunk, so ranks at the edges of both
SHAPES = [((20001, 6, 5), 7, 0), ((19457, 5, 4), 16, 1), ((5, 17000, 4), 33, 0),
          ((65, 9, 8), 65, 0), ((64, 63, 3), 128, 0), ((3, 130, 7), 100, 2),
          ((1100, 4, 3), 81, 1), ((2, 2, 2, 2), 3, 0), ((2, 3), 90, 0),
          ((2048, 5, 3), 64, 0), ((2047, 5, 3), 64, 1), ((19460, 3, 2), 70, 0)]


@pytest.mark.parametrize("nls", ["hals", "bpp", "admm"])
@pytest.mark.parametrize("dims,R,split", SHAPES)
def test_one_iteration_matches_oracle(dims, R, split, nls):
    if nls != "hals" and (R > 32 or max(dims) > 19457):
        pytest.skip("the other updates take R <= 32; one long shape is enough")
    if nls == "bpp" and max(dims) > 10000:
        pytest.skip("the oracle solves row by row")
    x, _ = synth.lowrank_plus_noise(dims, min(R, 4), seed=31, noise=0.05)
    H0 = synth.init_factors(dims, R, seed=32)
    ref = oracle.nncp_hals(x.astype(np.float64), dims, [h.astype(np.float64) for h in H0],
                           max_iters=1, use_dimtree=True, s=split or None, nls=nls)
    c = nncp.Context(dims, R, root_split=split)
    try:
        c.set_nls(nls)
        H = [torch.from_numpy(h.copy()).cuda() for h in H0]
        c.set_tensor(torch.from_numpy(x).cuda())
        c.set_factors(H)
        lam, k, fit = c.solve(1, 0.0)
    finally:
        c.close()
    assert k == 1
    assert rel_fro(lam, ref["lam"]) <= 1e-4
    for n in range(len(dims)):
        assert rel_fro(H[n].cpu().numpy(), ref["H"][n]) <= 1e-4, n
    # eps^2 = (alpha - 2 beta + gamma) / alpha of float32 factors cancels to a few 2^-23 of
    # its terms, which moves eps by that over 2 eps
    eps = max(1.0 - ref["fits"][-1], 1e-6)
    assert abs(fit - ref["fits"][-1]) <= max(1e-5, 2.0 ** -21 / (2.0 * eps))
