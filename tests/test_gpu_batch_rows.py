"""The root phases of a batch at the edges of their row blocks (four rows per thread,
row strides of every remainder by eight, one to 256 column groups) and rank groups:
one CTA per item gives the bits of the streamed kernels, whose threads take one row
each, and one iteration agrees with the float64 oracle."""
import numpy as np
import pytest
import torch

import oracle
from _util import ensure_built, rel_fro
from paper_1806_07985_gb300 import nncp, synth

pytestmark = pytest.mark.gpu
FIRST = (1, 2, 3, 4, 5, 6, 7, 8, 9, 13, 16, 17, 18, 24, 31, 32, 33, 36, 40, 63, 64, 65, 86, 100, 127, 128, 129,
         136, 255, 256)


def _solve(probs, iters, sched):
    b = nncp.Batch([p[0] for p in probs], [p[1] for p in probs], max_iters=iters)
    try:
        b.set_schedule(*sched)
        X = [torch.from_numpy(p[2]).cuda() for p in probs]
        H = [[torch.from_numpy(h.copy()).cuda() for h in p[3]] for p in probs]
        b.set_data(X, H)
        b.solve(iters, 0.0)
        return [[h.cpu().numpy() for h in hs] for hs in H]
    finally:
        b.close()


@pytest.mark.parametrize("ranks", [(1, 3, 4), (5, 8), (9, 13, 16), (17, 32), (33, 64), (2, 6, 64)])
@pytest.mark.parametrize("rest", [(37, 29), (150,), (5, 7, 11)])
def test_first_modes_and_ranks(rest, ranks):
    ensure_built()
    probs = []
    for t, i1 in enumerate(FIRST):
        dims, R = (i1, *rest), ranks[t % len(ranks)]
        x, _ = synth.lowrank_plus_noise(dims, min(R, 4), seed=900 + t, noise=0.05)
        probs.append((dims, R, x, synth.init_factors(dims, R, seed=950 + t)))
    got, ref = _solve(probs, 2, (0, 0)), _solve(probs, 2, (2, 2))
    for a, b in zip(got, ref):
        for x, y in zip(a, b):
            assert np.array_equal(x, y)
    one = _solve(probs, 1, (1, 1))
    for (dims, R, x, H0), H in zip(probs, one):
        exact = oracle.nncp_hals(x.astype(np.float64), dims, [h.astype(np.float64) for h in H0], max_iters=1,
                                 use_dimtree=True, s=1)
        for h, e in zip(H, exact["H"]):  # float32 rows, as for single problems
            assert rel_fro(h, e) <= 1e-4, (dims, R)
