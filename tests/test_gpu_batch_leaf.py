"""The batched leaf multi-TTV at the edges of its thread groups (slices of one read to
several blocks of outputs), ranks that are and are not multiples of four, and mode
digits carried over tiles of 64 rows, against the float64 oracle after one iteration
(float32 rows: 1e-4, as for single problems)."""
import numpy as np
import pytest
import torch

import oracle
from _util import ensure_built, rel_fro
from paper_1806_07985_gb300 import nncp, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ranks", [(4, 8, 16), (1, 3, 6), (5, 12, 64), (20, 33, 60)])
@pytest.mark.parametrize("shapes", [
    [(3, 1, 70), (4, 2, 63), (5, 7, 64), (2, 31, 65), (3, 32, 129), (2, 33, 40), (2, 64, 9), (3, 100, 5), (2, 256, 200)],
    [(3, 1, 9, 17), (2, 5, 63, 3), (2, 16, 64, 5), (3, 33, 65, 2), (2, 65, 1, 70), (2, 7, 130, 9)],
    [(2, 3, 4, 5, 6), (2, 17, 2, 33, 3), (3, 1, 66, 2, 3)]])
def test_leaf_shapes(shapes, ranks):
    ensure_built()
    probs = []
    for t, dims in enumerate(shapes):
        R = ranks[t % len(ranks)]
        x, _ = synth.lowrank_plus_noise(dims, min(R, 4), seed=400 + t, noise=0.05)
        probs.append((dims, R, x, synth.init_factors(dims, R, seed=450 + t)))
    b = nncp.Batch([p[0] for p in probs], [p[1] for p in probs], max_iters=1)
    try:
        X = [torch.from_numpy(p[2]).cuda() for p in probs]
        H = [[torch.from_numpy(h.copy()).cuda() for h in p[3]] for p in probs]
        b.set_data(X, H)
        b.solve(1, 0.0)
        got = [[h.cpu().numpy() for h in hs] for hs in H]
    finally:
        b.close()
    for (dims, R, x, H0), hs in zip(probs, got):
        exact = oracle.nncp_hals(x.astype(np.float64), dims, [h.astype(np.float64) for h in H0], max_iters=1,
                                 use_dimtree=True, s=1)
        for h, e in zip(hs, exact["H"]):
            assert rel_fro(h, e) <= 1e-4, (dims, R)
