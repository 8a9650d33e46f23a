"""contract_slow of a bf16 tensor, whose MN-major tiles go to the MMA as TMA stored
them: at the edges of the 64-output halves, of the 128-output tiles and of the
64-element stages, against float64 on the bf16 tensor.  Bound: the Khatri-Rao operand
is the sum of two bf16 numbers (2^-17 relative), and a K-element sum of nonnegative
terms takes ceil(K / 16) float32 accumulations that may truncate (2^-23 each)."""
import math

import numpy as np
import pytest
import torch

from _util import ensure_built, rel_fro
from paper_1806_07985_gb300 import nncp

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims,R", [
    ((8, 5), 3), ((56, 63), 16), ((64, 64), 17), ((72, 65), 33), ((120, 3, 21), 48), ((128, 64, 2), 64),
    ((136, 9, 15), 49), ((192, 31, 5), 32), ((264, 66, 3), 40), ((16, 200, 41), 24), ((4104, 7), 64)])
def test_edges(dims, R):
    ensure_built()
    rng = np.random.default_rng(sum(dims) + R)
    K = math.prod(dims[1:])
    X = torch.from_numpy(rng.random(math.prod(dims)).astype(np.float32)).cuda()
    Xb = torch.empty(X.numel(), dtype=torch.bfloat16, device="cuda")
    nncp.nncp_tensor_to_bf16(X, Xb)
    H = [rng.random((d, R)).astype(np.float32) for d in dims]
    krp = np.ones((1, R))
    for h in H[1:]:
        krp = (h.astype(np.float64)[:, None] * krp).reshape(-1, R)
    ref = Xb.double().cpu().numpy().reshape(K, dims[0]).T @ krp
    Hd = [torch.from_numpy(h).cuda() for h in H]
    c = nncp.Context(dims, R, precision="bf16_stored", root_split=1)
    try:
        c.set_tensor(Xb)
        c.set_factors(Hd)
        T = torch.full((dims[0], R), float("nan"), device="cuda")
        c.partial_mttkrp(0, T)
        torch.cuda.synchronize()
        assert rel_fro(T.cpu().numpy(), ref) <= 2.0 ** -17 + math.ceil(K / 16) * 2.0 ** -23
    finally:
        c.close()
