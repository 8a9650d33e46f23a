"""Khatri-Rao rows whose first mode is long and no multiple of a stage (it wraps inside
one), at the lengths where that path starts, against float64 on the tensor as stored.
Bounds: an operand's rounding (bf16 pair 2^-17, TF32 2^-11) on both factors of a product
and a float32 accumulation that may truncate (2^-23) every eight elements of nonnegative
terms."""
import math

import numpy as np
import pytest
import torch

from _util import ensure_built, rel_fro
from paper_1806_07985_gb300 import nncp

pytestmark = pytest.mark.gpu


def _krp(fs, R):
    k = np.ones((1, R))
    for f in fs:
        k = (f[:, None, :] * k[None, :, :]).reshape(-1, R)
    return k


@pytest.mark.parametrize("prec,unit", [("split_bf16x3", 2.0 ** -17), ("tf32", 2.0 ** -11), ("bf16_stored", 2.0 ** -17)])
@pytest.mark.parametrize("dims,R,split", [
    ((200, 193, 5), 17, 1), ((136, 195), 33, 1), ((192, 191, 3), 16, 1), ((264, 257, 3), 40, 1), ((16, 300, 5, 7), 64, 1),
    ((296, 3, 4, 130), 24, 2), ((8, 1001, 11), 48, 1), ((520, 12, 255), 32, 2), ((1000, 8, 3), 40, 1)])
def test_long_ragged_first_modes(dims, R, split, prec, unit):
    ensure_built()
    rng = np.random.default_rng(sum(dims) + R)
    X = torch.from_numpy(rng.random(math.prod(dims)).astype(np.float32)).cuda()
    if prec == "bf16_stored":
        Xb = torch.empty(X.numel(), dtype=torch.bfloat16, device="cuda")
        nncp.nncp_tensor_to_bf16(X, Xb)
        X = Xb
    H = [rng.random((d, R)).astype(np.float32) for d in dims]
    Hd = [torch.from_numpy(h).cuda() for h in H]
    H64 = [h.astype(np.float64) for h in H]
    L = math.prod(dims[:split])
    X64 = X.double().cpu().numpy().reshape(-1, L)
    refs = [X64.T @ _krp(H64[split:], R), X64 @ _krp(H64[:split], R)]
    c = nncp.Context(dims, R, precision=prec, root_split=split)
    try:
        c.set_tensor(X)
        c.set_factors(Hd)
        for side, ref in enumerate(refs):
            T = torch.full(ref.shape, float("nan"), device="cuda", dtype=torch.float32)
            c.partial_mttkrp(side, T)
            torch.cuda.synchronize()
            K = X64.size // ref.shape[0]
            assert rel_fro(T.cpu().numpy(), ref) <= 2 * unit + math.ceil(K / 8) * 2.0 ** -23, side
    finally:
        c.close()
