"""The work whose speed is measured: what users of this library have it do.

Five kinds of call, each through the package's public entry points:

  direct    one MTTKRP of every mode of a dense tensor, ``nncp_mttkrp_noalloc`` (what a gradient of
            the CP objective needs, and the call for a host that must not allocate);
  sweep     one block-coordinate sweep's MTTKRPs through the dimension tree, the factor updates being
            the caller's own (``Context.mttkrp_cached`` / ``factor_changed``: the local step of the
            distributed solver, or a user's own constraint on the factors);
  partials  both root contractions of the dimension tree alone (``Context.partial_mttkrp``), the two
            calls that read the tensor in every outer iteration, per tensor-core precision;
  solve     a whole nonnegative CP decomposition, ``Context.solve``: initialisation, a stated number
            of outer iterations, factors, weights and fit (tol = 0, so every run does the same work);
  batch     many small independent decompositions at once, ``Batch.solve``.

Tensors are nonnegative low rank plus noise, factors U[0, 1), as in the tests and the benchmark; mode
1 is the fastest in memory.  A solve overwrites its factors, so a pass first copies the starting
factors in, as a program with a new start does.
"""

import math
import random

import numpy as np
import torch

from paper_1806_07985_gb300 import nncp

L2_BYTES = 126 << 20  # a tensor that stays in L2 between two passes needs only one read from memory


def _solve(name, dims, R, precision, iters, split=0, nls="hals"):
    return {"name": name, "kind": "solve", "dims": dims, "R": R, "precision": precision,
            "iters": iters, "split": split, "nls": nls}


def listed():
    return [
        # the smallest calls: launches and latency; the size of the first configuration (64^3, R = 8)
        {"name": "sweep_64_r8_fp32", "kind": "sweep", "dims": "64x64x64", "R": 8,
         "precision": "fp32_simt", "split": 0},
        _solve("solve_64_r8_fp32", "64x64x64", 8, "fp32_simt", 20),
        # a gradient of the CP objective of a ragged 4-way tensor
        {"name": "direct_130x77x65x12_r20", "kind": "direct", "dims": "130x77x65x12", "R": 20},
        # the two tensor passes of the headline configuration
        {"name": "partials_512_r32_split", "kind": "partials", "dims": "512x512x512", "R": 32,
         "precision": "split_bf16x3", "split": 1},
        # a tensor kept in bf16, ragged, at a rank above 32
        {"name": "partials_600x404x330_r40_bf16", "kind": "partials", "dims": "600x404x330", "R": 40,
         "precision": "bf16_stored", "split": 0},
        # the headline configuration as a whole call: the largest case
        _solve("solve_512_r32_split", "512x512x512", 32, "split_bf16x3", 6, split=1),
        # a time-lapse image cube (rows, columns, bands, times), split in the middle
        _solve("solve_512x512x32x16_r24_split", "512x512x32x16", 24, "split_bf16x3", 6, split=2),
        # the default precision on a ragged tensor of ordinary size
        _solve("solve_301x257x199_r20_fp32", "301x257x199", 20, "fp32_simt", 6),
        # a rank above 64, which only the default precision takes
        _solve("solve_220x180x150_r100_fp32", "220x180x150", 100, "fp32_simt", 4),
        # one long mode (samples) against two short ones (channels, conditions)
        _solve("solve_40000x48x40_r16_fp32", "40000x48x40", 16, "fp32_simt", 4),
        # the paper's own update, exact nonnegative least squares of every row
        _solve("solve_512x384x256_r24_bpp", "512x384x256", 24, "split_bf16x3", 4, nls="bpp"),
        # many small tensors together (lengths 16 to 128, ranks 4, 8 and 16)
        {"name": "batch_1024_3way", "kind": "batch", "count": 1024, "order": 3, "lo": 16, "hi": 128,
         "ranks": "4,8,16", "iters": 8, "shape_seed": 1},
    ]


def _dims(case):
    return tuple(int(v) for v in case["dims"].split("x"))


# ---- drawn cases ---------------------------------------------------------------------------------

def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _shape(rng, elems, order, longest=60000):
    """Mode lengths with about `elems` elements: cube-like, or with one long mode anywhere."""
    w = [rng.uniform(0.6, 1.4) for _ in range(order)]
    if rng.random() < 0.25:
        w[rng.randrange(order)] *= rng.uniform(1.5, 3.0)
    d = [max(2, min(longest, round(elems ** (v / sum(w))))) for v in w]
    while math.prod(d) > 1.1 * elems and max(d) > 2:
        k = d.index(max(d))
        d[k] = max(2, int(d[k] * elems / math.prod(d)))
    return d


def _tileable(dims, precision):
    """Mode 1 as the tensor-core precisions take it: rows of whole 16-byte units."""
    q = 8 if precision == "bf16_stored" else 4
    return [max(q, dims[0] // q * q)] + dims[1:]


def draw(rng):
    kind = rng.choice(["direct", "sweep", "partials", "solve", "solve", "solve", "batch"])
    if kind == "batch":
        return {"kind": "batch", "count": round(_log(rng, 16, 1500)), "order": rng.choice([3, 3, 4]),
                "lo": rng.choice([4, 16]), "hi": rng.choice([40, 64, 128]),
                "ranks": rng.choice(["4,8,16", "3,5,12", "8,16,32", "10,24,64"]),
                "iters": rng.randint(3, 8), "shape_seed": rng.randrange(1 << 20)}
    order = rng.choice([3, 3, 3, 4, 4, 5])
    if kind == "direct":
        R = round(_log(rng, 2, 100))
        d = _shape(rng, _log(rng, 1 << 14, min(1 << 25, (1 << 30) / R)), order, 4000)
        return {"kind": kind, "dims": "x".join(map(str, d)), "R": R}
    if kind == "partials":
        precision = rng.choice(["split_bf16x3", "split_bf16x3", "tf32", "bf16_stored"])
        R = round(_log(rng, 4, 64))
        d = _tileable(_shape(rng, _log(rng, 1 << 20, 1 << 27), order, 20000), precision)
        return {"kind": kind, "dims": "x".join(map(str, d)), "R": R, "precision": precision,
                "split": rng.randint(0, order - 1)}
    precision = rng.choice(["fp32_simt", "fp32_simt", "split_bf16x3", "bf16_stored"])
    iters = rng.randint(2, 6)
    R = round(_log(rng, 2, 128 if precision == "fp32_simt" else 64))
    # no dearer than the largest listed case; float32 runs on the CUDA cores
    most = (1 << 27) * 32 * 6 / (max(R, 16) * (iters if kind == "solve" else 1))
    if precision == "fp32_simt":
        most /= 6
    d = _shape(rng, _log(rng, 1 << 15, min(1 << 27, most)), order)
    if precision != "fp32_simt":
        d = _tileable(d, precision)
    case = {"kind": kind, "dims": "x".join(map(str, d)), "R": R, "precision": precision,
            "split": rng.choice([0, 0, rng.randint(1, order - 1)])}
    if kind == "solve":
        case["iters"] = iters
        case["nls"] = rng.choice(["hals", "hals", "bpp", "admm"]) if R <= 32 else "hals"
        if case["nls"] != "hals" and max(d) > 4000:
            case["nls"] = "hals"
    return case


# ---- inputs --------------------------------------------------------------------------------------

def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) * 7919 + 11)
    return g


def _krp(factors):
    """Rows of the Khatri-Rao product, the first factor's index fastest."""
    k = factors[0]
    for f in factors[1:]:
        k = (f[:, None, :] * k[None, :, :]).reshape(-1, f.shape[1])
    return k


def _tensor(dims, rank, g):
    """Nonnegative low rank plus noise, flat, mode 1 fastest."""
    f = [torch.rand(d, rank, generator=g, device="cuda") for d in dims]
    x = _krp(f[1:]) @ f[0].T
    x.add_(torch.rand(x.shape, generator=g, device="cuda"), alpha=0.01)
    return x.reshape(-1)


class _Factors:
    """Starting factors and the factors a call updates, in two flat buffers of the same layout."""

    def __init__(self, shapes, g):
        off, place = 0, []
        for rows, R in shapes:
            place.append((off, rows, R))
            off += -(-rows * R // 64) * 64
        self.start = torch.rand(off, generator=g, device="cuda")
        self.live = self.start.clone()
        self.views = [self.live[o:o + n * R].view(n, R) for o, n, R in place]
        self.first = [self.start[o:o + n * R].view(n, R) for o, n, R in place]

    def restart(self):
        self.live.copy_(self.start)


def _batch_shapes(case):
    r = random.Random(case["shape_seed"])
    ranks = [int(v) for v in case["ranks"].split(",")]
    shapes, total = [], 0
    for _ in range(case["count"]):
        while True:
            d = tuple(round(_log(r, case["lo"], case["hi"])) for _ in range(case["order"]))
            if math.prod(d) <= 4 << 20:
                break
        R = r.choice(ranks)
        total += math.prod(d)
        if shapes and total > 180e6:
            break
        shapes.append((d, R))
    return shapes


def prepare(case, seed):
    g = _gen(seed)
    kind = case["kind"]
    s = {"case": dict(case), "kind": kind}
    if kind == "batch":
        shapes = _batch_shapes(case)
        s["X"] = [_tensor(d, R, g) for d, R in shapes]
        s["F"] = _Factors([(n, R) for d, R in shapes for n in d], g)
        N = case["order"]
        torch.cuda.synchronize()
        s["batch"] = nncp.Batch([d for d, _ in shapes], [R for _, R in shapes], case["iters"])
        v = s["F"].views
        s["batch"].set_data(s["X"], [v[t * N:(t + 1) * N] for t in range(len(shapes))])
        s["shapes"] = shapes
        return s
    dims, R = _dims(case), case["R"]
    X = _tensor(dims, min(R, 64), g)
    F = _Factors([(n, R) for n in dims], g)
    s.update(dims=dims, X=X, F=F)
    if kind == "direct":
        s["out"] = [torch.empty(n, R, device="cuda") for n in dims]
        return s
    if case["precision"] == "bf16_stored":
        s["X"] = torch.empty(X.numel(), dtype=torch.bfloat16, device="cuda")
        nncp.nncp_tensor_to_bf16(X, s["X"])
        del X
    # a plan prepares its workspace on a stream of its own: it is made once the inputs are
    torch.cuda.synchronize()
    ctx = nncp.Context(dims, R, precision=case["precision"], root_split=case["split"])
    ctx.set_tensor(s["X"])
    ctx.set_factors(F.views)
    s["ctx"] = ctx
    if kind == "solve":
        ctx.set_nls(case["nls"])
    elif kind == "sweep":
        s["out"] = [torch.empty(n, R, device="cuda") for n in dims]
    else:
        k = _split(case)
        s["out"] = [torch.empty(math.prod(dims[:k]), R, device="cuda"),
                    torch.empty(math.prod(dims[k:]), R, device="cuda")]
    torch.cuda.synchronize()
    return s


def _split(case):
    return case["split"] or nncp.nncp_default_split(_dims(case))


def run(s):
    kind = s["kind"]
    if kind == "direct":
        for n in range(len(s["dims"])):
            nncp.nncp_mttkrp_noalloc(s["dims"], s["case"]["R"], s["X"], s["F"].views, n + 1, s["out"][n])
        return s["out"]
    if kind == "sweep":
        ctx = s["ctx"]
        for n in range(len(s["dims"])):
            ctx.mttkrp_cached(n + 1, s["out"][n])
            ctx.factor_changed(n + 1)
        return s["out"]
    if kind == "partials":
        return [s["ctx"].partial_mttkrp(side, s["out"][side]) for side in (0, 1)]
    s["F"].restart()
    if kind == "solve":
        lam, iters, fit = s["ctx"].solve(s["case"]["iters"], 0.0)
        return {"H": s["F"].views, "lambda": np.array(lam), "iters": iters, "fit": fit}
    iters, fits, lams = s["batch"].solve(s["case"]["iters"], 0.0)
    return {"H": s["F"].live, "lambda": np.concatenate([np.array(v) for v in lams]),
            "iters": np.array(iters), "fit": np.array(fits)}


# ---- what a pass cannot do without ---------------------------------------------------------------

def work(case):
    """Tensor reads: one per call or, for an outer iteration (and a sweep), the two passes of the
    dimension tree, but only one in all where the tensor stays in L2.  Operations: 2 per tensor
    element and rank column of every contraction of the tensor."""
    kind = case["kind"]
    if kind == "batch":
        shapes = _batch_shapes(case)
        tb = 4 * sum(math.prod(d) for d, _ in shapes)
        fb = 4 * sum(sum(d) * R for d, R in shapes)
        fl = sum(4 * math.prod(d) * R for d, R in shapes) * case["iters"]
        return {"bytes": tb * (2 * case["iters"] if tb > L2_BYTES else 1) + 2 * fb, "flops": fl}
    dims, R = _dims(case), case["R"]
    el = math.prod(dims)
    tb = el * (2 if case.get("precision") == "bf16_stored" else 4)
    fb = 4 * sum(dims) * R
    if kind == "direct":
        passes = len(dims)
        outs, fl = fb, 2 * el * R * len(dims)
    elif kind == "sweep":
        passes, outs, fl = 2, fb, 4 * el * R
    elif kind == "partials":
        k = _split(case)
        passes, fl = 2, 4 * el * R
        outs = 4 * R * (math.prod(dims[:k]) + math.prod(dims[k:]))
    else:
        passes, outs, fl = 2 * case["iters"], fb, 4 * el * R * case["iters"]
    return {"bytes": tb * (passes if tb > L2_BYTES else 1) + fb + outs, "flops": fl}


# ---- results in 64 bits --------------------------------------------------------------------------

def _mttkrp(X, dims, H, n):
    L, Q = math.prod(dims[:n]), math.prod(dims[n + 1:])
    if L == 1:
        return X.view(Q, dims[n]).T @ _krp(H[n + 1:])
    T = (X.view(Q * dims[n], L) @ _krp(H[:n])).view(Q, dims[n], -1)
    if Q == 1:
        return T[0]
    return (T * _krp(H[n + 1:])[:, None, :]).sum(0)


def _nnls_rows(S, M):
    """min_{x >= 0} x S x / 2 - m x for every row m of M, by block principal pivoting."""
    n, R = M.shape
    F = torch.zeros(n, R, dtype=torch.bool, device=M.device)
    x, y = torch.zeros_like(M), -M
    best = torch.full((n,), R + 1, device=M.device)
    spare = torch.full((n,), 3, device=M.device)
    eye = torch.eye(R, dtype=M.dtype, device=M.device)
    for _ in range(50 * R + 50):
        bad = torch.where(F, x < 0, y < 0)
        count = bad.sum(1)
        if int(count.max()) == 0:
            break
        better = count < best
        full = better | (spare > 0)
        spare = torch.where(better, 3, torch.where(count > 0, spare - 1, spare)).clamp(min=0)
        best = torch.where(better, count, best)
        last = R - 1 - bad.flip(1).to(torch.int8).argmax(1)
        one = torch.zeros_like(bad).scatter_(1, last[:, None], True) & bad
        F = F ^ torch.where(full[:, None], bad, one)
        f = F.to(M.dtype)
        A = S * f[:, :, None] * f[:, None, :] + eye * (1 - f)[:, None, :]
        x = torch.linalg.solve(A, M * f) * f
        y = torch.where(F, torch.zeros_like(M), x @ S - M)
    return x


def _decompose(X, dims, H, iters, nls):
    """`iters` outer iterations in 64 bits: H normalised, weights, and the last fit."""
    N, R = len(dims), H[0].shape[1]
    lam = torch.ones(R, dtype=torch.float64, device="cuda")
    H = [h.clone() for h in H]
    for n in range(N):
        c = H[n].norm(dim=0)
        H[n] = H[n] / c
        lam = lam * c
    G = [h.T @ h for h in H]
    U = [torch.zeros_like(h) for h in H]
    alpha, fit = X.square().sum(), None
    for _ in range(iters):
        for n in range(N):
            M = _mttkrp(X, dims, H, n)
            S = torch.ones(R, R, dtype=torch.float64, device="cuda")
            for k in range(N):
                if k != n:
                    S = S * G[k]
            W = H[n] * lam
            if nls == "bpp":
                W = _nnls_rows(S, M)
            elif nls == "admm":
                rho = S.trace() / R
                A = S + rho * torch.eye(R, dtype=torch.float64, device="cuda")
                u = U[n] * lam
                for _k in range(5):  # the library's default number of inner steps
                    x = torch.linalg.solve(A, (M + rho * (W - u)).T).T
                    W = (x + u).clamp(min=0)
                    u = u + x - W
            else:
                for r in range(R):
                    # a column with S_rr = 0 (another factor's column is zero) stays as it is
                    step = torch.where(S[r, r] > 0, (M[:, r] - W @ S[:, r]) / S[r, r], 0.0)
                    W[:, r] = (W[:, r] + step).clamp(min=0)
            lam = W.norm(dim=0)
            inv = torch.where(lam > 0, 1 / lam, torch.zeros_like(lam))
            H[n] = W * inv
            if nls == "admm":
                U[n] = u * inv
            G[n] = H[n].T @ H[n]
        gamma = (lam[:, None] * S * G[N - 1] * lam[None, :]).sum()
        fit = 1 - ((alpha - 2 * (M * W).sum() + gamma).clamp(min=0) / alpha).sqrt()
    return H, lam, fit


def exact(case, seed):
    if case["kind"] == "batch":
        # the first tensors of the batch would do, but the outputs are whole: small batches only
        if case["count"] * case["iters"] > 300:
            return None
    s = prepare(case, seed)
    if case["kind"] == "batch":
        N, H, lams, fits = case["order"], torch.zeros_like(s["F"].start, dtype=torch.float64), [], []
        H.copy_(s["F"].start)
        off = 0
        for t, (d, R) in enumerate(s["shapes"]):
            h, lam, fit = _decompose(s["X"][t].double(), d,
                                     [f.double() for f in s["F"].first[t * N:(t + 1) * N]],
                                     case["iters"], "hals")
            for f in h:
                H[off:off + f.numel()] = f.reshape(-1)
                off += -(-f.numel() // 64) * 64
            lams.append(lam)
            fits.append(float(fit))
        return {"H": H, "lambda": torch.cat(lams), "iters": None, "fit": np.array(fits)}
    X, dims = s["X"].double(), s["dims"]
    H = [f.double() for f in s["F"].first]
    if case["kind"] in ("direct", "sweep"):
        return [_mttkrp(X, dims, H, n) for n in range(len(dims))]
    if case["kind"] == "partials":
        k = _split(case)
        IL, IR = math.prod(dims[:k]), math.prod(dims[k:])
        return [X.view(IR, IL).T @ _krp(H[k:]), X.view(IR, IL) @ _krp(H[:k])]
    H, lam, fit = _decompose(X, dims, H, case["iters"], case["nls"])
    return {"H": H, "lambda": lam, "iters": None, "fit": float(fit)}


def tolerance(case):
    """About four times the largest error against 64 bits seen over the listed and 150 drawn cases."""
    kind, precision = case["kind"], case.get("precision", "fp32_simt")
    if kind in ("direct", "sweep", "partials"):
        # the MTTKRP itself: float32 sums; bf16 hi + lo pairs; TF32 operands; a bf16 tensor against
        # hi + lo pairs with one long tensor-core accumulation
        return {"rel": {"fp32_simt": 1.2e-6, "split_bf16x3": 8e-6, "tf32": 3e-3, "bf16_stored": 6e-5}[precision]}
    if kind == "batch":
        return {"rel": 2e-5}
    # a few outer iterations on float32 factors carry the MTTKRP's error on; the exact updates
    # switch rows' supports
    if case["nls"] != "hals":
        return {"rel": 4e-4}
    return {"rel": 8e-5 if precision == "fp32_simt" else 1.2e-4}
