"""Timed cases: the calls that a user of this package makes, over the range of sizes it serves.

Every case goes through a public entry point: ``fit`` (the estimator, in its precisions and sketch
kinds), ``autograd.ols`` (training through the estimate), ``sketch``, ``grad`` and ``qr``.  Inputs
are drawn on the GPU from the seed; a program that calls an entry point repeatedly keeps its
workspace, so the larger cases do too.  ``exact`` gives the same results in 64 bits from plain torch.
"""
import math

import torch

import paper_2509_06856_gb300 as slse
from paper_2509_06856_gb300.autograd import ols

DTYPES = {"float32": torch.float32, "float64": torch.float64}
PAD = 16  # a ragged X can be a view into a wider row-major buffer


# ------------------------------------------------------------------------------------------ cases
def listed():
    return [
        # a small regression in double precision, called without a workspace: latency and launches
        # (the size of the `cfg1` workload)
        {"name": "fit_fp64_20000x50", "op": "fit", "N": 20000, "d": 50, "dtype": "float64", "prec": "fp64",
         "kind": "srht", "rows": "normal", "tol": 1e-12, "keep": False},
        # an ordinary single-precision table with an odd row count and an odd column count
        {"name": "fit_mixed_100003x37", "op": "fit", "N": 100003, "d": 37, "dtype": "float32", "prec": "mixed_bf16",
         "kind": "srht", "rows": "ar1", "tol": 1e-10, "keep": False},
        # the headline workload of the benchmark (`cfg3`): the largest problem, correlated columns
        {"name": "fit_mixed_4194304x512", "op": "fit", "N": 1 << 22, "d": 512, "dtype": "float32",
         "prec": "mixed_bf16", "kind": "srht", "rows": "ar1", "tol": 1e-10, "keep": True},
        # an ill-conditioned problem (cond 1e4) that wants double precision throughout (`cfg2`)
        {"name": "fit_fp64_1048576x256", "op": "fit", "N": 1 << 20, "d": 256, "dtype": "float64", "prec": "fp64",
         "kind": "srht", "rows": "cond1e4", "tol": 1e-13, "keep": True},
        # the CountSketch variant on a ragged number of rows
        {"name": "fit_countsketch_1500001x256", "op": "fit", "N": 1500001, "d": 256, "dtype": "float32",
         "prec": "mixed_bf16", "kind": "countsketch", "rows": "normal", "tol": 1e-10, "keep": True},
        # training through the estimate: forward fit and the gradients of X and Y (`cfg5`)
        {"name": "train_mixed_2097152x128", "op": "train", "N": 1 << 21, "d": 128, "dtype": "float32",
         "rows": "normal"},
        # one SRHT sketch of single-precision data, padded rows, stored in BF16
        {"name": "sketch_srht_bf16_3000000x384", "op": "sketch", "N": 3000000, "d": 384, "dtype": "float32",
         "prec": "mixed_bf16", "kind": "srht", "m": 1 << 18, "pad": False},
        # the same sketch in double precision, N just below a power of two
        {"name": "sketch_srht_fp64_1000000x200", "op": "sketch", "N": 1000000, "d": 200, "dtype": "float64",
         "prec": "fp64", "kind": "srht", "m": 1 << 16, "pad": False},
        # a Gaussian Hessian sketch (6 d rows) on the tensor cores
        {"name": "sketch_gauss_bf16_524288x512", "op": "sketch", "N": 1 << 19, "d": 512, "dtype": "float32",
         "prec": "mixed_bf16", "kind": "gaussian", "m": 3072, "pad": False},
        # one residual-gradient pass, single-precision data with compensated sums
        {"name": "grad_mixed_2097152x256", "op": "grad", "N": 1 << 21, "d": 256, "dtype": "float32",
         "prec": "mixed_bf16", "pad": False},
        # one residual-gradient pass in double precision on a view with a row stride
        {"name": "grad_fp64_700001x200", "op": "grad", "N": 700001, "d": 200, "dtype": "float64", "prec": "fp64",
         "pad": True},
        # the factor of a Hessian sketch of 6 d rows and its inverse
        {"name": "qr_3072x512", "op": "qr", "N": 3072, "d": 512, "dtype": "float64"},
    ]


def draw(rng):
    """One more case: an entry point, then sizes spread over the logarithm of its range."""
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    op = rng.choice(["fit_fp64", "fit_mixed", "fit_countsketch", "train", "sketch_bf16", "sketch_fp64",
                     "sketch_gauss", "grad_mixed", "grad_fp64", "qr"])
    d = size(10, 512)
    if rng.random() < 0.5:
        d = max(8, d // 8 * 8)
    # elements of the padded X: at most those of the listed case of the same kind
    most = {"fit_fp64": 28, "fit_mixed": 31, "fit_countsketch": 28, "train": 28, "sketch_bf16": 30, "sketch_fp64": 27,
            "sketch_gauss": 28, "grad_mixed": 29, "grad_fp64": 27, "qr": 21}[op]
    top = 1 << int(math.log2((1 << most) / d))
    if op == "qr":
        return {"op": "qr", "N": size(2 * d, 6 * d), "d": d, "dtype": "float64"}
    N = size(60 * d, min(top, 1 << 22))
    if rng.random() < 0.25:
        N = 1 << int(math.log2(N))
    if op.startswith("fit"):
        fp64 = op == "fit_fp64"
        return {"op": "fit", "N": max(N, 60 * d), "d": d, "dtype": "float64" if fp64 and rng.random() < 0.7 else "float32",
                "prec": "fp64" if fp64 else "mixed_bf16", "kind": "countsketch" if op == "fit_countsketch" else "srht",
                "rows": rng.choice(["normal", "ar1"]), "tol": 1e-12 if fp64 else 1e-10, "keep": rng.random() < 0.5}
    if op == "train":
        return {"op": "train", "N": max(N, 60 * d), "d": d, "dtype": "float32", "rows": rng.choice(["normal", "ar1"])}
    fp64 = op.endswith("fp64")
    case = {"op": "grad" if op.startswith("grad") else "sketch", "N": N, "d": d,
            "dtype": "float64" if fp64 and rng.random() < 0.7 else "float32",
            "prec": "fp64" if fp64 else "mixed_bf16", "pad": rng.random() < 0.3}
    if op.startswith("sketch"):
        case["kind"] = "gaussian" if op == "sketch_gauss" else "srht"
        case["m"] = 6 * d if op == "sketch_gauss" else size(2 * d, N // 2)
    return case


# ----------------------------------------------------------------------------------------- inputs
def _rows(rows, N, d, dtype, gen):
    """X (N x d): independent normals; AR(1) rows with correlation 0.5; or condition number 1e4."""
    if rows == "normal":
        return torch.randn(N, d, dtype=dtype, device="cuda", generator=gen)
    if rows == "ar1":
        i = torch.arange(d, dtype=torch.float64, device="cuda")
        L = torch.linalg.cholesky(0.5 ** (i[:, None] - i[None, :]).abs())
        return torch.randn(N, d, dtype=dtype, device="cuda", generator=gen) @ L.T.to(dtype)
    V, R = torch.linalg.qr(torch.randn(d, d, dtype=torch.float64, device="cuda", generator=gen))
    s = torch.logspace(0.0, -4.0, d, dtype=torch.float64, device="cuda")
    return torch.randn(N, d, dtype=dtype, device="cuda", generator=gen) @ (s[:, None] * (V * R.diagonal().sign()).T).to(dtype)


def _data(case, seed):
    """(X, Y, beta): Y = X beta + noise; X a view with a row stride where the case has "pad"."""
    gen = torch.Generator(device="cuda").manual_seed(int(seed))
    N, d, dtype = case["N"], case["d"], DTYPES[case["dtype"]]
    X = _rows(case.get("rows", "normal"), N, d, dtype, gen)
    if case.get("pad"):
        wide = torch.empty(N, d + PAD, dtype=dtype, device="cuda")
        wide[:, :d] = X
        X = wide[:, :d]
    beta = torch.randn(d, dtype=torch.float64, device="cuda", generator=gen)
    Y = X @ beta.to(dtype) + (0.01 if case.get("rows") == "cond1e4" else 0.1) * torch.randn(
        N, dtype=dtype, device="cuda", generator=gen)
    return X, Y, beta


def _direction(case, seed):
    """The loss gradient dL/d(beta-hat) of a training step."""
    gen = torch.Generator(device="cuda").manual_seed(int(seed) + (1 << 40))
    return torch.randn(case["d"], dtype=torch.float64, device="cuda", generator=gen)


def _iterate(case, seed, beta):
    """The iterate at which a gradient pass is taken: a tenth off the solution."""
    gen = torch.Generator(device="cuda").manual_seed(int(seed) + (1 << 41))
    return beta * (1.0 + 0.1 * torch.randn(case["d"], dtype=torch.float64, device="cuda", generator=gen))


def prepare(case, seed):
    s = dict(case, seed=int(seed) % (1 << 31))
    if case["op"] == "qr":
        gen = torch.Generator(device="cuda").manual_seed(int(seed))
        s["A"] = torch.randn(case["N"], case["d"], dtype=torch.float64, device="cuda", generator=gen)
        return s
    s["X"], s["Y"], beta = _data(case, seed)
    if case["op"] == "fit":
        s["schedule"] = slse.default_schedule(case["N"], case["d"], prec=case["prec"], tol=case["tol"], kind=case["kind"])
        s["workspace"] = slse.alloc_workspace(slse.workspace_size(s["X"], s["Y"], slse.OP_FIT, s["schedule"])) \
            if case["keep"] else None
    elif case["op"] == "train":
        s["v"] = _direction(case, seed)
        s["X"].requires_grad_(True)
        s["Y"].requires_grad_(True)
    elif case["op"] == "sketch":
        how = slse.Schedule(m=[], a=[], r=case["d"], mu=1.0, eta=0.0, prec=case["prec"], kind=slse.KIND[case["kind"]])
        s["workspace"] = slse.alloc_workspace(slse.workspace_size(s["X"], s["Y"], slse.OP_SKETCH, how, case["m"]))
    else:
        s["beta"] = _iterate(case, seed, beta)
        s["workspace"] = slse.alloc_workspace(slse.workspace_size(s["X"], s["Y"], slse.OP_GRAD))
    return s


# ------------------------------------------------------------------------------------------- runs
def run(s):
    if s["op"] == "fit":
        return {"beta": slse.fit(s["X"], s["Y"], s["schedule"], seed=s["seed"], workspace=s["workspace"]).beta}
    if s["op"] == "train":
        beta = ols(s["X"], s["Y"], seed=s["seed"])
        dX, dY = torch.autograd.grad(beta, (s["X"], s["Y"]), s["v"])
        return {"beta": beta.detach(), "dX": dX, "dY": dY}
    if s["op"] == "sketch":
        SX, SY = slse.sketch(s["X"], s["Y"], s["m"], seed=s["seed"], prec=s["prec"], kind=s["kind"],
                             workspace=s["workspace"], want_y=s["kind"] != "gaussian")
        return {"SX": SX} if SY is None else {"SX": SX, "SY": SY}
    if s["op"] == "grad":
        return {"g": slse.grad(s["X"], s["Y"], s["beta"], prec=s["prec"], workspace=s["workspace"])}
    R, H = slse.qr(s["A"])
    return {"R": R, "Hinv": H}


def work(case):
    """Each input read once, each output written once; the operations of the method's formulas."""
    N, d, e = case["N"], case["d"], 8 if case["dtype"] == "float64" else 4
    if case["op"] == "qr":
        return {"bytes": 8 * (N * d + 2 * d * d), "flops": 2 * N * d * d - 2 * d ** 3 / 3 + 4 * d ** 3 / 3}
    read = e * N * (d + 1)
    if case["op"] == "fit":  # one transform of [X | Y] and one exact pass
        adds = N * d * math.log2(N) if case["kind"] == "srht" else N * d
        return {"bytes": read + 8 * d, "flops": adds + 4 * N * d}
    if case["op"] == "train":
        return {"bytes": 2 * read + 8 * d, "flops": N * d * math.log2(N) + 4 * N * d + 8 * N * d}
    if case["op"] == "grad":
        return {"bytes": read + 16 * d, "flops": 4 * N * d}
    out = (8 if case["prec"] == "fp64" else 2) * case["m"] * (d + 1)
    if case["kind"] == "gaussian":
        return {"bytes": read + out, "flops": 2 * case["m"] * N * d}
    return {"bytes": read + out, "flops": N * d * math.log2(N)}


# ---------------------------------------------------------------------------- the same in 64 bits
def _blocks(N, d):
    step = max(1, (1 << 27) // d)
    return [(i, min(N, i + step)) for i in range(0, N, step)]


def _gradient(X, Y, beta):
    g = torch.zeros(X.shape[1], dtype=torch.float64, device="cuda")
    for lo, hi in _blocks(*X.shape):
        x = X[lo:hi].double()
        g += x.T @ (Y[lo:hi].double() - x @ beta)
    return g


def _least_squares(X, Y):
    """(beta, L): the least-squares solution and the Cholesky factor of X^T X, refined on the residual."""
    G = torch.zeros(X.shape[1], X.shape[1], dtype=torch.float64, device="cuda")
    for lo, hi in _blocks(*X.shape):
        x = X[lo:hi].double()
        G += x.T @ x
    L = torch.linalg.cholesky(G)
    beta = torch.zeros(X.shape[1], dtype=torch.float64, device="cuda")
    for _ in range(4):
        beta = beta + torch.cholesky_solve(_gradient(X, Y, beta)[:, None], L)[:, 0]
    return beta, L


def _philox(c0, c1, c2, c3, seed):
    """Philox4x32-10 on int64 tensors that hold 32-bit words."""
    mask = 0xFFFFFFFF

    def mul(a, x):
        return ((x * (a >> 16)) + ((x * (a & 0xFFFF)) >> 16)) >> 16, (x * a) & mask

    k0, k1 = seed & mask, (seed >> 32) & mask
    for _ in range(10):
        (h0, l0), (h1, l1) = mul(0xD2511F53, c0), mul(0xCD9E8D57, c2)
        c0, c1, c2, c3 = h1 ^ c1 ^ k0, l1, h0 ^ c3 ^ k1, l0
        k0, k1 = (k0 + 0x9E3779B9) & mask, (k1 + 0xBB67AE85) & mask
    return c0, c1, c2, c3


def _stream(n, stream, seed):
    i = torch.arange(n, dtype=torch.int64, device="cuda")
    return _philox(i & 0xFFFFFFFF, i >> 32, torch.full_like(i, stream), torch.zeros_like(i), seed)


def _permutation(n, stream, seed):
    w0, w1, _, _ = _stream(n, stream, seed)
    return torch.argsort(((w1 ^ 0x80000000) << 32) | w0, stable=True)  # unsigned order of (w1, w0)


def _srht(X, Y, m, seed):
    N, d = X.shape
    Np = 1 << max(0, int(N - 1).bit_length())
    D = 1.0 - 2.0 * (_stream(Np, 0, seed)[0] & 1).double()
    P, keep = _permutation(Np, 1, seed), _permutation(Np, 2, seed)[:m]
    live = P < N
    out = torch.empty(m, d + 1, dtype=torch.float64, device="cuda")
    step = max(1, (1 << 28) // Np)
    for c in range(0, d + 1, step):
        cols = [X[:, c:min(d, c + step)].double()] if c < d else []
        if c + step > d:
            cols.append(Y.double()[:, None])
        cols = torch.cat(cols, 1)
        z = torch.zeros(Np, cols.shape[1], dtype=torch.float64, device="cuda")
        z[live] = cols[P[live]]
        z *= D[:, None]
        h = 1
        while h < Np:
            v = z.view(Np // (2 * h), 2, h, -1)
            z = torch.stack((v[:, 0] + v[:, 1], v[:, 0] - v[:, 1]), 1).view(Np, -1)
            h *= 2
        out[:, c:c + cols.shape[1]] = z[keep] / math.sqrt(m)
    return {"SX": out[:, :d], "SY": out[:, d]}


def _gaussian(X, m, seed):
    N, d = X.shape
    out = torch.zeros(m, d, dtype=torch.float64, device="cuda")
    i = torch.arange(m, dtype=torch.int64, device="cuda")[:, None]
    step = max(8, (1 << 25) // m // 8 * 8)
    for lo in range(0, N, step):
        hi = min(N, lo + step)
        q = torch.arange(lo // 8, (hi + 7) // 8, dtype=torch.int64, device="cuda")[None, :].expand(m, -1)
        w = torch.stack(_philox(q & 0xFFFFFFFF, q >> 32, torch.full_like(q, 5), i.expand_as(q), seed), -1)
        rad = torch.sqrt(-2.0 * torch.log(((w & 0xFFFF).double() + 0.5) / 65536.0))
        ang = 2.0 * math.pi * ((w >> 16).double() + 0.5) / 65536.0
        G = torch.stack((rad * torch.cos(ang), rad * torch.sin(ang)), -1).reshape(m, -1)[:, :hi - lo]
        out += G @ X[lo:hi].double()
    return {"SX": out / math.sqrt(m)}


def exact(case, seed):
    if case["op"] == "qr":
        A = prepare(case, seed)["A"]
        R = torch.linalg.qr(A, mode="r").R
        R = R * torch.where(R.diagonal() < 0, -1.0, 1.0)[:, None].double()
        return {"R": R, "Hinv": torch.cholesky_inverse(R, upper=True)}
    X, Y, beta = _data(case, seed)
    if case["op"] == "fit":
        return {"beta": _least_squares(X, Y)[0]}
    if case["op"] == "train":
        beta, L = _least_squares(X, Y)
        v = _direction(case, seed)
        w = torch.cholesky_solve(v[:, None], L)[:, 0]
        for _ in range(3):  # refined: v - X^T X w is the gradient of a problem with Y = 0, plus v
            w = w + torch.cholesky_solve((v + _gradient(X, torch.zeros_like(Y), w))[:, None], L)[:, 0]
        dX, dY = torch.empty_like(X, dtype=torch.float64), torch.empty_like(Y, dtype=torch.float64)
        for lo, hi in _blocks(*X.shape):
            x = X[lo:hi].double()
            dY[lo:hi] = x @ w
            dX[lo:hi] = (Y[lo:hi].double() - x @ beta)[:, None] * w - dY[lo:hi, None] * beta
        return {"beta": beta, "dX": dX, "dY": dY}
    if case["op"] == "grad":
        return {"g": _gradient(X, Y, _iterate(case, seed, beta))}
    seed = int(seed) % (1 << 31)
    return _gaussian(X, case["m"], seed) if case["kind"] == "gaussian" else _srht(X, Y, case["m"], seed)
