"""What the performance of this package is measured on: calls of its public entry points over the
sizes, storage types and options its users run, each with inputs drawn from a seed, the work the
call cannot do without, and the 64-bit result it approximates.

A case names a `kind` (which entry points run) and their sizes and options:
    solve   sketch, factor and iterate to `tol` (lsq_sketch, lsq_factor, lsq_solve): x
    refresh lsq_solve with a fresh embedding every iteration: x
    sketch  lsq_sketch alone: SA
    factor  lsq_factor alone: R and W = R^{-1}
    pass    lsq_hmatvec, one fused pass over A (the step of the row-partitioned solver): A^T A p, p^T A^T A p
    grad    lstsq_solve and its backward: x, dL/dA, dL/db
    batch   lsq_solve_batched over uneven problems: every X

Data as in the package's workloads: A = G diag(sigma), G iid N(0, 1), sigma log-spaced from 1 to
SIGMA_MAX, optionally 5% of the rows x100, b = A^T (A x_true + 0.1 noise).  Tolerances lie above what
the arithmetic reaches: 1e-12 in FP64, 1e-11 in the mixed precision (whose exact residuals carry
about 45 bits), so that a solution is well defined to many digits.
"""
import math

import torch

import paper_1911_02675_gb300 as L

SIGMA_MAX = 1e4
NOISE = 0.1
MASK32 = 0xFFFFFFFF
L2_BYTES = 120e6  # a matrix smaller than this is read from memory once however often it is used


def listed():
    return [
        # the small dense problem: a fit of a few thousand samples, everything in FP64; latency counts
        dict(name="solve_f64_4096x64", kind="solve", n=4096, d=64, dtype="f64", sketch="gauss", m=256, s=8,
             sketch_precision="f64", method="pcg", precision="f64", tol=1e-12, outliers=False),
        # the same size with refreshed embeddings: a sketch, a factor and one step per iteration
        dict(name="refresh_polyak_4096x64", kind="refresh", n=4096, d=64, sketch="gauss", m=512, s=8,
             method="polyak", tol=1e-10),
        # plain FP64 at an odd size: rows and columns off every tile, a sparse embedding
        dict(name="solve_f64_300007x301", kind="solve", n=300007, d=301, dtype="f64", sketch="sjlt", m=1204, s=8,
             sketch_precision="f64", method="pcg", precision="f64", tol=1e-12, outliers=False),
        # the mixed-precision pipeline on a tall FP64 matrix (SRHT that also writes the FP32 copy)
        dict(name="solve_mixed_1048576x512", kind="solve", n=1 << 20, d=512, dtype="f64", sketch="srht", m=4096, s=8,
             sketch_precision="f32", method="pcg", precision="mixed", tol=1e-11, outliers=False),
        # the largest one: FP32 storage with high-leverage rows, the Gaussian embedding on the tensor cores
        dict(name="solve_mixed_4194304x1024_f32", kind="solve", n=1 << 22, d=1024, dtype="f32", sketch="gauss",
             m=4096, s=8, sketch_precision="bf16", method="pcg", precision="mixed", tol=1e-11, outliers=True),
        # embeddings of the tall FP64 matrix on their own, one of each kind
        dict(name="sketch_gauss_bf16_1048576x512", kind="sketch", n=1 << 20, d=512, dtype="f64", sketch="gauss",
             m=2048, s=8, sketch_precision="bf16"),
        dict(name="sketch_sjlt_f32_1048576x512", kind="sketch", n=1 << 20, d=512, dtype="f64", sketch="sjlt",
             m=2048, s=8, sketch_precision="f32"),
        dict(name="sketch_srht_f64_1048576x512", kind="sketch", n=1 << 20, d=512, dtype="f64", sketch="srht",
             m=1024, s=8, sketch_precision="f64"),
        # the preconditioner of the widest problems
        dict(name="factor_mixed_4096x1024", kind="factor", m=4096, d=1024, precision="mixed"),
        # one pass over a slab of rows, as each rank of a row-partitioned solve makes it
        dict(name="pass_f64_600011x333", kind="pass", n=600011, d=333, dtype="f64"),
        # a differentiable layer: forward solve, backward solve, dense gradient of A
        dict(name="grad_f32_262144x256", kind="grad", n=1 << 18, d=256, dtype="f32", m=1024, tol=1e-11),
        # many uneven problems with several right-hand sides each, one call
        dict(name="batch_256_f32", kind="batch", nprob=256, n_lo=1 << 12, n_hi=1 << 18, d_lo=32, d_hi=512, k_hi=16,
             dtype="f32", sketch_precision="bf16", tol=1e-11, shapes=10),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the same ranges: sizes log-uniform (odd ones among them, powers of two now
    and then), n well above d, embeddings of 2 d to 16 d rows."""
    kind = rng.choice(["solve", "solve", "solve", "sketch", "sketch", "sketch", "factor", "pass", "grad", "batch",
                       "batch", "refresh"])

    def width(lo, hi):
        d = _log(rng, lo, hi)
        return min(hi, 1 << (d.bit_length() - 1)) if rng.random() < 0.3 else d

    def rows(d, lo, hi, elems):
        n = _log(rng, max(lo, 8 * d), max(8 * d + 1, min(hi, elems // d)))
        return 1 << (n.bit_length() - 1) if rng.random() < 0.3 and (1 << (n.bit_length() - 1)) >= 8 * d else n

    if kind == "solve":
        if rng.random() < 0.4:  # FP64 throughout: the cost of its arithmetic keeps these smaller
            d = width(16, 400)
            n = rows(d, 1024, 1 << 19, 1 << 27)
            sketch = rng.choice(["gauss", "srht", "sjlt"]) if n * d < (1 << 20) else rng.choice(["srht", "sjlt"])
            return dict(kind=kind, n=n, d=d, dtype=rng.choice(["f64", "f64", "f32"]), sketch=sketch,
                        m=int(d * rng.uniform(3, 8)), s=8, sketch_precision="f64",
                        method=rng.choice(["pcg", "pcg", "polyak"]), precision="f64", tol=1e-12, outliers=False)
        d = width(32, 1024)
        n = rows(d, 1 << 14, 1 << 22, 1 << 30)
        sketch, prec = rng.choice([("srht", "f32"), ("sjlt", "f32"), ("gauss", "bf16"), ("sjlt", "bf16")])
        return dict(kind=kind, n=n, d=d, dtype=rng.choice(["f64", "f32"]), sketch=sketch,
                    m=min(8192, n, max(d + 8, int(d * rng.uniform(3, 8)))), s=8, sketch_precision=prec, method="pcg",
                    precision="mixed", tol=1e-11, outliers=rng.random() < 0.3)
    if kind == "refresh":
        d = width(8, 96)
        return dict(kind=kind, n=rows(d, 1024, 1 << 14, 1 << 20), d=d, sketch=rng.choice(["gauss", "srht"]),
                    m=int(d * rng.uniform(6, 12)), s=8, method=rng.choice(["ihs", "polyak"]), tol=1e-10)
    if kind == "sketch":
        d = width(32, 1024)
        sketch, prec = rng.choice([("gauss", "bf16"), ("gauss", "bf16"), ("sjlt", "f32"), ("sjlt", "f32"),
                                   ("sjlt", "bf16"), ("srht", "f32"), ("srht", "f64"), ("sjlt", "f64")])
        n = rows(d, 1 << 13, 1 << 21, 1 << 29)
        return dict(kind=kind, n=n, d=d, dtype=rng.choice(["f64", "f32"]), sketch=sketch,
                    m=min(4096, n, int(d * rng.uniform(2, 8))), s=rng.choice([4, 8, 8, 16]), sketch_precision=prec)
    if kind == "factor":
        d = width(16, 1024)
        return dict(kind=kind, m=min(8192, int(d * rng.uniform(2, 8))), d=d, precision=rng.choice(["f64", "mixed"]))
    if kind == "pass":
        d = width(16, 1024)
        return dict(kind=kind, n=rows(d, 1 << 12, 1 << 21, 1 << 28), d=d, dtype=rng.choice(["f64", "f32"]))
    if kind == "grad":
        d = width(32, 512)
        return dict(kind=kind, n=rows(d, 1 << 13, 1 << 19, 1 << 27), d=d, dtype=rng.choice(["f32", "f32", "f64"]),
                    m=int(d * rng.uniform(3, 8)), tol=1e-11)
    nprob = _log(rng, 16, 160)
    d_hi = rng.choice([64, 128, 256, 512])
    dtype = rng.choice(["f32", "f32", "f32", "f64"])
    return dict(kind=kind, nprob=nprob, n_lo=1 << 12, n_hi=1 << (rng.choice([14, 16, 18]) if dtype == "f32" else 14),
                d_lo=min(32, d_hi // 4), d_hi=d_hi, k_hi=rng.choice([1, 4, 16, 16]), dtype=dtype,
                sketch_precision=rng.choice(["f32", "bf16"]), tol=1e-11, shapes=rng.randrange(1 << 20))


# ---------------------------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------------------------
def _dtype(case):
    return torch.float64 if case.get("dtype", "f64") == "f64" else torch.float32


def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _sigma(d, dtype=torch.float64):
    if d == 1:
        return torch.ones(1, dtype=dtype, device="cuda")
    return (SIGMA_MAX ** (torch.arange(d, dtype=torch.float64, device="cuda") / (d - 1))).to(dtype)


def _matrix(n, d, dtype, g, outliers=False):
    A = torch.empty((n, d), dtype=dtype, device="cuda")
    sig = _sigma(d, dtype)
    step = max(1, (1 << 27) // d)
    for r in range(0, n, step):
        blk = A[r:r + step]
        torch.randn(blk.shape, generator=g, dtype=dtype, device="cuda", out=blk)
        blk *= sig
    if outliers:
        A[torch.rand(n, generator=g, device="cuda") < 0.05] *= 100
    return A


def _rhs(A, k, g):
    """k right-hand sides b = A^T (A x_true + noise), FP64, as rows."""
    n, d = A.shape
    xt = torch.randn((d, k), generator=g, dtype=torch.float64, device="cuda")
    b = torch.zeros((d, k), dtype=torch.float64, device="cuda")
    step = max(1, (1 << 27) // d)
    for r in range(0, n, step):
        blk = A[r:r + step].double()
        y = blk @ xt + NOISE * torch.randn((blk.shape[0], k), generator=g, dtype=torch.float64, device="cuda")
        b += blk.T @ y
    return b.T.contiguous()


def _batch_shapes(case):
    """(n, d, k) of every problem: n and d log-uniform in their ranges, k uniform; a property of the
    case, not of the seed (a program solves batches of the same shapes again and again)."""
    g = torch.Generator()
    g.manual_seed(case["shapes"])
    u = torch.rand((case["nprob"], 3), generator=g, dtype=torch.float64).tolist()
    out = []
    for a, b, c in u:
        n = math.exp(math.log(case["n_lo"]) + a * math.log(case["n_hi"] / case["n_lo"]))
        d = math.exp(math.log(case["d_lo"]) + b * math.log(case["d_hi"] / case["d_lo"]))
        out.append((int(n), int(d), 1 + int(c * case["k_hi"])))
    return out


def prepare(case, seed):
    """The inputs of one case on the GPU, with the context and the buffers a program keeps."""
    g = _gen(seed)
    kind = case["kind"]
    st = dict(case=case, ctx=L.Context(), seed=int(seed))
    if kind in ("solve", "refresh", "grad"):
        n, d, m = case["n"], case["d"], case["m"]
        st["A"] = _matrix(n, d, _dtype(case), g, case.get("outliers", False))
        st["b"] = _rhs(st["A"], 1, g).reshape(-1)
        if kind == "solve":
            st["SA"] = torch.empty((m, d), dtype=torch.float64, device="cuda")
            st["R"] = torch.empty((d, d), dtype=torch.float64, device="cuda")
            st["W"] = torch.empty((d, d), dtype=torch.float64, device="cuda")
            st["a32"] = None
            if case["precision"] == "mixed" and case["dtype"] == "f64":
                st["a32"] = L.narrow_buffer(st["A"])
            st["ctx"].set_deferred_checks(True)
        if kind == "grad":
            st["A"].requires_grad_(True)
            st["b"].requires_grad_(True)
            st["g"] = torch.randn(d, generator=g, dtype=torch.float64, device="cuda")
    elif kind == "sketch":
        st["A"] = _matrix(case["n"], case["d"], _dtype(case), g)
        st["SA"] = torch.empty((case["m"], case["d"]), dtype=torch.float64, device="cuda")
    elif kind == "factor":
        st["SA"] = _matrix(case["m"], case["d"], torch.float64, g)
    elif kind == "pass":
        st["A"] = _matrix(case["n"], case["d"], _dtype(case), g)
        st["p"] = torch.randn(case["d"], generator=g, dtype=torch.float64, device="cuda") / _sigma(case["d"])
    else:
        st["problems"] = []
        for n, d, k in _batch_shapes(case):
            A = _matrix(n, d, _dtype(case), g)
            st["problems"].append((A, _rhs(A, k, g)))
    return st


def run(st):
    """One pass through the entry points, as a program calls them."""
    case, ctx, kind = st["case"], st["ctx"], st["case"]["kind"]
    if kind == "solve":
        SA = L.lsq_sketch(ctx, st["A"], case["sketch"], case["m"], st["seed"], s=case["s"],
                          precision=case["sketch_precision"], out=st["SA"], a32=st["a32"])
        _, W = L.lsq_factor(ctx, SA, R=st["R"], W=st["W"], precision=case["precision"])
        x, _ = L.lsq_solve(ctx, st["A"], st["b"], case["method"], W, tol=case["tol"], maxit=1000, raise_on_maxit=True,
                           m=case["m"], precision=case["precision"], a32=st["a32"])
        return x
    if kind == "refresh":
        x, _ = L.lsq_solve(ctx, st["A"], st["b"], case["method"], None, tol=case["tol"], maxit=1000,
                           raise_on_maxit=True, refresh=1, sketch_type=case["sketch"], m=case["m"], seed=st["seed"])
        return x
    if kind == "sketch":
        return L.lsq_sketch(ctx, st["A"], case["sketch"], case["m"], st["seed"], s=case["s"],
                            precision=case["sketch_precision"], out=st["SA"])
    if kind == "factor":
        R, W = L.lsq_factor(ctx, st["SA"], precision=case["precision"])
        return {"R": R, "W": W}
    if kind == "pass":
        v, q = L.lsq_hmatvec(ctx, st["A"], st["p"])
        return {"v": v, "q": q}
    if kind == "grad":
        x = L.lstsq_solve(st["A"], st["b"], ctx, m=case["m"], seed=st["seed"], tol=case["tol"])
        gA, gb = torch.autograd.grad(x, (st["A"], st["b"]), st["g"])
        return {"x": x.detach(), "gA": gA, "gb": gb}
    X, _, _ = L.lsq_solve_batched(ctx, st["problems"], tol=case["tol"], maxit=1000, seed=st["seed"],
                                  sketch_precision=case["sketch_precision"],
                                  precision="mixed" if case["dtype"] == "f32" else "f64")
    return torch.cat([x.reshape(-1) for x in X])


# ---------------------------------------------------------------------------------------------
# the work a pass cannot do without
# ---------------------------------------------------------------------------------------------
def _iterations(d, m, tol):
    """Iterations of PCG to a relative error of tol: 2 sqrt(rho)^T <= tol with rho = d / m."""
    return max(1, math.ceil(math.log(2 / tol) / (0.5 * math.log(max(m / d, 1.01)))))


def _sketch_flops(kind, n, d, m, s):
    if kind == "gauss":
        return 2.0 * m * n * d
    return 2.0 * n * d * s if kind == "sjlt" else n * d * math.log2(max(2, n))


def _solve_work(n, d, m, s, sketch, e_stored, e_pass, k, its):
    """Sketch, factor and `its` iterations of k right-hand sides: A as stored once, then once more per
    iteration in the passes' element size unless it stays on the chip."""
    nbytes = n * d * e_stored + (its * n * d * e_pass if n * d * e_pass > L2_BYTES else 0) + 2 * 8 * d * k
    return dict(bytes=float(nbytes),
                flops=_sketch_flops(sketch, n, d, m, s) + m * d * d + 2 / 3 * d ** 3 + its * k * (4.0 * n * d + 2.0 * d * d))


def work(case):
    kind = case["kind"]
    e = 8 if case.get("dtype", "f64") == "f64" else 4
    if kind == "solve":
        ep = 4 if case["precision"] == "mixed" else e
        return _solve_work(case["n"], case["d"], case["m"], case["s"], case["sketch"], e, ep, 1,
                           _iterations(case["d"], case["m"], case["tol"]))
    if kind == "refresh":
        # each iteration: its own sketch and factor, one pass
        n, d, m = case["n"], case["d"], case["m"]
        its = _iterations(d, m, case["tol"])
        return dict(bytes=float(n * d * 8 + 16 * d),
                    flops=its * (_sketch_flops(case["sketch"], n, d, m, 8) + m * d * d + 2 / 3 * d ** 3 + 4.0 * n * d))
    if kind == "sketch":
        n, d, m = case["n"], case["d"], case["m"]
        return dict(bytes=float(n * d * e + m * d * 8), flops=_sketch_flops(case["sketch"], n, d, m, case["s"]))
    if kind == "factor":
        m, d = case["m"], case["d"]
        return dict(bytes=float(m * d * 8 + 2 * d * d * 8), flops=m * d * d + 2 / 3 * d ** 3)
    if kind == "pass":
        return dict(bytes=float(case["n"] * case["d"] * e + 16 * case["d"]), flops=4.0 * case["n"] * case["d"])
    if kind == "grad":
        n, d = case["n"], case["d"]
        w = _solve_work(n, d, case["m"], 8, "srht", e, 4, 1, 2 * _iterations(d, case["m"], case["tol"]))
        # dL/dA: A read and the gradient written once, two products in and two out per element
        return dict(bytes=w["bytes"] + 2.0 * n * d * e, flops=w["flops"] + 8.0 * n * d)
    total = dict(bytes=0.0, flops=0.0)
    for n, d, k in _batch_shapes(case):
        w = _solve_work(n, d, 4 * d, 8, "sjlt", e, e, k, _iterations(d, 4 * d, case["tol"]))
        # a small problem of a large batch does not stay on the chip between iterations
        w["bytes"] = n * d * e * (1.0 + _iterations(d, 4 * d, case["tol"])) + 16 * d * k
        total = {key: total[key] + w[key] for key in total}
    return total


# ---------------------------------------------------------------------------------------------
# the same results in 64 bits, without the package
# ---------------------------------------------------------------------------------------------
def _philox(c0, c1, c2, c3, seed):
    """Philox4x32-10 (Salmon et al., SC'11) on int64 tensors that hold 32-bit words."""
    k0, k1 = seed & MASK32, (seed >> 32) & MASK32
    for _ in range(10):
        p0, p1 = c0 * 0xD2511F53, c2 * 0xCD9E8D57
        c0, c1, c2, c3 = ((p1 >> 32) & MASK32) ^ c1 ^ k0, p1 & MASK32, ((p0 >> 32) & MASK32) ^ c3 ^ k1, p0 & MASK32
        k0, k1 = (k0 + 0x9E3779B9) & MASK32, (k1 + 0xBB67AE85) & MASK32
    return c0, c1, c2, c3


def _words(i, c1, tag, seed):
    z = torch.zeros_like(i)
    return _philox(i, z + c1, z, z + tag, seed)


def _exact_gauss(A, m, seed):
    n, d = A.shape
    q = torch.arange((m + 1) // 2, device="cuda")[:, None]
    SA = torch.zeros((m, d), dtype=torch.float64, device="cuda")
    step = max(64, (1 << 25) // m)
    for r in range(0, n, step):
        i = torch.arange(r, min(n, r + step), device="cuda")[None, :] + torch.zeros_like(q)
        w0, w1, w2, w3 = _words(i, q, 1, seed)
        u1 = (((w0 << 21) | (w1 >> 11)).double() + 0.5) * 2.0 ** -53
        u2 = (((w2 << 21) | (w3 >> 11)).double() + 0.5) * 2.0 ** -53
        rad = torch.sqrt(-2.0 * torch.log(u1))
        z = torch.stack((rad * torch.cos(2 * math.pi * u2), rad * torch.sin(2 * math.pi * u2)), dim=1)
        SA += z.reshape(-1, i.shape[1])[:m] @ A[r:r + step].double()
    return SA / math.sqrt(m)


def _exact_srht(A, m, seed):
    n, d = A.shape
    N = 1 << max(0, (n - 1).bit_length())
    i = torch.arange(N, device="cuda")
    k0, k1, _, _ = _words(i, 0, 3, seed)
    key = ((k0 - 0x80000000) << 32) | k1  # ordered as the unsigned 64-bit key
    rows = torch.sort(torch.sort(key, stable=True)[1][:m])[0]
    sign = 1.0 - 2.0 * (_words(i[:n], 0, 2, seed)[0] & 1).double()
    out = torch.empty((m, d), dtype=torch.float64, device="cuda")
    cols = max(1, (1 << 28) // N)
    for c in range(0, d, cols):
        x = torch.zeros((N, min(cols, d - c)), dtype=torch.float64, device="cuda")
        x[:n] = A[:, c:c + cols].double() * sign[:, None]
        h = 1
        while h < N:
            v = x.view(N // (2 * h), 2, h, -1)
            x = torch.stack((v[:, 0] + v[:, 1], v[:, 0] - v[:, 1]), dim=1).view(N, -1)
            h *= 2
        out[:, c:c + cols] = x[rows]
    return out / math.sqrt(m)


def _exact_sjlt(A, m, s, seed, t=0):
    """s distinct rows per column by Lemire's bounded integers, in draw order."""
    n, d = A.shape
    SA = torch.zeros((m, d), dtype=torch.float64, device="cuda")
    threshold = ((1 << 32) - m) % m
    step = max(64, (1 << 25) // d)
    for r in range(0, n, step):
        i = torch.arange(r, min(n, r + step), device="cuda")
        picked = torch.full((i.numel(), s), -1, dtype=torch.int64, device="cuda")
        got = torch.zeros(i.numel(), dtype=torch.int64, device="cuda")
        drawn = 0
        while bool((got < s).any()):
            for w in _words(i, drawn, 4, seed):
                prod = w * m
                v = (prod >> 32) & MASK32
                ok = ((prod & MASK32) >= threshold) & (got < s) & ~(picked == v[:, None]).any(1)
                at = torch.nonzero(ok)[:, 0]
                picked[at, got[at]] = v[at]
                got += ok
            drawn += 1
        bits = _words(i, 0, 5, seed)[0]
        rows64 = A[r:r + step].double()
        for k in range(s):
            sgn = 1.0 - 2.0 * ((bits >> k) & 1).double()
            SA.index_add_(0, picked[:, k], rows64 * sgn[:, None])
    return SA / math.sqrt(s)


def _gram_solver(A):
    """v -> H^{-1} v for H = A^T A by a Cholesky factor of the column-scaled Gram matrix with two
    steps of refinement against A itself."""
    n, d = A.shape
    step = max(1, (1 << 27) // d)
    G = torch.zeros((d, d), dtype=torch.float64, device="cuda")
    for r in range(0, n, step):
        blk = A[r:r + step].double()
        G += blk.T @ blk
    D = torch.sqrt(torch.diagonal(G)).reciprocal()
    C = torch.linalg.cholesky(G * D[:, None] * D[None, :])

    def apply(v):
        return D[:, None] * torch.cholesky_solve(D[:, None] * v, C)

    def solve(v):
        x = apply(v)
        for _ in range(2):
            hx = torch.zeros_like(v)
            for r in range(0, n, step):
                blk = A[r:r + step].double()
                hx += blk.T @ (blk @ x)
            x = x + apply(v - hx)
        return x

    return solve


def exact(case, seed):
    """What run() returns for these inputs, from plain torch in FP64."""
    st = prepare(case, seed)
    kind = case["kind"]
    st["ctx"].close()
    if kind in ("solve", "refresh"):
        return _gram_solver(st["A"])(st["b"][:, None])[:, 0].contiguous()
    if kind == "sketch":
        A, m = st["A"], case["m"]
        if case["sketch"] == "gauss":
            return _exact_gauss(A, m, st["seed"])
        return _exact_srht(A, m, st["seed"]) if case["sketch"] == "srht" else _exact_sjlt(A, m, case["s"], st["seed"])
    if kind == "factor":
        SA = st["SA"]
        R = torch.linalg.cholesky(SA.T @ SA).T.contiguous()
        W = torch.linalg.solve_triangular(R, torch.eye(case["d"], dtype=torch.float64, device="cuda"), upper=True)
        return {"R": R, "W": W}
    if kind == "pass":
        A64 = st["A"].double()
        y = A64 @ st["p"]
        return {"v": A64.T @ y, "q": (y @ y).reshape(1)}
    if kind == "grad":
        A = st["A"].detach()
        solve = _gram_solver(A)
        x, lam = solve(st["b"].detach()[:, None])[:, 0], solve(st["g"][:, None])[:, 0]
        A64 = A.double()
        gA = -((A64 @ x)[:, None] * lam[None, :] + (A64 @ lam)[:, None] * x[None, :])
        return {"x": x, "gA": gA.to(A.dtype), "gb": lam}
    return torch.cat([_gram_solver(A)(B.T.contiguous()).T.reshape(-1) for A, B in st["problems"]])
