"""The batched passes over FP32 A (stages in shared memory: TF32 MMAs for the FP32 passes, packed
double-FP32 for the exact ones) at the edges of their tiles: widths around every change of the
stage's shape and of the row spacing (odd d, 2 x odd, multiples of 4 and of 8), row counts around a
stage, 1 to 16 right-hand sides, rows with gaps and matrices off 16 bytes.

The first iterate depends on one FP32 pass (and, from a nonzero x0, on one exact pass for the initial
residual); its error is that of the pass, products to 2^-22 and FP32 sums of at most 256 rows a stage:
below 1e-6 of the iterate by the same count of roundings, tested at the 1e-5 of the package's
first-iteration test."""
import numpy as np
import pytest
import torch

import oracle as O
import workloads as W
from gpu_util import rel_fro, to_dev

pytestmark = pytest.mark.gpu

D = [1, 7, 8, 9, 15, 16, 17, 31, 33, 48, 62, 63, 64, 65, 100, 127, 128, 129, 136, 137, 255, 256, 257, 272, 273, 340,
     385, 510, 511, 512]


@pytest.fixture(scope="module")
def L():
    import paper_1911_02675_gb300 as lib
    return lib


@pytest.fixture(scope="module")
def ctx(L):
    c = L.Context(0)
    yield c
    c.close()


@pytest.mark.parametrize("layout", ["contiguous", "gap", "offset"])
@pytest.mark.parametrize("x0", [False, True])
def test_first_iterate(L, ctx, x0, layout):
    shapes = [(max(4 * d, 256) + (d * 37) % 300, d, 1 + (5 * i) % 16) for i, d in enumerate(D)]
    probs = W.make_batch(shapes, seed=23, scale_max=1e2, dtype=np.float32)
    dev = []
    for i, q in enumerate(probs):
        A = to_dev(q["A"])
        n, d = A.shape
        if layout == "gap":
            wide = torch.full((n, d + 1 + i % 4), float("nan"), dtype=torch.float32, device="cuda")
            wide[:, :d] = A
            A = wide[:, :d]
        elif layout == "offset":
            flat = torch.full((n * d + 1 + i % 3,), float("nan"), dtype=torch.float32, device="cuda")
            flat[1 + i % 3:] = A.reshape(-1)
            A = flat[1 + i % 3:].view(n, d)
        dev.append((A, to_dev(q["B"])))
    rng = np.random.default_rng(9)
    X0 = [rng.standard_normal(q["B"].shape) for q in probs] if x0 else None
    X, per, info = L.lsq_solve_batched(ctx, dev, tol=0.0, maxit=1, precision="mixed", sketch_precision="f64", seed=3,
                                       X0=[to_dev(v) for v in X0] if x0 else None)
    ref = O.solve_batched([(q["A"].astype(np.float64), q["B"]) for q in probs], kind="sjlt", s=8, m_factor=4.0, seed=3,
                          tol=0.0, maxit=1, X0=X0)
    for i, (sh, Xp, (Xr, its, sts), (it, st)) in enumerate(zip(shapes, X, ref, per)):
        assert it == 1 and st == L.LSQ_ERR_MAXIT, (sh, it, st)
        start = X0[i] if x0 else 0.0
        assert rel_fro(Xp.cpu().numpy() - start, Xr - start) < 1e-5, sh


@pytest.mark.parametrize("d,pad", [(33, 1), (64, 4), (255, 1), (512, 4)])
def test_rows_with_gaps_keep_fp32_sums(L, ctx, d, pad):
    """Batches whose rows have gaps take FP32 multiply-adds: the first iterate x = u <b, u> / ||A u||^2 shows
    ||A p||^2, whose roundings (of p, and of 20000 sums of d products) are as often up as down and average
    out below one unit of 2^-24 over the batch (the tensor cores' sums, cut off, lie 3e-7 low)."""
    g = torch.Generator(device="cuda").manual_seed(d)
    probs = []
    for _ in range(16):
        wide = torch.randn((20000, d + pad), generator=g, dtype=torch.float32, device="cuda")
        probs.append((wide[:, :d], torch.randn((2, d), generator=g, dtype=torch.float64, device="cuda")))
    X, _, _ = L.lsq_solve_batched(ctx, probs, tol=1e-12, maxit=1, precision="mixed", seed=4)
    err = []
    for (A, B), x in zip(probs, X):
        for xj, b in zip(x, B):
            u = xj / xj.norm()
            err.append(float(xj.norm() * (A.double() @ u).square().sum() / (b @ u)) - 1.0)
    assert np.sqrt(np.mean(np.square(err))) < 2.0 ** -24
