"""The FP64 SRHT of 2048-row blocks (integer-pipe transform) at the edges of its tiles, over wide
dynamic ranges and with infinities and NaNs, against the FP64 oracle.

Bound: the transform of a block is exact to 2^-73 of its largest element and is rounded once, and
the blocks' sums add in FP64, so a column is within (blocks + 2) 2^-53 of the exact result; the
oracle's own log2(N) levels of additions are within log2(N) 2^-53.  Both together stay below
40 * 2^-53 < 1e-14 for the sizes here (norm-wise per column)."""
import numpy as np
import pytest
import torch

import oracle as O
from gpu_util import to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def L():
    import paper_1911_02675_gb300 as lib
    return lib


@pytest.fixture(scope="module")
def ctx(L):
    c = L.Context(0)
    yield c
    c.close()


@pytest.mark.parametrize("n,d,m,dtype,pad", [
    (1025, 1, 5, np.float64, 0), (2048, 4, 256, np.float64, 0), (2049, 7, 257, np.float64, 1),
    (5000, 33, 1025, np.float32, 3), (20000, 6, 2049, np.float64, 0), (9000, 5, 5000, np.float32, 0)])
def test_edges(L, ctx, n, d, m, dtype, pad):
    g = np.random.default_rng(n + d)
    A = g.standard_normal((n, d)).astype(dtype)
    A[g.random(n) < 0.01] *= dtype(1e6)          # outlier rows: a block's scale is set by few elements
    A *= (10.0 ** g.uniform(-12, 12, size=d)).astype(dtype)
    wide = to_dev(np.concatenate([A, np.full((n, pad), 7, dtype=dtype)], axis=1))
    SA = L.lsq_sketch(ctx, wide[:, :d], "srht", m, 3, t=1).cpu().numpy()
    ref = O.sketch_srht(A.astype(np.float64), m, 3, 1)
    err = np.linalg.norm(SA - ref, axis=0) / np.linalg.norm(ref, axis=0)
    assert err.max() < 1e-14, err


def test_extreme_scales(L, ctx):
    """Columns near the ends of the FP64 range (subnormal elements in the last) and an all-zero one."""
    n, m = 3000, 200
    A = np.random.default_rng(5).standard_normal((n, 5)) * np.array([1e300, 1e-300, 0.0, 1.0, 3e-310])
    SA = L.lsq_sketch(ctx, to_dev(A), "srht", m, 9).cpu().numpy()
    ref = O.sketch_srht(A, m, 9, 0)
    assert np.all(SA[:, 2] == 0.0)
    for c in (0, 1, 3):
        assert np.linalg.norm(SA[:, c] / 2.0**900 - ref[:, c] / 2.0**900 if c == 0 else
                              (SA[:, c] - ref[:, c]) * 2.0**(900 if c == 1 else 0)) \
            <= 1e-14 * np.linalg.norm(ref[:, c] / 2.0**900 if c == 0 else ref[:, c] * 2.0**(900 if c == 1 else 0))
    # subnormal sums: one unit of 2^-1074 per rounding (two blocks and the scaling on either side)
    assert np.abs(SA[:, 4] - ref[:, 4]).max() <= 8 * 2.0**-1074 + 1e-14 * np.abs(ref[:, 4]).max()


def test_infinities_and_nans(L, ctx):
    n, d, m = 5000, 6, 300
    g = np.random.default_rng(2)
    A = g.standard_normal((n, d))
    plain = L.lsq_sketch(ctx, to_dev(A), "srht", m, 4).cpu().numpy()
    rows = [17, 900, 4100]  # 17 and 900 share a 2048-row block
    E = np.zeros((n, 3))
    for k, r in enumerate(rows):
        E[r, k] = 1.0
    s = np.sign(O.sketch_srht(E, m, 4, 0))       # the signs of S at those rows
    A[17, 1] = np.inf
    A[17, 2], A[900, 2] = np.inf, -np.inf
    A[900, 3] = np.nan
    A[17, 4], A[4100, 4] = -np.inf, -np.inf
    SA = L.lsq_sketch(ctx, to_dev(A), "srht", m, 4).cpu().numpy()
    assert np.array_equal(SA[:, [0, 5]], plain[:, [0, 5]])
    with np.errstate(invalid="ignore"):
        assert np.array_equal(SA[:, 1], s[:, 0] * np.inf)
        assert np.array_equal(SA[:, 2], s[:, 0] * np.inf - s[:, 1] * np.inf, equal_nan=True)
        assert np.isnan(SA[:, 3]).all()
        assert np.array_equal(SA[:, 4], -s[:, 0] * np.inf - s[:, 2] * np.inf, equal_nan=True)
