"""The FP64 Gaussian sketch from digit products against the FP64 oracle: every entry of S (A = I), sizes
around its tiles (64 x 64), stages (16 rows) and folds (128 rows), FP32 and strided A, columns over
+-1e100 with outlier rows, a row slab, and non-finite entries.

Bound: an entry of S differs from the oracle's by the errors of two FP64 evaluations (log, square root,
sine: a few units of 2^-53 each, the angle 2 pi u2 rounded once more) and 2^-58: below 1e-14 absolute; a
column of SA by sqrt(n) 2^-57 of its norm on top, below 1e-14 relative for the sizes here."""
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


def test_entries(L, ctx):
    n, m = 700, 130
    S = L.lsq_sketch(ctx, torch.eye(n, dtype=torch.float64, device="cuda"), "gauss", m, 11, t=3).cpu().numpy()
    ref = O.sketch_gauss(np.eye(n), m, 11, 3)
    assert np.abs(S - ref).max() * np.sqrt(m) < 1e-14


@pytest.mark.parametrize("n,d,m,dtype,pad", [(1, 1, 1, np.float64, 0), (15, 3, 2, np.float64, 1),
                                             (129, 64, 63, np.float64, 0), (1000, 65, 64, np.float32, 3),
                                             (2049, 33, 65, np.float64, 0), (5000, 130, 200, np.float64, 2)])
def test_sketch(L, ctx, n, d, m, dtype, pad):
    g = np.random.default_rng(n)
    A = g.standard_normal((n, d))
    A[g.random(n) < 0.05] *= 100.0
    A = (A * 10.0 ** g.uniform(-18, 18, size=d)).astype(dtype) if dtype == np.float32 else A * 10.0 ** g.uniform(-100, 100, size=d)
    wide = to_dev(np.concatenate([A, np.full((n, pad), np.nan, dtype=dtype)], axis=1))
    SA = L.lsq_sketch(ctx, wide[:, :d], "gauss", m, 5, t=1).cpu().numpy()
    ref = O.sketch_gauss(A.astype(np.float64), m, 5, 1)
    s = np.abs(ref).max(0)
    assert (np.linalg.norm((SA - ref) / s, axis=0) / np.linalg.norm(ref / s, axis=0)).max() < 1e-14
    if n >= 1000:
        k = 512
        top = L.lsq_sketch(ctx, wide[:k, :d], "gauss", m, 5, t=1, row0=0, n_total=n).cpu().numpy()
        bot = L.lsq_sketch(ctx, wide[k:, :d], "gauss", m, 5, t=1, row0=k, n_total=n).cpu().numpy()
        assert (np.linalg.norm((top + bot - ref) / s, axis=0) / np.linalg.norm(ref / s, axis=0)).max() < 1e-14


def test_columns_near_the_smallest_numbers(L, ctx):
    # entries of SA down to the subnormals: the bound of the columns above plus half a unit of 2^-1074
    # for the rounding of each entry here and in the oracle's sums (300 of them)
    A = np.random.default_rng(4).standard_normal((300, 6)) * np.array([1e-306, 3e-310, 0.0, 1e-305, 2.0 ** -1010, 1.0])
    SA = L.lsq_sketch(ctx, to_dev(A), "gauss", 70, 2).cpu().numpy()
    ref = O.sketch_gauss(A, 70, 2, 0)
    assert (np.abs(ref).max(0) > 0).tolist() == [True, True, False, True, True, True]
    assert np.all(np.abs(SA - ref) <= 1e-14 * np.abs(ref).max(0) * 10 + 301 * 2.0 ** -1074)


def test_uniform_next_to_one(L, ctx):
    # row 847055 of this instance draws u1 = 1 - 1.7e-10, where -2 ln u1 hangs on the last bit of u1;
    # 32 rows of ones around it, each entry within 1e-14
    i0, n = 847040, 1 << 20
    SA = L.lsq_sketch(ctx, torch.ones((32, 1), dtype=torch.float64, device="cuda"), "gauss", 2, 11, t=3, row0=i0,
                      n_total=n).cpu().numpy()[:, 0]
    ref = [sum(O.gauss_z(11, 3, j, i) for i in range(i0, i0 + 32)) / np.sqrt(2) for j in (0, 1)]
    assert np.abs(SA - ref).max() < 32e-14


def _entries(m, n, seed, t):
    """sqrt(m) S in extended precision, from the same uniforms"""
    w = O.philox4x32_10([(i, j, t, 1) for i in range(n) for j in range(m // 2)], (seed, 0)).astype(np.uint64)
    k1, k2 = ((w[:, 0] << 32 | w[:, 1]) >> 11), ((w[:, 2] << 32 | w[:, 3]) >> 11)
    u1, u2 = ((k.astype(np.float64) + 0.5) * 2.0 ** -53 for k in (k1, k2))
    pi = 4 * np.arctan(np.longdouble(1))
    rad = np.sqrt(-2 * np.log(u1.astype(np.longdouble)))
    h = np.rint(4 * u2)                                  # quarter turns, exact remainder
    a = 2 * pi * (u2 - h / 4).astype(np.longdouble)
    sn, cs = np.sin(a), np.cos(a)
    h = h.astype(int) % 4
    z = np.empty((m, n), dtype=np.longdouble)
    z[0::2] = (rad * np.choose(h, [cs, -sn, -cs, sn])).reshape(n, m // 2).T
    z[1::2] = (rad * np.choose(h, [sn, cs, -sn, -cs])).reshape(n, m // 2).T
    return z


@pytest.mark.parametrize("n,d", [(64, 3), (700, 67)])
def test_entries_that_hang_on_one_row(L, ctx, n, d):
    """Columns with one nonzero row, with one dominant row and even ones, entry by entry on the scale of
    sum_i |z(j, i) a_i|: FP64 entries of S are within 8 units (logarithm, square root, sine, their
    product), their products and sums within n."""
    m = 400
    g = np.random.default_rng(n)
    A = g.standard_normal((n, d))
    A[:, 0] = 0.0
    A[:, d // 2] *= 1e-9
    A[n // 3, [0, d // 2]] = 3.0
    SA = L.lsq_sketch(ctx, to_dev(A), "gauss", m, 9, t=2).cpu().numpy()
    z, A = _entries(m, n, 9, 2), A.astype(np.longdouble)
    ref, S = z @ A, np.abs(z) @ np.abs(A)
    err = np.abs(SA * np.sqrt(np.longdouble(m)) - ref)
    assert np.all(err <= (2 * 8 + n + 4) * 2.0 ** -53 * S)
    assert np.all(err[:, 0] <= (2 * 8 + 4) * 2.0 ** -53 * S[:, 0])


def test_non_finite(L, ctx):
    A = np.random.default_rng(3).standard_normal((300, 5))
    clean = L.lsq_sketch(ctx, to_dev(A), "gauss", 70, 2).cpu().numpy()
    E = np.zeros((300, 1))
    E[40] = 1.0
    z = O.sketch_gauss(E, 70, 2, 0)[:, 0]
    A[40, 1], A[7, 2], A[40, 3], A[41, 3] = np.inf, np.nan, np.inf, -np.inf
    SA = L.lsq_sketch(ctx, to_dev(A), "gauss", 70, 2).cpu().numpy()
    assert np.array_equal(SA[:, [0, 4]], clean[:, [0, 4]])
    assert np.array_equal(SA[:, 1], np.sign(z) * np.inf)
    assert np.isnan(SA[:, 2]).all()
    assert not np.isfinite(SA[:, 3]).any()


@pytest.mark.parametrize("kind", ["even", "dominant rows"])
def test_second_panel_of_rows(L, ctx, kind):
    """More rows than one panel of digits holds (2^18 at d <= 64), the second one short and off a stage:
    the bound of the columns above, sqrt(n) 2^-57 of their norm, against extended precision."""
    n, d, m = (1 << 18) + 1013, 3, 8
    A = np.random.default_rng(6).standard_normal((n, d))
    if kind != "even":
        A[[5, n - 3], [1, 2]] = 1e6
    SA = L.lsq_sketch(ctx, to_dev(A), "gauss", m, 9, t=2).cpu().numpy()
    ref = _entries(m, n, 9, 2) @ A.astype(np.longdouble)
    err = np.linalg.norm((SA * np.sqrt(np.longdouble(m)) - ref).astype(float), axis=0)
    assert np.all(err < 1e-14 * np.sqrt(m) * np.linalg.norm(A, axis=0))
