"""lsq_factor's Gram matrix from digit products, at the edges of its tiles (64 x 32), stages (32 rows)
and folds (128 rows), with columns scaled over +-1e120, dominant entries and a panel of rows that
does not end on a stage: R against numpy's Householder QR of the column-normalised SA.

Bound: H_S is within 2^-57 (mixed: 2^-49) of the columns' norms, its FP64 Cholesky within about
(d + 1) 2^-53 of them, numpy's QR within a few d 2^-53; R moves by that times the condition of the
normalised H_S (below 20 for these m >= 3 d).  (d + 1) 2^-53 * 20 < 2e-12 (mixed: 2^-49 * 20 more) for
d <= 520; entries compared on the scale of their column."""
import numpy as np
import pytest
import torch

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


@pytest.mark.parametrize("precision", ["f64", "mixed"])
@pytest.mark.parametrize("m,d", [(5, 1), (17, 5), (100, 31), (129, 33), (256, 64), (200, 65), (513, 97), (1000, 128),
                                 (1700, 511), (2050, 520)])
def test_r_of_scaled_columns(L, ctx, m, d, precision):
    g = np.random.default_rng(m)
    N = g.standard_normal((m, d))
    N[g.integers(0, m, size=d), np.arange(d)] *= 8.0   # an entry that sets its column's scale
    s = 10.0 ** g.uniform(-120, 120, size=d)
    s[0] = 1.0
    R, W = L.lsq_factor(ctx, to_dev(N * s), precision=precision)
    ref = np.linalg.qr(N, mode="r")
    ref *= np.sign(np.diagonal(ref))[:, None]
    got = R.cpu().numpy() / s
    assert np.abs(got - ref).max() <= 2e-12 * np.sqrt((ref ** 2).sum(0)).max()
    WR = (W.cpu().numpy() * s[:, None]) @ got
    assert np.abs(WR - np.eye(d)).max() < 1e-9


@pytest.mark.parametrize("precision", ["f64", "mixed"])
def test_second_panel_of_rows(L, ctx, precision):
    """More rows than one panel of digits holds (2^18 at d <= 64; 299520 with 7 digits), the second one short
    and off a stage, as above."""
    test_r_of_scaled_columns(L, ctx, 300101, 33, precision)


@pytest.mark.parametrize("precision", ["f64", "mixed"])
@pytest.mark.parametrize("d", [70, 300])
@pytest.mark.parametrize("kind", ["even", "2^10", "2^20", "2^30", "sparse", "scaled"])
def test_entries_where_columns_peak_in_different_rows(L, ctx, kind, d, precision):
    """H_S[0][b] = R[0][0] R[0][b] entry by entry, on the scale of sum_r |a_r b_r| and not of the columns'
    norms: FP64 multiply-adds err by at most m 2^-53 of it, double-FP32 ones by 2^-44 (45 bits of each
    element) and m 2^-46 (the FP32 sums of their tails), and R[0][0], R[0][b] by a few units more."""
    g = np.random.default_rng(11)
    m = 1024
    X = g.standard_normal((m, d))
    if kind == "sparse":
        X *= g.random((m, d)) < 0.05
    elif kind != "even":
        X[(7 * np.arange(d)) % m, np.arange(d)] = 2.0 ** {"2^10": 10, "2^20": 20, "2^30": 30, "scaled": 20}[kind]
    s = 10.0 ** g.uniform(-100, 100, size=d) if kind == "scaled" else np.ones(d)
    R, _ = L.lsq_factor(ctx, to_dev(X * s), precision=precision)
    X = (X * s).astype(np.longdouble)
    H, S = X[:, 0] @ X, np.abs(X[:, 0]) @ np.abs(X)
    got = R.cpu().numpy()[0].astype(np.longdouble)
    u = m * 2.0 ** -53 if precision == "f64" else 2.0 ** -44 + m * 2.0 ** -46
    assert np.all(np.abs(got[0] * got - H) <= (u + 8 * 2.0 ** -53) * S)


@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_non_finite_is_a_rank_error(L, ctx, bad):
    A = np.random.default_rng(1).standard_normal((300, 40))
    A[7, 39] = bad
    with pytest.raises(L.LsqError) as e:
        L.lsq_factor(ctx, to_dev(A))
    assert e.value.status == L.LSQ_ERR_RANK
