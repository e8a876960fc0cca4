"""The FP64 pass with its dot products from digit products (FP64 rows of 65 to 512 columns, 192 and
more a CTA; the other calls here keep FP64 sums), against extended precision: chunks of 32 columns and their remainders, tiles of 16 rows and theirs, both types,
strided rows, rows and columns of very different scales, zeros, subnormals, entries of p out of the digits'
range, infinities and NaNs.  Each v_j is a sum of n products a_ij w_i of d-term sums: with FP64
accumulators of n / (152 x 8) rows at most and a few hundred partial sums, the error is below
2^-53 (n / 1216 + d + 400) sum_i |a_ij| sum_k |a_ik p_k|."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

N = 304 * 384 + 1111


def _run(A, p, ld=None):
    import paper_1911_02675_gb300 as L

    ctx = L.Context()
    t = torch.from_numpy(A).cuda()
    if ld:
        wide = torch.full((A.shape[0], ld), float("nan"), dtype=t.dtype, device="cuda")
        wide[:, 1:1 + A.shape[1]] = t
        t = wide[:, 1:1 + A.shape[1]]
    v, q = L.lsq_hmatvec(ctx, t, torch.from_numpy(p).cuda())
    return v.cpu().numpy(), float(q)


def _check(A, p, ld=None):
    n, d = A.shape
    v, q = _run(A, p, ld)
    X = A.astype(np.longdouble)
    w = X @ p.astype(np.longdouble)
    S = np.abs(X) @ np.abs(p.astype(np.longdouble))
    u = 2.0 ** -53 * (n / 1216 + d + 400)
    with np.errstate(all="ignore"):
        ref, bound = X.T @ w, np.abs(X).T @ S
        assert np.all(np.abs(v - ref) <= u * bound + 1e-300)
        rq = w @ w
        assert abs(q - rq) <= 2 * u * (S @ S) + 1e-300


@pytest.mark.parametrize("dtype", [np.float64, np.float32])
@pytest.mark.parametrize("n,d,ld", [(N, 65, None), (N + 5, 96, None), (N, 130, 135), (2 * N + 3, 128, None)])
def test_sizes(n, d, ld, dtype):
    rng = np.random.default_rng(d)
    _check(rng.standard_normal((n, d)).astype(dtype), rng.standard_normal(d), ld)


@pytest.mark.parametrize("scaled", [False, True])
@pytest.mark.parametrize("nk", range(3, 17))
def test_each_dot_product(nk, scaled):
    """The w_i themselves, at every number of 32-column chunks: the last 24 columns hold a 1 in one row each
    and p is zero there, so that v_j = w_i.  A chunk drops less than 3 units of 2^-53 of its largest
    |a_ij p_j| (6 digit pairs of 255 x 128 on 2^40 of 2^114, for 32 columns) and rounds once as it is added;
    the sum of two lanes and of the odd and even chunks rounds twice more."""
    rng = np.random.default_rng(nk)
    n, d = 304 * 200 + 77, 32 * nk - (0 if nk % 3 == 0 else rng.integers(1, 32))
    A, p = rng.standard_normal((n, d)), rng.standard_normal(d)
    if scaled:
        s = 10.0 ** rng.uniform(-60, 60, d)
        A, p = A * s, p / s
        A *= 10.0 ** rng.uniform(-30, 30, (n, 1))
    rows = np.concatenate([np.arange(16), [200, 201, 402, 30007, n - 78, n - 17, n - 2, n - 1]])
    A[:, d - 24:] = 0.0
    A[rows, np.arange(d - 24, d)] = 1.0
    p[d - 24:] = 0.0
    v, _ = _run(A, p)
    P = A[rows].astype(np.longdouble) * p.astype(np.longdouble)
    assert np.all(np.abs(v[d - 24:] - P.sum(1)) <= (nk + 6) * 2.0 ** -53 * np.abs(P).sum(1))
    S = np.abs(A) @ np.abs(p)
    assert np.all(np.abs(v - A.T @ (A @ p)) <= 1e-12 * (np.abs(A).T @ S))


def test_widest_rows():
    rng = np.random.default_rng(1)
    n = 152 * 384 + 77
    _check(rng.standard_normal((n, 545)), rng.standard_normal(545))


@pytest.mark.parametrize("kind", ["columns", "rows", "both", "sparse", "tiny p", "huge p", "tiny A", "one entry"])
def test_scales(kind):
    rng = np.random.default_rng(7)
    d = 81
    A, p = rng.standard_normal((N, d)), rng.standard_normal(d)
    if kind in ("columns", "both"):
        s = 10.0 ** rng.uniform(-100, 100, d)
        A, p = A * s, p / s
        if kind == "both":
            A *= 10.0 ** rng.uniform(-40, 40, (N, 1))
    elif kind == "rows":
        A *= 10.0 ** rng.uniform(-140, 140, (N, 1))
    elif kind == "sparse":
        A *= rng.random((N, d)) < 0.02
        A[::7] = 0.0
        A[3::11] *= 5e-320
        p[::3] = 0.0
    elif kind == "tiny p":
        p *= 1e-250
    elif kind == "huge p":
        p *= 1e190
        A *= 1e-150
    elif kind == "tiny A":
        A *= 1e-290
        p *= 1e150
    else:
        p[:] = 0.0
        p[40] = 3.0
    _check(A, p)


@pytest.mark.parametrize("kind", ["zeros of p", "zeros past d", "subnormal p", "chunks of zeros"])
def test_elements_that_meet_no_product(kind):
    """The scale of a row and 32 columns comes from its products: neither from elements that meet a zero of
    p (or lie past d), nor from subnormal entries of p; bounds as above."""
    rng = np.random.default_rng(8)
    d = 81
    A, p = rng.standard_normal((N, d)), rng.standard_normal(d)
    if kind == "zeros of p":
        p *= 1e-125
        p[[0, 40, 70]] = 0.0
        A[:, [0, 40, 70]] *= 1e290
    elif kind == "zeros past d":
        p *= 1e-125
        p[80] = 0.0
        A[:, 80] *= 1e290
    elif kind == "subnormal p":
        p *= 1e-150
        p[33] = 1e-320
        A[:, :33] = A[:, 34:] = 0.0
        A[:, 33] *= 1e200
    else:
        p[:64] = 0.0
        A[::3, 64:] = 0.0
    _check(A, p)


@pytest.mark.parametrize("d", [70, 160, 333])
def test_integers_are_exact(d):
    """Small integers with signs: every product and sum is exact in FP64, and in the digits."""
    rng = np.random.default_rng(d)
    A, p = rng.integers(-9, 10, (N, d)).astype(float), rng.integers(-300, 301, d).astype(float)
    v, q = _run(A, p)
    w = A @ p
    assert np.array_equal(v, A.T @ w) and q == w @ w


def test_null_vector():
    """A p = 0 exactly over integers, which the solvers see as q = 0."""
    A = np.random.default_rng(5).integers(-9, 10, (N, 96)).astype(float)
    A[:, 48:] = -A[:, :48]
    v, q = _run(A, np.full(96, 3.0))
    assert q == 0.0 and not v.any()


@pytest.mark.parametrize("bad", [np.inf, -np.inf, np.nan])
@pytest.mark.parametrize("where", ["A", "p"])
def test_not_finite(bad, where):
    rng = np.random.default_rng(9)
    A, p = rng.standard_normal((N, 70)), rng.standard_normal(70)
    if where == "A":
        A[50001, 66] = bad
        p[12] = 0.0
    else:
        p[13] = bad
    v, q = _run(A, p)
    with np.errstate(all="ignore"):
        w = (A * p).sum(1)
        ref, rq = (A * w[:, None]).sum(0), (w * w).sum()
    for got, want in ((v, ref), (np.array([q]), np.array([rq]))):
        assert np.array_equal(np.isnan(got), np.isnan(want))
        assert np.array_equal(np.isinf(got), np.isinf(want))
