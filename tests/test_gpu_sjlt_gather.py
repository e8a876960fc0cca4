"""The FP32 SJLT (entries sorted by target row, then gathered) against the oracle's SJLT on small
integers, where every sum is exact: the result times sqrt(s) rounds to the oracle's integer, for
sizes at the edges of its chunks (2048 rows, fewer for s > 8), target slices (4096), pairs of
threads sharing a target (m <= 128) and unaligned rows; and it repeats bit for bit."""
import numpy as np
import pytest
import torch

import oracle as O
from gpu_util import int_matrix, to_dev

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


@pytest.mark.parametrize("n,d,m,s,dtype,pad", [
    (1, 1, 1, 1, np.float64, 0), (2047, 3, 8, 8, np.float32, 0), (2049, 9, 32, 8, np.float64, 1),
    (4096, 8, 128, 8, np.float32, 0), (5000, 17, 129, 5, np.float64, 0), (3000, 16, 256, 16, np.float32, 4),
    (1025, 12, 257, 32, np.float64, 0), (7000, 10, 1000, 8, np.float32, 1), (20001, 5, 2049, 8, np.float64, 0),
    (9000, 4, 4097, 3, np.float32, 0), (6000, 2, 40000, 32, np.float64, 0)])
def test_exact_on_integers(L, ctx, n, d, m, s, dtype, pad):
    A = int_matrix(n, d, n + m)
    wide = to_dev(np.concatenate([A, np.full((n, pad), 99.0)], axis=1).astype(dtype))
    SA = L.lsq_sketch(ctx, wide[:, :d], "sjlt", m, 6, t=2, s=s, precision="f32")
    again = L.lsq_sketch(ctx, wide[:, :d], "sjlt", m, 6, t=2, s=s, precision="f32")
    assert torch.equal(SA, again)
    got = SA.cpu().numpy() * np.sqrt(s)
    ref = np.rint(O.sketch_sjlt(A, m, s, 6, 2) * np.sqrt(s))
    assert np.array_equal(np.rint(got), ref)
    assert np.abs(got - ref).max() <= 1e-12 * max(1.0, np.abs(ref).max())


@pytest.mark.parametrize("n,d,m,s,dtype,pad", [
    (2049, 17, 129, 4, np.float64, 1), (16385, 33, 256, 8, np.float32, 3), (40000, 130, 1025, 16, np.float64, 0),
    (300001, 17, 64, 32, np.float32, 0), (5000, 600, 4096, 4, np.float64, 0), (610000, 101, 9000, 16, np.float32, 0),
    (33000, 130, 2049, 32, np.float64, 0), (1 << 19, 9, 512, 8, np.float32, 0), (70001, 20, 300, 3, np.float64, 0)])
def test_gathered_sizes(L, ctx, n, d, m, s, dtype, pad):
    """The sizes that are gathered, either side of one and two slices of targets and of a tile, as above."""
    test_exact_on_integers(L, ctx, n, d, m, s, dtype, pad)


@pytest.mark.parametrize("n,d,m,s,dtype,pad", [
    (60000, 4, 16, 16, np.float64, 0), (100003, 12, 60, 8, np.float32, 1), (2047, 40, 2000, 1, np.float64, 0),
    (9000, 25, 6400, 8, np.float32, 3), (60001, 9, 51200, 8, np.float64, 0)])
def test_scattered_sizes(L, ctx, n, d, m, s, dtype, pad):
    """Sizes whose lists would cost more than their additions, with one to four columns a tile, as above."""
    test_exact_on_integers(L, ctx, n, d, m, s, dtype, pad)
