"""Mixed solve over FP32 rows of 129 to 256 columns: the pass that stages rows by bulk copies and the
pass with register loads (rows that are not 16-byte aligned) add in one order, so the solutions agree
bit for bit, also where a warp has fewer rows than ring slots."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,d", [(600, 132), (5003, 196), (40000, 252), (9001, 256)])
def test_staged_rows_match_register_rows(n, d):
    import paper_1911_02675_gb300 as L

    rng = np.random.default_rng(n + d)
    A = torch.from_numpy(rng.standard_normal((n, d)).astype(np.float32)).cuda()
    b = torch.from_numpy(rng.standard_normal(d)).cuda()
    buf = torch.empty(n * d + 1, dtype=torch.float32, device="cuda")
    shifted = buf[1:].view(n, d)  # 4 bytes off a 16-byte boundary
    shifted.copy_(A)
    ctx = L.Context()
    m = min(n, 4 * d)
    _, W = L.lsq_factor(ctx, L.lsq_sketch(ctx, A, "gauss", m, 7, precision="f32"))
    xs = [L.lsq_solve(ctx, M, b, "pcg", W, tol=1e-11, maxit=500, m=m, precision="mixed")[0] for M in (A, shifted)]
    assert torch.equal(xs[0], xs[1])
    A64 = A.cpu().double()
    xr = torch.linalg.solve(A64.T @ A64, b.cpu())
    assert torch.linalg.norm(xs[0].cpu() - xr) <= 1e-8 * torch.linalg.norm(xr)
