"""Right-hand sides of the tall solve side by side (cqr_lstsq.cu): each does the arithmetic of its own
solve, so the bits are those of one at a time.  One CTA per side, several, so many that only some
fit at once, and more sides than one launch takes; the adjoint's solves the same."""
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2311_11943_gb300 import binding as B  # noqa: E402


@pytest.mark.parametrize("m,n,p_r,p_c,f,dtype,k", [(40, 8, 4, 4, 1, "f64", 4), (1003, 132, 6, 4, 2, "f32", 7),
                                                   (4000, 1600, 5, 4, 2, "f32", 5), (900, 516, 6, 4, 2, "f64", 3)])
def test_sides_together_match_one_at_a_time(m, n, p_r, p_c, f, dtype, k):
    td = torch.float64 if dtype == "f64" else torch.float32
    g = torch.Generator(device="cuda").manual_seed(m)
    A = torch.randn((n, m), generator=g, device="cuda", dtype=td).t()
    y = torch.randn((k, m + 3), generator=g, device="cuda", dtype=td).t()[:m]
    q = B.CodedQR(m, n, p_r, p_c, f, 64, dtype=dtype, nrhs_max=k, seed=4)
    q.encode(A)
    q.factor(0, -1)
    x = B.colmajor_empty(n, k, td, ld=n + 5)
    q.solve_ls(y, x)
    one = B.colmajor_empty(n, k, td)
    for j in range(k):
        q.solve_ls(y[:, j:j + 1], one[:, j:j + 1])
    torch.cuda.synchronize()
    assert q.sync_status() == 0 and torch.isfinite(x).all()
    assert torch.equal(x, one)
    xb = torch.randn((k, n), generator=g, device="cuda", dtype=td).t()
    Ab = [B.colmajor_empty(m, n, td).zero_() for _ in range(2)]
    yb = [B.colmajor_empty(m, k, td).zero_() for _ in range(2)]
    yc, xc = y.t().contiguous().t(), x.t().contiguous().t()
    q.adjoint_lstsq(A, yc, xc, xb, Ab[0], yb[0])
    for j in range(k):
        s = slice(j, j + 1)
        q.adjoint_lstsq(A, yc[:, s], xc[:, s], xb[:, s], Ab[1], yb[1][:, s])
    torch.cuda.synchronize()
    assert q.sync_status() == 0
    # the matrix products around the solves take other tiles for another k: n terms in each
    u = 2.0 ** -53 if dtype == "f64" else 2.0 ** -24
    assert (yb[0] - yb[1]).norm() <= 4 * n * u * A.norm() * (yb[1].norm() / A.norm() + xb.norm())
    q.close()
