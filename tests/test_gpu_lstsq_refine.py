"""The tall solve by iterative refinement (cqr_lstsq.cu) against FP64 least squares: one CTA, several
CTAs with a ragged last one, vectors that are not a multiple of their padding, rows read from
global memory (too many for shared memory), several right-hand sides, y = 0.
Tolerance: n u kappa (1 + |G~|^2), the forward error of factors good to n u kappa through
I - Q_2^T Q_2, whose condition number is at most 1 + |G~|^2."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2311_11943_gb300 import binding as B  # noqa: E402


@pytest.mark.parametrize("m,n,p_r,p_c,f,dtype,mma", [
    (40, 8, 4, 4, 1, "f64", "simt"), (40, 8, 4, 4, 1, "f32", "simt"),
    (1003, 132, 6, 4, 2, "f64", "simt"), (1003, 132, 6, 4, 2, "f32", "3xtf32"),
    (2999, 516, 8, 6, 3, "f32", "3xtf32"), (4600, 3800, 5, 4, 2, "f32", "3xtf32")])
def test_tall_solve_matches_fp64_least_squares(m, n, p_r, p_c, f, dtype, mma):
    td = torch.float64 if dtype == "f64" else torch.float32
    g = torch.Generator(device="cuda").manual_seed(5)
    A = torch.randn((n, m), generator=g, device="cuda", dtype=td).t()
    y = torch.randn((3, m), generator=g, device="cuda", dtype=td).t()
    y[:, 1] = 0.0
    q = B.CodedQR(m, n, p_r, p_c, f, 64, dtype=dtype, mma=mma, nrhs_max=3, seed=4,
                  reorth_block=mma != "simt")
    q.encode(A)
    q.factor(0, -1)
    x = B.colmajor_empty(n, 3, td)
    q.solve_ls(y, x)
    torch.cuda.synchronize()
    assert q.sync_status() == 0
    Gt, _ = q.generator()
    q.close()
    A64, y64 = A.double(), y.double()
    Q, R = torch.linalg.qr(A64)
    ref = torch.linalg.solve_triangular(R, Q.t() @ y64, upper=True)
    s = torch.linalg.svdvals(R)
    u = (np.finfo(np.float64).eps if dtype == "f64" else np.finfo(np.float32).eps) / 2
    tol = n * u * (8 if mma == "3xtf32" else 1) * float(s[0] / s[-1]) * (1 + np.linalg.norm(Gt, 2) ** 2)
    err = torch.linalg.norm(x.double() - ref, dim=0)
    assert float(err[1]) == 0.0
    assert float(err[0] / torch.linalg.norm(ref[:, 0])) < tol
    assert float(err[2] / torch.linalg.norm(ref[:, 2])) < tol
