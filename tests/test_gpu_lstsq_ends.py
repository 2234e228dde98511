"""How the tall solve ends (cqr_lstsq.cu, and the conjugate gradients for long vectors): what is not
finite comes out as NaN and not as a finite x, and a correction that makes the residual larger is not
kept."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2311_11943_gb300 import binding as B  # noqa: E402


def handle(m, n, f, dtype, k=1):
    td = torch.float64 if dtype == "f64" else torch.float32
    g = torch.Generator(device="cuda").manual_seed(5)
    A = torch.randn((n, m), generator=g, device="cuda", dtype=td).t()
    y = torch.randn((k, m), generator=g, device="cuda", dtype=td).t()
    q = B.CodedQR(m, n, 6, 4, f, 32, dtype=dtype, nrhs_max=k, seed=4)
    q.encode(A)
    q.factor(0, -1)
    return q, A, y, B.colmajor_empty(n, k, td)


@pytest.mark.parametrize("dtype", ["f64", "f32"])
@pytest.mark.parametrize("f", [0, 2])
@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
def test_a_right_hand_side_that_is_not_finite(dtype, f, bad):
    q, A, y, x = handle(1003, 96, f, dtype, 2)
    y[7, 1] = bad
    q.solve_ls(y, x)
    torch.cuda.synchronize()
    assert q.sync_status() == 0
    assert bool(torch.isfinite(x[:, 0]).all())
    assert not bool(torch.isfinite(x[:, 1]).any())
    q.close()


def test_a_right_hand_side_that_is_not_finite_with_long_vectors():
    # 8192 columns: the vectors of the refinement do not fit shared memory
    m, n = 8448, 8192
    A = torch.zeros((n, m), device="cuda").t()
    A[:n].fill_diagonal_(1.0)
    A[n:] = 0.01
    q = B.CodedQR(m, n, 4, 4, 1, 256, dtype="f32", mma="3xtf32", seed=4)
    q.encode(A)
    q.factor(0, -1)
    y = torch.ones((1, m), device="cuda").t()
    x = B.colmajor_empty(n, 1, torch.float32)
    q.solve_ls(y, x)
    assert q.sync_status() == 0
    assert bool(torch.isfinite(x).all())
    y[5, 0] = float("nan")
    q.solve_ls(y, x)
    assert q.sync_status() == 0
    assert not bool(torch.isfinite(x).any())
    q.close()


@pytest.mark.parametrize("dtype", ["f64", "f32"])
def test_a_checksum_row_that_is_not_finite(dtype):
    q, A, y, x = handle(1003, 96, 2, dtype)
    Q, _ = q.factors()
    Q[q.geo["m_pad"] + 3, 11] = float("nan")
    q.solve_ls(y, x)
    torch.cuda.synchronize()
    assert not bool(torch.isfinite(x).any())
    q.close()


@pytest.mark.parametrize("dtype", ["f64", "f32"])
@pytest.mark.parametrize("scale", [1.3, 2.0, 3.0])
def test_a_correction_that_makes_the_residual_larger_is_not_kept(dtype, scale):
    # checksum rows times `scale`: I - Q_2^T Q_2 is indefinite and conjugate gradients break down
    q, A, y, x = handle(1003, 96, 2, dtype)
    Q, R = q.factors()
    g = q.geo
    Q2 = Q[g["m_pad"]: g["M"], :96]
    Q2 *= scale
    q.solve_ls(y, x)
    torch.cuda.synchronize()
    z = Q[:1003, :96].double().t() @ y.double()
    w = torch.triu(R[:96, :96]).double() @ x.double()
    Q2 = Q2.double()
    r = z - (w - Q2.t() @ (Q2 @ w))
    # w = 0 leaves |z|; x in the storage precision through R (condition number below 2)
    u = np.finfo(np.float64 if dtype == "f64" else np.float32).eps
    lim = float(torch.linalg.norm(z)) + 96 * 4 * u * float(torch.linalg.norm(w)) * (1 + scale ** 2)
    assert float(torch.linalg.norm(r)) <= lim
    q.close()
