"""The 3xTF32 update where a column's large part is taken out exactly: what is left keeps its digits.
The first panel is the identity on its rows, the columns behind it hold integers there (up to 2^g) and
N(0,1) entries below; R's first rows are those integers, the rest is the QR of what lies below.
Tolerance: n u kappa of that part, u = 8 times FP32's (as for every 3xTF32 factor)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2311_11943_gb300 import binding as B  # noqa: E402

U3X = 8 * np.finfo(np.float32).eps / 2


@pytest.mark.parametrize("g", [0, 10, 24, 40])
@pytest.mark.parametrize("b", [64, 128])
@pytest.mark.parametrize("mma", ["simt", "3xtf32"])
def test_what_is_left_of_a_column_keeps_its_digits(mma, b, g):
    m, n = 900, 500
    rng = np.random.default_rng(3)
    A = np.zeros((m, n))
    A[:b, :b] = np.eye(b)
    A[:b, b:] = rng.integers(-1000, 1001, (b, n - b)) * 2.0 ** (g - 10)
    Z = rng.standard_normal((m - b, n - b)).astype(np.float32).astype(np.float64)
    A[b:, b:] = Z
    q = B.CodedQR(m, n, 1, 1, 0, b, dtype="f32", mma=mma, seed=1)
    Ad = B.colmajor_empty(m, n, torch.float32)
    Ad.copy_(torch.from_numpy(A))
    q.encode(Ad)
    q.factor(0, -1)
    Q, R = q.factors()
    torch.cuda.synchronize()
    st = q.sync_status()
    Q, R = Q.double().cpu().numpy(), R.double().cpu().numpy()
    q.close()
    assert st == 0
    Q0, R0 = np.linalg.qr(Z)
    d = np.sign(np.diag(R0))
    tol = n * U3X * np.linalg.cond(Z)
    assert np.abs(R[:b, b:n] - A[:b, b:]).max() <= 0.0 if g else True
    assert np.abs(R[b:n, b:n] - d[:, None] * R0).max() < tol * np.abs(R0).max()
    assert np.abs(Q[b:m, b:n] - Q0 * d).max() < tol
