"""The FP64 trailing update by integer slices on the tensor cores (cqr_f64_gemm.cu) against products in
extended precision where numpy has them (else FP64): one panel of an uncoded problem, Rbar and
the updated columns.  Ragged rows, panel widths and trailing widths, columns of very different
size, a zero column, the largest magnitude at a power of two; an infinite entry must reach the status.
Bounds: an FP64 product sum of K terms is off by at most K u |q| |b| (u = 2^-53), the update by
(b + 2) u (|C| + |Q| |R|); the slices add at most 2 u of the largest products, and
max |q| max |b| <= |q| |b|."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2311_11943_gb300 import binding as B  # noqa: E402

U = 2.0 ** -53


def one_panel(A, b):
    m, n = A.shape
    q = B.CodedQR(m, n, 1, 1, 0, b, dtype="f64", seed=1)
    Ad = B.colmajor_empty(m, n, torch.float64)
    Ad.copy_(torch.from_numpy(A))
    q.encode(Ad)
    q.profile_read()
    q.factor(0, 1)
    Q, R = q.factors()
    torch.cuda.synchronize()
    st, prof = q.sync_status(), q.profile_read()
    Q, R = Q.cpu().numpy(), R.cpu().numpy()
    q.close()
    return Q, R, st, prof


@pytest.mark.parametrize("m,n,b", [(3001, 613, 33), (2049, 260, 128), (9000, 259, 130),
                                   (1111, 1100, 64)])
def test_integer_slices_match_extended_products(m, n, b):
    rng = np.random.default_rng(m)
    A = rng.standard_normal((m, n)) * 10.0 ** rng.uniform(-9, 9, n)[None, :]
    A[:, n - 2] = 0.0
    A[:, n - 3] = np.sign(A[:, n - 3])
    A = np.asfortranarray(A)
    Q, R, st, prof = one_panel(A, b)
    assert st == 0
    assert prof["tc_rbar"][1] > 0 and prof["gemm_rbar_simt"][1] == 0  # the path under test ran
    cols = np.unique(np.r_[b, b + 1, n - 3, n - 2, n - 1, rng.integers(b, n, 6)])
    Qb, Ac = Q[:, :b].astype(np.longdouble), A[:, cols].astype(np.longdouble)
    Rr = Qb.T @ Ac
    Rc = R[:b][:, cols].astype(np.longdouble)
    nq, na = np.linalg.norm(Q[:, :b], axis=0), np.linalg.norm(A[:, cols], axis=0)
    assert (np.abs(Rc - Rr) <= (m + 2) * U * np.outer(nq, na)).all()
    assert (Rc[:, cols == n - 2] == 0).all()
    scale = np.abs(Ac) + np.abs(Qb) @ np.abs(Rc)
    # the slices: 2 u of the largest product per term
    big = np.abs(Q[:, :b]).max(1)[:, None] * np.abs(R[:b][:, cols]).max(0)[None, :]
    assert (np.abs(Q[:, cols] - (Ac - Qb @ Rc)) <= (b + 2) * U * scale + 2 * b * U * big).all()


def test_an_infinite_entry_is_reported():
    rng = np.random.default_rng(1)
    A = np.asfortranarray(rng.standard_normal((2049, 256)))
    A[77, 200] = np.inf
    q = B.CodedQR(2049, 256, 1, 1, 0, 128, dtype="f64", seed=1)
    Ad = B.colmajor_empty(2049, 256, torch.float64)
    Ad.copy_(torch.from_numpy(A))
    q.encode(Ad)
    q.factor(0, -1)
    assert q.sync_status() == B.CQR_EBREAKDOWN
    q.close()
