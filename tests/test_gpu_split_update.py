"""The 3xTF32-grade trailing update by scaled FP16 halves (cqr_tc_gemm.cu): one panel of an uncoded
problem.  With a panel of unit vectors, Rbar is the panel's rows of the trailing columns and the
update leaves zeros there and every other entry as it was: the split itself is seen, entry by
entry.  Two halves of 11 bits are off by 2^-22 of an entry and, below the subnormal step, by
2^-25 of a column scaled to a norm of at least 2^9; the unit's own rounding is 2^-23.  Ragged
rows, panel and trailing widths, column norms over the whole FP32 range, a zero column; an
infinite entry spoils its own column only.  A random panel against extended precision: K terms in
FP32 chains of 16-term steps, three products each."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2311_11943_gb300 import binding as B  # noqa: E402


def one_panel(A, b, t1=1, reorth=False):
    m, n = A.shape
    q = B.CodedQR(m, n, 1, 1, 0, b, dtype="f32", mma="3xtf32", reorth_block=reorth, seed=1)
    Ad = B.colmajor_empty(m, n, torch.float32)
    Ad.copy_(torch.from_numpy(np.ascontiguousarray(A)))
    q.encode(Ad)
    q.factor(0, t1)
    Q, R = q.factors()
    torch.cuda.synchronize()
    Q, R = Q.cpu().numpy().astype(np.float64), R.cpu().numpy().astype(np.float64)
    q.close()
    return Q, R


def trailing(rng, m, n):
    A = rng.standard_normal((m, n)) * 2.0 ** rng.uniform(-100, 100, n)[None, :]
    A[:, n - 2] = 0.0
    return A.astype(np.float32)


@pytest.mark.parametrize("m,n,b", [(1000, 333, 32), (517, 300, 128), (901, 641, 256), (300, 260, 96)])
def test_split_is_exact_to_its_bits(m, n, b):
    rng = np.random.default_rng(m)
    A = trailing(rng, m, n)
    rows = np.sort(rng.permutation(m)[:b])
    A[:, :b] = 0.0
    A[rows, np.arange(b)] = 2.0 ** rng.integers(-20, 20, b)
    Q, R = one_panel(A, b)
    T = A[:, b:].astype(np.float64)
    tol = 2.0 ** -21 * np.abs(T) + 2.0 ** -33 * np.linalg.norm(T, axis=0)[None, :]
    assert (np.abs(R[:b, b:n] - T[rows]) <= tol[rows]).all()
    keep = np.ones(m, bool)
    keep[rows] = False
    assert (Q[:m, b:n][keep] == T[keep]).all()
    assert (np.abs(Q[rows, b:n]) <= 2 * tol[rows]).all()


@pytest.mark.parametrize("m,n,b", [(1000, 333, 32), (901, 641, 256)])
def test_products_match_extended_precision(m, n, b):
    rng = np.random.default_rng(m + 1)
    A = trailing(rng, m, n)
    A[:, :b] = rng.standard_normal((m, b))
    A[3, n - 1] = np.inf
    Q, R = one_panel(A, b)
    assert not np.isfinite(Q[:m, n - 1]).all()
    A, Rc = A[:, :n - 1].astype(np.longdouble), R[:b, b:n - 1].astype(np.longdouble)
    T, Qb = A[:, b:], Q[:m, :b].astype(np.longdouble)
    na = np.linalg.norm(T.astype(np.float64), axis=0)[None, :]
    assert np.isfinite(R[:b, :n - 1]).all() and np.isfinite(Q[:m, :n - 1]).all()
    assert (np.abs(Rc - Qb.T @ T) <= (3 * m / 16 + 24) * 2.0 ** -23 * na).all()
    assert (np.abs(Q[:m, b:n - 1] - (T - Qb @ Rc)) <= (3 * b / 16 + 8) * 2.0 ** -23 * na).all()


def test_block_pass_scales_shrunk_columns():
    """Second panel = first panel's span plus a part 2^-12 as large: after the block pass it is
    orthogonal to the first to FP32 accuracy of what is left (16-term steps over m rows)."""
    m, b = 700, 64
    rng = np.random.default_rng(5)
    A = rng.standard_normal((m, 2 * b))
    A[:, b:] = A[:, :b] @ rng.standard_normal((b, b)) / 8 + 2.0 ** -12 * A[:, b:]
    Q, _ = one_panel(A.astype(np.float32), b, t1=2, reorth=True)
    S = Q[:m, :b].T @ Q[:m, b:2 * b]
    assert np.abs(S).max() <= (3 * m / 16 + 24) * 2.0 ** -23
    assert np.linalg.norm(S) <= 32 * b * 2.0 ** -24
