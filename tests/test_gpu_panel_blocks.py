"""The panel in sub-blocks (cqr_panel_blk.cu: one reduction per 16 FP32 or 8 FP64 columns) against
the oracle's column recurrence, at the edges of its tiles: rows that leave a slice ragged, one
CTA, sub-blocks cut by the panel's width, columns that fail the ICGS test (projected once more as
a block), nearly dependent columns (the column recurrence inside the kernel), a zero column.
Tolerance: n u kappa, as for every Gram-Schmidt factor."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2311_11943_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2311_11943_gb300 import binding as B  # noqa: E402


def correlated(m, n, seed):
    """Columns with a common direction of twice their own size: about half of each column's
    squared norm goes with its first projections, so most columns fail the ICGS test."""
    rng = np.random.default_rng(seed)
    A = rng.standard_normal((m, n))
    return A + 2.0 * rng.standard_normal((m, 1))


def dependent(m, n, seed):
    A = synth.gaussian(m, n, seed)
    A[:, 1::7] = A[:, 0::7][:, : A[:, 1::7].shape[1]] + 1e-3 * A[:, 1::7]
    return A


KINDS = {"kappa": lambda m, n, s: synth.kappa_matrix(m, n, 10.0, s), "correlated": correlated,
         "dependent": dependent}


@pytest.mark.parametrize("kind", list(KINDS))
@pytest.mark.parametrize("dtype", ["f64", "f32"])
@pytest.mark.parametrize("m,n,p_r,p_c,f,b", [(21, 8, 4, 4, 1, 8), (203, 96, 8, 4, 2, 20),
                                             (331, 60, 5, 4, 1, 1), (1001, 120, 7, 4, 0, 120),
                                             (2500, 160, 10, 4, 2, 64)])
def test_sub_block_panel_matches_the_column_recurrence(kind, dtype, m, n, p_r, p_c, f, b):
    A = KINDS[kind](m, n, 11)
    td = torch.float64 if dtype == "f64" else torch.float32
    A = np.asfortranarray(A.astype(np.float32).astype(np.float64))  # the same values on both sides
    q = B.CodedQR(m, n, p_r, p_c, f, b, dtype=dtype, seed=3)
    Ad = B.colmajor_empty(m, n, td)
    Ad.copy_(torch.from_numpy(A))
    q.encode(Ad)
    q.factor(0, -1)
    Qc, Rc = q.factors()
    torch.cuda.synchronize()
    assert q.sync_status() == 0
    Q, R, st = Qc.double().cpu().numpy(), Rc.double().cpu().numpy(), q.stats()
    q.close()
    ref = O.run(A, p_r, p_c, f, b, seed=3)
    u = (np.finfo(np.float64).eps if dtype == "f64" else np.finfo(np.float32).eps) / 2
    tol = n * u * np.linalg.cond(A)
    assert np.abs(R - ref["R"]).max() < tol * max(1.0, np.abs(ref["R"]).max())
    assert np.abs(Q[: ref["geom"].M, :n] - ref["Q"][:, :n]).max() < tol
    if dtype == "f64":  # the test is taken on the same quantity: borderline columns apart
        assert abs(st["n_reorth"] - ref["n_reorth"]) <= 1 + n // 20
    if kind != "kappa" and b > 1 and n > 8:
        assert st["n_reorth"] > 0


@pytest.mark.parametrize("dtype", ["f64", "f32"])
@pytest.mark.parametrize("col", [0, 5, 19])
def test_zero_column_breaks_down(dtype, col):
    A = synth.gaussian(200, 40, 5)
    A[:, col] = 0.0
    td = torch.float64 if dtype == "f64" else torch.float32
    q = B.CodedQR(200, 40, 4, 4, 1, 20, dtype=dtype, seed=3)
    Ad = B.colmajor_empty(200, 40, td)
    Ad.copy_(torch.from_numpy(A))
    q.encode(Ad)
    q.factor(0, -1)
    assert q.sync_status() == B.CQR_EBREAKDOWN
    # the handle goes on with a new matrix
    Ad.copy_(torch.from_numpy(synth.gaussian(200, 40, 6)))
    q.encode(Ad)
    q.factor(0, -1)
    assert q.sync_status() == 0
    q.close()
