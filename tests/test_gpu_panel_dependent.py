"""Nearly dependent columns in the sub-block panel (cqr_panel_blk.cu): columns that repeat the one before
to within eps, and columns that are all one direction to within eps, from what a second projection
mends to below the rounding of the storage type; ICGS and MGS, ragged rows and widths.
Bounds: A = Q R to n u (each column takes at most n projections); Q^T Q = I to 4 n u within a panel
while the part that is left of a column is well above its rounding (ICGS, "twice is enough").
Without the second projection (MGS) equal columns may leave nothing at all: a breakdown.
Time: such columns cost at most four times what N(0,1) columns do."""
import numpy as np
import pytest

from paper_2311_11943_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2311_11943_gb300 import binding as B  # noqa: E402


def pairs(m, n, eps, seed):
    A = synth.gaussian(m, n, seed)
    A[:, 1::2] = A[:, 0::2][:, : n // 2] + eps * A[:, 1::2]
    return A


def one_direction(m, n, eps, seed):
    A = synth.gaussian(m, n, seed)
    return A[:, :1] + eps * A


@pytest.mark.parametrize("panel", ["icgs", "mgs"])
@pytest.mark.parametrize("dtype", ["f64", "f32"])
@pytest.mark.parametrize("kind", [pairs, one_direction])
@pytest.mark.parametrize("eps", [1e-1, 1e-2, 1e-3, 1e-5, 3e-8, 1e-12])
@pytest.mark.parametrize("m,n,b", [(1003, 120, 40), (2500, 160, 160)])
def test_nearly_dependent_columns(m, n, b, eps, kind, dtype, panel):
    td = torch.float64 if dtype == "f64" else torch.float32
    u = (np.finfo(np.float64).eps if dtype == "f64" else np.finfo(np.float32).eps) / 2
    A = kind(m, n, eps, 11).astype(np.float32 if dtype == "f32" else np.float64).astype(np.float64)
    q = B.CodedQR(m, n, 5, 4, 1, b, dtype=dtype, seed=3, panel=panel)
    Ad = B.colmajor_empty(m, n, td)
    Ad.copy_(torch.from_numpy(A))
    q.encode(Ad)
    q.factor(0, -1)
    Q, R = q.factors()
    torch.cuda.synchronize()
    st = q.sync_status()
    if panel == "mgs" and eps < u and st == B.CQR_EBREAKDOWN:
        q.close()
        return
    assert st == 0
    Q, R = Q[:, :n].double().cpu().numpy(), R[:n, :n].double().cpu().numpy()
    q.close()
    assert np.linalg.norm(A - Q[:m] @ R) < n * u * np.linalg.norm(A)
    if panel == "icgs" and eps > 1e3 * u and b >= n:
        assert np.abs(Q.T @ Q - np.eye(n)).max() < 4 * n * u


@pytest.mark.parametrize("panel", ["icgs", "mgs"])
def test_nearly_dependent_columns_cost_little_more(panel):
    m, n = 4096, 1024
    q = B.CodedQR(m, n, 8, 4, 1, 128, dtype="f32", mma="3xtf32", seed=3, panel=panel)
    ms = []
    for A in (synth.gaussian(m, n, 1), pairs(m, n, 1e-3, 1)):
        Ad = B.colmajor_empty(m, n, torch.float32)
        Ad.copy_(torch.from_numpy(A))
        best = np.inf
        for _ in range(4):
            q.encode(Ad)
            a, b = torch.cuda.Event(True), torch.cuda.Event(True)
            a.record()
            q.factor(0, -1)
            b.record()
            torch.cuda.synchronize()
            best = min(best, a.elapsed_time(b))
        ms.append(best)
    q.close()
    assert ms[1] < 4 * ms[0], ms
