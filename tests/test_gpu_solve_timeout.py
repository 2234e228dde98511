"""The waits of the tall solve by refinement (cqr_lstsq.cu) are bounded like the panel's (needs a GB300).
Nothing here faults or hangs a GPU: the launch is correct, only the bound of its waits between
CTAs is set to a few hundred SM cycles, so that its first sum runs out; every CTA leaves and the
status comes back within a second.  With the default bound the same factors solve again."""
import time

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2311_11943_gb300 import binding as B  # noqa: E402


@pytest.mark.parametrize("dtype,k", [("f64", 1), ("f32", 1), ("f32", 6)])
def test_expired_wait_of_the_solve(dtype, k):
    m, n = 3000, 480
    td = torch.float64 if dtype == "f64" else torch.float32
    g = torch.Generator(device="cuda").manual_seed(8)
    A = torch.randn((n, m), generator=g, device="cuda", dtype=td).t()
    y = torch.randn((k, m), generator=g, device="cuda", dtype=td).t()
    x, ref = B.colmajor_empty(n, k, td), B.colmajor_empty(n, k, td)
    q = B.CodedQR(m, n, 6, 4, 2, 64, dtype=dtype, nrhs_max=k, seed=4)
    q.encode(A)
    q.factor(0, -1)
    q.solve_ls(y, ref)
    assert q.sync_status() == 0
    q.set_wait_limit(200)
    t0 = time.perf_counter()
    q.solve_ls(y, x)
    st = q.sync_status()
    assert st == B.CQR_ETIMEOUT, B.errstr(st)
    assert time.perf_counter() - t0 < 1.0
    q.set_wait_limit(0)
    q.solve_ls(y, x)
    assert q.sync_status() == 0
    assert torch.equal(x, ref)
    q.close()
