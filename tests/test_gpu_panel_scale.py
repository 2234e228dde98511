"""The sub-block panel does not depend on the size of its columns: a matrix times a power of two gives
the same Q and stats and that power of two times R, bit for bit, also where the squares of the
columns leave the range of a float (2^-80, 2^80) and where columns are nearly dependent, so that
the test of what a sub-block amplifies decides which columns go one at a time."""
import numpy as np
import pytest

from paper_2311_11943_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2311_11943_gb300 import binding as B  # noqa: E402


def dependent(m, n, seed):
    A = synth.gaussian(m, n, seed)
    A[:, 1::7] = A[:, 0::7][:, : A[:, 1::7].shape[1]] + 1e-5 * A[:, 1::7]
    return A


def factors(A, shape, dtype):
    m, n, p_r, p_c, f, b = shape
    td = torch.float64 if dtype == "f64" else torch.float32
    q = B.CodedQR(m, n, p_r, p_c, f, b, dtype=dtype, seed=3)
    Ad = B.colmajor_empty(m, n, td)
    Ad.copy_(torch.from_numpy(A))
    q.encode(Ad)
    q.factor(0, -1)
    Q, R = q.factors()
    torch.cuda.synchronize()
    assert q.sync_status() == 0
    out = Q[:, :n].double().cpu().numpy(), R.double().cpu().numpy(), q.stats()["n_reorth"]
    q.close()
    return out


@pytest.mark.parametrize("dtype,e", [("f64", -80), ("f64", 80), ("f64", -200), ("f32", -20), ("f32", 20)])
@pytest.mark.parametrize("kind", ["kappa", "dependent"])
@pytest.mark.parametrize("shape", [(203, 96, 8, 4, 2, 20), (2049, 260, 3, 4, 1, 128)])
def test_a_power_of_two_changes_nothing_else(shape, kind, dtype, e):
    m, n = shape[:2]
    A = dependent(m, n, 7) if kind == "dependent" else synth.kappa_matrix(m, n, 1e3, 7)
    Q, R, k = factors(A, shape, dtype)
    Qs, Rs, ks = factors(np.ldexp(A, e), shape, dtype)
    assert k == ks
    assert np.array_equal(Q, Qs)
    assert np.array_equal(np.ldexp(R, e), Rs)
