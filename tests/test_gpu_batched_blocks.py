"""The batched panel in sub-blocks of 16 columns (cqr_batched.cu) against the oracle where it can go
wrong: ragged rows and columns, a cluster's CTA with few rows, panels cut by their width, nearly
dependent and strongly correlated columns (the column recurrence takes over inside the panel), a
zero column (the status of that instance alone).  Tolerance: 50 n u kappa, as for every batch."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2311_11943_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2311_11943_gb300 import binding as B  # noqa: E402

P_R, P_C, F, SEED = 8, 4, 2, 7


def to_dev(A):
    d = B.colmajor_empty(A.shape[0], A.shape[1], torch.float32)
    d.copy_(torch.from_numpy(A))
    return d


def inputs():
    rng = np.random.default_rng(3)
    A = [synth.gaussian(m, n, 20 + m) for m, n in ((65, 8), (259, 36), (1031, 68), (2050, 20))]
    c = synth.gaussian(700, 64, 1) + 2.0 * rng.standard_normal((700, 1))   # correlated
    d = synth.gaussian(901, 60, 2)
    d[:, 21::9] = d[:, 20::9][:, : d[:, 21::9].shape[1]] + 1e-2 * d[:, 21::9]  # nearly dependent
    return [np.asfortranarray(x.astype(np.float32).astype(np.float64)) for x in A + [c, d]]


@pytest.mark.parametrize("cluster,b", [(1, 16), (2, 32), (8, 64), (2, 20)])
def test_sub_block_panels_match_the_oracle(cluster, b):
    As = inputs()
    bt = B.CodedQRBatch([a.shape for a in As], P_R, P_C, F, b=0, seed=SEED)
    bt.set_tuning(cluster, [b] * len(As))
    bt.encode([to_dev(a) for a in As])
    bt.factor()
    torch.cuda.synchronize()
    st, bad, reorth = bt.sync_status()
    assert (st, bad) == (0, -1) and reorth > 0
    u = np.finfo(np.float32).eps / 2
    for i, a in enumerate(As):
        ref = O.run(a, P_R, P_C, F, b, seed=SEED)
        n = a.shape[1]
        tol = 50 * n * u * np.linalg.cond(a)
        Q, R = (t.double().cpu().numpy() for t in bt.factors(i))
        assert np.abs(Q[:, :n] - ref["Q"][:, :n]).max() < tol, i
        assert np.abs(R - ref["R"]).max() < tol * max(1.0, np.abs(ref["R"]).max()), i
    bt.close()


def test_a_zero_column_stops_its_instance_only():
    As = inputs()
    As[2][:, 33] = 0.0
    bt = B.CodedQRBatch([a.shape for a in As], P_R, P_C, F, b=0, seed=SEED)
    bt.encode([to_dev(a) for a in As])
    bt.factor()
    torch.cuda.synchronize()
    st, bad, _ = bt.sync_status()
    assert (st, bad) == (B.CQR_EBREAKDOWN, 2)
    ref = O.run(As[1], P_R, P_C, F, bt.tuning()[1][1], seed=SEED)
    R = bt.factors(1)[1].double().cpu().numpy()
    tol = 50 * As[1].shape[1] * np.finfo(np.float32).eps * np.linalg.cond(As[1])
    assert np.abs(R - ref["R"]).max() < tol * max(1.0, np.abs(ref["R"]).max())
    bt.close()
