"""A handle that met a breakdown factors the next matrix as a fresh handle does, bit for bit: with
the block pass, the tensor-core modes and panel widths that are not a multiple of a stage of K
(64 columns of 16-bit operands, 32 of TF32), whose second product reads columns behind the last
computed one.  The first matrix has entries above 16 and a zero column, or an infinite entry."""
import numpy as np
import pytest

from paper_2311_11943_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2311_11943_gb300 import binding as B  # noqa: E402


def factors(q, A):
    Ad = B.colmajor_empty(*A.shape, torch.float32)
    Ad.copy_(torch.from_numpy(A))
    q.encode(Ad)
    q.factor(0, -1)
    st = q.sync_status()
    Q, R = q.factors()
    return st, Q[:, : A.shape[1]].clone(), R.clone()


@pytest.mark.parametrize("bad", ["zero", "inf"])
@pytest.mark.parametrize("mma,b", [("3xtf32", 32), ("3xtf32", 96), ("3xtf32", 48), ("3xtf32", 120),
                                   ("bf16x3", 32), ("tf32", 48)])
def test_the_next_factorisation_is_that_of_a_fresh_handle(mma, b, bad):
    m, n = 520, 480
    A = synth.gaussian(m, n, 5) * 100.0
    A[:, 3] = 0.0
    if bad == "inf":
        A = synth.gaussian(m, n, 5) * 100.0
        A[17, 3] = np.inf
    good = synth.gaussian(m, n, 6)
    args = dict(dtype="f32", mma=mma, reorth_block=True, seed=3)
    q = B.CodedQR(m, n, 4, 4, 1, b, **args)
    assert factors(q, A)[0] == B.CQR_EBREAKDOWN
    st, Q, R = factors(q, good)
    q.close()
    q = B.CodedQR(m, n, 4, 4, 1, b, **args)
    st0, Q0, R0 = factors(q, good)
    q.close()
    assert st0 == 0 and st == 0
    assert torch.equal(Q, Q0) and torch.equal(R, R0)
