"""A last panel narrower than b on the tensor-core update: the operand planes keep the stride of
their tensor maps.  The checksum columns of the coded Q lie in the span of the factored columns, so
the last update leaves only rounding there: per panel, chains of 16-term steps over the m rows
(three products each with split operands; with one TF32 product 2^-10 of the terms, in norm)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2311_11943_gb300 import binding as B  # noqa: E402


@pytest.mark.parametrize("mma,unit", [("3xtf32", 2.0 ** -23), ("bf16x3", 2.0 ** -15), ("tf32", 2.0 ** -10)])
@pytest.mark.parametrize("n,b", [(200, 128), (440, 192), (300, 64)])
def test_checksum_columns_vanish_after_a_narrow_last_panel(mma, unit, n, b):
    p, f, m = 4, 1, 640
    q = B.CodedQR(m, n, p, p, f, b, dtype="f32", mma=mma, reorth_block=True, seed=3)
    rng = np.random.default_rng(n)
    A = B.colmajor_empty(m, n, torch.float32)
    A.copy_(torch.from_numpy(rng.standard_normal((m, n)).astype(np.float32)))
    q.encode(A)
    Q, _ = q.factors()
    before = Q[:, n:].double().norm(dim=0).clone()
    q.factor()
    Q, _ = q.factors()
    left = Q[:, n:].double().norm(dim=0)
    torch.cuda.synchronize()
    steps = 3 * (m // p * (p + f)) / 16 + 24 if mma == "3xtf32" else 1
    bound = -(-n // b) * steps * unit * (b ** 0.5 if mma != "3xtf32" else 1) * before
    assert Q.shape[1] > n and (before > 0).all()
    assert (left <= bound).all(), (left / before).max().item()
    q.close()
