"""The FP64 update by integer slices over more columns than it holds digits of (1 GB: 3776 columns of
20,000 rows), so in two blocks: Rbar and the updated columns on both sides of the boundary against
FP64 products.  Bounds as in test_gpu_f64_update.py (m u |q| |a|, and (b + 2) u (|C| + |Q| |R|) with 2 b u of
the largest products), twice for the FP64 reference's own rounding."""
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2311_11943_gb300 import binding as B  # noqa: E402

U = 2.0 ** -53


def test_two_blocks_of_columns():
    m, n, b = 20000, 4200, 72
    block = (1 << 30) // (7 * 20032 * 2) // 64 * 64
    assert b < block < n - b
    g = torch.Generator(device="cuda").manual_seed(6)
    A = torch.randn((n, m), generator=g, device="cuda", dtype=torch.float64).t()
    q = B.CodedQR(m, n, 1, 1, 0, b, dtype="f64", seed=1)
    q.encode(A)
    q.profile_read()
    q.factor(0, 1)
    launches = q.profile_read()["tc_update"][1]
    Q, R = q.factors()
    torch.cuda.synchronize()
    assert q.sync_status() == 0 and launches == 4  # two blocks, digits and product each
    Qb, Rb = Q[:, :b], R[:b, b:n]
    ref = Qb.t() @ A[:, b:]
    nq, na = torch.linalg.norm(Qb, dim=0), torch.linalg.norm(A[:, b:], dim=0)
    assert bool(((Rb - ref).abs() <= 2 * (m + 2) * U * nq[:, None] * na[None, :]).all())
    C = A[:, b:] - Qb @ Rb
    scale = A[:, b:].abs() + Qb.abs() @ Rb.abs()
    big = Qb.abs().amax(1)[:, None] * Rb.abs().amax(0)[None, :]
    assert bool(((Q[:, b:] - C).abs() <= 2 * (b + 2) * U * scale + 2 * b * U * big).all())
    q.close()
