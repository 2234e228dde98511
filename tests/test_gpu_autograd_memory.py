"""The differentiable batch takes its workspaces from the caller's stream: calls one after the other
take the same blocks, although each has side streams of its own."""
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2311_11943_gb300 import binding as B  # noqa: E402
from paper_2311_11943_gb300.autograd import coded_lstsq  # noqa: E402


def test_calls_one_after_the_other_take_the_same_workspaces():
    count, m, n = 12, 4096, 512
    torch.cuda.empty_cache()
    g = torch.Generator(device="cuda").manual_seed(2)
    A = torch.randn((count, m, n), generator=g, device="cuda", requires_grad=True)
    y = torch.randn((count, m, 1), generator=g, device="cuda")
    q = B.CodedQR(m, n, 8, 8, 1, 64, dtype="f32", mma="3xtf32")
    ws = B.coded_qr_workspace_size(q.cfg)
    q.close()
    grads = []
    for _ in range(3):
        Q, R, x = coded_lstsq(A, y, 8, 8, 1, 64)
        grads.append(torch.autograd.grad(Q.sum() + x.sum(), A)[0])
        del Q, R, x
    torch.cuda.synchronize()
    mine = torch.cuda.current_stream().cuda_stream
    blocks = [(s["stream"], b["size"]) for s in torch.cuda.memory_snapshot() for b in s["blocks"]]
    big = [s for s, size in blocks if ws <= size < 2 * ws and size < 4 * count * m * n]
    assert all(s == mine for s in big) and len(big) <= count + 1
    assert torch.equal(grads[0], grads[1]) and torch.equal(grads[0], grads[2])


def test_an_allocation_that_cannot_be_had_keeps_its_error():
    from paper_2311_11943_gb300 import autograd
    cfg = B.make_config(400000, 300000, 8, 8, 1, 64, dtype="f32", mma="3xtf32")  # a matrix of 480 GB
    with pytest.raises(B.CodedQRError) as e:
        autograd._workspaces(1, cfg)
    assert e.value.status == B.CQR_ENOMEM
