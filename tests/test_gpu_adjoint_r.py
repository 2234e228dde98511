"""The gradient of a loss in R on a tensor-core handle: R Rbar^T, which every later product builds on, is
an FP32 product.  2048 x 512, kappa = 4, against FP64: 3.9e-6 off with it in FP32 (what the
3xTF32 products behind it leave), 6.2e-6 with it in 3xTF32 too; the bound lies between."""
import pytest

from paper_2311_11943_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2311_11943_gb300.autograd import coded_lstsq  # noqa: E402


def test_gradient_of_a_loss_in_r():
    m, n, p = 2048, 512, 8
    A = torch.from_numpy(synth.kappa_matrix(m, n, 4.0, seed=5)).float().cuda().requires_grad_()
    y = torch.zeros(m, 1, device="cuda")
    W = torch.randn((n, n), generator=torch.Generator(device="cuda").manual_seed(1), device="cuda")
    # f = 0: G_0 is the identity
    _, R, _ = coded_lstsq(A, y, p, p, 0, 64, mma="3xtf32")
    got, = torch.autograd.grad((W * R).sum(), A)
    A64 = A.detach().double().requires_grad_()
    _, R64 = torch.linalg.qr(A64)
    d = torch.sign(torch.diagonal(R64)).detach()
    ref, = torch.autograd.grad((W.double() * torch.triu(d[:, None] * R64)).sum(), A64)
    assert float((got - ref).norm() / ref.norm()) < 5e-6
