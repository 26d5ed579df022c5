"""The gradient of a training's minibatch repeats bit for bit."""
import pytest

from paper_2112_00864_gb300 import learned

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 256, 257, 777, 1024])
def test_same_sums_in_every_call(n):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2112_00864_gb300 import bcfmm
    from paper_2112_00864_gb300.build import build
    build()
    gen = torch.Generator().manual_seed(n)
    params = torch.tensor(learned.init_params(5), device="cuda")
    feat = (torch.randn((n, 12), generator=gen) * 0.8).cuda()
    qhat = torch.rand((n, 16), generator=gen).cuda() + 0.2
    chat = (0.03 * torch.randn((n,), generator=gen)).cuda()
    ref = None
    for _ in range(50):
        grad, loss = torch.empty_like(params), torch.empty(1, device="cuda")
        bcfmm.mlp_grad(params, feat, qhat, chat, grad, loss)
        if ref is None:
            ref = (grad, loss)
        assert torch.equal(grad, ref[0]) and torch.equal(loss, ref[1])
