"""How the minibatch gradient is summed over its CTAs."""
import numpy as np
import pytest

from paper_2112_00864_gb300 import learned

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,tol", [(512, 1.6e-7), (513, 1.6e-7), (1024, 1.1e-7), (1216, 1.1e-7), (2433, 1.1e-7), (4099, 1.1e-7), (20000, 1.8e-7)])
def test_gradient_error(n, tol):
    """Against FP64 autograd, mean of five calls.  The rounding of the pairs' own
    values averages out (0.7e-7 of the norm at 1,024 pairs, less above, 1.5e-7 at a few hundred); what
    grows is the number of FP32 additions to a parameter's running sum, one per
    128 to 512 pairs, each within half of 2^-24 of it: 1.8e-7 at 20,000 pairs.
    One addition per 8 to 32 pairs gives 1.7e-7 to 3.6e-7 from 1,024 pairs on."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2112_00864_gb300 import bcfmm
    from paper_2112_00864_gb300.build import build
    build()
    gen = torch.Generator().manual_seed(n)
    params = torch.tensor(learned.init_params(3), device="cuda")
    feat = (torch.randn((n, 12), generator=gen) * 0.8).cuda()
    qhat = torch.rand((n, 16), generator=gen) + 0.2
    qhat = (qhat / qhat.sum(1, keepdim=True)).cuda().contiguous()
    chat = (0.03 * torch.randn((n,), generator=gen)).cuda()
    P = params.to(torch.bfloat16).double().requires_grad_(True)
    W1, b1, W2, b2, W3, b3 = torch.split(P, [768, 64, 4096, 64, 1024, 16])
    h = torch.nn.functional.gelu(feat.double() @ W1.view(64, 12).T + b1)
    h = torch.nn.functional.gelu(h @ W2.view(64, 64).T + b2)
    pred = ((h @ W3.view(16, 64).T + b3) * qhat.double()).sum(1)
    ref, = torch.autograd.grad(((pred - chat.double()) ** 2).mean(), P)
    err = []
    for _ in range(5):
        grad, loss = torch.empty_like(params), torch.empty(1, device="cuda")
        bcfmm.mlp_grad(params, feat, qhat, chat, grad, loss)
        err.append(((grad - ref).norm() / ref.norm()).item())
    assert np.mean(err) <= tol, err
