"""Gradient and prediction kernels of the learned correction at the edges of
their tiles (pairs per CTA 8, 16, 32; 32 and 128) against FP64 autograd on the
BF16-rounded weights."""
import numpy as np
import pytest

from paper_2112_00864_gb300 import learned

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def bc():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2112_00864_gb300 import bcfmm
    from paper_2112_00864_gb300.build import build
    build()
    return bcfmm


@pytest.mark.parametrize("n", [1, 7, 8, 9, 31, 1216, 1217, 2432, 2433, 4099, 19455, 19456, 19457])
def test_against_fp64(bc, n):
    """FP32 products and sums of at most a few hundred terms a pair: 2e-6 of the
    largest value (predictions), 2e-5 of the gradient's norm (atomics over pairs)."""
    rng = np.random.default_rng(n)
    params = torch.tensor(learned.init_params(n % 97), device="cuda")
    feat = torch.tensor(rng.normal(0, 0.8, (n, 12)).astype(np.float32), device="cuda")
    qhat = torch.tensor(rng.uniform(0.2, 1.0, (n, 16)).astype(np.float32), device="cuda")
    qhat = (qhat / qhat.sum(1, keepdim=True)).contiguous()
    chat = torch.tensor(rng.normal(0, 0.03, n).astype(np.float32), device="cuda")
    P = params.to(torch.bfloat16).double().requires_grad_(True)
    W1, b1, W2, b2, W3, b3 = torch.split(P, [768, 64, 4096, 64, 1024, 16])
    h = torch.nn.functional.gelu(feat.double() @ W1.view(64, 12).T + b1)
    h = torch.nn.functional.gelu(h @ W2.view(64, 64).T + b2)
    pred = ((h @ W3.view(16, 64).T + b3) * qhat.double()).sum(1)
    loss = ((pred - chat.double()) ** 2).mean()
    g, = torch.autograd.grad(loss, P)
    out, grad, l = torch.empty_like(chat), torch.full_like(params, 7.0), torch.full((1,), 7.0, device="cuda")
    bc.mlp_predict(params, feat, qhat, out)
    bc.mlp_grad(params, feat, qhat, chat, grad, l)
    assert (out - pred).abs().max() <= 2e-6 * pred.abs().max().clamp(min=0.1)
    assert abs(l.item() - loss.item()) <= 2e-5 * loss.item()
    assert (grad - g).norm() <= 2e-5 * g.norm()
