"""FP32 sums over the interaction list at order 8.

Orders 8 and 9 both keep a compensated sum over a target's list, entry by entry
(order 8 in the sibling-group kernel, order 9 in the kernel with one CTA per
target), so apart from the truncation, which the FP64 form of the same order
shares, the two orders are rounded alike.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_order8_is_as_accurate_as_order9():
    """Positive sources on one side, potentials on the other: no near field, long
    sums of one sign.  The error of order 8 is at most 1.25 times that of order 9
    (the two differ by a few of some hundred roundings; plain FP32 sums over the
    chunks of the list give 1.6 times)."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2112_00864_gb300 import bcfmm
    from paper_2112_00864_gb300.build import build
    from paper_2112_00864_gb300.inputs import ball_bc_mesh
    build()
    m = ball_bc_mesh(level=3, radial=0.5)
    c = m.verts[m.tets].mean(1)
    far = c[:, 0] > 0.4
    base = np.where(c[:, 0] < -0.4, 1.0 + 0.3 * np.sin(5 * c[:, 1]), 0.0)
    f = base * np.random.default_rng(0).uniform(0.5, 1.5, (4, m.ntet))
    err = {}
    for q in (8, 9):
        u = {}
        for prec in ("fp64", "fp32"):
            ctx = bcfmm.Context.from_mesh(m, p=q, eta0=0.6, leaf_size=64, precision=prec, near_n=1, near_k=0)
            ctx.set_density(bcfmm.VOLUME, f)
            u[prec] = ctx.eval_vtv().cpu().numpy()[:, far]
            ctx.close()
        err[q] = np.sqrt(np.mean((u["fp32"] / u["fp64"] - 1) ** 2))
    assert err[8] <= 1.25 * err[9], err
