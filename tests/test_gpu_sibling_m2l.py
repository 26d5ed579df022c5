"""The sibling-group M2L (Taylor form) against the FP64 CPU oracle's FMM with
the same tree and orders: every order the kernel is instantiated for, the
first one past it, groups of one to eight siblings and ragged last chunks."""
import numpy as np
import pytest

import oracle as O
from paper_2112_00864_gb300.inputs import ball_bc_mesh, cube_bc_mesh, densities

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


@pytest.mark.parametrize("q", [1, 2, 3, 4, 5, 6, 7, 8, 9])
@pytest.mark.parametrize("mesh,leaf,eta0", [("cube", 24, 0.5), ("ball", 9, 0.7)])
def test_every_order_against_oracle(bc, q, mesh, leaf, eta0):
    """FP64: rounding of sums of at most a few thousand terms, 1e-12 of the
    result's norm; FP32: 2^-24 per product and per chunk sum, the norms of the
    terms within ten times the result's, 3e-6."""
    m = cube_bc_mesh(0.25, 0.25) if mesh == "cube" else ball_bc_mesh(level=1, radial=0.6)
    f, g = densities(m, "random", ndens=3, seed=q)
    for task, dens, kind in (("vtv", f, 0), ("vtb", f, 0), ("btv", g, 1)):
        ref = np.concatenate([np.atleast_2d(O.fmm(task, m, dens[i:i + 1], p=q, leaf_size=leaf, eta0=eta0)) for i in range(3)])
        for prec, tol in (("fp64", 1e-12), ("fp32", 3e-6)):
            ctx = bc.Context.from_mesh(m, p=q, leaf_size=leaf, eta0=eta0, precision=prec)
            ctx.set_density(kind, dens)
            u = ctx.eval(task).cpu().numpy()
            ctx.close()
            assert np.linalg.norm(u - ref) <= tol * np.linalg.norm(ref), (task, prec, np.linalg.norm(u - ref) / np.linalg.norm(ref))
