"""P2M, M2M and L2L (outer-product moments, axis-by-axis shifts of all the
children of a box at once) against the FP64 CPU oracle's FMM: orders at the
edges of the kernels' instantiations, one density, a part of a group of
four densities and more than one group, boxes with one to eight children."""
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


@pytest.mark.parametrize("p", [0, 1, 7, 8, 11, 12])
@pytest.mark.parametrize("nd", [1, 3, 6])
def test_against_oracle(bc, p, nd):
    """FP64 rounding of sums of a few thousand terms: 1e-12 of the norm."""
    for m, leaf in ((cube_bc_mesh(0.25, 0.25), 20), (ball_bc_mesh(level=1, radial=0.6), 7)):
        f, g = densities(m, "random", ndens=nd, seed=p)
        ctx = bc.Context.from_mesh(m, p=p, leaf_size=leaf, precision="fp64")
        ctx.set_density(bc.VOLUME, f)
        ctx.set_density(bc.BOUNDARY, g)
        for task, dens in (("vtv", f), ("btv", g)):
            u = ctx.eval(task).cpu().numpy()
            for i in (0, nd - 1):
                ref = np.atleast_2d(O.fmm(task, m, dens[i:i + 1], p=p, leaf_size=leaf))[0]
                assert np.linalg.norm(u[i] - ref) <= 1e-12 * np.linalg.norm(ref), (task, i)
        ctx.close()
