"""The FP32 near field with several densities (symmetric form up to four, packed
chunk blocks above and for VtB and BtV) against the FP64 context on the same
tree and orders: every count of densities the kernels are instantiated for and
paddings of it, leaves at the edges of the lane layouts, split leaves, a batch."""
import numpy as np
import pytest

from paper_2112_00864_gb300.inputs import ball_bc_mesh, batch_meshes, cube_bc_mesh, densities

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


@pytest.mark.parametrize("nd", [2, 3, 4, 5, 8, 16])
@pytest.mark.parametrize("mesh,leaf", [("cube", 24), ("ball", 7), ("ball", 33), ("ball", 65), ("ball", 97), ("ball", 128), ("batch", 64)])
def test_against_fp64(bc, mesh, leaf, nd):
    """Positive densities, different ones: rounding (2^-23 for the reciprocal
    root, 2^-24 for products and sums) stays below 3e-7 of the result, element
    by element below 2e-6."""
    ms = dict(cube=lambda: [cube_bc_mesh(0.25, 0.125)], ball=lambda: [ball_bc_mesh(level=2, radial=0.6)],
              batch=lambda: batch_meshes(2, seed=4, hs=(1 / 8,)))[mesh]()
    rng = np.random.default_rng(leaf + nd)
    f = rng.uniform(0.5, 2.0, (nd, sum(m.ntet for m in ms)))
    g = rng.uniform(0.5, 2.0, (nd, sum(m.ntri for m in ms)))
    u = {}
    for prec in ("fp32", "fp64"):
        ctx = bc.Context.from_meshes(ms, p=5, leaf_size=leaf, eta0=0.6, precision=prec, near_n=1, near_k=0)
        ctx.set_density(bc.VOLUME, f)
        ctx.set_density(bc.BOUNDARY, g)
        u[prec] = {t: ctx.eval(t).cpu().numpy() for t in ("vtv", "vtb", "btv")}
        if prec == "fp32":
            again = ctx.eval_graph(("vtv", "vtb", "btv"))
            for t in ("vtv", "btv"):
                np.testing.assert_array_equal(u[prec][t], again[t].cpu().numpy())
        ctx.close()
    for t in ("vtv", "vtb", "btv"):
        d = u["fp32"][t] - u["fp64"][t]
        for i in range(nd):
            r = np.linalg.norm(d[i]) / np.linalg.norm(u["fp64"][t][i])
            assert r <= 3e-7, (t, i, r)
        assert np.abs(d / u["fp64"][t]).max() <= 2e-6, (t, np.abs(d / u["fp64"][t]).max())
