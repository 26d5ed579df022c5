"""The symmetric FP32 near field of VtV (each pair of points once, owner blocks,
slots gathered per point) against the FP64 context on the same tree and
orders: leaves of 1 to 128 points (every count of point pairs a lane holds),
owners cut into several blocks, leaves on different levels, a batch."""
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


@pytest.mark.parametrize("mesh,leaf", [("cube", 24), ("cube", 60), ("ball", 17), ("ball", 33), ("ball", 48), ("ball", 49),
                                       ("ball", 64), ("ball", 65), ("ball", 81), ("ball", 97), ("ball", 113), ("ball", 128),
                                       ("ball3", 128), ("batch", 100)])
def test_against_fp64(bc, mesh, leaf):
    """Positive densities: every sum's terms have one sign, so rounding (2^-23
    for the reciprocal root, 2^-24 for products and sums) stays below 3e-7
    of the result, point by point below 2e-6."""
    ms = dict(cube=lambda: [cube_bc_mesh(0.25, 0.125)], ball=lambda: [ball_bc_mesh(level=2, radial=0.6)],
              ball3=lambda: [ball_bc_mesh(level=3, radial=0.5)], batch=lambda: batch_meshes(3, seed=4, hs=(1 / 4, 1 / 8)))[mesh]()
    f = np.concatenate([densities(m, "one")[0] + 0.5 * np.abs(densities(m, "random", seed=leaf)[0]) for m in ms], axis=1)
    u = {}
    for prec in ("fp32", "fp64"):
        ctx = bc.Context.from_meshes(ms, p=5, leaf_size=leaf, eta0=0.6, precision=prec, near_n=1, near_k=0)
        ctx.set_density(bc.VOLUME, f)
        u[prec] = ctx.eval_vtv().cpu().numpy()
        again = ctx.eval_graph(("vtv", "vtb"))["vtv"].cpu().numpy()
        np.testing.assert_array_equal(u[prec], again)
        ctx.close()
    d = u["fp32"] - u["fp64"]
    assert np.linalg.norm(d) <= 3e-7 * np.linalg.norm(u["fp64"]), np.linalg.norm(d) / np.linalg.norm(u["fp64"])
    assert np.abs(d / u["fp64"]).max() <= 2e-6, np.abs(d / u["fp64"]).max()
