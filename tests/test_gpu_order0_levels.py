"""The level schedule q_l = q0 + L - l with a largest order of zero: every level has
order zero, as without the schedule."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
def test_schedule_is_capped_at_p0(prec):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2112_00864_gb300 import bcfmm
    from paper_2112_00864_gb300.build import build
    from paper_2112_00864_gb300.inputs import cube_bc_mesh, densities
    build()
    m = cube_bc_mesh(0.25, 0.125)
    f, g = densities(m, "sine")
    out = []
    for q0 in (0, 3):
        ctx = bcfmm.Context.from_mesh(m, p=0, q0=q0, leaf_size=32, precision=prec, near_n=1, near_k=0)
        assert set(ctx.stats()["level_order"]) == {0}
        ctx.set_density(bcfmm.VOLUME, f)
        ctx.set_density(bcfmm.BOUNDARY, g)
        out.append([ctx.eval(t).cpu().numpy() for t in ("vtv", "vtb", "btv")])
        ctx.close()
    for a, b in zip(*out):
        np.testing.assert_array_equal(a, b)
