"""The no-allocation entry point at expansion order 8.

The chunk sums of order 8 may need more room than the library's fixed array
(a chunk of at most 32 entries serves at most 128 boxes of a target's list
and holds 168 floats); such a mesh is evaluated all the same, with the sums
in the context's own buffer, and equals the ordinary entry point.
"""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mesh,large", [("cube", False), ("ball", True)])
def test_noalloc_order8_equals_eval(mesh, large):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2112_00864_gb300 import bcfmm
    from paper_2112_00864_gb300.build import build
    from paper_2112_00864_gb300.inputs import ball_bc_mesh, cube_bc_mesh, densities
    build()
    m = ball_bc_mesh(4, radial=0.35) if large else cube_bc_mesh(0.25, 0.125)
    ctx = bcfmm.Context.from_mesh(m, p=8, leaf_size=64, precision="fp32")
    f = torch.tensor(densities(m, "sine")[0], device="cuda")
    ctx.set_density(bcfmm.VOLUME, f)
    if large:
        assert ctx.stats()["vtv"]["m2l_pairs"] / 128 * 168 * 4 > 64 << 20
    for task, n in (("vtv", m.ntet), ("vtb", m.ntri)):
        ref = ctx.eval(task)[0].clone()
        out = torch.full((n,), float("nan"), dtype=torch.float64, device="cuda")
        ctx.eval_noalloc(task, f[0].contiguous(), out)
        torch.cuda.synchronize()
        assert torch.equal(out, ref)
