"""The no-allocation entry point on a mesh whose Taylor-form partial sums exceed the
fixed array of the tensor-core form: they stand in the context's own buffer."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kw", [dict(p=7), dict(p=7, q0=6)])
def test_partial_sums_above_the_fixed_array(kw):
    """A chunk holds at most 32 entries, each of which serves at most 32 box pairs, and
    its eight targets at least 84 floats each where the order is 6 or 7: above 64 MiB from 25 M
    pairs on, more than half of that in either order alone."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2112_00864_gb300 import bcfmm
    from paper_2112_00864_gb300.build import build
    from paper_2112_00864_gb300.inputs import ball_bc_mesh, densities
    build()
    m = ball_bc_mesh(4, radial=0.35)
    ctx = bcfmm.Context.from_mesh(m, leaf_size=64, precision="fp32", near_n=1, near_k=0, **kw)
    f = torch.tensor(densities(m, "sine")[0], device="cuda")
    ctx.set_density(bcfmm.VOLUME, f)
    assert ctx.stats()["vtv"]["m2l_pairs"] > 25_000_000
    for task, n in (("vtv", m.ntet), ("vtb", m.ntri)):
        ref = ctx.eval(task)[0].clone()
        out = torch.full((n,), float("nan"), dtype=torch.float64, device="cuda")
        ctx.eval_noalloc(task, f[0].contiguous(), out)
        torch.cuda.synchronize()
        assert torch.equal(out, ref)
    ctx.close()
