"""A single task on a stream that is being captured: its parts run on streams of the
context's own, which join the capture and leave it again."""
import pytest

from paper_2112_00864_gb300.inputs import cube_bc_mesh, densities

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp64", "fp32", "bf16x2"])
def test_captured_tasks_replay(prec):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2112_00864_gb300 import bcfmm
    from paper_2112_00864_gb300.build import build
    build()
    m = cube_bc_mesh(0.25, 0.125)
    f, g = (torch.tensor(x, device="cuda") for x in densities(m, "sine"))
    torch.cuda.synchronize()
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        ctx = bcfmm.Context.from_mesh(m, p=5, leaf_size=32, precision=prec, near_n=1, near_k=0, stream=s)
        ctx.set_density(bcfmm.VOLUME, f)
        ctx.set_density(bcfmm.BOUNDARY, g)
        ref = {t: ctx.eval(t).clone() for t in ("vtv", "vtb", "btv")}
        out = {t: torch.empty_like(r) for t, r in ref.items()}
    s.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=s):
        for t in out:
            ctx.eval(t, out[t])
    for _ in range(2):
        for o in out.values():
            o.fill_(float("nan"))
        torch.cuda.synchronize()
        graph.replay()
        torch.cuda.synchronize()
        for t in out:
            assert torch.equal(out[t], ref[t]), t
    with torch.cuda.stream(s):
        assert torch.equal(ctx.eval("vtv"), ref["vtv"])       # and without a capture again
    s.synchronize()
    ctx.close()
