"""Labels of a strided sample of the near-singular pairs: neighbouring pairs of the
sample have different target elements."""
import time

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("task", ["vtv", "vtb", "btv"])
def test_sample_costs_about_what_its_share_of_all_pairs_costs(task):
    """A sample of 4,000 pairs does 1/k of the work of all n = 4,000 k pairs.  Per
    pair it may cost four times as much (fewer pairs in flight, shared points not
    shared), besides 0.6 ms for the call; a warp in four at work and the barriers
    of a CTA for every pair cost ten to twenty times as much."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2112_00864_gb300 import bcfmm
    from paper_2112_00864_gb300.build import build
    from paper_2112_00864_gb300.inputs import ball_bc_mesh
    build()
    m = ball_bc_mesh(level=3, radial=0.5)
    ctx = bcfmm.Context.from_mesh(m, p=3, leaf_size=64, precision="fp32", near_mode="none")
    n = ctx.stats()[task]["near_singular"]

    def seconds(k):
        best = 1e9
        for _ in range(4):
            torch.cuda.synchronize()
            t = time.perf_counter()
            d = ctx.mlp_dataset(task, k)
            torch.cuda.synchronize()
            best = min(best, time.perf_counter() - t)
        assert len(d["chat"]) == k
        return best

    few, every = seconds(4000), seconds(n)
    ctx.close()
    assert few <= 6e-4 + 4 * every * 4000 / n, (few, every, n)
