"""Training data: the near-singular pairs in CSR order, the same in every build."""
import numpy as np
import pytest

from paper_2112_00864_gb300.inputs import ball_bc_mesh

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("task", ["vtv", "vtb", "btv"])
def test_pairs_are_evenly_spaced_in_csr_order(task):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2112_00864_gb300 import bcfmm
    from paper_2112_00864_gb300.build import build
    build()
    m = ball_bc_mesh(level=2, radial=0.5)
    got = []
    for _ in range(2):
        ctx = bcfmm.Context.from_mesh(m, p=3, leaf_size=64, precision="fp32", near_mode="none", near_n=1, near_k=0)
        n = ctx.stats()[task]["near_singular"]
        every, few = ctx.mlp_dataset(task, n), ctx.mlp_dataset(task, 1000)
        ctx.close()
        pairs = every["pairs"].cpu().numpy().astype(np.int64)
        key = pairs[:, 0] * (1 << 32) + pairs[:, 1]
        assert len(key) == n > 1000 and np.all(np.diff(key) > 0)
        np.testing.assert_array_equal(few["pairs"].cpu().numpy(), pairs[(np.arange(1000.0) * n / 1000.0).astype(np.int64)])
        got.append({k: v.cpu().numpy() for k, v in every.items()})
    for k in got[0]:
        np.testing.assert_array_equal(got[0][k], got[1][k])
