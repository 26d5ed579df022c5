"""Host check of the symmetric near field's schedule: every pair of near leaves in one
block, every slot written and gathered once, blocks in the launches' order."""
import pytest

from paper_2112_00864_gb300 import bcfmm
from paper_2112_00864_gb300.inputs import ball_bc_mesh, batch_meshes, cube_bc_mesh


@pytest.fixture(scope="module", autouse=True)
def lib():
    from paper_2112_00864_gb300.build import build
    build()
    return bcfmm.load()


@pytest.mark.parametrize("mesh", ["cube", "ball", "batch", "one"])
@pytest.mark.parametrize("leaf,eta0", [(3, 0.9), (17, 0.6), (33, 0.6), (64, 0.5), (65, 0.3), (128, 0.6)])
def test_blocks_and_slots(mesh, leaf, eta0):
    cube = cube_bc_mesh(0.25, 0.125)
    if mesh == "one":
        cube.tets, cube.tris = cube.tets[:1], cube.tris[:0]
    ms = dict(cube=[cube], one=[cube], ball=[ball_bc_mesh(2, radial=0.6)],
              batch=[cube, ball_bc_mesh(1, radial=0.5), *batch_meshes(2, seed=3, hs=(1 / 4, 1 / 8))])[mesh]
    blocks = []
    for chunk in (1, 200, 4096, 1 << 40):
        out = bcfmm.debug_sym_coverage(ms, chunk, leaf_size=leaf, eta0=eta0)
        assert list(out[:3]) == [0, 0, 0], (chunk, out)
        blocks.append(out[3])
    assert blocks == sorted(blocks, reverse=True)
    if mesh != "one":
        assert blocks[0] > blocks[-1] > 0


def test_tiny_leaves_stay_with_the_directed_kernel():
    m = [ball_bc_mesh(1, radial=0.5)]
    assert bcfmm.debug_sym_coverage(m, 512, leaf_size=1)[4] == 0
    assert bcfmm.debug_sym_coverage(m, 512, leaf_size=64)[4] == 1
