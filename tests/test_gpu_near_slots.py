"""Which kernel VtV's FP32 near field takes, and the memory of its slots: held for the
counts of densities that read them, given up when other buffers need the room,
and taken again when there is some."""
import numpy as np
import pytest

from paper_2112_00864_gb300.inputs import ball_bc_mesh, densities

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
KW = dict(p=5, leaf_size=64, eta0=0.6, near_n=1, near_k=0)


@pytest.fixture(scope="module")
def bc():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2112_00864_gb300 import bcfmm
    from paper_2112_00864_gb300.build import build
    build()
    return bcfmm


@pytest.fixture(scope="module")
def ball(bc):
    m = ball_bc_mesh(level=2, radial=0.6)
    f = densities(m, "one")[0] + 0.5 * np.abs(densities(m, "random", ndens=16, seed=3)[0])
    ctx = bc.Context.from_mesh(m, precision="fp64", **KW)
    ctx.set_density(bc.VOLUME, f)
    ref = ctx.eval_vtv().cpu().numpy()
    ctx.close()
    return m, f, ref


def sym(ctx):
    return ctx.stats()["vtv"]["near_sym"]


def slot_bytes(s, nd):
    return nd * (4 * s["src_slots"] + 8 * s["tgt_slots"])


def check(bc, ctx, ball, nd, dens):
    m, f, ref = ball
    ctx.set_density(bc.VOLUME, f[:nd])
    assert sym(ctx)["densities"] == dens
    u = ctx.eval_vtv().cpu().numpy()
    np.testing.assert_array_equal(u, ctx.eval_graph(("vtv",))["vtv"].cpu().numpy())
    assert np.linalg.norm(u - ref[:nd]) <= 3e-7 * np.linalg.norm(ref[:nd])


def test_slots_follow_the_densities(bc, ball):
    ctx = bc.Context.from_mesh(ball[0], precision="fp32", **KW)
    s = sym(ctx)
    assert s["blocks"] > 0 and 0 < s["large"] <= s["blocks"] and s["src_slots"] > 0 and s["densities"] == 0
    for nd, dens in ((16, 0), (5, 0), (2, 2), (1, 2), (3, 4), (8, 4), (4, 4)):
        check(bc, ctx, ball, nd, dens)
    ctx.close()
    assert bc.Context.from_mesh(ball[0], precision="fp64", **KW).stats()["vtv"]["near_sym"]["blocks"] == 0


def test_work_buffers_of_one_set_do_not_grow_with_the_other(bc, ball):
    """Boundary densities alone: no slots for more than one density, partial sums
    for BtV's lists only (a third of VtV's boxes have triangles)."""
    a, b = (bc.Context.from_mesh(ball[0], precision="fp32", **KW) for _ in range(2))
    base = a.stats()["device_bytes"]
    a.set_density(bc.VOLUME, ball[1])
    b.set_density(bc.BOUNDARY, np.ones((16, ball[0].ntri)))
    assert sym(b)["densities"] == 1
    assert b.stats()["device_bytes"] - base - slot_bytes(sym(b), 1) < 0.75 * (a.stats()["device_bytes"] - base)
    a.close()
    b.close()


def test_no_room_for_the_slots(bc, ball):
    full = bc.Context.from_mesh(ball[0], precision="fp32", **KW)
    full.set_density(bc.VOLUME, ball[1][:1])
    need = full.stats()["device_bytes"]
    slots = slot_bytes(sym(full), 1)
    full.close()
    ctx = bc.Context.from_mesh(ball[0], precision="fp32", **KW)
    assert ctx._lib.bcfmm_debug_memory_limit(ctx._ctx, need - slots // 2) == 0
    check(bc, ctx, ball, 1, 0)
    check(bc, ctx, ball, 1, 0)
    assert ctx._lib.bcfmm_debug_memory_limit(ctx._ctx, 0) == 0
    check(bc, ctx, ball, 2, 2)                 # room again
    ctx.close()


def test_other_buffers_take_the_slots_room(bc, ball):
    plain = bc.Context.from_mesh(ball[0], precision="fp32", **KW)
    plain.set_density(bc.VOLUME, ball[1])
    need = plain.stats()["device_bytes"]       # sixteen densities, no slots
    assert sym(plain)["densities"] == 0
    plain.close()
    ctx = bc.Context.from_mesh(ball[0], precision="fp32", **KW)
    check(bc, ctx, ball, 4, 4)
    assert ctx._lib.bcfmm_debug_memory_limit(ctx._ctx, need) == 0
    check(bc, ctx, ball, 16, 0)
    assert ctx._lib.bcfmm_debug_memory_limit(ctx._ctx, -1) == -1
    ctx.close()
