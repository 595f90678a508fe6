"""Gravity cell sweeps at the edges of their units, cells and leaves.

Units of 16 and of 8 particles per warp: leaves that are no multiple of a unit,
leaves of a handful of particles, chaining-mesh cells above 256 particles (no RCB cells
inside, more cells of 32 than one leaf of 128 holds) and leaves of up to 1024,
against the FP64 oracle at the gates of the other gravity tests.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import oracle as O
from paper_2310_16122_gb300 import workloads as W
from tests._errors import check
from tests.test_gpu_parity import boundary_pairs, cut_boundary_particles

pytestmark = pytest.mark.gpu

N = 70001

BOXES = {
    "leaf37": lambda: W.random_box(N, 33.0, 0.5, 301, max_leaf=37, h=1.0),
    "leaf128": lambda: W.random_box(N, 33.0, 0.5, 302, max_leaf=128, h=1.0),
    "leaf1024": lambda: W.random_box(N, 33.0, 0.5, 303, max_leaf=1024, h=1.0),
    "mesh6": lambda: W.random_box(N, 33.0, 0.5, 304, h=1.0, leaf_mode=0, cells=6),
}


@pytest.mark.parametrize("variant", [1, 8], ids=["tiles", "split8"])
@pytest.mark.parametrize("name", sorted(BOXES))
def test_cell_sweeps(name, variant):
    from paper_2310_16122_gb300 import api
    from paper_2310_16122_gb300.build import build_library

    build_library()
    b = BOXES[name]()
    ctx = api.Context(0)
    for k in ("gravity", "gravity_adjoint"):
        ctx.set_variant(k, variant)
    db = api.DeviceBox(b)
    lv = api.build_leaves(ctx, db.x, db.y, db.z, db.species, db.h, db.L, db.lp)
    a, cnt = api.grav_short(ctx, lv, db.gp, db.m, count=True)
    gx, gm = api.grav_short_adjoint(ctx, lv, db.gp, db.m, 2.0 * a)
    I = O.from_box(b)
    ref, npairs = O.gravity(I)
    where = f"gravity_cells/{name}/v{variant}"
    check(where, "acc", a.cpu().numpy().T, ref)
    assert abs(int(cnt.item()) - npairs) <= boundary_pairs(b, False)
    ogx, ogm = O.gravity_adjoint(I, 2.0 * ref)
    check(where, "grav_gx", gx.cpu().numpy().T, ogx, "gx", exclude=cut_boundary_particles(I.pos, b.L, b.r_cut))
    check(where, "grav_gm", gm.cpu().numpy(), ogm, "gm")
