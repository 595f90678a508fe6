"""Kernel orders of RCB leaves of at most 128 members (the rank bisection) at the edges of its words.

Leaves of exactly 128 members (7-bit ranks used up), 127, 33 and 9, all gas, some gas and no gas,
with coordinates on a coarse grid (ties along every axis): the canonical leaf order against the
oracle bit for bit, and what depends on the kernel orders (volumes in the gas order, forces and
their gradients in the gravity order) against the oracle at the usual gates.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import oracle as O
from paper_2310_16122_gb300 import workloads as W
from tests._errors import check

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("gas", [0.0, 0.37, 1.0])
@pytest.mark.parametrize("n,max_leaf", [(1024, 128), (1016, 127), (1000, 33), (777, 9), (130, 128)])
def test_rank_bisection(n, max_leaf, gas):
    from paper_2310_16122_gb300 import api
    from paper_2310_16122_gb300.build import build_library

    build_library()
    b = W.random_box(n, 12.0, gas, 400 + n, max_leaf=max_leaf, h=1.1)
    for c in (b.x, b.y, b.z):
        c[: n // 2] = np.float32(0.25) * np.floor(c[: n // 2] * np.float32(4.0))
    db = api.DeviceBox(b)
    ctx = api.Context(0)
    lv = api.build_leaves(ctx, db.x, db.y, db.z, db.species, db.h, db.L, db.lp)
    I = O.from_box(b)
    perm, start = O.leaves_rcb(I, max_leaf)
    got = lv.export()
    assert np.array_equal(got["perm"], perm) and np.array_equal(got["leaf_start"], start)
    where = f"leaf_orders/{n}/{max_leaf}/{gas}"
    a, _ = api.grav_short(ctx, lv, db.gp, db.m)
    ref, _ = O.gravity(I)
    check(where, "acc", a.cpu().numpy().T, ref)
    V, rho, _ = api.geometry(ctx, lv, db.m)
    g = b.species == 0
    if g.any():
        oV, orho, _ = O.geometry(I)
        check(where, "V", V.cpu().numpy()[g], oV[g])
        check(where, "rho", rho.cpu().numpy()[g], orho[g])
    assert not V.cpu().numpy()[~g].any()
