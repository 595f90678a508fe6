"""A rebuild of particles that have clustered since the build: the leaf-pair lists keep room for 32 pairs a leaf.

Dark matter, uniform at the build, then 36 of its 64 leaves' worth in a clump smaller than r_cut: 2006 leaf
pairs (the oracle's count), between the 1920 that an estimate from the mean leaf size would hold and 32 a leaf.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import oracle as O
from paper_2310_16122_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def test_clustered_rebuild_fits():
    from paper_2310_16122_gb300 import api
    from paper_2310_16122_gb300.build import build_library

    build_library()
    b = W.random_box(8192, 64.0, 0.0, 9, h=1.0)
    b.r_cut = 0.5
    ctx = api.Context(0)
    db = api.DeviceBox(b)
    lv = api.build_leaves(ctx, db.x, db.y, db.z, db.species, db.h, db.L, db.lp)
    rng = np.random.default_rng(4)
    for k in ("x", "y", "z"):
        getattr(b, k)[:36 * 128] = (20.0 + 0.2 * rng.random(36 * 128)).astype(np.float32)
        getattr(db, k).copy_(torch.as_tensor(getattr(b, k)))
    api.rebuild_leaves(ctx, lv, db)
    assert lv.status() == 0
    I = O.from_box(b)
    perm, start = O.leaves_rcb(I, b.max_leaf)
    ptr, pairs = O.leaf_pairs(I, perm, start, False)
    assert 1920 < len(pairs) <= 32 * (len(start) - 1)
    e = lv.export()
    assert np.array_equal(e["perm"], perm) and np.array_equal(e["grav_ptr"], ptr) and np.array_equal(e["grav_list"], pairs)
