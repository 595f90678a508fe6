"""Leaf-pair images near the cut: the FP32 gaps decide all but the images within their margin of it.

* "touch": particles on a lattice of spacing 1/2 and r_cut = 3, so that gaps equal to the cut (out: the
  range test is strict) and one rounding below it both occur; the pair lists equal the oracle's.
* "wrap": a box little wider than two cuts, so that leaves see each other through several images; the
  lists equal the oracle's and the accelerations those of the oracle's sum over all pairs.
Whole numbers, compared exactly; the accelerations by the gate of the other boxes.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import oracle as O
from paper_2310_16122_gb300 import workloads as W
from tests._errors import check

pytestmark = pytest.mark.gpu


def _box(kind, max_leaf, mode):
    if kind == "wrap":
        return W.random_box(401, 6.25, 0.5, 5, max_leaf=max_leaf, h=1.5, leaf_mode=mode, cells=3)
    b = W.random_box(24 ** 3, 12.0, 0.5, 6, max_leaf=max_leaf, h=0.75, leaf_mode=mode, cells=4)
    g = np.stack(np.meshgrid(*[np.arange(24)] * 3, indexing="ij"), -1).reshape(-1, 3) * 0.5
    g = g.astype(np.float32)
    g[::7] = np.nextafter(g[::7], np.float32(100.0), dtype=np.float32)
    b.x, b.y, b.z = (np.ascontiguousarray(g[:, k]) for k in range(3))
    return b


@pytest.mark.parametrize("kind", ["touch", "wrap"])
@pytest.mark.parametrize("max_leaf,mode", [(8, 1), (64, 1), (128, 0)])
def test_pair_lists(kind, max_leaf, mode):
    from paper_2310_16122_gb300 import api
    from paper_2310_16122_gb300.build import build_library

    build_library()
    b = _box(kind, max_leaf, mode)
    I = O.from_box(b)
    perm, start = O.leaves_rcb(I, max_leaf) if mode == 1 else O.leaves_mesh(I, b.cells_per_side)
    ctx = api.Context(0)
    db = api.DeviceBox(b)
    lv = api.build_leaves(ctx, db.x, db.y, db.z, db.species, db.h, db.L, db.lp)
    ex = lv.export()
    assert np.array_equal(ex["perm"], perm) and np.array_equal(ex["leaf_start"], start)
    for hyd, key in ((False, "grav"), (True, "hydro")):
        ptr, lst = O.leaf_pairs(I, perm, start, hydro=hyd)
        assert np.array_equal(ex[key + "_ptr"], ptr) and np.array_equal(ex[key + "_list"], lst), key
    if kind == "wrap":
        acc, _ = api.grav_short(ctx, lv, db.gp, db.m)
        ref, _ = O.gravity(I, brute=True)
        check(f"leaf_images/{kind}/{max_leaf}/{mode}", "acc", acc.cpu().numpy().T, ref)
