"""RCB trees whose levels are split between the streamed, the one-block-per-segment and the shared-memory
kernels: sizes around the largest segment each of them takes (16384 and 2048 entries), odd sizes, small
leaves (more levels), coordinates with ties, and a batch in which some boxes are leaves long before others.
Leaves are whole numbers, equal to the oracle's.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import oracle as O
from paper_2310_16122_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _box(n, max_leaf, seed):
    L = max(8.0, float(np.cbrt(n / 2.0)))
    b = W.random_box(n, L, 0.5, seed, max_leaf=max_leaf, h=1.0)
    b.x[::3] = np.float32(0.5) * np.floor(b.x[::3] * np.float32(2.0))
    b.y[: n // 2] = b.y[n // 2 : n // 2 + 1]
    return b


@pytest.mark.parametrize("n,max_leaf", [(2049, 128), (4097, 32), (16384, 128), (16385, 128), (32769, 100),
                                        (65537, 128), (40001, 24)])
def test_levels(n, max_leaf):
    from paper_2310_16122_gb300 import api
    from paper_2310_16122_gb300.build import build_library

    build_library()
    b = _box(n, max_leaf, n)
    db = api.DeviceBox(b)
    lv = api.build_leaves(api.Context(0), db.x, db.y, db.z, db.species, db.h, db.L, db.lp)
    perm, start = O.leaves_rcb(O.from_box(b), max_leaf)
    got = lv.export()
    assert np.array_equal(got["leaf_start"], start) and np.array_equal(got["perm"], perm)


def test_levels_batch():
    from paper_2310_16122_gb300 import api

    boxes = [_box(n, 128, 70 + n) for n in (5, 140, 17000, 2050, 33000, 128, 9001)]
    lv = api.build_leaves_batch(api.Context(0), api.DeviceBatch(boxes))
    got = lv.export()
    n0 = leaf0 = 0
    for b in boxes:
        perm, start = O.leaves_rcb(O.from_box(b), 128)
        assert np.array_equal(got["perm"][n0 : n0 + b.n], perm + n0)
        assert np.array_equal(got["leaf_start"][leaf0 : leaf0 + start.size], start + n0)
        n0, leaf0 = n0 + b.n, leaf0 + start.size - 1
