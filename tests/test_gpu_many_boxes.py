"""Batches of many boxes, nearly all of them empty: the same leaves as the batch of the occupied boxes alone.

The box numbers of the particles then need one to four 8-bit digits of the sort by box (2^24 + 1 boxes: four),
and the box tables are written by the host instead of a kernel above 64 boxes.
"""
import types

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2310_16122_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nbox", [64, 65, 257, 65537, 2 ** 24 + 1])
def test_empty_boxes_change_nothing(nbox):
    from paper_2310_16122_gb300 import api
    from paper_2310_16122_gb300.build import build_library

    build_library()
    boxes = [W.random_box(n, L, 0.5, 600 + n, h=0.8) for n, L in ((700, 9.0), (401, 8.0), (1203, 12.0))]
    ctx = api.Context(0)
    few = api.DeviceBatch(boxes)
    ref = api.build_leaves_batch(ctx, few)
    at = [0, nbox // 3, nbox - 1]
    count = np.zeros(nbox, np.int64)
    side = np.full(nbox, 10.0, np.float32)
    for k, b in zip(at, boxes):
        count[k], side[k] = b.n, b.L
    many = types.SimpleNamespace(**vars(few))
    many.box_start = np.concatenate([[0], np.cumsum(count)])
    many.box_side = side
    lv = api.build_leaves_batch(ctx, many)
    assert lv.status() == 0
    a, b = lv.export(), ref.export()
    for k in b:
        assert np.array_equal(a[k], b[k]), k
