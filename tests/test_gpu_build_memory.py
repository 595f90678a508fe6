"""Device memory of a leaf build: the rank columns reuse the buffers of the axis sorts.

Per particle and with 1/8 headroom: 12 ints of sort buffers, 3 more rank columns, 3 ranks, 3 of node numbers
and members, 1.4 of counts and sums (20.4 x 4.5 = 92 bytes); leaves of 20 bytes of orders, 32 of positions and 4 of
cell boxes; and per leaf of 122 particles 2.7 KB of image and pair lists (22): 170 bytes.  The nine other rank
columns in scratch of their own (40 bytes) would exceed the limit of 200.
"""
import gc

import pytest

torch = pytest.importorskip("torch")

from paper_2310_16122_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def test_bytes_per_particle():
    from paper_2310_16122_gb300 import api
    from paper_2310_16122_gb300.build import build_library

    build_library()
    n = 4000001
    db = api.DeviceBox(W.random_box(n, (n / 2.0) ** (1.0 / 3.0), 0.0, 84, h=1.0))
    tiny = api.DeviceBox(W.random_box(2001, 10.0, 0.0, 84, h=1.0))
    ctx = api.Context(0)
    api.build_leaves(ctx, tiny.x, tiny.y, tiny.z, tiny.species, tiny.h, tiny.L, tiny.lp)  # kernels loaded
    ctx.close()
    ctx = api.Context(0)
    gc.collect()
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    before = torch.cuda.mem_get_info()[0]
    lv = api.build_leaves(ctx, db.x, db.y, db.z, db.species, db.h, db.L, db.lp)
    torch.cuda.synchronize()
    used = before - torch.cuda.mem_get_info()[0]
    assert lv.status() == 0
    assert used <= 200 * n, used / n
