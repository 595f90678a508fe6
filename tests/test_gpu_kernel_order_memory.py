"""Single gas calls on large boxes when device memory runs short.

The columns of the kernel-order form (17 of Corrections: 68 MB on 1M particles) and the rows they pass through
(64 MB) are an advantage, not a need: without room for either the call runs directly, with the same bits; and
the columns that an earlier call left with the context are given back when another allocation needs the room.
Memory is filled by one tensor; everything else of the test is in place before.
"""
import gc

import pytest

torch = pytest.importorskip("torch")

from paper_2310_16122_gb300 import workloads as W

pytestmark = pytest.mark.gpu

MB = 1 << 20


def _box(api, n, seed):
    L = (n / 2.0) ** (1.0 / 3.0)
    return api.DeviceBox(W.random_box(n, L, 0.5, seed, h=1.2 * L / (n * 0.5) ** (1.0 / 3.0)))


def _build(api, ctx, db):
    return api.build_leaves(ctx, db.x, db.y, db.z, db.species, db.h, db.L, db.lp)


def _fill(left):
    """A tensor that leaves about `left` MB of device memory."""
    gc.collect()
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    return torch.empty(torch.cuda.mem_get_info()[0] - left * MB, dtype=torch.uint8, device="cuda")


@pytest.fixture
def api():
    from paper_2310_16122_gb300 import api as A
    from paper_2310_16122_gb300.build import build_library

    build_library()
    yield A
    gc.collect()
    torch.cuda.empty_cache()


@pytest.mark.parametrize("left", [92, 40])
def test_no_room_for_rows_or_columns(api, left):
    from paper_2310_16122_gb300 import native as N

    db = _box(api, 1000001, 79)
    warm = api.Context(0)
    lw = _build(api, warm, db)
    V = api.geometry(warm, lw, db.m)[0]
    ref = [t.clone() for t in api.corrections(warm, lw, V)[:4]]
    lw.free()
    warm.close()
    ctx = api.Context(0)
    lv = _build(api, ctx, db)
    out = [torch.full_like(t, float("nan")) for t in ref]
    hog = _fill(left)
    rc = N.lib().crk_corrections(ctx.handle, lv.handle, V.data_ptr(), *[t.data_ptr() for t in out], None)
    torch.cuda.synchronize()
    del hog
    assert rc == N.CRK_OK
    for a, r in zip(out, ref):
        assert torch.equal(a, r)


def test_columns_are_given_back(api):
    db, small = _box(api, 1000001, 80), _box(api, 150001, 81)
    ctx = api.Context(0)
    lv = _build(api, ctx, db)
    V = api.geometry(ctx, lv, db.m)[0]
    ref = [t.clone() for t in api.corrections(ctx, lv, V)[:4]]
    hog = _fill(24)
    ls = _build(api, ctx, small)  # its lists alone take more than is left
    del hog
    assert ls.status() == 0 and ls.n_leaves > 0
    for a, r in zip(api.corrections(ctx, lv, V)[:4], ref):
        assert torch.equal(a, r)
