"""A box of a large batch gives the same bits as the box alone (no kernel splits its sums by the total size)."""
import pytest

torch = pytest.importorskip("torch")

from paper_2310_16122_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sides", [[12, 40, 24, 33], [48, 13]])
def test_batch_equals_boxes(sides):
    from paper_2310_16122_gb300 import api
    from paper_2310_16122_gb300.build import build_library

    build_library()
    boxes = [W.clustered_box(s, max(1, int(round(200 * (s / 64) ** 3))), 300 + s) for s in sides]
    ctx = api.Context(0)
    dbt = api.DeviceBatch(boxes)
    io = api.StepIO(ctx, dbt)
    api.step(ctx, api.build_leaves_batch(ctx, dbt), dbt, io)
    for k, b in enumerate(boxes):
        sl = slice(int(dbt.box_start[k]), int(dbt.box_start[k + 1]))
        db = api.DeviceBox(b)
        one = api.StepIO(ctx, db)
        api.step(ctx, api.build_leaves(ctx, db.x, db.y, db.z, db.species, db.h, db.L, db.lp), db, one)
        torch.cuda.synchronize()
        for name in ("acc", "gx_grav", "gm_grav", "dv", "du", "gx_geom", "gm_geom"):
            assert torch.equal(getattr(io, name)[..., sl], getattr(one, name)), (k, name)
