"""Single gas calls captured in a CUDA graph of the caller, after a crk_step on the same context and nothing else.

A call that would permute its columns on a large box must not allocate the room for them inside the capture:
it runs in its direct form there, with the bits of the eager call in the kernel order.
"""
import pytest

torch = pytest.importorskip("torch")

from paper_2310_16122_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def test_captured_calls_allocate_nothing():
    from paper_2310_16122_gb300 import api
    from paper_2310_16122_gb300.build import build_library

    build_library()
    n = 1700001
    L = (n / 2.0) ** (1.0 / 3.0)
    b = W.random_box(n, L, 0.5, 78, h=1.2 * L / (n * 0.5) ** (1.0 / 3.0))
    st = torch.cuda.Stream()
    with torch.cuda.stream(st):
        ctx = api.Context(0, stream=st)
        db = api.DeviceBox(b)
        lv = api.build_leaves(ctx, db.x, db.y, db.z, db.species, db.h, db.L, db.lp)
        io = api.StepIO(ctx, db)
        api.step(ctx, lv, db, io)
        st.synchronize()

        def calls():
            A, B, gA, gB, _ = api.corrections(ctx, lv, io.V)
            dv, du, cons, _ = api.hydro(ctx, lv, db.hp, db.m, db.v3, db.u, io.V, io.rho, A, B, gA, gB)
            return A, B, gA, gB, dv, du, cons

        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=st):
            got = calls()
        for t in got:
            t.fill_(float("nan"))
        g.replay()
        ref = calls()
        st.synchronize()
    for a, r in zip(got, ref):
        assert torch.equal(a, r)
