"""Every single gas call that can run in the kernel order, against its direct form on the same inputs.

The eager call permutes its columns on these boxes (the launch count says so); captured in a graph it runs
directly.  Both run the same kernels on the same order of pairs, so every output, the conservation sums, the
signal velocity and the singular count agree bit for bit.
"""
import ctypes

import pytest

torch = pytest.importorskip("torch")

from paper_2310_16122_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _setup(n, st):
    from paper_2310_16122_gb300 import api
    from paper_2310_16122_gb300.build import build_library

    build_library()
    L = (n / 2.0) ** (1.0 / 3.0)
    b = W.random_box(n, L, 0.5, 83, h=1.2 * L / (n * 0.5) ** (1.0 / 3.0))
    ctx = api.Context(0, stream=st)
    db = api.DeviceBox(b)
    return api, ctx, db, api.build_leaves(ctx, db.x, db.y, db.z, db.species, db.h, db.L, db.lp)


def _flat(x):
    if isinstance(x, torch.Tensor):
        return [x]
    if isinstance(x, dict):
        x = x.values()
    return [t for v in x if v is not None for t in _flat(v)]


def _launches(api, ctx):
    c = ctypes.c_int64(0)
    ctx.check(api.N.lib().crk_launch_count(ctx.handle, ctypes.byref(c)))
    return c.value


def _both_forms(api, ctx, st, name, call):
    n0 = _launches(api, ctx)
    eager = _flat(call())
    n1 = _launches(api, ctx)
    st.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=st):
        direct = _flat(call())
    n2 = _launches(api, ctx)
    g.replay()
    st.synchronize()
    assert n1 - n0 > n2 - n1, name  # the eager call permuted its columns
    assert len(eager) == len(direct)
    for k, (a, r) in enumerate(zip(eager, direct)):
        assert torch.equal(a, r), (name, k)
    assert any(bool(t.any()) for t in eager), name


def test_both_forms_agree():
    st = torch.cuda.Stream()
    with torch.cuda.stream(st):
        api, ctx, db, lv = _setup(1700001, st)
        V, rho, _ = api.geometry(ctx, lv, db.m)
        A, B, gA, gB, ns = api.corrections(ctx, lv, V)
        rho_r, dvdx, _ = api.extras(ctx, lv, db.m, db.v3, V, A, B, gA, gB)
        assert int(ns) == 0
        g = torch.Generator(device="cuda").manual_seed(5)
        gas = (db.species == 0).float()
        cot = lambda k: torch.randn(k, lv.n, generator=g, device="cuda") * gas
        vs, dvb, dub, cb = cot(3), cot(3), cot(1), [cot(k) for k in (1, 3, 3, 9)]
        args = (db.m, db.v3, db.u, V, rho, A, B, gA, gB)
        calls = dict(
            corrections=lambda: api.corrections(ctx, lv, V),
            extras=lambda: api.extras(ctx, lv, db.m, db.v3, V, A, B, gA, gB),
            hydro=lambda: api.hydro(ctx, lv, db.hp, *args, count=True),
            limited=lambda: api.hydro_limited(ctx, lv, db.hp, *args, dvdx),
            accel=lambda: api.hydro_accel(ctx, lv, db.hp, *args),
            accel_limited=lambda: api.hydro_accel(ctx, lv, db.hp, *args, dvdx=dvdx),
            energy=lambda: api.hydro_energy(ctx, lv, db.hp, *args, db.v3),
            energy_limited=lambda: api.hydro_energy(ctx, lv, db.hp, *args, vs, dvdx=dvdx),
            corrections_adjoint=lambda: api.corrections_adjoint(ctx, lv, V, *cb),
            hydro_adjoint=lambda: api.hydro_adjoint(ctx, lv, db.hp, *args, dvb, dub))
        for name, call in calls.items():
            _both_forms(api, ctx, st, name, call)


def test_geometry_adjoint():
    st = torch.cuda.Stream()
    with torch.cuda.stream(st):
        api, ctx, db, lv = _setup(8500001, st)
        V, rho, _ = api.geometry(ctx, lv, db.m)
        _both_forms(api, ctx, st, "geometry_adjoint", lambda: api.geometry_adjoint(ctx, lv, db.m, V, rho))
        _both_forms(api, ctx, st, "geometry_adjoint_V", lambda: api.geometry_adjoint(ctx, lv, db.m, V, rho, V))
