"""Which form a single gas call takes: in the kernel order (columns permuted by extra launches) or directly.

A call on a large box with little gas must not permute the columns of all particles around a kernel that reads
few of them; the calls whose outputs are many scattered columns gain at any gas share.  The form is read off
the number of kernels that the call launches, against the same call on a box below the size where it switches.
"""
import pytest

torch = pytest.importorskip("torch")

from paper_2310_16122_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _launches(n, share):
    import ctypes

    from paper_2310_16122_gb300 import api, native as N
    from paper_2310_16122_gb300.build import build_library

    build_library()
    L = (n / 2.0) ** (1.0 / 3.0)
    b = W.random_box(n, L, share, 77, h=1.2 * L / (n * share) ** (1.0 / 3.0))
    ctx = api.Context(0)
    db = api.DeviceBox(b)
    lv = api.build_leaves(ctx, db.x, db.y, db.z, db.species, db.h, db.L, db.lp)
    V, rho, _ = api.geometry(ctx, lv, db.m)
    A, B, gA, gB, _ = api.corrections(ctx, lv, V)
    _, dvdx, _ = api.extras(ctx, lv, db.m, db.v3, V, A, B, gA, gB)
    args = (db.m, db.v3, db.u, V, rho, A, B, gA, gB)
    calls = dict(corrections=lambda: api.corrections(ctx, lv, V),
                 extras=lambda: api.extras(ctx, lv, *args[:2], V, A, B, gA, gB),
                 hydro=lambda: api.hydro(ctx, lv, db.hp, *args),
                 limited=lambda: api.hydro_limited(ctx, lv, db.hp, *args, dvdx),
                 accel=lambda: api.hydro_accel(ctx, lv, db.hp, *args, dvdx=dvdx),
                 energy=lambda: api.hydro_energy(ctx, lv, db.hp, *args, db.v3),
                 geometry_adjoint=lambda: api.geometry_adjoint(ctx, lv, db.m, V, rho),
                 corrections_adjoint=lambda: api.corrections_adjoint(ctx, lv, V, A, B, gA, gB),
                 hydro_adjoint=lambda: api.hydro_adjoint(ctx, lv, db.hp, *args, db.v3, db.u))
    out = {}
    for name, call in calls.items():
        c0, c1 = ctypes.c_int64(0), ctypes.c_int64(0)
        ctx.check(N.lib().crk_launch_count(ctx.handle, ctypes.byref(c0)))
        call()
        ctx.check(N.lib().crk_launch_count(ctx.handle, ctypes.byref(c1)))
        out[name] = c1.value - c0.value
    return out


@pytest.mark.parametrize("n,share,permuted", [
    (1000001, 0.02, {"corrections", "corrections_adjoint"}),
    (1700001, 0.5, {"corrections", "extras", "hydro", "limited", "accel", "energy", "corrections_adjoint",
                    "hydro_adjoint"}),
    (2500001, 0.1, {"corrections", "corrections_adjoint", "hydro_adjoint"})])
def test_form(n, share, permuted):
    small, large = _launches(100001, share), _launches(n, share)
    assert {k for k in large if large[k] > small[k]} == permuted
