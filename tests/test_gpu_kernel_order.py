"""Single calls on boxes large enough to run in the kernel order (columns permuted in bundles).

The same box through the single calls and through crk_step, which keeps its intermediates in the
kernel order: both run the same kernels on the same order of pairs, so every output agrees bit for
bit; an odd particle count just above the size where the calls switch, and one just below it.
"""
import pytest

torch = pytest.importorskip("torch")

from paper_2310_16122_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [900001, 899999])
def test_single_calls_equal_step(n):
    from paper_2310_16122_gb300 import api
    from paper_2310_16122_gb300.build import build_library

    build_library()
    L = (n / 2.0) ** (1.0 / 3.0)
    h = 1.2 * L / (n * 0.4) ** (1.0 / 3.0)
    b = W.random_box(n, L, 0.4, 501, h=h)
    ctx = api.Context(0)
    db = api.DeviceBox(b)
    lv = api.build_leaves(ctx, db.x, db.y, db.z, db.species, db.h, db.L, db.lp)
    io = api.StepIO(ctx, db, extras=True)
    api.step(ctx, lv, db, io)
    V, rho, _ = api.geometry(ctx, lv, db.m)
    A, B, gA, gB, _ = api.corrections(ctx, lv, V)
    rho_r, dvdx, _ = api.extras(ctx, lv, db.m, db.v3, V, A, B, gA, gB)
    dv, du, _, _ = api.hydro_limited(ctx, lv, db.hp, db.m, db.v3, db.u, V, rho_r, A, B, gA, gB, dvdx)
    rhobar = (db.species == 0).float()
    gx, gm = api.geometry_adjoint(ctx, lv, db.m, V, rhobar)
    for name, got, ref in (("V", V, io.V), ("rho", rho, io.rho), ("A", A, io.A), ("B", B, io.B), ("gA", gA, io.gA),
                           ("gB", gB, io.gB), ("rho_r", rho_r, io.rho_r), ("dvdx", dvdx, io.dvdx), ("dv", dv, io.dv),
                           ("du", du, io.du), ("gx", gx, io.gx_geom), ("gm", gm, io.gm_geom)):
        assert torch.equal(got, ref), name
    # the widest bundle (the limited Energy pass reads 35 columns), against the pass on v itself
    args = (db.m, db.v3, db.u, V, rho_r, A, B, gA, gB)
    e1, _, _ = api.hydro_energy(ctx, lv, db.hp, *args, db.v3, dvdx=dvdx)
    e2, _, _ = api.hydro_energy(ctx, lv, db.hp, *args, db.v3.clone(), dvdx=dvdx)
    assert torch.equal(e1, e2) and float(e1.abs().max()) > 0.0
    dark = db.species != 0
    assert not bool(e1[dark].any()) and not bool(dv[:, dark].any())
