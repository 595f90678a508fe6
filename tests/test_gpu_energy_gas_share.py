"""The Energy pass on both sides of the gas share (a sixteenth) at which the layout of its records changes.

Against the FP64 oracle on the same FP32 inputs, with the gate of du/dt (E <= 5e-5): the layout moves no rounding.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import oracle as O
from paper_2310_16122_gb300 import workloads as W
from tests._errors import check

pytestmark = pytest.mark.gpu

HP = (W.GAMMA, W.AV_ALPHA, W.AV_BETA, W.AV_ETA2)


@pytest.mark.parametrize("limited", [False, True])
@pytest.mark.parametrize("variant", [0, 1])
@pytest.mark.parametrize("n_gas", [149, 150])
def test_energy(n_gas, variant, limited):
    from paper_2310_16122_gb300 import api
    from paper_2310_16122_gb300.build import build_library

    build_library()
    n, L = 2400, 20.0
    b = W.random_box(n, L, 0.5, 89, h=1.0)
    rng = np.random.default_rng(n_gas)
    gas = np.zeros(n, bool)
    gas[rng.permutation(n)[:n_gas]] = True
    b.species = np.where(gas, 0, 1).astype(np.uint8)
    b.m = np.where(gas, 0.2, 1.0).astype(np.float32)
    b.h = np.where(gas, 1.2 * L / n_gas ** (1.0 / 3.0), 0.0).astype(np.float32)
    b.u = np.where(gas, rng.uniform(0.6, 1.8, n), 0.0).astype(np.float32)
    for c in ("vx", "vy", "vz"):
        setattr(b, c, np.where(gas, rng.normal(0.0, 0.05, n), 0.0).astype(np.float32))
    vstar = np.where(gas[:, None], np.stack([b.vx, b.vy, b.vz], 1) + rng.normal(0.0, 0.02, (n, 3)), 0.0)
    vstar = vstar.astype(np.float32).astype(np.float64)
    f32 = lambda a: np.asarray(a, np.float32).astype(np.float64)
    I = O.from_box(b)
    V, rho = (f32(a) for a in O.geometry(I)[:2])
    A, B, gA, gB = (f32(a) for a in O.corrections(I, V)[:4])
    dvg = None
    if limited:
        rho, dvg = (f32(a) for a in O.extras(I, V, A, B, gA, gB)[:2])
    ref = O.hydro_compatible(I, V, rho, A, B, gA, gB, *HP, vstar=vstar, dvg=dvg)[1]
    ctx = api.Context(0)
    ctx.set_variant("energy", variant)
    db = api.DeviceBox(b)
    lv = api.build_leaves(ctx, db.x, db.y, db.z, db.species, db.h, db.L, db.lp)
    t = lambda a: torch.as_tensor(np.ascontiguousarray(a.T, np.float32), device="cuda")
    du, _, _ = api.hydro_energy(ctx, lv, db.hp, db.m, db.v3, db.u, t(V), t(rho), t(A), t(B), t(gA), t(gB), t(vstar),
                                dvdx=t(dvg) if limited else None)
    g = du.cpu().numpy()
    check(f"energy_gas/{n_gas}/v{variant}/lim{int(limited)}", "du", g[gas], ref[gas])
    assert np.all(g[~gas] == 0)
