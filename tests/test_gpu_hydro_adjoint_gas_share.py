"""The hydro adjoint on both sides of the gas share (an eighth) at which the layout of its records changes.

Against the FP64 oracle, with the gate of the other adjoint tests (E <= 2e-5): the layout moves no rounding.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import oracle as O
from paper_2310_16122_gb300 import workloads as W
from tests._errors import check

pytestmark = pytest.mark.gpu

HP = (W.GAMMA, W.AV_ALPHA, W.AV_BETA, W.AV_ETA2)


@pytest.mark.parametrize("variant", [0, 1])
@pytest.mark.parametrize("n_gas", [299, 300])
def test_hydro_adjoint(n_gas, variant):
    from paper_2310_16122_gb300 import api
    from paper_2310_16122_gb300.build import build_library

    build_library()
    n, L = 2400, 20.0
    b = W.random_box(n, L, 0.5, 88, h=1.0)
    rng = np.random.default_rng(n_gas)
    gas = np.zeros(n, bool)
    gas[rng.permutation(n)[:n_gas]] = True
    b.species = np.where(gas, 0, 1).astype(np.uint8)
    b.m = np.where(gas, 0.2, 1.0).astype(np.float32)
    b.h = np.where(gas, 1.2 * L / n_gas ** (1.0 / 3.0), 0.0).astype(np.float32)
    b.u = np.where(gas, rng.uniform(0.6, 1.6, n), 0.0).astype(np.float32)
    for c in ("vx", "vy", "vz"):
        setattr(b, c, np.where(gas, rng.normal(0.0, 0.3, n), 0.0).astype(np.float32))
    I = O.from_box(b)
    V, rho, _ = O.geometry(I)
    ins = [np.asarray(a, np.float32).astype(np.float64) for a in (V, rho, *O.corrections(I, V)[:4])]
    dvbar = np.where(gas[:, None], rng.normal(size=(n, 3)), 0.0).astype(np.float32).astype(np.float64)
    dubar = np.where(gas, rng.normal(size=n), 0.0).astype(np.float32).astype(np.float64)
    ref = O.hydro_adjoint(I, *ins, *HP, dvbar, dubar)
    ctx = api.Context(0)
    ctx.set_variant("hydro", variant)
    db = api.DeviceBox(b)
    lv = api.build_leaves(ctx, db.x, db.y, db.z, db.species, db.h, db.L, db.lp)
    t = lambda a: torch.as_tensor(np.ascontiguousarray(a.T, np.float32), device="cuda")
    got = api.hydro_adjoint(ctx, lv, db.hp, db.m, db.v3, db.u, *[t(a) for a in ins], t(dvbar), t(dubar))
    for k, v in got.items():
        g = v.cpu().numpy()
        g = g.T if g.ndim == 2 else g
        check(f"hydro_adjoint_gas/{n_gas}/v{variant}", k + "bar", g[gas], ref[k][gas], "adj")
        assert np.all(g[~gas] == 0), k
