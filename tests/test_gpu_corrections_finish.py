"""The per-particle solve of Corrections and its reverse: float pairs, and FP64 near singular particles.

* A change of the length unit by a power of two changes no rounding: A keeps its bits, B, grad A and
  grad B (and the gradients of the reverse) are the same bits times the power.  Exact, no tolerance.
* A sheet of particles of relative thickness d has det m2 / tr^3 ~ d^2 / 5: the thicknesses below put
  its particles in the float-pair solve, on both sides of the line (1e-6) and in the FP64 solve, and a
  flat sheet is singular throughout.  With the normal direction measured in units of the thickness the
  solve is an ordinary one (condition number of the order of 100), each sum of ~30 FP32 terms is good to
  30 * 2^-24 = 2e-6, and dB is a product of three such factors: 1e-3 on each component's relative L2.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import oracle as O
from paper_2310_16122_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def api():
    from paper_2310_16122_gb300 import api as A
    from paper_2310_16122_gb300.build import build_library

    build_library()
    return A


def _run(api, b, V, cot):
    ctx = api.Context(0)
    db = api.DeviceBox(b)
    lv = api.build_leaves(ctx, db.x, db.y, db.z, db.species, db.h, db.L, db.lp)
    t = lambda a: torch.as_tensor(np.ascontiguousarray(a, np.float32), device="cuda")
    A, B, gA, gB, ns = api.corrections(ctx, lv, t(V))
    gx, gV, gns = api.corrections_adjoint(ctx, lv, t(V), *[t(c) for c in cot])
    return [a.cpu().numpy() for a in (A, B, gA, gB, gx, gV)], int(ns.cpu()), int(gns.cpu())


@pytest.mark.parametrize("k", [-9, -4, 5, 9])
def test_length_unit(api, k):
    f = np.float32(2.0 ** k)
    b = W.clustered_box(12, 1, 91)
    gas = b.species == 0
    rng = np.random.default_rng(3)
    V = np.where(gas, rng.uniform(0.5, 2.0, b.n), 0.0).astype(np.float32)
    cot = [np.where(gas, rng.normal(size=s), 0.0).astype(np.float32) for s in ((b.n,), (3, b.n), (3, b.n), (9, b.n))]
    ref, ns, gns = _run(api, b, V, cot)
    for a in ("x", "y", "z", "h"):
        setattr(b, a, getattr(b, a) * f)
    b.L, b.r_cut = float(b.L * 2.0 ** k), float(b.r_cut * 2.0 ** k)
    got, ns2, gns2 = _run(api, b, V * f ** 3, [cot[0], cot[1] * f, cot[2] * f, cot[3] * f * f])
    assert (ns, gns) == (ns2, gns2) == (0, 0)
    for name, a, r, s in zip(("A", "B", "gA", "gB", "xbar", "Vbar"), got, ref, (0, -1, -1, -2, -1, -3)):
        assert np.array_equal(a, r * f ** s), name
        assert np.all(np.isfinite(a)) and np.any(a != 0), name


@pytest.mark.parametrize("d", [3e-2, 3e-3, 1e-4, 0.0])
def test_sheets(api, d):
    n, L = 1201, 20.0
    rng = np.random.default_rng(17)
    h = 1.8 * L / np.sqrt(n)
    b = W.random_box(n, L, 1.0, 17, h=h)
    b.z = (1.0 + d * h * rng.uniform(-1.0, 1.0, n)).astype(np.float32)
    I = O.from_box(b)
    V = np.full(n, np.float32(L * L / n * h), np.float64).astype(np.float32).astype(np.float64)
    A, B, gA, gB, ns = O.corrections(I, V)[:5]
    zero = [np.zeros(s) for s in ((n,), (3, n), (3, n), (9, n))]
    got, gns, _ = _run(api, b, V, zero)
    assert gns == ns == (0 if d else n)
    if d:
        for name, a, r in (("A", got[0][None], A[:, None]), ("B", got[1], B), ("gA", got[2], gA), ("gB", got[3], gB)):
            for c in range(a.shape[0]):
                e = np.linalg.norm(a[c] - r[:, c]) / np.linalg.norm(r[:, c])
                assert e <= 1e-3, (name, c, e)
