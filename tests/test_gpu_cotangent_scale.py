"""The reverse of Corrections is linear in its cotangents: powers of two of them come out as the same power.

With the volumes at 2^30 of their size m0 is about 2^30, and a cotangent 2^-55 of grad A meets A^2 = 2^-60 in
the per-particle step: intermediate products there lie below the FP32 normal numbers although the polynomial
coefficients (above 2^-121) and the results (about 2^-85) do not.  Powers of two change no rounding, so the
results agree to one FP32 rounding, 2^-23 in relative L2.
"""
import pytest

torch = pytest.importorskip("torch")

from paper_2310_16122_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("part,volume,ks", [(2, 30, (-55, -40, 20)), (3, -20, (-110, -60, 40)), (0, 0, (-90, 60))])
def test_powers_of_two(part, volume, ks):
    from paper_2310_16122_gb300 import api
    from paper_2310_16122_gb300.build import build_library

    build_library()
    b = W.clustered_box(12, 1, 91)
    gas = torch.as_tensor(b.species == 0, device="cuda")
    ctx = api.Context(0)
    db = api.DeviceBox(b)
    lv = api.build_leaves(ctx, db.x, db.y, db.z, db.species, db.h, db.L, db.lp)
    V = api.geometry(ctx, lv, db.m)[0] * 2.0 ** volume
    g = torch.Generator(device="cuda").manual_seed(7)
    cot = [torch.zeros(s, b.n, device="cuda") for s in (1, 3, 3, 9)]
    cot[part] = torch.randn(cot[part].shape, generator=g, device="cuda") * gas
    ref = [t.double() for t in api.corrections_adjoint(ctx, lv, V, *cot)[:2]]
    for k in ks:
        got = api.corrections_adjoint(ctx, lv, V, *[c * 2.0 ** k for c in cot])[:2]
        for name, a, r in zip(("xbar", "Vbar"), got, ref):
            e = float((a.double() * 2.0 ** -k - r).norm() / r.norm())
            assert e <= 2.0 ** -23, (k, name, e)
    zero = api.corrections_adjoint(ctx, lv, V, *[torch.zeros_like(c) for c in cot])[:2]
    assert not bool(zero[0].any()) and not bool(zero[1].any())
