"""The time step (Eq. 55) and the force (Eq. 18) against numpy, at sizes on both sides of where
a context's levels stop sharing a launch, with one and two levels; the force and the time of a
coarse step, formed the same way, against the calls.

Tolerances.  The time step is the reciprocal of a maximum: FP64 within 2^-42 of it
(double-float sound speed and velocity, 2^-44 each), FP32 20 roundings of 2^-24.  The force sums
terms in FP64: 2^-40 of the sum of their magnitudes (numpy's own terms are rounded to 2^-52,
the deviations it takes from the fields to 2^-52 of rho0, 1e-2 here).
"""
import numpy as np
import pytest

from paper_1812_03191_gb300 import binding
from paper_1812_03191_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [binding.DF_FP64, binding.DF_FP32_STATE],
                         ids=["fp64", "fp32"])
@pytest.mark.parametrize("levels", [1, 2])
# chunks a level, time step / force: 8 / 4, 693 / 347, 720 / 360, 1366 / 683, 1421 / 711,
# 2944 / 1472, 3136 / 1568
@pytest.mark.parametrize("n", [(20, 20, 20), (96, 88, 84), (96, 96, 80), (116, 112, 108),
                               (116, 112, 112), (112, 128, 212), (112, 128, 224)], ids=str)
def test_time_step_and_force(n, levels, precision):
    from paper_1812_03191_gb300 import build as B
    B.build()
    half = tuple(4.0 * m / 32 for m in n)
    lo = tuple(-h for h in half)
    p = I.base_params(mach=0.8, flow_dir=(-0.6, 0.48, 0.64), eps=0.3, chi=0.01)
    sim = binding.Sim(levels, n, lo, half, I.DEFAULT_G, p, precision=precision)
    e0 = p["cs"] ** 2 * p["rho0"] / (p["gamma"] * (p["gamma"] - 1.0))
    for l in range(levels):
        for f in range(5):
            q = sim.get_field(l, f)
            sim.set_field(l, f, q + I.smooth_perturbation(q.shape, 3 + 5 * l + f, 0.01))
    dt, lev = sim.compute_dt()
    F = np.asarray(sim.force_now())
    want, total = np.zeros(3), np.zeros(3)
    for l in range(levels):
        dx = [2.0 * half[d] / n[d] / 2**l for d in range(3)]
        rho, e = sim.get_field(l, 0), sim.get_field(l, 1)
        cs = np.sqrt(p["gamma"] * (p["gamma"] - 1.0) * e / rho)
        pad = sim.full_shape(l)
        limit = min(p["cfl_diff"] / (2.0 * p["chi"] * sum(1.0 / d**2 for d in dx)), 1e300)
        G = I.DEFAULT_G
        for d in range(3):
            v = np.abs(sim.get_full(l, 2 + d).reshape(pad))
            here = v[G:G + n[2], G:G + n[1], G:G + n[0]]
            up = [slice(G, G + n[2]), slice(G, G + n[1]), slice(G, G + n[0])]
            up[2 - d] = slice(G + 1, G + n[d] + 1)
            limit = min(limit, p["cfl"] * dx[d] / (cs + np.maximum(here, v[tuple(up)])).max())
        assert abs(lev[l] - limit) <= (2.0**-42 if precision == binding.DF_FP64 else
                                       20 * 2.0**-24) * limit, (l, lev[l], limit)
        x, y, z = ((np.arange(n[d]) + 0.5) * dx[d] - half[d] / 2**l for d in range(3))
        Z, Y, X = np.meshgrid(z, y, x, indexing="ij")
        w = p["GM"] * dx[0] * dx[1] * dx[2] / (X**2 + Y**2 + Z**2 + p["eps"] ** 2) ** 1.5
        if l + 1 < levels:
            w[n[2] // 4:3 * n[2] // 4, n[1] // 4:3 * n[1] // 4, n[0] // 4:3 * n[0] // 4] = 0.0
        for d, r in enumerate((X, Y, Z)):
            terms = (rho - p["rho0"]) * w * r
            want[d] += terms.sum()
            total[d] += np.abs(terms).sum()
    assert np.all(np.abs(F - want) <= 2.0**-40 * total), (F, want)
    assert dt == min(lev[l] * 2**l for l in range(levels))
    # a coarse step takes that time step, and ends with the force of its state
    sim.step(2)
    assert np.array_equal(np.asarray(sim.force()[0]), np.asarray(sim.force_now()))
    dt2 = sim.status()[1]
    t2 = sim.status()[0]
    assert t2 == dt + dt2
    sim.close()
