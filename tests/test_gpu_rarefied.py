"""One coarse step of a gas whose density falls to 1e-4 of the background, against the FP64
oracle: there the sums of the background and a deviation that the stencils divide by
(rho0 + drho, rho0 + drho of a face) cancel.

Tolerance.  A stored deviation near -rho0 has a grid of 2^-47 rho0, and the double-float
operations round to about that: relative to the density that is 2^-47 / 1e-4 = 7.1e-11.  A
cell passes about 50 roundings a sweep, three sweeps, and 50 in the kicks, the compression and
the diffusion; all 200 the same way give 1.5e-8, of rho and e relative to themselves, of the
velocities in units of the sound speed.  (A quotient whose error grew with the square of the
cancellation would be off by (2^-24 / 1e-4)^2 = 3.6e-7.)
"""
import numpy as np
import pytest

from oracle import Oracle
from paper_1812_03191_gb300 import binding
from paper_1812_03191_gb300 import inputs as I

pytestmark = pytest.mark.gpu

RHO_MIN = 1e-4
TOL = 200 * 2.0**-47 / RHO_MIN


@pytest.mark.parametrize("transport", [binding.TRANSPORT_FUSED, binding.TRANSPORT_SEPARATE],
                         ids=["fused", "separate"])
def test_fp64_state_keeps_its_accuracy_in_rarefied_gas(transport):
    from paper_1812_03191_gb300 import build as B
    B.build()
    n, half = (32, 24, 28), (4.0, 3.0, 3.5)
    lo, hi = tuple(-h for h in half), half
    p = I.base_params(mach=0.6, flow_dir=(-0.6, 0.48, 0.64), chi=0.5, bc=(I.BC_PERIODIC,) * 6)
    sim = binding.Sim(1, n, lo, hi, I.DEFAULT_G, p, precision=binding.DF_FP64)
    sim.set_transport(transport)
    orc = Oracle(1, n, lo, hi, I.DEFAULT_G, p)
    shape = sim.get_field(0, 0).shape
    # rho from 1e-4 to 1 of the background, e in proportion: a sound speed of about 1
    s = I.smooth_perturbation(shape, 11, 1.0)
    rho = RHO_MIN ** ((s.max() - s) / (s.max() - s.min()))
    e0 = sim.get_field(0, 1).flat[0]
    sim.set_field(0, 0, rho)
    sim.set_field(0, 1, e0 * rho * (1.0 + I.smooth_perturbation(shape, 12, 0.2)))
    for f in range(2, 5):
        sim.set_field(0, f, sim.get_field(0, f) + I.smooth_perturbation(shape, 11 + f, 0.3))
    for f in range(5):
        orc.set_field(0, f, sim.get_field(0, f))
    sim.step(1)
    orc.step(1)
    for f in range(5):
        a, b = sim.get_field(0, f), orc.get_field(0, f)
        scale = np.abs(b) if f < 2 else 1.0
        err = (np.abs(a - b) / scale).max()
        print(f"field {f}: {err:.2e} (bound {TOL:.2e})")
        assert err <= TOL, (f, err)
    sim.close()
    orc.close()
