"""The boxes that a level step gives its operators (fused sweeps): against the same run
sweeping whole arrays, over the operators that can be off and the sub-cycling search, and
against the oracle over ghost widths, where the boxes are clipped at the array.

Tolerances.  FP64 own boxes against whole arrays: the same bits (double-float arithmetic does
not depend on how the compiler contracts).  FP32: the two forms of a sweep may be contracted
differently, so test_gpu_sweep.py's 3.6e-6 (2000 roundings of 2^-24 x 0.03).  Against the
oracle: the same, and the parity tests' 1e-10 in FP64.
"""
import numpy as np
import pytest

from oracle import Oracle
from paper_1812_03191_gb300 import binding
from paper_1812_03191_gb300 import inputs as I

pytestmark = pytest.mark.gpu

PRECISIONS = [binding.DF_FP64, binding.DF_FP32_STATE]
TOL = {binding.DF_FP64: 1e-10, binding.DF_FP32_STATE: 3.6e-6}
N, HALF = (24, 28, 32), (3.0, 3.5, 4.0)
LO = tuple(-h for h in HALF)


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1812_03191_gb300 import build as B
    B.build()
    binding.load()


def _perturb(sim, levels, orc=None):
    for l in range(levels):
        for f in range(5):
            q = sim.get_field(l, f)
            sim.set_field(l, f, q + I.smooth_perturbation(q.shape, 9 + 5 * l + f, 0.02))
            if orc:
                orc.set_field(l, f, sim.get_field(l, f))


@pytest.mark.parametrize("precision", PRECISIONS, ids=["fp64", "fp32"])
@pytest.mark.parametrize("over", [
    dict(chi=0.0), dict(chi=0.0, L=0.0), dict(hydro_on=0), dict(hydro_on=0, chi=0.0, dt_fixed=2e-3),
    dict(chi=0.0, xi_mode=1), dict(xi_mode=1), dict(),
], ids=str)
def test_own_boxes_equal_whole_arrays(over, precision):
    p = I.base_params(**{**dict(mach=0.9, flow_dir=(-0.6, 0.48, 0.64), eps=0.25, chi=0.6,
                                L=0.03, lum_sigma=0.25), **over})
    own, whole = (binding.Sim(3, N, LO, HALF, I.DEFAULT_G, p, precision=precision)
                  for _ in range(2))
    whole.debug_full_boxes(True)
    for s in (own, whole):
        _perturb(s, 3)
        for l in range(2):
            s.prolong(l)
        s.step(3)
    for l in range(3):
        for f in range(5):
            a, b = own.get_field(l, f), whole.get_field(l, f)
            if precision == binding.DF_FP64:
                assert np.array_equal(a, b), (l, f)
            else:
                assert np.abs(a - b).max() <= TOL[precision], (l, f)
    own.close()
    whole.close()


@pytest.mark.parametrize("precision", PRECISIONS, ids=["fp64", "fp32"])
@pytest.mark.parametrize("G", [2, 4, 6, 10])
@pytest.mark.parametrize("levels,chi", [(1, 0.5), (3, 0.5), (3, 0.0)], ids=str)
def test_ghost_widths_match_the_oracle(levels, chi, G, precision):
    flow = (-0.6, 0.48, 0.64)
    p = I.base_params(mach=0.7, flow_dir=flow, eps=0.25, chi=chi, bc=I.wind_bcs(flow))
    sim = binding.Sim(levels, N, LO, HALF, G, p, precision=precision)
    orc = Oracle(levels, N, LO, HALF, G, p)
    _perturb(sim, levels, orc)
    sim.step(3)
    orc.step(3)
    for l in range(levels):
        for f in range(5):
            err = np.abs(sim.get_field(l, f) - orc.get_field(l, f)).max()
            assert err <= TOL[precision], (l, f, err)
    sim.close()
    orc.close()
