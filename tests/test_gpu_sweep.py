"""The fused transport sweeps at the sizes where their layout can go wrong, against the
FP64 oracle: rows that end inside a warp and ones longer than several, boxes with fewer
positions than one warp owns, chunks of one plane and a short last chunk, walls at the
array's ends, and frontier faces next to a warp's halo.

Tolerances.  FP64 state: the parity tests' 1e-10.  FP32 state: a field of deviations up to
0.03 passes about 50 roundings a sweep, 3 sweeps and 2 kicks a level step, 2^(l) level
steps of 3 coarse steps; 2000 roundings of 2^-24 x 0.03 add up to 3.6e-6 if they all fall
the same way.
"""
import numpy as np
import pytest

from oracle import Oracle
from paper_1812_03191_gb300 import binding
from paper_1812_03191_gb300 import inputs as I

pytestmark = pytest.mark.gpu

TOL = {binding.DF_FP64: 1e-10, binding.DF_FP32_STATE: 3.6e-6}
PERIODIC = (I.BC_PERIODIC,) * 6
WALLS = (I.BC_REFLECT,) * 6


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    if not torch.cuda.is_available():
        pytest.fail("GPU tests need a CUDA device")
    from paper_1812_03191_gb300 import build as B
    B.build()
    binding.load()


@pytest.mark.parametrize("precision", [binding.DF_FP64, binding.DF_FP32_STATE],
                         ids=["fp64", "fp32"])
@pytest.mark.parametrize("full_boxes", [False, True], ids=["own_boxes", "whole_arrays"])
@pytest.mark.parametrize("levels,n,bc", [
    (1, (8, 8, 8), PERIODIC), (1, (12, 8, 44), WALLS), (1, (148, 12, 8), PERIODIC),
    (1, (8, 100, 12), None), (2, (20, 24, 28), None), (3, (36, 20, 24), PERIODIC),
], ids=str)
def test_sweeps_match_the_oracle(levels, n, bc, full_boxes, precision):
    half = tuple(4.0 * m / 32 for m in n)
    lo, hi = tuple(-h for h in half), half
    flow = (-0.6, 0.48, 0.64)
    p = I.base_params(mach=0.7, flow_dir=flow, GM=0.01, eps=0.25, chi=0.5,
                      bc=I.wind_bcs(flow) if bc is None else bc)
    sim = binding.Sim(levels, n, lo, hi, I.DEFAULT_G, p, precision=precision)
    sim.set_transport(binding.TRANSPORT_FUSED)
    sim.debug_full_boxes(full_boxes)
    orc = Oracle(levels, n, lo, hi, I.DEFAULT_G, p)
    for l in range(levels):
        for f in range(5):
            q = sim.get_field(l, f)
            sim.set_field(l, f, q + I.smooth_perturbation(q.shape, 7 + 5 * l + f, 0.02))
            orc.set_field(l, f, sim.get_field(l, f))
    sim.step(3)
    orc.step(3)
    for l in range(levels):
        for f in range(5):
            err = np.abs(sim.get_field(l, f) - orc.get_field(l, f)).max()
            assert err <= TOL[precision], (l, f, err)
    sim.close()
    orc.close()
