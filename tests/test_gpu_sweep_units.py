"""Double-float sweeps whose columns are laid end to end and cut evenly (a unit may end one
column and begin the next), against the FP64 oracle, within the parity tests' 1e-10: boxes
of each aspect, walls at the array's ends, and frontier faces.  The sizes are ones for which
sweep_split takes that form along one axis or more."""
import numpy as np
import pytest

from oracle import Oracle
from paper_1812_03191_gb300 import binding
from paper_1812_03191_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    if not torch.cuda.is_available():
        pytest.fail("GPU tests need a CUDA device")
    from paper_1812_03191_gb300 import build as B
    B.build()
    binding.load()


@pytest.mark.parametrize("levels,n,whole", [
    (2, (200, 48, 120), False), (2, (64, 160, 96), False), (2, (160, 128, 64), True),
    (1, (144, 144, 144), False),
], ids=str)
def test_sweeps_cut_across_columns_match_the_oracle(levels, n, whole):
    half = tuple(4.0 * m / 32 for m in n)
    lo, hi = tuple(-h for h in half), half
    flow = (-0.6, 0.48, 0.64)
    p = I.base_params(mach=0.7, flow_dir=flow, GM=0.01, eps=0.25, chi=0.5,
                      bc=(I.BC_REFLECT,) * 6 if whole else I.wind_bcs(flow))
    sim = binding.Sim(levels, n, lo, hi, I.DEFAULT_G, p, precision=binding.DF_FP64)
    sim.debug_full_boxes(whole)
    orc = Oracle(levels, n, lo, hi, I.DEFAULT_G, p)
    for l in range(levels):
        for f in range(5):
            q = sim.get_field(l, f)
            sim.set_field(l, f, q + I.smooth_perturbation(q.shape, 3 + 5 * l + f, 0.02))
            orc.set_field(l, f, sim.get_field(l, f))
    sim.step(2)
    orc.step(2)
    for l in range(levels):
        for f in range(5):
            err = np.abs(sim.get_field(l, f) - orc.get_field(l, f)).max()
            assert err <= 1e-10, (l, f, err)
    sim.close()
    orc.close()
