"""The one-launch ghost fill against the oracle's axis-by-axis fill, over every pair of
boundary types on an axis and mixtures of them across axes, on whole padded arrays of
random values (ghosts included, so what must stay untouched is checked too).

Tolerances: the fill copies values or forms -v - 2V.  FP64: one rounding of a stored
deviation (47 bits) and the oracle's of the full value, below 1e-13 for values below 2.
FP32 state: one rounding of a deviation below 4, 2^-22, and of the stored input, 2.4e-7.
"""
import numpy as np
import pytest

from oracle import Oracle
from paper_1812_03191_gb300 import binding
from paper_1812_03191_gb300 import inputs as I

pytestmark = pytest.mark.gpu

TOL = {binding.DF_FP64: 1e-13, binding.DF_FP32_STATE: 4.8e-7}


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
@pytest.mark.parametrize("pair", range(16))
def test_fill_matches_the_axis_by_axis_fill(pair, precision):
    lo_t, hi_t = divmod(pair, 4)
    bc = (lo_t, hi_t, hi_t, lo_t, (lo_t + 1) % 4, (hi_t + 2) % 4)
    n, half = (12, 8, 20), (3.0, 2.0, 5.0)
    flow = (0.48, -0.6, 0.64)
    p = I.base_params(mach=0.9, flow_dir=flow, bc=bc)
    lo = tuple(-h for h in half)
    sim = binding.Sim(1, n, lo, half, I.DEFAULT_G, p, precision=precision)
    orc = Oracle(1, n, lo, half, I.DEFAULT_G, p)
    rng = np.random.default_rng(pair)
    for f in range(5):
        q = sim.get_full(0, f)
        sim.set_full(0, f, q + rng.uniform(-0.2, 0.2, q.shape))
        orc.set_full(0, f, sim.get_full(0, f))
    sim.fill_bc()
    orc.fill_bc()
    for f in range(5):
        err = np.abs(sim.get_full(0, f) - orc.get_full(0, f)).max()
        assert err <= TOL[precision], (bc, f, err)
    sim.close()
    orc.close()
