"""CommMean and the ghost fill of another level in one launch: deep mirrored hierarchies,
where the fill is the parent's or that of a level below the child, against the oracle, with
the parity tests' bounds."""
import pytest

from oracle import Oracle
from paper_1812_03191_gb300 import binding
from paper_1812_03191_gb300 import inputs as I
from test_gpu_mirror import _built, _geometry, _params  # noqa: F401
from test_gpu_parity import assert_parity

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mirror,n_levels,over", [
    ((True, True), 4, {}), ((True, False), 5, {}), ((True, True), 4, dict(xi_mode=1)),
], ids=str)
def test_deep_mirrored_hierarchies_match_the_oracle(mirror, n_levels, over):
    p = _params(mirror, **over)
    n, lo, hi = _geometry(mirror)
    sim = binding.Sim(n_levels, n, lo, hi, I.DEFAULT_G, p, precision=binding.DF_FP64)
    orc = Oracle(n_levels, n, lo, hi, I.DEFAULT_G, p)
    sim.step(4)
    orc.step(4)
    assert_parity(sim, orc, p)
    sim.close()
    orc.close()
