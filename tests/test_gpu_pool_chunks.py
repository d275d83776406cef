"""A run gives bitwise the same result alone in a pool as beside a run so much larger that the
pool's sweeps take longer chunks, over ghost widths and the artificial viscosity, with which
the sweeps' boxes reach the ends of the array (there a chunk may take another form of the
sweep)."""
import numpy as np
import pytest

from paper_1812_03191_gb300 import binding
from paper_1812_03191_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [binding.DF_FP64, binding.DF_FP32_STATE],
                         ids=["fp64", "fp32"])
@pytest.mark.parametrize("G,av", [(2, 0.0), (4, 0.0), (6, 0.0), (8, 0.0), (8, 2.0), (12, 0.0)],
                         ids=str)
@pytest.mark.parametrize("levels", [1, 2])
def test_runs_do_not_depend_on_the_chunks_of_their_pool(levels, G, av, precision):
    from paper_1812_03191_gb300 import build as B
    B.build()
    n, half = 48, 6.0
    p = I.base_params(mach=0.9, flow_dir=(-0.6, 0.48, 0.64), eps=0.3, chi=0.6, av_c2=av)
    alone, mix = (binding.Pool(1 << 34, precision=precision) for _ in range(2))
    a = alone.admit(levels, n, (-half,) * 3, (half,) * 3, G, p)
    m = mix.admit(levels, n, (-half,) * 3, (half,) * 3, G, p)
    # 160^3 cells make the chunks of the mix twice as long (alone they are the shortest)
    assert mix.admit(1, 160, (-20.0,) * 3, (20.0,) * 3, I.DEFAULT_G, p) is not None
    for l in range(levels):
        for f in range(5):
            q = alone.get_field(a, l, f)
            q = q + I.smooth_perturbation(q.shape, 5 * l + f, 0.05)
            alone.set_field(a, l, f, q)
            mix.set_field(m, l, f, q)
    alone.step(3)
    mix.step(3)
    assert np.array_equal(alone.query()[a], mix.query()[m])
    for l in range(levels):
        for f in range(5):
            assert np.array_equal(alone.get_field(a, l, f), mix.get_field(m, l, f)), (l, f)
    alone.close()
    mix.close()
