"""Field I/O on host buffers that the device reaches itself (pinned), on pageable ones and on
a misaligned view of pinned memory (both through the staging copy): the same bytes."""
import ctypes

import numpy as np
import pytest

from paper_1812_03191_gb300 import binding
from paper_1812_03191_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [binding.DF_FP64, binding.DF_FP32_STATE],
                         ids=["fp64", "fp32"])
@pytest.mark.parametrize("n", [(8, 12, 20), (64, 36, 40)], ids=str)
def test_pinned_pageable_and_misaligned_buffers_agree(n, precision):
    import torch

    from paper_1812_03191_gb300 import build as B
    B.build()
    half = tuple(4.0 * m / 32 for m in n)
    sim = binding.Sim(1, n, tuple(-h for h in half), half, I.DEFAULT_G, I.base_params(),
                      precision=precision)
    cells = n[0] * n[1] * n[2]
    pinned = torch.empty(8 * cells + 8, dtype=torch.uint8, pin_memory=True)

    def at(offset):
        return ctypes.cast(pinned.data_ptr() + offset, ctypes.POINTER(ctypes.c_double))

    def values(offset):
        return pinned[offset:offset + 8 * cells].numpy().tobytes()

    rng = np.random.default_rng(3)
    for f in range(5):
        q = sim.get_field(0, f)
        sim.set_field(0, f, q + rng.uniform(-0.1, 0.1, q.shape))
        ref = sim.get_field(0, f).tobytes()
        for offset in (0, 4):
            assert sim.lib.df_get_field(sim.h, 0, f, at(offset)) == 0
            assert values(offset) == ref
            # written back from there, the state is what it was
            sim.set_field(0, f, q)
            assert sim.lib.df_set_field(sim.h, 0, f, at(offset)) == 0
            assert sim.get_field(0, f).tobytes() == ref
    state = torch.empty(sim.state_size(), dtype=torch.float64, pin_memory=True)
    sim.get_state(state.numpy())
    assert state.numpy().tobytes() == sim.get_state()[0].tobytes()
    sim.close()
