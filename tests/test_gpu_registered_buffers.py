"""Field I/O on buffers registered with CUDA, in one piece and in two side by side: the bytes
of a pageable buffer."""
import ctypes
import mmap

import numpy as np
import pytest

from paper_1812_03191_gb300 import binding
from paper_1812_03191_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("pieces", [1, 2])
def test_registered_buffers(pieces):
    import torch

    from paper_1812_03191_gb300 import build as B
    B.build()
    n = (32, 32, 16)
    sim = binding.Sim(1, n, (-4.0, -4.0, -2.0), (4.0, 4.0, 2.0), I.DEFAULT_G, I.base_params())
    nbytes = 8 * n[0] * n[1] * n[2]
    page = max(65536, mmap.PAGESIZE)
    assert nbytes == 2 * page
    mem = mmap.mmap(-1, 4 * page)
    base = ctypes.addressof(ctypes.c_char.from_buffer(mem))
    base += -base % page  # page-aligned, with three pages left
    rt = torch.cuda.cudart()
    parts = [(base, nbytes)] if pieces == 1 else [(base, page), (base + page, page)]
    for at, size in parts:
        assert int(rt.cudaHostRegister(at, size, 0)) == 0
    buf = np.frombuffer((ctypes.c_char * nbytes).from_address(base), dtype=np.float64)
    ptr = ctypes.cast(base, ctypes.POINTER(ctypes.c_double))
    rng = np.random.default_rng(5)
    try:
        for f in range(5):
            q = sim.get_field(0, f)
            sim.set_field(0, f, q + rng.uniform(-0.1, 0.1, q.shape))
            ref = sim.get_field(0, f)
            assert sim.lib.df_get_field(sim.h, 0, f, ptr) == 0
            assert buf.tobytes() == ref.tobytes()
            sim.set_field(0, f, q)
            assert sim.lib.df_set_field(sim.h, 0, f, ptr) == 0
            assert sim.get_field(0, f).tobytes() == ref.tobytes()
    finally:
        for at, _ in parts:
            rt.cudaHostUnregister(at)
    sim.close()
