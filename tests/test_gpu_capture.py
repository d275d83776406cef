"""Calls while the caller's stream is being captured: a step whose plan has to be built, and the
operators on demand, cannot be part of a capture; they fail, and what follows them gives the
results of a context that never saw the attempt."""
import numpy as np
import pytest

from paper_1812_03191_gb300 import binding
from paper_1812_03191_gb300 import inputs as I

pytestmark = pytest.mark.gpu

N, HALF = (24, 20, 28), (3.0, 2.5, 3.5)
LO = tuple(-h for h in HALF)


def _pair(precision):
    import torch

    from paper_1812_03191_gb300 import build as B
    B.build()
    stream = torch.cuda.Stream()
    p = I.base_params(mach=0.7, chi=0.4, eps=0.3)
    sims = [binding.Sim(2, N, LO, HALF, I.DEFAULT_G, p, precision=precision,
                        stream=stream.cuda_stream) for _ in range(2)]
    return stream, p, sims


def _attempt(stream, mode, call):
    """`call` within a capture of the stream; it has to fail"""
    import torch
    graph = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.stream(stream):
        graph.capture_begin(capture_error_mode=mode)
        with pytest.raises(binding.DfError):
            call()
        try:
            graph.capture_end()
        except RuntimeError:
            pass  # the failed call may have ended the capture
    torch.cuda.synchronize()


def _perturb(sim):
    for l in range(2):
        for f in range(5):
            q = sim.get_field(l, f)
            sim.set_field(l, f, q + I.smooth_perturbation(q.shape, 5 * l + f, 0.02))


@pytest.mark.parametrize("mode", ["global", "relaxed"])
@pytest.mark.parametrize("precision", [binding.DF_FP64, binding.DF_FP32_STATE],
                         ids=["fp64", "fp32"])
def test_a_plan_is_not_built_within_a_capture(precision, mode):
    stream, p, (sim, ref) = _pair(precision)
    for s in (sim, ref):
        _perturb(s)
        s.step(1)
        s.status()
        # other parameters: the next step builds a new plan
        s.set_params({**p, "rho0": 1.5, "mach": 1.1, "cfl": 0.3, "chi": 0.2})
        _perturb(s)
    _attempt(stream, mode, lambda: sim.step(1))
    for s in (sim, ref):
        s.step(3)
    assert sim.status() == ref.status()
    for l in range(2):
        for f in range(5):
            assert np.array_equal(sim.get_field(l, f), ref.get_field(l, f)), (l, f)
    for s in (sim, ref):
        s.close()


@pytest.mark.parametrize("call", ["compute_dt", "force_now", "fill_bc"])
def test_operators_within_a_capture_leave_nothing_behind(call):
    stream, p, (sim, ref) = _pair(binding.DF_FP64)
    for s in (sim, ref):
        _perturb(s)
    _attempt(stream, "relaxed", getattr(sim, call))
    for s in (sim, ref):
        s.fill_bc()
    for _ in range(2):
        a, b = sim.compute_dt(), ref.compute_dt()
        assert a[0] == b[0] and np.array_equal(a[1], b[1])
        assert np.array_equal(sim.force_now(), ref.force_now())
    for s in (sim, ref):
        s.step(2)
    assert sim.status() == ref.status()
    for s in (sim, ref):
        s.close()
