"""The fused sweeps' lane layout and the double-float sums they use, on the CPU (host
code compiled with nvcc; no GPU needed)."""
import pytest

from test_index_math_cpu import _run_check


@pytest.mark.parametrize("name", ["sweep_lanes_check", "df64_sums_check"])
def test_host_check(tmp_path, name):
    _run_check(tmp_path, name)
