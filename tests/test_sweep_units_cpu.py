"""How a fused sweep is cut into units, on the CPU (host code compiled with nvcc; no GPU
needed)."""
from test_index_math_cpu import _run_check


def test_units_cover_every_plane_of_every_column_once(tmp_path):
    _run_check(tmp_path, "sweep_units_check")
