"""The sizes of test_gpu_sweep_units.py take the columns laid end to end, on the CPU (host code
compiled with nvcc; no GPU needed)."""
from test_index_math_cpu import _run_check


def test_the_sizes_take_columns_cut_evenly(tmp_path):
    _run_check(tmp_path, "sweep_ends_check")
