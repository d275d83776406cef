"""Double-float quotients by sums that cancel, on the CPU (host code compiled with nvcc; no GPU
needed)."""
from test_index_math_cpu import _run_check


def test_quotients_by_cancelling_sums_keep_a_linear_error(tmp_path):
    _run_check(tmp_path, "df64_divisor_check")
