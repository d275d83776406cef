"""Which host buffers a kernel may reach itself and how long, on the CPU (host code compiled
with nvcc; no GPU needed)."""
from test_index_math_cpu import _run_check


def test_only_buffers_registered_from_end_to_end_are_reached(tmp_path):
    _run_check(tmp_path, "hostbuf_check")


def test_a_failed_transfer_leaves_none_in_flight(tmp_path):
    _run_check(tmp_path, "transfer_all_check")
