"""The Givens rotation that the host-driven and the device-side GMRES cycles
share keeps its accuracy over the whole range of doubles.  The header the CUDA
kernels include is compiled for the host."""
from test_native_sums_cpu import run_check


def test_rotation_over_the_whole_range(tmp_path):
    run_check("givens_check", tmp_path)
