"""The bench's CSR line (CPU only): the kernel it names, the traffic figure of the kernel that runs
and the bytes it counts."""
import os
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)
import bench  # noqa: E402


def _lay(index_bytes, staged, weight_bytes=0):
    return dict(index_bytes=index_bytes, weight_bytes=weight_bytes, staged=staged)


@pytest.mark.parametrize("index_bytes,staged,n,k,kernel", [
    (2, 1, 65536, 100, "csr_sliced_step_kernel"), (4, 1, 65536, 100, "csr_chunk_step_kernel"),
    (2, 0, 65536, 55, "csr_direct_step_kernel"), (2, 0, 65536, 56, "csr_step_kernel"),
    (2, 0, 40000, 500, "csr_direct_step_kernel"), (4, 0, 65536, 31, "csr_direct_step_kernel"),
    (4, 0, 65536, 32, "csr_step_kernel")])
def test_csr_kernel_of_a_layout(index_bytes, staged, n, k, kernel):
    assert bench.csr_kernel(_lay(index_bytes, staged), n, n * k) == kernel


@pytest.mark.parametrize("key", ["c3_k100", "c3_k1000"])
def test_traffic_of_the_staged_line_is_the_sliced_kernels(key):
    kernel = bench.csr_kernel(_lay(2, 1), 65536, 65536 * 100)
    assert bench.traffic_for(key, kernel, "graph", dict(csr_staging=2, csr_lanes_per_row=8))
    assert bench.traffic_for(key, kernel, "graph", dict(csr_staging=1)) is None


def test_csr_bytes_do_not_depend_on_the_staging():
    n, nnz = 65536, 6553600
    assert bench.csr_bytes_per_timestep(_lay(2, 1), n, nnz) == bench.csr_bytes_per_timestep(_lay(2, 0), n, nnz)
    assert bench.csr_bytes_per_timestep(_lay(2, 1, 4), n, nnz) == 6 * nnz + 4 * (n + 1) + 140 * n
