"""Row pointers of structures whose Jacobian has more than 2^31 rows: the scan kernel alone, on counts that no test could
afford to search for."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from paper_2609_05709_b200 import build

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

PROGRAM = r"""
#include "neighbor_kernels.cuh"
extern "C" int rows_order(int wide, const int* rows, const int* pairs, int C, int ctas, long long* row_ptr, int* order, void* counters) {
    return soap::launch_cluster(wide ? soap::rows_order_kernel<long long> : soap::rows_order_kernel<int>, ctas, 1024, nullptr, true, rows, pairs, C, row_ptr, order, (soap::Counters*)counters, (soap::Counters*)nullptr);
}
"""


@pytest.fixture(scope="module")
def rows_order(tmp_path_factory):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    d = tmp_path_factory.mktemp("rows")
    (d / "rows.cu").write_text(PROGRAM)
    subprocess.run([os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc"), "-gencode", "arch=compute_100a,code=sm_100a", "-std=c++17", "-shared",
                    "-Xcompiler", "-fPIC", "-I", build.CSRC, str(d / "rows.cu"), "-o", str(d / "rows.so")], check=True)
    lib = ctypes.CDLL(str(d / "rows.so"))
    lib.rows_order.argtypes = [ctypes.c_int] + [ctypes.c_void_p] * 2 + [ctypes.c_int] * 2 + [ctypes.c_void_p] * 3
    return lib.rows_order


def check(rows_order, wide, rows, ctas):
    n_centers, rng = rows.size, np.random.default_rng(rows.size)
    pairs = rng.integers(0, 2000, n_centers).astype(np.int32)
    d_rows, d_pairs = torch.from_numpy(rows).cuda(), torch.from_numpy(pairs).cuda()
    ptr = torch.zeros(n_centers + 1, dtype=torch.int64, device="cuda")
    order = torch.full((n_centers,), -1, dtype=torch.int32, device="cuda")
    counters = torch.zeros(3, dtype=torch.int64, device="cuda")              # status, pairs, rows
    torch.cuda.synchronize()
    assert rows_order(wide, d_rows.data_ptr(), d_pairs.data_ptr(), n_centers, ctas, ptr.data_ptr(), order.data_ptr(), counters.data_ptr()) == 0
    torch.cuda.synchronize()
    assert np.array_equal(ptr.cpu().numpy(), np.concatenate([[0], np.cumsum(rows.astype(np.int64))]))
    assert counters[2].item() == rows.astype(np.int64).sum()
    assert np.array_equal(np.sort(order.cpu().numpy()), np.arange(n_centers))


@pytest.mark.parametrize("n_centers,ctas,mean", [(1, 1, 2_000_000_000), (4096, 1, 800_000), (4097, 8, 8_000_000), (65536, 8, 400_000)])
def test_totals_beyond_32_bits(rows_order, n_centers, ctas, mean):
    check(rows_order, 1, np.random.default_rng(n_centers).integers(mean // 2, mean + mean // 16, n_centers).astype(np.int32), ctas)


@pytest.mark.parametrize("n_centers,ctas", [(1, 1), (4096, 1), (4097, 8), (65536, 8)])
def test_the_most_that_32_bits_hold(rows_order, n_centers, ctas):
    """All centres at the most atoms that the narrow sums are launched with."""
    check(rows_order, 0, np.full(n_centers, (2 ** 31 - 1) // -(-n_centers // ctas), np.int32), ctas)
