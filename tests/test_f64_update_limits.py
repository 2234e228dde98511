"""The FP64 update by integer slices is offered only where its integer sums are exact (CPU: the
library's own rule, no device call).  A work unit adds the accumulators up every 256 of K; its 16-bit
remainders hold sixteen readings of at most 4095, so a unit takes at most 4096 of K: Rbar's rows
in at most eight splits, the update's panel width in one."""
import ctypes as C

import pytest

from paper_2311_11943_gb300 import build

READING, REMAINDER = 256, 4095


@pytest.fixture(scope="module")
def offered():
    fn = C.CDLL(build.build())._ZN3cqr14f64_gemm_bytesElll
    fn.restype, fn.argtypes = C.c_size_t, [C.c_int64] * 3
    return lambda M, N, b: fn(M, N, b) > 0


@pytest.mark.parametrize("b", [128, 4096, 4097, 4160, 8192, 20000])
def test_the_panel_width_fits_one_sum(offered, b):
    M, N = 30000, b + 6000
    exact = -(-b // READING) * REMAINDER < 1 << 16
    assert offered(M, N, b) == exact


@pytest.mark.parametrize("M", [4608, 32768, 32769, 60000])
def test_the_rows_fit_eight_splits(offered, M):
    assert offered(M, 4000, 128) == (M <= 8 * 4096)
