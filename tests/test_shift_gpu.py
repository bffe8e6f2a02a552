"""Operands of any alignment through the bulk-copy engine (column classes):
leading dimensions and base pointers of every residue, row-block edges (252,
508, 1020 rows in binary32; 254, 510 in binary64), stage edges (16 inner
indices), classes with no column (n < 4), every column width, any grid.

Bound: the componentwise 2 gamma_n(u) |A||B| of the other parity tests; exact
equality for small integers."""
import numpy as np
import pytest

import tsm2_inputs as ti

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from gpu_util import DevMat, assert_parity, call  # noqa: E402


def product(op, dtype, m, n, k, lda, offA, grid=0, gen=ti.uniform_pm1, exact=False, want="simple_"):
    import paper_2002_03258_gb300 as pkg
    A = gen(3, ti.MID_A, m, n, dtype)
    B = gen(3, ti.MID_B, n, k, dtype)
    dA, dB = DevMat(A, lda, offA), DevMat(B, n + 1, 1)  # NaN around both
    dC = DevMat(np.full((m, k), np.nan, dtype), m + 1, 1, fill=-7.0)
    pkg.tsm2_set_path(0)
    pkg.tsm2_set_grid(grid)
    try:
        assert call(op, dtype, m, n, k, dA, dB, dC) == 0, pkg.tsm2_get_last_error_string()
        assert pkg.tsm2_get_device_status(0) == 0
    finally:
        pkg.tsm2_set_grid(0)
    cfg = pkg.tsm2_last_config()
    assert cfg.startswith(want), cfg
    assert np.all(dC.padding() == -7.0), "C written outside its m x k extent"
    got = dC.numpy()
    assert_parity(got, A, B, dtype, exact=exact)
    return got


@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("pad,offA", [(0, 0), (0, 1), (1, 0), (1, 2), (2, 3), (3, 1), (4, 1)])
def test_every_residue(pad, offA, dtype):
    m = 1021 if (pad, offA) != (4, 1) else 1020
    product("r", dtype, m, 83, 4, m + pad, offA)


@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("op,m,n,k", [
    ("r", 1, 1, 1), ("l", 5, 2, 2), ("l", 251, 3, 3), ("l", 253, 15, 4), ("r", 255, 16, 5), ("l", 509, 17, 9),
    ("r", 511, 33, 17), ("l", 1021, 31, 23), ("l", 33333, 31, 31), ("r", 4081, 1000, 16), ("l", 777, 33, 40),
    ("r", 999, 5001, 12), ("l", 650001, 8, 8), ("l", 650001, 24, 2), ("r", 10001, 4099, 5),
])
def test_shapes(op, m, n, k, dtype):
    product(op, dtype, m, n, k, m, 1)


@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("m,n,k", [(3001, 4099, 16), (50001, 31, 29)])
def test_small_integers_bit_exact(m, n, k, dtype):
    product("r" if n > 64 else "l", dtype, m, n, k, m + 2, 0, gen=ti.int_small, exact=True)


@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("grid", [1, 7, 151])
def test_any_grid_and_repeatable(grid, dtype):
    first = product("r", dtype, 3001, 1003, 3, 3001, 1, grid)
    assert np.array_equal(product("r", dtype, 3001, 1003, 3, 3001, 1, grid), first)


def test_binary64_digits_through_column_classes():
    product("r", np.float64, 2001, 777, 13, 2001, 1, want="simple_f64_tc")
    product("l", np.float64, 2001, 77, 8, 2003, 0, want="simple_f64_tc")


def test_timeout_reports_and_recovers():
    import paper_2002_03258_gb300 as pkg
    for dtype, k in ((np.float32, 8), (np.float64, 2), (np.float64, 16)):
        A = ti.uniform_pm1(4, ti.MID_A, 3001, 999, dtype)
        B = ti.uniform_pm1(4, ti.MID_B, 999, k, dtype)
        dA, dB, dC = DevMat(A, 3001, 1), DevMat(B), DevMat(np.zeros((3001, k), dtype))
        pkg.tsm2_set_wait_budget_ns(-1)
        try:
            assert call("r", dtype, 3001, 999, k, dA, dB, dC) == 0
            st = pkg.tsm2_get_device_status(0)
        finally:
            pkg.tsm2_set_wait_budget_ns(1_000_000_000)
        assert st == pkg.ERR_TIMEOUT
        assert call("r", dtype, 3001, 999, k, dA, dB, dC) == 0
        assert pkg.tsm2_get_device_status(0) == 0
        assert_parity(dC.numpy(), A, B, dtype)


@pytest.mark.parametrize("k", [3, 20])
def test_a_that_no_tensor_map_describes(k):
    """One column with a leading dimension of 2 TB: strides of 2^40 bytes and
    more have no tensor map; the element-wise kernel needs none."""
    import paper_2002_03258_gb300 as pkg
    m = 1001
    A, B = ti.uniform_pm1(3, ti.MID_A, m, 1, np.float32), ti.uniform_pm1(3, ti.MID_B, 1, k, np.float32)
    dA, dB, dC = DevMat(A), DevMat(B), DevMat(np.full((m, k), np.nan, np.float32))
    st = pkg.tsm2l_s(m, 1, k, dA.ptr, (1 << 39) + 1, dB.ptr, 1, dC.ptr, m, 0)
    assert st == 0, pkg.tsm2_get_last_error_string()
    assert pkg.tsm2_last_config() == "simple_f32"
    assert_parity(dC.numpy(), A, B, np.float32)
