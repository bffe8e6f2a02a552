"""The binary64 kernels on the FMA units (tsm2_set_path(2)): what runs for the
smallest products, in a capture without scratch, without memory for it, and
where a caller asks for it.  Exact configuration names, so that no case passes
on the tensor cores.

Bound: the componentwise 2 gamma_n(2^-53) |A||B| of the other parity tests;
exact equality for small integers."""
import numpy as np
import pytest

import tsm2_inputs as ti

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from gpu_util import DevMat, assert_parity, call  # noqa: E402


@pytest.fixture(autouse=True)
def _fma_path():
    import paper_2002_03258_gb300 as pkg
    pkg.tsm2_set_path(2)
    pkg.tsm2_set_grid(0)
    yield
    pkg.tsm2_set_path(0)
    pkg.tsm2_set_grid(0)
    pkg.tsm2_set_balance(0)


def even(x):
    return (x + 1) // 2 * 2


def product(op, m, n, k, cfg, pad=True, grid=0, gen=ti.uniform_pm1, exact=False, dtype=np.float64):
    import paper_2002_03258_gb300 as pkg
    A, B = gen(5, ti.MID_A, m, n, dtype), gen(5, ti.MID_B, n, k, dtype)
    dA = DevMat(A, even(m)) if pad else DevMat(A, m, 1)
    dB, dC = DevMat(B, even(n)), DevMat(np.full((m, k), np.nan, dtype), even(m) + 2, fill=-7.0)
    pkg.tsm2_set_grid(grid)
    assert call(op, dtype, m, n, k, dA, dB, dC) == 0, pkg.tsm2_get_last_error_string()
    assert pkg.tsm2_get_device_status(0) == 0
    assert pkg.tsm2_last_config() == cfg
    assert np.all(dC.padding() == -7.0), "C written outside its m x k extent"
    got = dC.numpy()
    assert_parity(got, A, B, dtype, exact=exact)
    return got


@pytest.mark.parametrize("op,m,n,k,cfg", [
    ("r", 31, 33, 3, "r_f64_kc4"), ("r", 1000, 1023, 8, "r_f64_kc8"), ("r", 1023, 1000, 16, "r_f64_kc16"),
    ("r", 4097, 300, 2, "r_f64_kc2"), ("r", 3001, 2000, 12, "r_f64_kc12"), ("r", 2500, 1500, 28, "r_f64_kc12"),
    ("r", 300, 5000, 7, "r_f64_kc8"), ("r", 5000, 16, 16, "r_f64_kc16"),
    ("l", 65537, 16, 16, "l_f64_kc16"), ("l", 33333, 32, 32, "l_f64_kc32"), ("l", 5000, 64, 64, "l_f64_kc32"),
    ("l", 4096, 24, 2, "l_f64_kc2"), ("l", 70001, 17, 9, "l_f64_kc12"), ("l", 50001, 24, 24, "l_f64_kc24"),
    ("l", 100003, 8, 8, "l_f64_kc8"), ("l", 1, 20, 20, "l_f64_kc24"),
    ("l", 5000, 65, 8, "lt_f64_kc8"), ("l", 30001, 300, 32, "lt_f64_kc32"), ("l", 2049, 1000, 3, "lt_f64_kc4"),
    ("l", 10, 200, 64, "lt_f64_kc32"), ("l", 30001, 300, 24, "lt_f64_kc24"), ("l", 5000, 100, 12, "lt_f64_kc12"),
    ("l", 100003, 100, 16, "lt_f64_kc16"),
])
def test_products(op, m, n, k, cfg):
    product(op, m, n, k, cfg)
    product(op, m, n, k, cfg, gen=ti.int_small, exact=True)


@pytest.mark.parametrize("grid", [1, 7, 151])
@pytest.mark.parametrize("op,m,n,k,cfg", [("r", 3001, 2000, 12, "r_f64_kc12"), ("l", 70001, 17, 9, "l_f64_kc12"),
                                          ("l", 20001, 150, 24, "lt_f64_kc24")])
def test_any_grid(op, m, n, k, cfg, grid):
    product(op, m, n, k, cfg, grid=grid)


def test_claimed_row_blocks_give_the_bits_of_the_static_partition():
    import paper_2002_03258_gb300 as pkg
    out = []
    for mode in (1, 0):
        pkg.tsm2_set_balance(mode)
        out.append(product("l", 500001, 16, 16, "l_f64_kc16"))
    assert np.array_equal(*out)


@pytest.mark.parametrize("m,n,k,cfg", [(100, 37, 3, "t_f64_kc4"), (1000, 1023, 8, "t_f64_kc8"), (4097, 300, 16, "t_f64_kc16"),
                                       (2048, 64, 17, "t_f64_kc2"), (257, 4000, 2, "t_f64_kc2"), (5000, 31, 33, "t_f64_kc2")])
def test_transposed(m, n, k, cfg):
    import paper_2002_03258_gb300 as pkg
    A, D = ti.uniform_pm1(1, ti.MID_A, m, n, np.float64), ti.uniform_pm1(1, ti.MID_B, m, k, np.float64)
    dA, dD, out = DevMat(A, even(m) + 2), DevMat(D, even(m)), DevMat(np.full((n, k), np.nan), n + 1, 1, fill=-5.0)
    assert pkg.tsm2r_t_d(m, n, k, dA.ptr, dA.ld, dD.ptr, dD.ld, out.ptr, out.ld, 0) == 0
    assert pkg.tsm2_get_device_status(0) == 0
    assert pkg.tsm2_last_config() == cfg
    assert np.all(out.padding() == -5.0)
    assert_parity(out.numpy(), np.asfortranarray(A.T), D, np.float64)


@pytest.mark.parametrize("m,n,k", [(1, 1, 1), (1000, 300, 8), (1025, 67, 16), (4099, 129, 3), (777, 65, 40), (2048, 2048, 8)])
def test_rankk(m, n, k):
    import paper_2002_03258_gb300 as pkg
    D, B = ti.uniform_pm1(1, ti.MID_A, m, k, np.float64), ti.uniform_pm1(1, ti.MID_B, n, k, np.float64)
    dD, dB, out = DevMat(D, even(m)), DevMat(B), DevMat(np.full((m, n), np.nan), m + 1, 1, fill=-5.0)
    assert pkg.tsm2_rankk_d(m, n, k, dD.ptr, dD.ld, dB.ptr, dB.ld, out.ptr, out.ld, 0) == 0
    assert pkg.tsm2_last_config() == "rankk_f64"
    assert np.all(out.padding() == -5.0)
    assert_parity(out.numpy(), D, np.asfortranarray(B.T), np.float64)


# Unaligned, every width; row blocks of 254 and 510 rows.
@pytest.mark.parametrize("m", [253, 254, 255, 509, 510, 511])
@pytest.mark.parametrize("k,kc", [(2, 2), (3, 4), (7, 8), (16, 16)])
def test_unaligned_row_block_edges(m, k, kc):
    product("r", m, 83, k, f"simple_shift_f64_kc{kc}_r1", pad=False)


@pytest.mark.parametrize("m,n,k,cfg", [
    (20401, 601, 2, "simple_shift_f64_kc2_r2"), (20399, 603, 4, "simple_shift_f64_kc4_r2"), (20400, 601, 8, "simple_shift_f64_kc8_r2"),
    (20401, 999, 13, "simple_shift_f64_kc16_r2"), (4081, 1000, 33, "simple_shift_f64_kc2_r1"), (50001, 8, 8, "simple_f64"),
])
def test_unaligned(m, n, k, cfg):
    product("r", m, n, k, cfg, pad=False)
    product("r", m, n, k, cfg, pad=False, gen=ti.int_small, exact=True)


@pytest.mark.parametrize("m,n,k,kc,r", [(251, 83, 3, 4, 1), (252, 83, 8, 8, 1), (253, 83, 16, 16, 1), (1020, 64, 2, 2, 1),
                                        (40801, 300, 8, 8, 4), (20399, 601, 30, 32, 2), (1021, 64, 20, 24, 1)])
def test_unaligned_binary32(m, n, k, kc, r):
    product("r", m, n, k, f"simple_shift_f32_kc{kc}_r{r}", pad=False, dtype=np.float32)


@pytest.mark.parametrize("op,m,n,k,cfg,pad", [
    ("r", 3000, 6000, 8, "r_f64_kc8", True), ("l", 1 << 19, 16, 16, "l_f64_kc16", True), ("l", 1 << 17, 200, 16, "lt_f64_kc16", True),
    ("r", 20401, 999, 13, "simple_shift_f64_kc16_r2", False),
])
def test_waits_that_run_out(op, m, n, k, cfg, pad):
    import paper_2002_03258_gb300 as pkg
    from test_timeouts_gpu import expect_timeout_then_recover
    A, B = ti.uniform_pm1(4, ti.MID_A, m, n, np.float64), ti.uniform_pm1(4, ti.MID_B, n, k, np.float64)
    dA = DevMat(A, even(m)) if pad else DevMat(A, m, 1)
    dB, dC = DevMat(B), DevMat(np.zeros((m, k)))
    expect_timeout_then_recover(lambda: call(op, np.float64, m, n, k, dA, dB, dC),
                                lambda: assert_parity(dC.numpy(), A, B, np.float64))
    assert pkg.tsm2_last_config() == cfg


def test_cancelling_sums_keep_the_digits_of_the_small_terms():
    """1 - 1 and then terms of 2^-40: inside gamma_n |A||B| either way, but only
    multiply-adds in this order keep the terms to the last bit (see Accuracy in
    the header)."""
    m, n, k = 300, 512, 8
    rng = np.random.default_rng(1)
    A = np.asfortranarray(rng.uniform(0.5, 1, (m, n)) * 2.0 ** -40)
    A[:, 0], A[:, 1] = 1.0, -1.0
    B = np.asfortranarray(rng.uniform(0.5, 1, (n, k)))
    B[0] = B[1] = 1.0
    dA, dB, dC = DevMat(A), DevMat(B), DevMat(np.full((m, k), np.nan))
    import paper_2002_03258_gb300 as pkg
    assert call("l", np.float64, m, n, k, dA, dB, dC) == 0 and pkg.tsm2_last_config() == "lt_f64_kc8"
    want = (A[:, 2:].astype(np.longdouble) @ B[2:].astype(np.longdouble)).astype(np.float64)
    assert np.all(np.abs(dC.numpy() - want) <= 512 * 2.0 ** -53 * want)
