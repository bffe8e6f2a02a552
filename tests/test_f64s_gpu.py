"""Binary64 products with an inner dimension of at most 32 on the tensor cores
(TSM2L, short TSM2R, rank-k): every edge of the kernel (tiles of 128 rows, 8, 16
and 32 inner indices, column groups of 16 of which four stay on chip, passes of
32 in the rank-k update), parts cut anywhere, and the inputs whose outputs its
flags cannot certify.

Bound: the componentwise 2 gamma_n(2^-53) |A||B| of the other parity tests;
exact equality for integers."""
import threading

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from gpu_util import DevMat, assert_parity, call  # noqa: E402
from test_f64tc_gpu import even, inputs, product  # noqa: E402


def rankk(D, B, tc=True):
    import paper_2002_03258_gb300 as pkg
    (m, k), n = D.shape, B.shape[0]
    dD, dB = DevMat(D, even(m)), DevMat(B, n + 1, 1)
    out = DevMat(np.full((m, n), np.nan), m + 1, 1, fill=-7.0)
    assert pkg.tsm2_rankk_d(m, n, k, dD.ptr, dD.ld, dB.ptr, dB.ld, out.ptr, out.ld, 0) == 0
    assert pkg.tsm2_get_device_status(0) == 0
    assert (pkg.tsm2_last_config() == "rankk_f64_tc") == tc, pkg.tsm2_last_config()
    assert np.all(out.padding() == -7.0)
    return out.numpy()


@pytest.mark.parametrize("m,n,k", [
    (1, 16, 16), (127, 8, 8), (128, 9, 9), (129, 16, 17), (300, 17, 15), (1000, 32, 32), (1000, 31, 33), (50001, 24, 20),
    (500, 4, 64), (640, 25, 65), (200000, 32, 3), (300, 2, 200), (20001, 12, 100),
])
def test_short_inner_dimension(m, n, k):
    for op in "lr":
        A, B = inputs("normal", m, n, k)
        assert_parity(product(op, A, B), A, B, np.float64)
        rng = np.random.default_rng(1)
        A = np.asfortranarray(rng.integers(-1000, 1001, (m, n)).astype(float))
        B = np.asfortranarray(rng.integers(-1000, 1001, (n, k)).astype(float))
        assert_parity(product(op, A, B), A, B, np.float64, exact=True)


@pytest.mark.parametrize("kind", ["uneven", "growing", "sparse", "tiny", "ends", "digits", "special"])
@pytest.mark.parametrize("m,n,k", [(600, 16, 40), (3000, 32, 16), (3000, 5, 20)])
def test_inputs_off_the_fast_path(kind, m, n, k):
    A, B = inputs(kind, m, n, k)
    with np.errstate(invalid="ignore"):
        assert_parity(product("l", A, B), A, B, np.float64)
        D = np.asfortranarray(B.T)
        assert_parity(rankk(A, D), A, D.T, np.float64)


@pytest.mark.parametrize("m,n,k", [(1, 16, 1), (1025, 67, 16), (4099, 129, 3), (130, 1000, 32), (777, 65, 33), (500, 300, 70),
                                   (2000, 16, 2), (300, 8, 8)])
def test_rankk(m, n, k):
    rng = np.random.default_rng(k)
    D, B = np.asfortranarray(rng.normal(size=(m, k))), np.asfortranarray(rng.normal(size=(n, k)))
    assert_parity(rankk(D, B), D, B.T, np.float64)


@pytest.mark.parametrize("grid", [1, 2, 7, 40, 151])
def test_any_grid(grid):
    """Tiles and column groups cut anywhere: the same bits."""
    A, B = inputs("normal", 3001, 20, 150)
    assert np.array_equal(product("l", A, B, grid), product("l", A, B))


def test_capture_without_room_takes_the_fma_kernels():
    import paper_2002_03258_gb300 as pkg
    m, n, k = 500, 64, 16
    A, B = inputs("normal", m, k, n)
    D = np.asfortranarray(B.T)
    dA, dB, dC = DevMat(A), DevMat(D), DevMat(np.zeros((m, n)))
    assert pkg.tsm2_rankk_d(m, n, k, dA.ptr, m, dB.ptr, n, dC.ptr, m, 0) == 0  # (code loaded before the capture)
    torch.cuda.synchronize()
    s, g = torch.cuda.Stream(), torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        st = pkg.tsm2_rankk_d(m, n, k, dA.ptr, m, dB.ptr, n, dC.ptr, m, s.cuda_stream)
    assert st == 0, pkg.tsm2_get_last_error_string()
    assert pkg.tsm2_last_config() == "rankk_f64"
    g.replay()
    torch.cuda.synchronize()
    assert_parity(dC.numpy(), A, B, np.float64)


def test_threads_on_one_stream():
    """The digits of one thread's call are not another's."""
    import paper_2002_03258_gb300 as pkg
    lib, s = pkg.lib(), torch.cuda.Stream()
    work = []
    for i in range(4):
        rng = np.random.default_rng(i)
        A, B = np.asfortranarray(rng.normal(size=(1000, 16))), np.asfortranarray(rng.normal(size=(16, 32)))
        work.append((A, B, DevMat(A), DevMat(B), [DevMat(np.zeros((1000, 32))) for _ in range(50)]))
    torch.cuda.synchronize()

    def run(A, B, dA, dB, outs):
        for o in outs:
            assert lib.tsm2l_d(1000, 16, 32, dA.ptr, 1000, dB.ptr, 16, o.ptr, 1000, s.cuda_stream) == 0
    threads = [threading.Thread(target=run, args=w) for w in work]
    [t.start() for t in threads]
    [t.join() for t in threads]
    s.synchronize()
    for A, B, dA, dB, outs in work:
        first = outs[0].numpy()
        assert_parity(first, A, B, np.float64)
        assert all(np.array_equal(o.numpy(), first) for o in outs[1:])


def test_wait_that_runs_out():
    from test_timeouts_gpu import expect_timeout_then_recover
    A, B = inputs("normal", 5000, 32, 100)
    dA, dB, dC = DevMat(A), DevMat(B), DevMat(np.zeros((5000, 100)))
    expect_timeout_then_recover(lambda: call("l", np.float64, 5000, 32, 100, dA, dB, dC),
                                lambda: assert_parity(dC.numpy(), A, B, np.float64))


@pytest.mark.parametrize("kind", ["normal", "uneven", "special"])
@pytest.mark.parametrize("m,n,k,pad,off", [
    (1, 16, 16, 0, 1), (125, 15, 10, 0, 0), (126, 17, 20, 1, 1), (127, 32, 16, 2, 1), (253, 31, 100, 0, 1), (1000, 5, 24, 1, 0),
    (50001, 9, 12, 0, 0), (4000, 1, 24, 1, 0), (100001, 8, 7, 0, 0),
])
def test_unaligned_rows(kind, m, n, k, pad, off):
    """Tiles of 126 rows by column classes, every residue of base and stride."""
    import paper_2002_03258_gb300 as pkg
    A, B = inputs(kind if n > 3 and m > 10 else "normal", m, n, k)
    dA, dB = DevMat(A, m + pad, off), DevMat(B, n + 1, 1)
    dC = DevMat(np.full((m, k), np.nan), m + 1, 1, fill=-7.0)
    assert call("l", np.float64, m, n, k, dA, dB, dC) == 0, pkg.tsm2_get_last_error_string()
    assert pkg.tsm2_get_device_status(0) == 0
    assert dA.ptr % 16 == 0 and dA.ld % 2 == 0 or pkg.tsm2_last_config() == "simple_f64_s_tc"
    assert np.all(dC.padding() == -7.0), "C written outside its m x k extent"
    with np.errstate(invalid="ignore"):
        assert_parity(dC.numpy(), A, B, np.float64)


@pytest.mark.parametrize("how", ["l", "unaligned", "rankk"])
def test_few_outputs_not_certified(how):
    """Two rows of a tile in all columns, one column in all rows: each left to
    multiply-adds once (the rank-k update adds its second pass)."""
    import paper_2002_03258_gb300 as pkg
    rng = np.random.default_rng(9)
    m, n, k = 300, 32 if how != "rankk" else 40, 37
    A, B = rng.uniform(0.5, 1, (m, n)), rng.uniform(0.5, 1, (n, k))
    B[2] *= 1e4                   # the columns' largest element ...
    A[[5, 130], 2] = 1e-3         # ... where these rows are small
    A[[5, 130], 3] = 1e-6
    B[:, 20] = 10.0 ** rng.uniform(-30, 0, n)
    if how == "unaligned":
        dA, dB, dC = DevMat(np.asfortranarray(A), m, 1), DevMat(np.asfortranarray(B)), DevMat(np.full((m, k), np.nan), m + 1, 1, fill=-7.0)
        assert call("l", np.float64, m, n, k, dA, dB, dC) == 0, pkg.tsm2_get_last_error_string()
        assert pkg.tsm2_last_config() == "simple_f64_s_tc"
        assert np.all(dC.padding() == -7.0)
        got = dC.numpy()
    elif how == "l":
        got = product("l", np.asfortranarray(A), np.asfortranarray(B))
    else:
        got = rankk(np.asfortranarray(A), np.asfortranarray(B.T))
    assert pkg.tsm2_get_device_status(0) == 0
    assert_parity(got, A, B, np.float64)


def test_columns_in_slices():
    """More columns than the workspace holds digits for (20 KB per 16, 256 MB), in two passes of the inner dimension."""
    rng = np.random.default_rng(4)
    m, n, k = 130, 210001, 40
    D, B = np.asfortranarray(rng.normal(size=(m, k))), np.asfortranarray(rng.normal(size=(n, k)))
    assert_parity(rankk(D, B), D, B.T, np.float64)


def test_scratch_is_bounded():
    import paper_2002_03258_gb300 as pkg
    from test_f64tc_gpu import random_cols, scratch_of
    m, n, k = 600, 400000, 32
    D, B, out = random_cols(m, k, 1), random_cols(n, k, 2), torch.empty((n, m), dtype=torch.float64, device="cuda")
    f = pkg.lib().tsm2_rankk_d
    a = (m, n, k, D.data_ptr(), m, B.data_ptr(), n, out.data_ptr(), m)
    assert f(*a, 0) == 0 and pkg.tsm2_last_config() == "rankk_f64_tc"
    assert scratch_of(lambda s: f(*a, s)) < 420 << 20


@pytest.mark.parametrize("m,n,k,cfg", [(64, 70000, 4, "rankk_f64"), (64, 70000, 5, "rankk_f64_tc"), (66, 70000, 4, "rankk_f64_tc"),
                                       (64, 60000, 4, "rankk_f64_tc"), (2, 70000, 2, "rankk_f64")])
def test_rankk_of_few_rows(m, n, k, cfg):
    """Both sides of the rule, with the same bound."""
    rng = np.random.default_rng(k)
    D, B = np.asfortranarray(rng.normal(size=(m, k))), np.asfortranarray(rng.normal(size=(n, k)))
    assert_parity(rankk(D, B, cfg == "rankk_f64_tc"), D, B.T, np.float64)
