"""Binary64 products on the tensor cores (integer digits): every shape edge of
the kernel (row blocks of 256, stages of 16 and chunks of 64 inner indices,
column passes of 16) and the inputs that leave its fast path (uneven
magnitudes, growing scales, zeros, subnormals, infinities, NaN, large digits).

Bound: the componentwise 2 gamma_n(2^-53) |A||B| of the other parity tests,
which the kernel's certificate guarantees for any input; exact equality for
integers and for sums of one product."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from gpu_util import DevMat, assert_parity, call  # noqa: E402


def even(x):
    return (x + 1) // 2 * 2


def product(op, A, B, grid=0):
    import paper_2002_03258_gb300 as pkg
    (m, n), k = A.shape, B.shape[1]
    dA, dB = DevMat(A, even(m)), DevMat(B, even(n))
    dC = DevMat(np.full((m, k), np.nan), even(m) + 2, fill=-7.0)
    pkg.tsm2_set_path(0)
    pkg.tsm2_set_grid(grid)
    try:
        assert call(op, np.float64, m, n, k, dA, dB, dC) == 0, pkg.tsm2_get_last_error_string()
        assert pkg.tsm2_get_device_status(0) == 0
    finally:
        pkg.tsm2_set_grid(0)
    assert "_f64_tc" in pkg.tsm2_last_config(), pkg.tsm2_last_config()
    assert np.all(dC.padding() == -7.0), "C written outside its m x k extent"
    return dC.numpy()


def inputs(kind, m, n, k):
    rng = np.random.default_rng(m * 31 + n)
    A, B = rng.normal(size=(m, n)), rng.normal(size=(n, k))
    if kind == "uneven":      # 40 decades inside every sum
        A *= 10.0 ** rng.uniform(-20, 20, (m, n))
        B *= 10.0 ** rng.uniform(-20, 20, (n, k))
    elif kind == "growing":   # the scale of every row changes again and again
        A *= 2.0 ** (np.arange(n) / 6.0)
    elif kind == "sparse":
        A *= rng.random((m, n)) < 0.01
        B *= rng.random((n, k)) < 0.1
        A[5] = 0.0
        B[:, 1] = 0.0
    elif kind == "tiny":
        A *= 1e-310
    elif kind == "ends":      # products near both ends of the exponent range
        A *= 1e-200
        B *= 1e-120
        A[::3] *= 1e300
        B[:, ::2] *= 1e200
    elif kind == "digits":    # every digit as large as it can be
        A[:] = -float(0x80808080808080) * 2.0 ** -60
        B[:] = float(0x80808080808080)
    elif kind == "special":
        A[7, n // 2] = np.nan
        A[8, 0] = -np.inf
        A[9, n - 1] = np.inf
        B[n // 3, 2] = np.inf
    return np.asfortranarray(A), np.asfortranarray(B)


@pytest.mark.parametrize("op,m,n,k", [
    ("r", 1, 16, 5), ("r", 255, 17, 16), ("r", 256, 64, 8), ("r", 257, 65, 7), ("r", 513, 128, 16), ("r", 300, 4097, 9),
    ("r", 5001, 129, 37), ("r", 40000, 16, 16), ("l", 1000, 24, 16), ("l", 30001, 33, 48), ("l", 5000, 300, 6),
])
def test_shapes(op, m, n, k):
    A, B = inputs("normal", m, n, k)
    assert_parity(product(op, A, B), A, B, np.float64)
    rng = np.random.default_rng(1)
    A = np.asfortranarray(rng.integers(-1000, 1001, (m, n)).astype(float))
    B = np.asfortranarray(rng.integers(-1000, 1001, (n, k)).astype(float))
    assert_parity(product(op, A, B), A, B, np.float64, exact=True)


@pytest.mark.parametrize("kind", ["uneven", "growing", "sparse", "tiny", "ends", "digits", "special"])
@pytest.mark.parametrize("m,n,k", [(600, 1000, 8), (300, 77, 16)])
def test_inputs_off_the_fast_path(kind, m, n, k):
    A, B = inputs(kind, m, n, k)
    with np.errstate(invalid="ignore"):
        assert_parity(product("r", A, B), A, B, np.float64)


@pytest.mark.parametrize("grid", [1, 2, 7, 40, 151])
def test_any_grid_and_repeatable(grid):
    """Row blocks cut anywhere; the same bits on every call."""
    A, B = inputs("normal", 1537, 3001, 13)
    first = product("r", A, B, grid)
    assert_parity(first, A, B, np.float64)
    assert np.array_equal(product("r", A, B, grid), first)


def test_one_product_is_exact():
    rng = np.random.default_rng(3)
    m, n, k = 400, 96, 8
    A = np.zeros((m, n), order="F")
    A[np.arange(m), rng.integers(0, n, m)] = rng.normal(size=m)
    B = np.asfortranarray(rng.normal(size=(n, k)))
    assert np.array_equal(product("r", A, B), A @ B)  # one rounding each


def test_capture_without_room_takes_the_fma_kernel():
    """A stream whose workspace suffices for the FMA kernel but not for the
    digits: the captured call still runs."""
    import paper_2002_03258_gb300 as pkg
    lib = pkg.lib()
    m, n, k = 64, 8192, 16
    A, B = inputs("normal", m, n, k)
    dA, dB, dC = DevMat(A), DevMat(B), DevMat(np.zeros((m, k)))
    assert lib.tsm2r_d(m, n, k, dA.ptr, m, dB.ptr, n, dC.ptr, m, 0) == 0
    torch.cuda.synchronize()
    s = torch.cuda.Stream()
    # a binary32 product leaves a workspace of a few MB on the stream
    mm = 8192
    big = torch.ones((512, mm), device="cuda")
    out = torch.empty((16, mm), device="cuda")
    bb = torch.ones((16, 512), device="cuda")
    torch.cuda.synchronize()
    assert lib.tsm2r_s(mm, 512, 16, big.data_ptr(), mm, bb.data_ptr(), 512, out.data_ptr(), mm, s.cuda_stream) == 0
    s.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        st = lib.tsm2r_d(m, n, k, dA.ptr, m, dB.ptr, n, dC.ptr, m, s.cuda_stream)
    assert st == 0, pkg.tsm2_get_last_error_string()
    dC.view.fill_(float("nan"))
    torch.cuda.synchronize()
    g.replay()
    torch.cuda.synchronize()
    assert pkg.tsm2_get_device_status(0) == 0
    assert_parity(dC.numpy(), A, B, np.float64)


@pytest.mark.parametrize("kind", ["normal", "uneven", "growing", "sparse", "special"])
@pytest.mark.parametrize("m,n,k", [(16, 256, 16), (1000, 257, 8), (4099, 300, 9), (77, 600, 16), (40002, 130, 16)])
def test_transposed(kind, m, n, k):
    """dB = A^T dC with A read by swizzled lines."""
    import paper_2002_03258_gb300 as pkg
    A, D = inputs(kind, n, m, k)  # A^T, dC
    dA, dD = DevMat(np.asfortranarray(A.T), even(m) + 2), DevMat(D, even(m))
    out = DevMat(np.full((n, k), np.nan), n + 1, 1, fill=-5.0)
    assert pkg.tsm2r_t_d(m, n, k, dA.ptr, dA.ld, dD.ptr, dD.ld, out.ptr, out.ld, 0) == 0
    assert pkg.tsm2_get_device_status(0) == 0
    assert pkg.tsm2_last_config() == "t_f64_tc_kc16"
    assert np.all(out.padding() == -5.0)
    with np.errstate(invalid="ignore"):
        assert_parity(out.numpy(), A, D, np.float64)


@pytest.mark.parametrize("zero", ["none", "row", "column"])
def test_certificate_of_eight_products(zero):
    """Sums of absolute values between a seventh and a half of the scales after
    eight products, certified only if none of the eight is zero; n = 40: the
    bound allows 2 gamma_40 of the sum, a piece may be as short as 16."""
    m, n, k = 777, 40, 16
    rng = np.random.default_rng(5)
    A = np.asfortranarray(rng.uniform(0.25, 0.3, (m, n)) * rng.choice([-1.0, 1.0], (m, n)))
    B = np.asfortranarray(rng.uniform(0.09, 0.11, (n, k)))
    B[n - 1] = 1.0
    if zero == "row":
        A[::2, 3] = 0.0
    if zero == "column":
        B[7, 1::2] = 0.0
    for grid in (0, 7):
        assert_parity(product("r", A, B, grid), A, B, np.float64)


def short_waits(run, ns=2_000_000):
    """`run` with every pipeline wait bounded by 2 ms: nothing in the pipeline may take that long."""
    import paper_2002_03258_gb300 as pkg
    pkg.tsm2_set_wait_budget_ns(ns)
    try:
        return run()
    finally:
        pkg.tsm2_set_wait_budget_ns(1_000_000_000)


def test_rows_of_zeros_do_not_hold_up_the_pipeline():
    """A row of zeros (of either sign) in a piece of 32768 inner indices, and one of magnitudes below the smallest scale."""
    m, n, k = 256, 32768, 8
    A, B = inputs("normal", m, n, k)
    A[3] = 0.0
    A[100] = -0.0
    A[200] *= 1e-300
    A[200, :n - 1] = 0.0
    A[255] = 0.0
    A[255, n // 2] = 5e-324
    got = short_waits(lambda: product("r", A, B, 1))
    assert_parity(got, A, B, np.float64)
    assert np.array_equal(got[[3, 100]], np.zeros((2, k)))
    assert np.array_equal(got[[200, 255]], A[[200, 255]] @ B)  # one product each


def hard_inputs(kind, m, n, k):
    """Inputs whose outputs the product kernel leaves to others: all of them, or few."""
    rng = np.random.default_rng(m * 31 + n)
    A, B = rng.uniform(-1, 1, (m, n)), rng.uniform(-1, 1, (n, k))
    i, j = np.arange(m)[:, None], np.arange(n)[None, :]
    if kind == "band":          # few products each
        A *= np.abs(j - i) <= 2
    elif kind == "eye":
        A = (i == j).astype(float)
    elif kind == "late":        # certified by what comes late
        A[:, :n - 40] *= rng.random((m, n - 40)) < 0.002
    elif kind == "outlier":     # one product outweighs the others
        A[:, n // 3] *= 1e4
        B[n // 3] *= 1e-3
    elif kind == "rows":        # a few rows only, one of them special
        A[m // 2, :] = 0.0
        A[m // 2, n - 1] = 3.0
        A[m - 1, ::2] *= 1e-9
        A[0, 1] = np.inf
    elif kind == "columns":     # all rows of some columns
        B[:, ::3] *= rng.random((n, B[:, ::3].shape[1])) < 0.001
        B[n // 2, 1] = np.nan
    return np.asfortranarray(A), np.asfortranarray(B)


@pytest.mark.parametrize("kind", ["band", "eye", "late", "outlier", "rows", "columns"])
@pytest.mark.parametrize("how", ["cut", "whole", "unaligned", "transposed", "transposed whole"])
def test_outputs_that_are_not_certified(kind, how):
    import paper_2002_03258_gb300 as pkg
    m, n, k = 1023, 1500, 11
    A, B = hard_inputs(kind, m, n, k)
    with np.errstate(invalid="ignore"):
        if how in ("cut", "whole"):
            got = product("r", A, B, 0 if how == "cut" else 1)
        else:
            transposed = how.startswith("transposed")
            dA = DevMat(np.asfortranarray(A.T), even(n) + 2) if transposed else DevMat(A, m, 1)
            dB, out = DevMat(B, even(n)), DevMat(np.full((m, k), np.nan), m + 1, 1, fill=-5.0)
            pkg.tsm2_set_grid(1 if how.endswith("whole") else 0)
            try:
                if transposed:
                    st = pkg.tsm2r_t_d(n, m, k, dA.ptr, dA.ld, dB.ptr, dB.ld, out.ptr, out.ld, 0)
                else:
                    st = call("r", np.float64, m, n, k, dA, dB, out)
            finally:
                pkg.tsm2_set_grid(0)
            assert st == 0, pkg.tsm2_get_last_error_string()
            assert pkg.tsm2_last_config() == ("t_f64_tc_kc16" if transposed else "simple_f64_tc_kc16")
            assert pkg.tsm2_get_device_status(0) == 0
            assert np.all(out.padding() == -5.0)
            got = out.numpy()
        assert_parity(got, A, B, np.float64)
    if kind == "eye":
        assert np.array_equal(got, B[:m])


@pytest.mark.parametrize("kind", ["eye", "outlier", "late"])
def test_outputs_that_are_not_certified_do_not_hold_up_the_pipeline(kind):
    m, n, k = 256, 32768, 16
    A, B = hard_inputs(kind, m, n, k)
    assert_parity(short_waits(lambda: product("r", A, B, 1)), A, B, np.float64)


def test_digits_of_b_do_not_count_against_the_wait_bound():
    """Digits of 2^18 rows of B take longer than the bound of the waits in the product beside them."""
    m, n, k = 256, 1 << 18, 16
    rng = np.random.default_rng(2)
    A, B = np.asfortranarray(rng.uniform(-1, 1, (m, n))), np.asfortranarray(rng.uniform(-1, 1, (n, k)))
    assert_parity(short_waits(lambda: product("r", A, B), 60_000), A, B, np.float64)


def scratch_of(run):
    """Device memory that the library takes for `run` on a stream it has not seen."""
    s = torch.cuda.Stream()
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    run(s.cuda_stream)
    s.synchronize()
    return free - torch.cuda.mem_get_info()[0]


def random_cols(rows, cols, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return torch.empty((cols, rows), dtype=torch.float64, device="cuda").uniform_(-1, 1, generator=g)


@pytest.mark.parametrize("how", ["r", "unaligned", "transposed"])
def test_inner_dimension_in_slices(how):
    """More inner indices than the workspace holds digits for: 576 bytes each, 256 MB."""
    import paper_2002_03258_gb300 as pkg
    m, n, k = 67, 470001, 9
    rng = np.random.default_rng(11)
    A, B = rng.uniform(-1, 1, (m, n)), np.asfortranarray(rng.uniform(-1, 1, (n, k)))
    A[3] = 0.0
    A[5, 400000:] = 0.0
    A[7, n - 1] = np.inf
    dB, out = DevMat(B, even(n)), DevMat(np.full((m, k), np.nan), m + 1, 1, fill=-5.0)
    if how == "transposed":
        dA = DevMat(np.asfortranarray(A.T), even(n))
        st = pkg.tsm2r_t_d(n, m, k, dA.ptr, dA.ld, dB.ptr, dB.ld, out.ptr, out.ld, 0)
    else:
        dA = DevMat(np.asfortranarray(A), m + 1, 0) if how == "r" else DevMat(np.asfortranarray(A), m, 1)
        st = call("r", np.float64, m, n, k, dA, dB, out)
    assert st == 0, pkg.tsm2_get_last_error_string()
    assert pkg.tsm2_last_config().endswith("f64_tc_kc16")
    assert pkg.tsm2_get_device_status(0) == 0
    assert np.all(out.padding() == -5.0)
    with np.errstate(invalid="ignore"):
        assert_parity(out.numpy(), A, B, np.float64)


def test_rows_in_slices():
    """2^22 rows and some: the rows of the second slice, and those around the cut."""
    import paper_2002_03258_gb300 as pkg
    m, n, k = (1 << 22) + 300, 40, 16
    A, B, out = random_cols(m, n, 1), random_cols(n, k, 2), torch.full((k, m), float("nan"), dtype=torch.float64, device="cuda")
    assert pkg.tsm2l_d(m, n, k, A.data_ptr(), m, B.data_ptr(), n, out.data_ptr(), m, 0) == 0, pkg.tsm2_get_last_error_string()
    assert pkg.tsm2_last_config() == "l_f64_tc_kc16"
    assert pkg.tsm2_get_device_status(0) == 0
    assert not torch.isnan(out).any()
    rows = torch.cat([torch.arange(0, 300), torch.arange((1 << 22) - 300, m)]).cuda()
    assert_parity(np.asfortranarray(out.t()[rows].cpu().numpy()), np.asfortranarray(A.t()[rows].cpu().numpy()),
                  np.asfortranarray(B.t().cpu().numpy()), np.float64)


def test_scratch_is_bounded():
    import paper_2002_03258_gb300 as pkg
    m, n, k = 1 << 20, 64, 16
    A, D, out = random_cols(m, n, 1), random_cols(m, k, 2), torch.empty((k, n), dtype=torch.float64, device="cuda")
    f = pkg.lib().tsm2r_t_d
    a = (m, n, k, A.data_ptr(), m, D.data_ptr(), m, out.data_ptr(), n)
    assert f(*a, 0) == 0 and pkg.tsm2_last_config() == "t_f64_tc_kc16"
    assert scratch_of(lambda s: f(*a, s)) < 420 << 20


@pytest.mark.parametrize("kind", ["normal", "band", "rows", "columns", "late", "outlier"])
@pytest.mark.parametrize("m,n,k,grid", [(1023, 64, 16, 4), (15361, 57, 9, 0), (3000, 64, 24, 7), (300, 41, 16, 1)])
def test_short_rows_settled_where_they_are(kind, m, n, k, grid):
    """Inner dimensions of up to 64, all row blocks whole or some cut."""
    A, B = inputs(kind, m, n, k) if kind == "normal" else hard_inputs(kind, m, n, k)
    with np.errstate(invalid="ignore"):
        assert_parity(product("l", A, B, grid), A, B, np.float64)


def test_short_pieces_against_the_exact_sum():
    """Pieces of one stage (16 of 100 inner indices): all outputs within n u
    |A||B|, the bound that is promised, of the exact sum."""
    from fractions import Fraction
    m, n, k = 515, 100, 4
    rng = np.random.default_rng(8)
    A, B = rng.uniform(0.02, 1, (m, n)) * rng.choice([-1, 1], (m, n)), rng.uniform(0.02, 1, (n, k))
    A[:, 50] *= 6.0
    A, B = np.asfortranarray(A), np.asfortranarray(B)
    for grid in (21, 13):
        got = product("l", A, B, grid)
        for i in range(0, m, 7):
            for c in range(k):
                terms = [Fraction(A[i, j]) * Fraction(B[j, c]) for j in range(n)]
                err = abs(Fraction(got[i, c]) - sum(terms))
                assert err <= Fraction(n, 2 ** 53) * sum(abs(t) for t in terms)


@pytest.mark.parametrize("n", [17, 23, 33, 100, 1990, 2001])
@pytest.mark.parametrize("grid", [0, 1, 3, 7, 29, 60, 150])
def test_short_last_stage_goes_with_the_one_before(n, grid):
    """Fewer than eight inner indices in the last stage, cuts anywhere."""
    A, B = inputs("normal", 1537, n, 9)
    got = product("r", A, B, grid)
    assert_parity(got, A, B, np.float64)
    assert np.array_equal(product("r", A, B, grid), got)
