"""Cases of the binary64 tensor-core and unaligned kernels against the
bounds-checking build (TSM2_DEBUG=1), in a child process of
tests/test_debug_f64_gpu.py.  Every case must match the oracle and leave the
device status clean."""
import os
import sys

import numpy as np

HERE = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, HERE)
sys.path.insert(0, os.path.dirname(HERE))

import torch  # noqa: E402

import paper_2002_03258_gb300 as pkg  # noqa: E402
from gpu_util import DevMat, assert_parity, call  # noqa: E402
from test_f64tc_gpu import even, hard_inputs, inputs  # noqa: E402


def check(A, B, out, cfg):
    assert pkg.tsm2_get_device_status(0) == 0, pkg.tsm2_get_last_error_string()
    assert pkg.tsm2_last_config() == cfg, pkg.tsm2_last_config()
    assert np.all(out.padding() == -3.0)
    with np.errstate(invalid="ignore"):
        assert_parity(out.numpy(), A, B, A.dtype.type)
    return 1


def product(op, A, B, cfg, grid=0, pad=True):
    (m, n), k = A.shape, B.shape[1]
    dA = DevMat(A, even(m)) if pad else DevMat(A, m, 1)
    dB, out = DevMat(B, even(n)), DevMat(np.zeros((m, k), A.dtype), m + 3, 1, fill=-3.0)
    pkg.tsm2_set_grid(grid)
    assert call(op, A.dtype.type, m, n, k, dA, dB, out) == 0, pkg.tsm2_get_last_error_string()
    return check(A, B, out, cfg)


def transposed(A, B, grid):
    (m, n), k = A.shape, B.shape[1]
    dA, dB, out = DevMat(np.asfortranarray(A.T), even(n)), DevMat(B, even(n)), DevMat(np.zeros((m, k)), m + 3, 1, fill=-3.0)
    pkg.tsm2_set_grid(grid)
    assert pkg.tsm2r_t_d(n, m, k, dA.ptr, dA.ld, dB.ptr, dB.ld, out.ptr, out.ld, 0) == 0
    return check(A, B, out, "t_f64_tc_kc16")


def rankk(D, B):
    (m, k), n = D.shape, B.shape[0]
    dD, dB, out = DevMat(D, even(m)), DevMat(B), DevMat(np.zeros((m, n)), m + 3, 1, fill=-3.0)
    pkg.tsm2_set_grid(0)
    assert pkg.tsm2_rankk_d(m, n, k, dD.ptr, dD.ld, dB.ptr, dB.ld, out.ptr, out.ld, 0) == 0
    return check(D, np.asfortranarray(B.T), out, "rankk_f64_tc")


def main():
    assert pkg.DEBUG and pkg.lib().tsm2_debug_checks() == 1, "not the debug build"
    pkg.tsm2_set_path(0)
    n = 0
    for grid in (0, 1, 7):
        for make, kind in ((inputs, "normal"), (inputs, "special"), (hard_inputs, "band"), (hard_inputs, "rows")):
            A, B = make(kind, 1023, 1500, 11)
            n += product("r", A, B, "r_f64_tc_kc16", grid) + product("r", A, B, "simple_f64_tc_kc16", grid, False)
            n += transposed(A, B, grid)
    A, B = inputs("normal", 30001, 33, 48)
    n += product("l", A, B, "l_f64_tc_kc16")
    for kind in ("normal", "uneven", "special"):
        A, B = inputs(kind, 3001, 20, 150)
        n += product("l", A, B, "l_f64_kc32_s_f64_tc") + product("l", A, B, "simple_f64_s_tc", 0, False)
        D = np.asfortranarray(inputs(kind, 777, 33, 65)[0])
        n += rankk(D, np.asfortranarray(inputs(kind, 33, 65, 65)[0].T))
    rng = np.random.default_rng(0)
    for dtype, m, k, cfg in ((np.float64, 511, 3, "simple_shift_f64_kc4_r1"), (np.float32, 1021, 5, "simple_shift_f32_kc8_r1"),
                             (np.float32, 40801, 30, "simple_shift_f32_kc32_r2")):
        A, B = (np.asfortranarray(rng.uniform(-1, 1, s).astype(dtype)) for s in ((m, 283), (283, k)))
        n += product("r", A, B, cfg, 0, False)
    torch.cuda.synchronize()
    print(f"DEBUG-F64-OK {n}", flush=True)


if __name__ == "__main__":
    main()
