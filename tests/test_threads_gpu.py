"""Host threads that share a stream: every entry point that keeps something in
the stream's workspace (digits or pieces of B, partial sums, counters), from
threads of their own on one new stream, with sizes that split row blocks, so
that the workspace grows while others use it.  Every call must give the bits
that it gives alone."""
import threading

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

CALLS = 60


def colmajor(rows, cols, dtype, seed, ld=None, off=0):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    ld = ld or rows
    buf = torch.empty(cols * ld + off, dtype=dtype, device="cuda").uniform_(-1, 1, generator=g)
    return buf[off:].view(cols, ld), buf


def entry(kind, m, n, k, seed):
    """A call of one entry point: f(out pointer, stream), and its output's shape and type."""
    import paper_2002_03258_gb300 as pkg
    lib = pkg.lib()
    dtype = torch.float64 if "_d" in kind else torch.float32
    if kind == "tsm2r_bf16":
        X, _ = colmajor(m, n, torch.float32, seed)
        hi, lo = (torch.empty((n, m), dtype=torch.bfloat16, device="cuda") for _ in range(2))
        assert pkg.tsm2_split_bf16(m, n, X.data_ptr(), m, hi.data_ptr(), lo.data_ptr(), m, 0) == 0
        B, _ = colmajor(n, k, torch.float32, seed + 1)
        return (lambda o, s: lib.tsm2r_bf16(m, n, k, hi.data_ptr(), lo.data_ptr(), m, B.data_ptr(), n, o, m, s)), (k, m), dtype
    if "unaligned" in kind:
        f = getattr(lib, kind.replace("_unaligned", ""))
        A, keep = colmajor(m, n, dtype, seed, m + 1, 1)
        B, _ = colmajor(n, k, dtype, seed + 1)
        return (lambda o, s, keep=keep: f(m, n, k, A.data_ptr(), m + 1, B.data_ptr(), n, o, m, s)), (k, m), dtype
    f = getattr(lib, kind)
    if "rankk" in kind:
        A, B, ldb, rows, cols = colmajor(m, k, dtype, seed)[0], colmajor(n, k, dtype, seed + 1)[0], n, m, n
    elif "tsm2r_t" in kind:
        A, B, ldb, rows, cols = colmajor(m, n, dtype, seed)[0], colmajor(m, k, dtype, seed + 1)[0], m, n, k
    else:
        A, B, ldb, rows, cols = colmajor(m, n, dtype, seed)[0], colmajor(n, k, dtype, seed + 1)[0], n, m, k
    return (lambda o, s: f(m, n, k, A.data_ptr(), m, B.data_ptr(), ldb, o, rows, s)), (cols, rows), dtype


@pytest.mark.parametrize("kinds", [
    [("tsm2r_d", 512, 2048, 16), ("tsm2r_s", 2048, 2048, 16), ("tsm2r_bf16", 1024, 4096, 16), ("tsm2r_t_s", 2048, 1024, 8)],
    [("tsm2l_d", 4000, 32, 32), ("tsm2r_s_unaligned", 1001, 4001, 12), ("tsm2_rankk_d", 500, 600, 16), ("tsm2l_s", 100000, 16, 16)],
    [("tsm2r_t_d", 2048, 1024, 8), ("tsm2r_d_unaligned", 1001, 2001, 9), ("tsm2r_s", 4096, 1024, 8), ("tsm2r_bf16", 512, 8192, 8)],
])
def test_threads_of_different_entry_points_on_one_stream(kinds):
    import paper_2002_03258_gb300 as pkg
    pkg.tsm2_set_path(0)
    pkg.tsm2_set_grid(0)
    work = []
    for i, (kind, m, n, k) in enumerate(kinds):
        f, shape, dtype = entry(kind, m, n, k, 10 * i)
        alone = torch.full(shape, float("nan"), dtype=dtype, device="cuda")
        assert f(alone.data_ptr(), 0) == 0, pkg.tsm2_get_last_error_string()
        assert pkg.tsm2_last_config() not in ("simple_f32", "simple_f64"), (kind, pkg.tsm2_last_config())
        work.append((f, alone, [torch.full_like(alone, float("nan")) for _ in range(CALLS)]))
    torch.cuda.synchronize()
    assert pkg.tsm2_get_device_status(0) == 0
    s = torch.cuda.Stream()
    status = []

    def run(f, outs):
        for o in outs:
            status.append(f(o.data_ptr(), s.cuda_stream))
    threads = [threading.Thread(target=run, args=(f, outs)) for f, _, outs in work]
    [t.start() for t in threads]
    [t.join() for t in threads]
    s.synchronize()
    assert status == [0] * (CALLS * len(kinds))
    assert pkg.tsm2_get_device_status(s.cuda_stream) == 0
    for (kind, *_), (_, alone, outs) in zip(kinds, work):
        assert not torch.isnan(alone).any(), kind
        assert all(torch.equal(o, alone) for o in outs), kind
