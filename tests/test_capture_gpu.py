"""Stream capture and the per-stream workspace (include/tsm2.h, "Scratch").

The split-reduction workspace of a stream grows with cudaMalloc after a
synchronise, neither of which may run while the stream is captured into a
CUDA graph.  A call that would grow it during capture must return
TSM2_ERR_UNSUPPORTED and leave the capture valid; once the stream has run
the largest shape, the same call captures and replays correctly.
"""
import numpy as np
import pytest

import tsm2_inputs as ti

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from gpu_util import DevMat, assert_parity  # noqa: E402


def test_workspace_growth_refused_during_capture_then_captures():
    import paper_2002_03258_gb300 as pkg
    pkg.tsm2_set_path(0)
    pkg.tsm2_set_grid(0)
    lib = pkg.lib()
    m, n, k = 4096, 4096, 16  # row blocks split between blocks: needs the workspace
    A = ti.uniform_pm1(8, ti.MID_A, m, n, np.float32)
    B = ti.uniform_pm1(8, ti.MID_B, n, k, np.float32)
    dA, dB, dC = DevMat(A), DevMat(B), DevMat(np.zeros((m, k), np.float32))
    # library state initialised outside any capture (device attributes, status word)
    assert lib.tsm2r_s(m, n, k, dA.ptr, m, dB.ptr, n, dC.ptr, m, 0) == 0
    torch.cuda.synchronize()

    s = torch.cuda.Stream()  # a stream the library has no workspace for
    x = torch.zeros(1, device="cuda")
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        st = lib.tsm2r_s(m, n, k, dA.ptr, m, dB.ptr, n, dC.ptr, m, s.cuda_stream)
        x.add_(1.0)
    assert st == pkg.ERR_UNSUPPORTED
    assert "capture" in pkg.tsm2_get_last_error_string()
    g.replay()  # the capture itself stayed valid
    torch.cuda.synchronize()
    assert x.item() == 1.0

    # the largest shape once on the stream, then the call captures
    assert lib.tsm2r_s(m, n, k, dA.ptr, m, dB.ptr, n, dC.ptr, m, s.cuda_stream) == 0
    s.synchronize()
    g2 = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g2, stream=s):
        st2 = lib.tsm2r_s(m, n, k, dA.ptr, m, dB.ptr, n, dC.ptr, m, s.cuda_stream)
    assert st2 == 0, pkg.tsm2_get_last_error_string()
    dC.view.fill_(float("nan"))
    torch.cuda.synchronize()
    g2.replay()
    torch.cuda.synchronize()
    assert pkg.tsm2_get_device_status(0) == 0
    assert_parity(dC.numpy(), A, B, np.float32)


def random(rows, cols, dtype, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return torch.empty((cols, rows), dtype=dtype, device="cuda").uniform_(-1, 1, generator=g)


def bf16_pair(m, n):
    import paper_2002_03258_gb300 as pkg
    X = random(m, n, torch.float32, 3)
    hi, lo = (torch.empty((n, m), dtype=torch.bfloat16, device="cuda") for _ in range(2))
    assert pkg.tsm2_split_bf16(m, n, X.data_ptr(), m, hi.data_ptr(), lo.data_ptr(), m, 0) == 0
    return hi, lo


def entry(kind, seed=0):
    """f(out, stream) for one entry point, an output, and the configuration that runs it."""
    import paper_2002_03258_gb300 as pkg
    lib = pkg.lib()
    d, s = torch.float64, torch.float32
    if kind == "r_d":
        A, B, out = random(1000, 2000, d, seed), random(2000, 16, d, seed + 1), torch.empty((16, 1000), dtype=d, device="cuda")
        return (lambda o, st: lib.tsm2r_d(1000, 2000, 16, A.data_ptr(), 1000, B.data_ptr(), 2000, o.data_ptr(), 1000, st),
                out, "r_f64_tc_kc16")
    if kind == "t_d":
        A, B, out = random(2000, 1000, d, seed), random(2000, 16, d, seed + 1), torch.empty((16, 1000), dtype=d, device="cuda")
        return (lambda o, st: lib.tsm2r_t_d(2000, 1000, 16, A.data_ptr(), 2000, B.data_ptr(), 2000, o.data_ptr(), 1000, st),
                out, "t_f64_tc_kc16")
    if kind == "l_d":
        A, B, out = random(4000, 32, d, seed), random(32, 32, d, seed + 1), torch.empty((32, 4000), dtype=d, device="cuda")
        return (lambda o, st: lib.tsm2l_d(4000, 32, 32, A.data_ptr(), 4000, B.data_ptr(), 32, o.data_ptr(), 4000, st),
                out, "l_f64_kc32_s_f64_tc")
    if kind == "rankk_d":
        A, B, out = random(500, 16, d, seed), random(600, 16, d, seed + 1), torch.empty((600, 500), dtype=d, device="cuda")
        return (lambda o, st: lib.tsm2_rankk_d(500, 600, 16, A.data_ptr(), 500, B.data_ptr(), 600, o.data_ptr(), 500, st),
                out, "rankk_f64_tc")
    if kind == "bf16":
        (hi, lo), B = bf16_pair(1024, 4096), random(4096, 16, s, seed + 1)
        out = torch.empty((16, 1024), dtype=s, device="cuda")
        return (lambda o, st: lib.tsm2r_bf16(1024, 4096, 16, hi.data_ptr(), lo.data_ptr(), 1024, B.data_ptr(), 4096,
                                             o.data_ptr(), 1024, st), out, "tc_bf16_hilo")
    assert kind == "l_s"
    A, B, out = random(100000, 16, s, seed), random(16, 16, s, seed + 1), torch.empty((16, 100000), dtype=s, device="cuda")
    return (lambda o, st: lib.tsm2l_s(100000, 16, 16, A.data_ptr(), 100000, B.data_ptr(), 16, o.data_ptr(), 100000, st),
            out, "l_f32_kc16")


def capture(calls, stream):
    import paper_2002_03258_gb300 as pkg
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=stream):
        for f, out, cfg in calls:
            assert f(out, stream.cuda_stream) == 0, pkg.tsm2_get_last_error_string()
            assert pkg.tsm2_last_config() == cfg
    return g


KINDS = ["r_d", "t_d", "l_d", "rankk_d", "bf16", "l_s"]


@pytest.mark.parametrize("kind", KINDS)
def test_captured_call_replays_after_the_workspace_has_grown(kind):
    """The same bits as alone, replay after replay, also when a larger call has
    replaced the workspace that the stream had at the capture."""
    import paper_2002_03258_gb300 as pkg
    s = torch.cuda.Stream()
    f, out, cfg = entry(kind)
    torch.cuda.synchronize()
    assert f(out, s.cuda_stream) == 0
    s.synchronize()
    want = out.clone()
    assert not torch.isnan(want).any()
    g = capture([(f, out, cfg)], s)
    big = random(3000, 6000, torch.float64, 7), random(6000, 16, torch.float64, 8)
    other = torch.empty((16, 3000), dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    for _ in range(3):
        out.fill_(float("nan"))
        g.replay()
        torch.cuda.synchronize()
        assert torch.equal(out, want)
        assert pkg.tsm2r_d(3000, 6000, 16, big[0].data_ptr(), 3000, big[1].data_ptr(), 6000, other.data_ptr(), 3000,
                           s.cuda_stream) == 0
        s.synchronize()
    assert pkg.tsm2_get_device_status(0) == 0


def test_graphs_captured_on_one_stream_replay_beside_each_other():
    import paper_2002_03258_gb300 as pkg
    s = torch.cuda.Stream()
    calls = [entry(kind, 20 * i) for i, kind in enumerate(KINDS)]
    torch.cuda.synchronize()
    for f, out, _ in calls:
        assert f(out, s.cuda_stream) == 0
    s.synchronize()
    want = [out.clone() for _, out, _ in calls]
    graphs = [capture([c] * 3, s) for c in calls]
    streams = [torch.cuda.Stream() for _ in calls]
    torch.cuda.synchronize()
    for _ in range(20):
        for g, st in zip(graphs, streams):
            with torch.cuda.stream(st):
                g.replay()
    torch.cuda.synchronize()
    assert pkg.tsm2_get_device_status(0) == 0
    for (_, out, cfg), w in zip(calls, want):
        assert torch.equal(out, w), cfg


def test_scratch_of_a_graph_is_given_back():
    import gc
    import paper_2002_03258_gb300 as pkg
    s = torch.cuda.Stream()
    f, out, cfg = entry("r_d")
    torch.cuda.synchronize()
    assert f(out, s.cuda_stream) == 0
    s.synchronize()
    used = []
    for _ in range(6):
        g = capture([(f, out, cfg)], s)
        g.replay()
        torch.cuda.synchronize()
        del g
        gc.collect()
        assert f(out, s.cuda_stream) == 0
        torch.cuda.synchronize()
        used.append(torch.cuda.mem_get_info()[0])
    # (the scratch of one such graph is 20 MB or more; the pool and the driver may keep a little)
    assert used[2] - used[-1] < 16 << 20, used
    assert pkg.tsm2_get_device_status(0) == 0


def test_scratch_of_a_graph_is_what_its_calls_need():
    """Small calls captured on a stream whose workspace is large: the first
    shares nothing with a later, larger one, which the next small one then uses."""
    import paper_2002_03258_gb300 as pkg
    lib, s = pkg.lib(), torch.cuda.Stream()
    m, n = 1 << 20, 64
    A, D, out = random(m, n, torch.float64, 1), random(m, 16, torch.float64, 2), torch.empty((16, n), dtype=torch.float64, device="cuda")
    small = [entry(k, 40 + i) for i, k in enumerate(("l_s", "rankk_d", "r_d", "rankk_d"))]
    torch.cuda.synchronize()
    assert lib.tsm2r_t_d(m, n, 16, A.data_ptr(), m, D.data_ptr(), m, out.data_ptr(), n, s.cuda_stream) == 0
    for f, o, _ in small:
        assert f(o, s.cuda_stream) == 0
    s.synchronize()
    want = [o.clone() for _, o, _ in small]
    free = torch.cuda.mem_get_info()[0]
    g = capture(small, s)
    assert free - torch.cuda.mem_get_info()[0] < 96 << 20
    for _, o, _ in small:
        o.fill_(float("nan"))
    g.replay()
    torch.cuda.synchronize()
    assert pkg.tsm2_get_device_status(0) == 0
    assert all(torch.equal(o, w) for (_, o, _), w in zip(small, want))
