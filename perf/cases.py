"""The work that users of this library have it do, as cases that can be timed.

Shapes come from the paper's sweeps that the tests and the benchmark run
(TSM2R n x n x k, TSM2L m x n x n), from the 1024 x 1024 x 8 example, from the
differentiable, batched and bfloat16 workloads, and from ragged sizes without
padding.  Every case goes through the Python entry points on column-major
torch tensors; inputs are drawn on the GPU from the seed alone.
"""
import math

import torch

import paper_2002_03258_gb300 as tsm2
import paper_2002_03258_gb300.batched as batched
from paper_2002_03258_gb300.autograd import tsm2r_mm

DTYPES = {"f32": torch.float32, "f64": torch.float64}
SIZES = {"f32": 4, "f64": 8}


def listed():
    return [
        # One small product in double precision (a block of an orthogonalisation
        # or of a small solver): latency, launches and host work count.
        {"name": "r_f64_1024x1024x8", "kind": "r", "dtype": "f64", "m": 1024, "n": 1024, "k": 8, "pad": False},
        # The paper's TSM2R in double precision: a large square A against a block of vectors.
        {"name": "r_f64_20480x20480x16", "kind": "r", "dtype": "f64", "m": 20480, "n": 20480, "k": 16, "pad": False},
        # TSM2R in single precision, the middle of the sweep.
        {"name": "r_f32_10240x10240x8", "kind": "r", "dtype": "f32", "m": 10240, "n": 10240, "k": 8, "pad": False},
        # TSM2R in single precision, the largest of the sweep.
        {"name": "r_f32_30720x30720x16", "kind": "r", "dtype": "f32", "m": 30720, "n": 30720, "k": 16, "pad": False},
        # A matrix as a program happens to have it: odd sizes, no padding of the leading dimensions.
        {"name": "r_f32_10001x4099x5", "kind": "r", "dtype": "f32", "m": 10001, "n": 4099, "k": 5, "pad": False},
        # TSM2L, the smallest of the sweep (k-means, tall factors): a call of some ten microseconds.
        {"name": "l_f32_1048576x8x8", "kind": "l", "dtype": "f32", "m": 1 << 20, "n": 8, "k": 8, "pad": False},
        # TSM2L, the largest of the sweep.
        {"name": "l_f32_8388608x32x32", "kind": "l", "dtype": "f32", "m": 1 << 23, "n": 32, "k": 32, "pad": False},
        # TSM2L in double precision.
        {"name": "l_f64_1048576x32x32", "kind": "l", "dtype": "f64", "m": 1 << 20, "n": 32, "k": 32, "pad": False},
        # A training step on a TSM2R layer: forward, dA and dB through autograd.
        {"name": "grad_f32_16384x16384x8", "kind": "grad", "dtype": "f32", "m": 16384, "n": 16384, "k": 8, "pad": False},
        # The same in double precision, as for gradient checks and scientific models.
        {"name": "grad_f64_4096x4096x16", "kind": "grad", "dtype": "f64", "m": 4096, "n": 4096, "k": 16, "pad": False},
        # A batch of uneven problems in one launch, leading dimensions rounded up to 512 bytes.
        {"name": "batch_f32_64", "kind": "batch", "dtype": "f32", "count": 64, "shapes": 0},
        # A kept as a bfloat16 hi + lo pair, binary32 accumulation.
        {"name": "bf16_hilo_16384x16384x16", "kind": "bf16", "dtype": "bf16", "m": 16384, "n": 16384, "k": 16, "lo": True},
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["r", "r", "r", "l", "l", "l", "grad", "grad", "batch", "bf16"])
    if kind == "batch":
        return {"kind": kind, "dtype": "f32", "count": _log_int(rng, 8, 40), "shapes": rng.randrange(1, 1 << 20)}
    if kind == "bf16":
        return {"kind": kind, "dtype": "bf16", "m": _log_int(rng, 1024, 16384) // 8 * 8, "n": _log_int(rng, 1024, 16384),
                "k": rng.randint(2, 16), "lo": rng.random() < 0.5}
    dtype = rng.choice(["f32", "f64"])
    pad = rng.random() < 0.6
    if kind == "r":
        top = 30720 if dtype == "f32" else 20480
        return {"kind": kind, "dtype": dtype, "m": _log_int(rng, 512, top), "n": _log_int(rng, 512, top),
                "k": rng.randint(2, 16), "pad": pad}
    if kind == "l":
        n = rng.randint(4, 32)
        top = 1 << 23 if dtype == "f32" else 1 << 22
        return {"kind": kind, "dtype": dtype, "m": _log_int(rng, 1 << 14, top), "n": n,
                "k": n if rng.random() < 0.7 else rng.randint(2, 32), "pad": pad}
    top = 16384 if dtype == "f32" else 6144
    return {"kind": kind, "dtype": dtype, "m": _log_int(rng, 512, top), "n": _log_int(rng, 512, top),
            "k": rng.randint(2, 16), "pad": True}


def _round_up(x, to):
    return (x + to - 1) // to * to


def _colmajor(rows, cols, dtype, pad, elem):
    """Column-major rows x cols; `pad`: the leading dimension rounded up to 512 bytes."""
    return tsm2.empty_colmajor(rows, cols, dtype, "cuda", _round_up(rows, 512 // elem) if pad else rows)


def _uniform(gen, rows, cols, dtype, pad, elem):
    x = _colmajor(rows, cols, dtype, pad, elem)
    x.t().uniform_(-1.0, 1.0, generator=gen)
    return x


def _batch_shapes(case):
    """Half TSM2R (n x n x k), half TSM2L (m x n x n), as in the batched workload."""
    gen = torch.Generator()
    gen.manual_seed(case["shapes"])
    out = []
    for i in range(case["count"]):
        a, b = torch.rand(2, generator=gen, dtype=torch.float64).tolist()
        if i % 2 == 0:
            n = 512 + int(a * (8192 - 512 + 1))
            out.append(("r", n, n, 2 + int(b * 15)))
        else:
            m = (1 << 14) + int(a * ((1 << 20) - (1 << 14) + 1))
            n = 4 + int(b * 29)
            out.append(("l", m, n, n))
    return out


def prepare(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    kind = case["kind"]
    if kind in ("r", "l"):
        dt, e = DTYPES[case["dtype"]], SIZES[case["dtype"]]
        return {"kind": kind, "A": _uniform(gen, case["m"], case["n"], dt, case["pad"], e),
                "B": _uniform(gen, case["n"], case["k"], dt, case["pad"], e)}
    if kind == "grad":
        dt, e = DTYPES[case["dtype"]], SIZES[case["dtype"]]
        A, B, dC = (_colmajor(r, c, dt, case["pad"], e)
                    for r, c in ((case["m"], case["n"]), (case["n"], case["k"]), (case["m"], case["k"])))
        scale = 1.0 / math.sqrt(case["n"])
        A.t().normal_(0.0, scale, generator=gen)
        B.t().normal_(0.0, scale, generator=gen)
        dC.t().normal_(0.0, 1.0, generator=gen)
        return {"kind": kind, "A": A.requires_grad_(True), "B": B.requires_grad_(True), "dC": dC}
    if kind == "batch":
        mats, probs = [], []
        for op, m, n, k in _batch_shapes(case):
            A, B = (_uniform(gen, r, c, torch.float32, True, 4) for r, c in ((m, n), (n, k)))
            C = _colmajor(m, k, torch.float32, True, 4)
            mats.append((A, B, C))
            probs.append(batched.problem(op, m, n, k, A.data_ptr(), A.stride(1), B.data_ptr(), B.stride(1),
                                         C.data_ptr(), C.stride(1)))
        return {"kind": kind, "mats": mats, "plan": batched.BatchPlan(probs)}
    # bfloat16: random signs, magnitudes log-uniform in [1e-3, 1e3]
    m, n, k = case["m"], case["n"], case["k"]
    X = _colmajor(m, n, torch.float32, False, 4)
    X.t().uniform_(-1.0, 1.0, generator=gen)
    X = X.sign() * torch.exp((X.abs() * 2.0 - 1.0) * math.log(1e3))
    hi = X.to(torch.bfloat16)
    lo = (X - hi.float()).to(torch.bfloat16) if case["lo"] else None
    return {"kind": kind, "hi": hi, "lo": lo, "B": _uniform(gen, n, k, torch.float32, False, 4)}


def run(state):
    kind = state["kind"]
    if kind == "r":
        return tsm2.tsm2r(state["A"], state["B"])
    if kind == "l":
        return tsm2.tsm2l(state["A"], state["B"])
    if kind == "grad":
        C = tsm2r_mm(state["A"], state["B"])
        dA, dB = torch.autograd.grad(C, (state["A"], state["B"]), state["dC"])
        return [C, dA, dB]
    if kind == "batch":
        state["plan"].graph_launch(torch.cuda.current_stream().cuda_stream)
        return [C for _, _, C in state["mats"]]
    hi, lo, B = state["hi"], state["lo"], state["B"]
    (m, n), k = hi.shape, B.shape[1]
    C = tsm2.empty_colmajor(m, k, torch.float32, hi.device)
    tsm2.check(tsm2.tsm2r_bf16(m, n, k, hi.data_ptr(), lo.data_ptr() if lo is not None else None, hi.stride(1),
                               B.data_ptr(), B.stride(1), C.data_ptr(), C.stride(1),
                               torch.cuda.current_stream().cuda_stream))
    return C


def work(case):
    if case["kind"] == "batch":
        shapes = _batch_shapes(case)
        return {"bytes": sum(4 * (m * n + n * k + m * k) for _, m, n, k in shapes),
                "flops": sum(2 * m * n * k for _, m, n, k in shapes)}
    m, n, k = case["m"], case["n"], case["k"]
    if case["kind"] == "bf16":
        return {"bytes": (4 if case["lo"] else 2) * m * n + 4 * (n * k + m * k), "flops": 2 * m * n * k}
    e = SIZES[case["dtype"]]
    if case["kind"] == "grad":  # in: A, B, dC; out: C, dA, dB
        return {"bytes": e * 2 * (m * n + n * k + m * k), "flops": 6 * m * n * k}
    return {"bytes": e * (m * n + n * k + m * k), "flops": 2 * m * n * k}


def _halves(x):
    """x = high + low, each short enough that products of two of them are exact (Veltkamp's split)."""
    t = x * 134217729.0
    high = t - (t - x)
    return high, x - high


def _product(A, B):
    """A @ B in 64 bits.  binary32 and bfloat16 inputs: the inner dimension in short blocks, so that
    the rounding of the sums stays small.  binary64 inputs: every product and every sum with its
    rounding error (Dekker, Knuth), so that the result is right to about its last bit."""
    out = torch.zeros((A.shape[0], B.shape[1]), dtype=torch.float64, device=A.device)
    n = A.shape[1]
    if A.dtype != torch.float64:
        for j in range(0, n, 256):
            out += A[:, j:j + 256].double() @ B[j:j + 256].double()
        return out
    (Ah, Al), (Bh, Bl) = _halves(A), _halves(B)
    low = torch.zeros_like(out)
    for j in range(n):
        a, ah, al = A[:, j:j + 1], Ah[:, j:j + 1], Al[:, j:j + 1]
        b, bh, bl = B[j:j + 1], Bh[j:j + 1], Bl[j:j + 1]
        p = a * b
        low += ((ah * bh - p) + ah * bl + al * bh) + al * bl
        s = out + p
        t = s - out
        low += (out - (s - t)) + (p - t)
        out = s
    return out + low


def exact(case, seed):
    s = prepare(case, seed)
    if s["kind"] in ("r", "l"):
        return _product(s["A"], s["B"])
    if s["kind"] == "grad":
        A, B, dC = s["A"].detach(), s["B"].detach(), s["dC"]
        return [_product(A, B), _product(dC, B.t()), _product(A.t(), dC)]
    if s["kind"] == "batch":
        return [_product(A, B) for A, B, _ in s["mats"]]
    A = s["hi"].double()
    if s["lo"] is not None:
        A += s["lo"].double()
    return _product(A, s["B"])
