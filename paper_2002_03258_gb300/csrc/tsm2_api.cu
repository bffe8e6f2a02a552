// C ABI of the library (declared in include/tsm2.h): argument checking,
// choice of kernel path and configuration, tensor-map encoding, workspace
// management and the device status word.
#include "common.cuh"
#include "f64s.h"
#include "f64tc.h"
#include "internal.h"
#include "shift.h"
#include "tsm2.h"

#include <cuda.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
#include <cstdarg>
#include <cstdio>
#include <cstring>
#include <map>
#include <memory>
#include <mutex>
#include <string>
#include <utility>
#include <vector>

namespace tsm2 {
namespace {

__device__ unsigned int g_status_word;  // per device; bits kStatusTimeout, kStatusBounds set by kernels

thread_local std::string t_last_error = "no error";
thread_local const char *t_last_config = "none";
thread_local const char *t_last_host_copy = "none";  // copy path of the last host-operand call

int64_t g_wait_ns = 1000000000LL;
int g_path = 0;                    // 0: automatic; 1: element-wise; 2: FMA units (no tensor cores for binary64)
int g_grid_override = 0;
int g_host_copy = 0;               // 0: SM copies for device-mapped page-locked host buffers; 1: copy engines
int g_balance = 0;                 // 0: TSM2L row blocks claimed at run time; 1: static; 2: 0 + batched shares always adapted
thread_local int t_grid_cap = 0;   // > 0: upper bound of the product kernels' persistent grid (this thread)
unsigned long long *g_trace = nullptr;
int64_t g_trace_blocks = 0;

tsm2_status set_error(tsm2_status s, const char *fmt, ...) {
    char buf[512];
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(buf, sizeof buf, fmt, ap);
    va_end(ap);
    t_last_error = buf;
    return s;
}

tsm2_status cuda_error(cudaError_t e, const char *what) {
    return set_error(TSM2_ERR_CUDA, "%s: %s (%s)", what, cudaGetErrorName(e), cudaGetErrorString(e));
}

// ---- per-device state ------------------------------------------------------

struct DeviceState {
    bool init = false;
    int sm_count = 0;
    unsigned *status = nullptr;  // device address of g_status_word
};

std::mutex g_mu;
DeviceState g_dev[64];

struct Workspace {
    std::mutex mu;  // held from workspace() to the last launch of the call (taken after g_mu where both are)
    void *ptr = nullptr;
    size_t bytes = 0;
    size_t counter_bytes = 0;
};
std::map<std::pair<int, uintptr_t>, Workspace> g_ws;  // (device, stream) -> workspace; entries stay

// A call's hold on its stream's workspace.  Calls of several kernels pass data
// from one to the next there (digits or pieces of B, partial sums), and any
// call may grow it, so no other host thread's call on the same stream may come
// between workspace() and the last launch.
struct Scratch {
    void *ws = nullptr;       // 256-byte aligned
    int *counters = nullptr;  // zero between launches
    std::unique_lock<std::mutex> hold;
};

tsm2_status device_state(DeviceState **out) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return cuda_error(e, "cudaGetDevice");
    if (dev < 0 || dev >= 64) return set_error(TSM2_ERR_UNSUPPORTED, "device ordinal %d out of range", dev);
    std::lock_guard<std::mutex> lk(g_mu);
    DeviceState &d = g_dev[dev];
    if (!d.init) {
        e = cudaDeviceGetAttribute(&d.sm_count, cudaDevAttrMultiProcessorCount, dev);
        if (e != cudaSuccess) return cuda_error(e, "cudaDeviceGetAttribute");
        void *p = nullptr;
        e = cudaGetSymbolAddress(&p, g_status_word);
        if (e != cudaSuccess) return cuda_error(e, "cudaGetSymbolAddress(status)");
        d.status = static_cast<unsigned *>(p);
        d.init = true;
    }
    *out = &d;
    return TSM2_SUCCESS;
}

// The workspace of (current device, stream), locked for this call.
tsm2_status lock_workspace(cudaStream_t stream, Scratch &s, Workspace **out) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return cuda_error(e, "cudaGetDevice");
    Workspace *w = nullptr;
    {
        std::lock_guard<std::mutex> lk(g_mu);
        w = &g_ws[{dev, reinterpret_cast<uintptr_t>(stream)}];
    }
    s.hold = std::unique_lock<std::mutex>(w->mu);
    *out = w;
    return TSM2_SUCCESS;
}

tsm2_status is_capturing(cudaStream_t stream, bool *capturing) {
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    cudaError_t e = cudaStreamIsCapturing(stream, &cap);
    if (e == cudaErrorStreamCaptureImplicit) {  // (the legacy stream, while another is captured)
        (void)cudaGetLastError();
        e = cudaSuccess;
        cap = cudaStreamCaptureStatusNone;
    }
    if (e != cudaSuccess) return cuda_error(e, "cudaStreamIsCapturing");
    *capturing = cap != cudaStreamCaptureStatusNone;
    return TSM2_SUCCESS;
}

// Scratch of captured calls.  A graph is replayed on any stream, beside others
// and after the stream's workspace has been grown (freed), so the calls that
// are captured on a stream share an allocation that belongs to their graph:
// a user object of the graph marks it unused when the last of the graph and
// its executables is gone, and a later call frees it.
struct GraphScratch {
    int dev = 0;
    unsigned long long capture = 0;
    cudaStream_t stream = nullptr;
    void *ptr = nullptr;
    size_t bytes = 0, counter_bytes = 0;
    std::atomic<bool> unused{false};
};
std::mutex g_graph_mu;  // (not taken by graph_is_gone, so held over CUDA calls too)
std::vector<std::unique_ptr<GraphScratch>> &g_graph_scratch = *new std::vector<std::unique_ptr<GraphScratch>>;
std::atomic<int> g_graph_unused{0};

void CUDART_CB graph_is_gone(void *p) {  // (may not call CUDA)
    static_cast<GraphScratch *>(p)->unused = true;
    ++g_graph_unused;
}

// cudaMalloc and cudaFree are not recorded in a graph and harm no capture, but
// are refused while one goes on anywhere unless the thread says so.
struct RelaxedCapture {
    cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
    RelaxedCapture() { cudaThreadExchangeStreamCaptureMode(&mode); }
    ~RelaxedCapture() { cudaThreadExchangeStreamCaptureMode(&mode); }
};

void free_unused_graph_scratch() {
    std::lock_guard<std::mutex> lk(g_graph_mu);
    RelaxedCapture relaxed;
    int cur = 0;
    cudaGetDevice(&cur);
    for (size_t i = 0; i < g_graph_scratch.size();) {
        if (!g_graph_scratch[i]->unused) {
            ++i;
            continue;
        }
        cudaSetDevice(g_graph_scratch[i]->dev);
        cudaFree(g_graph_scratch[i]->ptr);  // (waits for replays still running)
        g_graph_scratch.erase(g_graph_scratch.begin() + (int64_t)i);
        --g_graph_unused;
    }
    cudaSetDevice(cur);
}

// Zeroes memory now, whatever is captured on other streams.
cudaError_t zero_now(void *p, size_t bytes) {
    cudaStream_t side = nullptr;
    cudaError_t e = cudaStreamCreateWithFlags(&side, cudaStreamNonBlocking);
    if (e != cudaSuccess) return e;
    e = cudaMemsetAsync(p, 0, bytes, side);
    const cudaError_t e2 = cudaStreamSynchronize(side);
    cudaStreamDestroy(side);
    return e != cudaSuccess ? e : e2;
}

// Scratch of the graph that `stream` is being captured into, for a call that
// needs `slot_bytes` (the calls of a stream come one after the other, so the
// largest serves those after it; `w`, the stream's workspace, would do).
tsm2_status graph_scratch(cudaStream_t stream, const Workspace &w, size_t slot_bytes, Scratch &s) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return cuda_error(e, "cudaGetDevice");
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    unsigned long long id = 0;
    cudaGraph_t graph = nullptr;
    e = cudaStreamGetCaptureInfo(stream, &cap, &id, &graph);
    if (e != cudaSuccess) return cuda_error(e, "cudaStreamGetCaptureInfo");
    GraphScratch *g = nullptr;
    {
        std::lock_guard<std::mutex> lk(g_graph_mu);
        for (auto &have : g_graph_scratch)
            if (have->dev == dev && have->capture == id && have->stream == stream && !have->unused &&
                have->bytes >= w.counter_bytes + slot_bytes)
                g = have.get();
    }
    if (!g) {
        RelaxedCapture relaxed;
        auto fresh = std::make_unique<GraphScratch>();
        fresh->dev = dev;
        fresh->capture = id;
        fresh->stream = stream;
        fresh->bytes = w.counter_bytes + slot_bytes;
        fresh->counter_bytes = w.counter_bytes;
        e = cudaMalloc(&fresh->ptr, fresh->bytes);
        if (e != cudaSuccess) return cuda_error(e, "cudaMalloc(scratch of a captured graph)");
        cudaUserObject_t owner = nullptr;
        if (w.counter_bytes) e = zero_now(fresh->ptr, w.counter_bytes);
        if (e == cudaSuccess) e = cudaUserObjectCreate(&owner, fresh.get(), graph_is_gone, 1, cudaUserObjectNoDestructorSync);
        if (e != cudaSuccess) {
            cudaFree(fresh->ptr);
            return cuda_error(e, "scratch of a captured graph");
        }
        g = fresh.get();
        {
            std::lock_guard<std::mutex> lk(g_graph_mu);
            g_graph_scratch.push_back(std::move(fresh));
        }
        e = cudaGraphRetainUserObject(graph, owner, 1, cudaGraphUserObjectMove);
        if (e != cudaSuccess) {
            cudaUserObjectRelease(owner, 1);  // (unused from here on)
            return cuda_error(e, "cudaGraphRetainUserObject");
        }
    }
    s.counters = static_cast<int *>(g->ptr);
    s.ws = static_cast<char *>(g->ptr) + g->counter_bytes;
    return TSM2_SUCCESS;
}

// At least `slot_bytes` behind `counter_bytes` that are zero: of `w`, which the
// caller has locked, or while the stream is captured of the graph's own.  The
// counters return to zero after every completed launch, so they are only
// cleared when (re)allocated.
tsm2_status grow_workspace(cudaStream_t stream, Workspace &w, size_t counter_bytes, size_t slot_bytes, Scratch &s) {
    counter_bytes = (counter_bytes + 255) / 256 * 256;
    bool capturing = false;
    const tsm2_status st = is_capturing(stream, &capturing);
    if (st != TSM2_SUCCESS) return st;
    if (!capturing && g_graph_unused > 0) free_unused_graph_scratch();
    if (!w.ptr || w.counter_bytes < counter_bytes || w.bytes < w.counter_bytes + slot_bytes) {
        // Growing needs a synchronize, which may not run while the stream is
        // being captured into a graph.
        if (capturing)
            return set_error(TSM2_ERR_UNSUPPORTED,
                             "the stream's workspace must grow, which cannot happen during stream capture: call the "
                             "largest shape once on this stream before capturing");
        const size_t cb = std::max(counter_bytes, w.counter_bytes);
        const size_t nb = std::max((cb + slot_bytes) * 5 / 4 + 4096, w.bytes);
        cudaError_t e;
        if (w.ptr) {
            // Pending work of this stream may still use the old buffer.
            e = cudaStreamSynchronize(stream);
            if (e != cudaSuccess) return cuda_error(e, "cudaStreamSynchronize(workspace)");
            cudaFree(w.ptr);
            w.ptr = nullptr;
            w.bytes = w.counter_bytes = 0;
        }
        void *p = nullptr;
        e = cudaMalloc(&p, nb);
        if (e != cudaSuccess) return cuda_error(e, "cudaMalloc(workspace)");
        e = cudaMemsetAsync(p, 0, cb, stream);
        if (e != cudaSuccess) {
            cudaFree(p);
            return cuda_error(e, "cudaMemsetAsync(workspace counters)");
        }
        w.ptr = p;
        w.bytes = nb;
        w.counter_bytes = cb;
    }
    if (capturing) return graph_scratch(stream, w, slot_bytes, s);
    s.counters = static_cast<int *>(w.ptr);
    s.ws = static_cast<char *>(w.ptr) + w.counter_bytes;
    return TSM2_SUCCESS;
}

tsm2_status workspace(cudaStream_t stream, size_t counter_bytes, size_t slot_bytes, Scratch &s) {
    Workspace *w = nullptr;
    const tsm2_status st = lock_workspace(stream, s, &w);
    return st == TSM2_SUCCESS ? grow_workspace(stream, *w, counter_bytes, slot_bytes, s) : st;
}

// Claim counters of the resident-B schedules: the first two counters of the
// stream's workspace (zero between launches; the kernel rearms them).  While
// the stream is being captured a workspace cannot be created, and the launch
// then keeps the static partition (nullptr).
tsm2_status claim_counters(cudaStream_t stream, int **claims, Scratch &s) {
    *claims = nullptr;
    if (g_balance == 1) return TSM2_SUCCESS;
    Workspace *w = nullptr;
    tsm2_status st = lock_workspace(stream, s, &w);
    if (st != TSM2_SUCCESS) return st;
    if (!w->ptr || w->counter_bytes < 2 * sizeof(int)) {
        bool capturing = false;
        st = is_capturing(stream, &capturing);
        if (st != TSM2_SUCCESS || capturing) return st;
    }
    st = grow_workspace(stream, *w, 2 * sizeof(int), 0, s);
    if (st == TSM2_SUCCESS) *claims = s.counters;
    return st;
}

// ---- tensor maps -----------------------------------------------------------

typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                  const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_fn() {
    static EncodeTiledFn fn = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<EncodeTiledFn>(p);
    });
    return fn;
}

tsm2_status encode_2d_ex(CUtensorMap *map, CUtensorMapDataType dtype, int elem, const void *base, int64_t rows,
                         int64_t cols, int64_t ld, int box_rows, int box_cols, CUtensorMapSwizzle swizzle) {
    EncodeTiledFn fn = encode_fn();
    if (!fn) return set_error(TSM2_ERR_CUDA, "cuTensorMapEncodeTiled unavailable from the driver");
    const cuuint64_t dims[2] = {(cuuint64_t)rows, (cuuint64_t)cols};
    const cuuint64_t strides[1] = {(cuuint64_t)(ld * elem)};
    const cuuint32_t box[2] = {(cuuint32_t)box_rows, (cuuint32_t)box_cols};
    const cuuint32_t estr[2] = {1, 1};
    const auto encode = [&]() {
        return fn(map, dtype, 2, const_cast<void *>(base), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, swizzle,
                  CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    };
    CUresult r = encode();
    int dev = 0;
    // A host thread that has made no runtime call yet has no context.
    if (r == CUDA_ERROR_INVALID_CONTEXT && cudaGetDevice(&dev) == cudaSuccess && cudaSetDevice(dev) == cudaSuccess) r = encode();
    if (r != CUDA_SUCCESS) return set_error(TSM2_ERR_CUDA, "cuTensorMapEncodeTiled failed (CUresult %d)", (int)r);
    return TSM2_SUCCESS;
}

tsm2_status encode_2d(CUtensorMap *map, int elem, const void *base, int64_t rows, int64_t cols, int64_t ld,
                      int box_rows, int box_cols) {
    return encode_2d_ex(map, elem == 8 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT64 : CU_TENSOR_MAP_DATA_TYPE_FLOAT32, elem, base, rows,
                        cols, ld, box_rows, box_cols, CU_TENSOR_MAP_SWIZZLE_NONE);
}

// ---- C-column widths --------------------------------------------------------

// Smallest compiled C-column width (KC) that holds a chunk of k columns: the
// kernels compute all KC columns (padding columns of B read as zero), so a
// close fit saves FMAs in the FMA-bound shapes.
int kc_for(int k) {
    static const int widths[] = {2, 4, 8, 12, 16, 24, 32};
    for (int w : widths)
        if (w >= k) return w;
    return 32;
}

// ---- argument checks ---------------------------------------------------------

bool ranges_overlap(const void *a, size_t abytes, const void *b, size_t bbytes) {
    if (!a || !b || !abytes || !bbytes) return false;
    const uintptr_t a0 = (uintptr_t)a, b0 = (uintptr_t)b;
    return a0 < b0 + bbytes && b0 < a0 + abytes;
}

size_t span_bytes(int64_t rows, int64_t cols, int64_t ld, int elem) {
    if (rows <= 0 || cols <= 0) return 0;
    return (size_t)(((cols - 1) * ld + rows) * elem);
}

tsm2_status check_args(const char *fn, int64_t m, int64_t n, int64_t k, const void *A, int64_t lda, const void *B,
                       int64_t ldb, const void *C, int64_t ldc, int elem) {
    if (m < 0 || n < 0 || k < 0)
        return set_error(TSM2_ERR_INVALID_VALUE, "%s: negative dimension (m=%lld n=%lld k=%lld)", fn, (long long)m,
                         (long long)n, (long long)k);
    if (lda < (m > 1 ? m : 1)) return set_error(TSM2_ERR_INVALID_VALUE, "%s: lda=%lld < max(1,m)", fn, (long long)lda);
    if (ldb < (n > 1 ? n : 1)) return set_error(TSM2_ERR_INVALID_VALUE, "%s: ldb=%lld < max(1,n)", fn, (long long)ldb);
    if (ldc < (m > 1 ? m : 1)) return set_error(TSM2_ERR_INVALID_VALUE, "%s: ldc=%lld < max(1,m)", fn, (long long)ldc);
    if (m > 0 && k > 0 && C == nullptr) return set_error(TSM2_ERR_INVALID_VALUE, "%s: C is NULL", fn);
    if (m > 0 && n > 0 && k > 0 && A == nullptr) return set_error(TSM2_ERR_INVALID_VALUE, "%s: A is NULL", fn);
    if (m > 0 && n > 0 && k > 0 && B == nullptr) return set_error(TSM2_ERR_INVALID_VALUE, "%s: B is NULL", fn);
    if (m > 0 && k > 0) {
        const size_t cb = span_bytes(m, k, ldc, elem);
        if ((n > 0 && ranges_overlap(C, cb, A, span_bytes(m, n, lda, elem))) ||
            (n > 0 && ranges_overlap(C, cb, B, span_bytes(n, k, ldb, elem))))
            return set_error(TSM2_ERR_INVALID_VALUE, "%s: C overlaps A or B", fn);
    }
    return TSM2_SUCCESS;
}

bool aligned16(const void *p) { return ((uintptr_t)p & 15u) == 0; }

// The column classes of A (shift.h): P maps that start at 16-byte boundaries.
tsm2_status column_classes(ColumnClasses *out, int elem, const void *A, int64_t m, int64_t n, int64_t lda,
                           int box_rows = 256) {
    const int P = 16 / elem;
    for (int r = 0; r < P; ++r) {
        const uintptr_t start = (uintptr_t)A + (uintptr_t)r * (uintptr_t)lda * elem;
        const uintptr_t base = start & ~(uintptr_t)15;
        out->shift[r] = (int)((start - base) / elem);
        out->cols[r] = (int)((n - r + P - 1) / P);
        if (r >= n) {
            out->shift[r] = out->shift[0];
            out->cols[r] = 0;
            out->map[r] = out->map[0];
            continue;
        }
        const tsm2_status st = encode_2d(&out->map[r], elem, reinterpret_cast<const void *>(base), m + out->shift[r],
                                         out->cols[r], P * lda, box_rows, kShiftStep / P);
        if (st != TSM2_SUCCESS) return st;
    }
    return TSM2_SUCCESS;
}

// ---- binary64 products with a short inner dimension ------------------------------

// The digits of B of a call: at most this much of the workspace, which a stream
// keeps; larger products run in slices.
constexpr int64_t kDigitBytes = 256 << 20;

// C(M x N) [+]= A(M x K) B(K x N), K <= kF64SMaxK, on the tensor cores
// (tsm2_f64s.cu); B's element (j, c) at B[j bes + c bcs].  A must be 16-byte
// aligned with 16-byte rows, or with split any multiple of 8 bytes.  *ran = false: not done (no tensor map describes A,
// or the workspace cannot grow: no memory, or stream capture).
tsm2_status product_f64s(DeviceState *dev, int64_t M, int64_t N, int64_t K, const void *A, int64_t lda, const void *B,
                         int64_t bes, int64_t bcs, void *C, int64_t ldc, bool accumulate, bool split,
                         const char *name, cudaStream_t stream, bool *ran) {
    *ran = false;
    F64SLaunch L;
    std::memset(&L, 0, sizeof L);
    tsm2_status st = split ? column_classes(&L.a, 8, A, M, K, lda, f64s_tile())
                           : encode_2d(&L.a.map[0], 8, A, M, K, lda, f64s_tile(), f64s_step());
    L.split = split;
    if (st != TSM2_SUCCESS) return TSM2_SUCCESS;
    const int64_t slice = std::min(N, kDigitBytes / (int64_t)f64s_digit_bytes(f64s_cols(), (int)K) * f64s_cols());
    Scratch scratch;
    st = workspace(stream, 0, f64s_digit_bytes(slice, (int)K), scratch);
    if (st != TSM2_SUCCESS) {
        (void)cudaGetLastError();  // (of the allocation)
        return TSM2_SUCCESS;
    }
    L.M = M;
    L.K = (int)K;
    L.A = static_cast<const double *>(A);
    L.lda = lda;
    L.bes = bes;
    L.bcs = bcs;
    L.ldc = ldc;
    L.accumulate = accumulate;
    L.digits = scratch.ws;
    L.status = dev->status;
    L.wait_ns = g_wait_ns;
    int grid = g_grid_override > 0 ? g_grid_override : dev->sm_count;
    if (t_grid_cap > 0 && grid > t_grid_cap) grid = t_grid_cap;
    L.blocks = grid < 1 ? 1 : grid;
    L.trace = g_trace;
    L.trace_blocks = g_trace_blocks;
    t_last_config = name;
    for (int64_t c = 0; c < N; c += slice) {
        L.N = std::min(slice, N - c);
        L.B = static_cast<const double *>(B) + c * bcs;
        L.C = static_cast<double *>(C) + c * ldc;
        const cudaError_t e = f64s_launch(L, stream);
        if (e != cudaSuccess) return cuda_error(e, "binary64 tensor-core kernel launch");
    }
    *ran = true;
    return TSM2_SUCCESS;
}

bool f64s_fits(int64_t M, int64_t N, int64_t K) {
    return K <= kF64SMaxK && M < (1ll << 31) - 4096 && N < (1ll << 30) &&
           (M / f64s_rows(true) + 1) * (N / f64s_cols() + 1) < (1ll << 30);
}

// Whether an m x n by n x k product with a short inner dimension goes there,
// else to the FMA kernels, whose time is that of n (in eights) times k (as
// compiled) FMAs per row, 1.8 us a unit for 2^20 rows; the tensor cores take
// 66 us (4 x 4) to 220 us (32 x 32) for them.  Measured on GB300 (FMA / tensor
// cores, us): 2^20 rows 4 x 4 62 / 66, 8 x 8 119 / 83, 16 x 4 119 / 76, 32 x 2
// 121 / 117, 16 x 16 455 / 114, 32 x 32 1732 / 222; 2^14 rows 4 x 4 9.0 / 8.9,
// 8 x 8 12.7 / 8.7, 32 x 32 79 / 16.  At 64 units there is a range of m that
// the FMA kernels do in one wave, 65536 rows 4 x 8 12.7 / 13.2, 16 x 4 12.7 /
// 14.6 (131072: 20.9 / 17.4, 21.0 / 18.3).
// An unaligned A (split) has the element-wise kernel beside it: 1048577 x 32 x
// 32 1742 / 227, x 16 x 16 442 / 117, x 8 x 8 115 / 87, 200001 x 16 x 4 27 / 21,
// but 50001 x 8 x 8 10.6 / 10.7, 16385 x 32 x 4 8.5 / 10.9, x 12 x 12 12.6 / 9.4.
bool f64s_pays(int64_t m, int64_t n, int64_t k, bool split) {
    const int64_t units = (n + 7) / 8 * 8 * kc_for((int)std::min<int64_t>(k, 32));
    if (!f64s_fits(m, k, n) || units < (n > 16 ? 96 : 64)) return false;
    return m >= 100000 || (split ? units >= 160 : units > 64 || m <= 40000);
}

// The same for the rank-k update, C(M x N) of K products each, whose FMA kernel
// takes 117 us for 2^20 rows of 64 products: 10^6 x 8 x 4 62 / 80, 12 x 4
// 90 / 89, 16 x 2 117 / 99, 8 x 8 117 / 80; 2048^2 x 2 37 / 31, 4096^2 x 2
// 134 / 88, x 16 515 / 80, 512^2 x 2 36 / 11 (any N from 16 on).  A tile is 128
// rows and writes the digits of B besides: few rows of many columns, 64 x 10^6 x
// 4 543 / 686, x 8 1012 / 710, 96 x 10^6 x 4 849 / 665, 64 x 20000 x 4 27 / 25,
// 16 x 1000 x 4 27 / 11.
bool f64s_pays_rankk(int64_t M, int64_t N, int64_t K) {
    if (M <= 64 && K <= 4 && N >= (1 << 16)) return false;
    return f64s_fits(M, N, K) && (N >= 16 || N * std::max<int64_t>(K, 4) >= 64);
}

// ---- the multiply ------------------------------------------------------------

// One column chunk with operands of any alignment (tsm2_shift.cu).  *ran =
// false: not done (no tensor map describes A, or the workspace cannot grow: no
// memory, or stream capture), the caller takes the element-wise kernel, which
// needs neither.
tsm2_status gemm_shift(DeviceState *dev, int elem, const GemmArgs &g, cudaStream_t stream, bool *ran) {
    *ran = false;
    int kc = 2;
    while (kc < g.k) kc = kc == 16 ? 24 : kc == 24 ? 32 : kc * 2;
    // Several rows per lane once that leaves every SM four stages and few idle
    // rows; below, one row per lane.  Measured on GB300, several / one, us:
    // 1000001 x 8 x 8 17.5 / 25.4, 300001 x 31 x 31 35.7 / 42.2, 20001 x 601 x 4
    // (5 stages per SM) 15.5 / 16.0, 601 x 20001 x 10 124 / 49.
    const int64_t upr = (g.n + kShiftStep - 1) / kShiftStep;
    const ShiftShape *shape = shift_shape(elem, kc, true);
    if (!shape) return set_error(TSM2_ERR_UNSUPPORTED, "no kernel configuration for k chunk %d", g.k);
    if (g.m < 4 * shape->rows || (g.m + shape->rows - 1) / shape->rows * upr < 4ll * dev->sm_count)
        shape = shift_shape(elem, kc, false);
    ShiftLaunch L;
    std::memset(&L, 0, sizeof L);
    L.g = g;
    tsm2_status st = column_classes(&L.a, elem, g.A, g.m, g.n, g.lda);
    if (st != TSM2_SUCCESS) return TSM2_SUCCESS;
    const int64_t num_rb = (g.m + shape->rows - 1) / shape->rows;
    int64_t grid = g_grid_override > 0 ? g_grid_override : dev->sm_count;
    if (t_grid_cap > 0 && grid > t_grid_cap) grid = t_grid_cap;
    L.splits = shift_splits(shape, num_rb, upr, (int)grid);
    grid = std::min<int64_t>(grid, num_rb * L.splits);
    Scratch scratch;
    if (L.splits > 1) {
        st = workspace(stream, (size_t)num_rb * sizeof(int), shift_slot_bytes(shape, num_rb, L.splits), scratch);
        if (st != TSM2_SUCCESS) {
            (void)cudaGetLastError();  // (of the allocation)
            return TSM2_SUCCESS;
        }
        L.slots = scratch.ws;
        L.counters = scratch.counters;
    }
    L.status = dev->status;
    L.wait_ns = g_wait_ns;
    L.grid = (int)grid;
    t_last_config = shape->name;
    const cudaError_t e = shift_launch(shape, L, stream);
    if (e != cudaSuccess) return cuda_error(e, "unaligned kernel launch");
    *ran = true;
    return TSM2_SUCCESS;
}

// Whether a binary64 column chunk (kc: its compiled width) goes to the tensor
// cores.  Their time hardly depends on k (A streamed at 4 TB/s when large, 25
// to 60 us when small), the FMA kernels' is 2 m n kc / 1.25 TFLOP/s and, from
// 8 columns on, a slow combine.  Measured on GB300, FMA kernel / tensor cores
// in us, on dense data (what is not certified costs more: see settle there):
//   TSM2R  kc 16: 20480^2 10790 / 787, 1024^2 80 / 26; kc 8: 4096^2 232 / 62,
//          1024^2 43 / 25, 512^2 42 / 21: always.
//          kc 4: 4096^2 121 / 61, 2048^2 41 / 34, 1024^2 25 / 26, 512 x 4096
//          29 / 34, 20480 x 512 80 / 58; short n in favour of the FMA kernels:
//          2^20 x 40 287 / 382.
//          kc 2: 8192^2 228 / 144, 4096^2 67 / 60, 2048^2 25 / 33, 20480 x 512
//          46 / 56, 200001 x 100 78 / 146.
//   TSM2L  n > 64: 2^20 x 200 x 16 5573 / 700, 16384 x 100 x 2 58 / 35, 131072 x
//          100 x 2 111 / 112: always.  n <= 64: every 256 rows end a row block,
//          which costs as much as the products of 24 inner indices or more:
//          2^20 x 64 x 16 1794 / 359, x 8 897 / 555, x 2 234 / 414; 131072 x 64 x
//          8 134 / 100, 40 x 8 85 / 90; 16384 x 40 x 8 46 / 37, 64 x 4 38 / 19.
// n below 16 leaves most of a stage empty.  An unaligned A (split) has the
// element-wise kernel beside it, which keeps the FMA units busy at small n;
// measured, element-wise / tensor cores: 4097^2 x 2 83 / 66, 20001 x 200 x 4
// 56 / 43, x 2 31 / 43, 200001 x 100 x 4 148 / 134, x 50 x 8 144 / 113, x 24 x 16
// 140 / 125, x 24 x 8 72 / 89.
// Transposed (m columns of A, 256 to a row block): 16384^2 x 16 6984 / 511, x 2
// 885 / 496, 4096^2 x 16 490 / 62, 1024^2 x 8 51 / 26; few columns of many rows
// leave most of a row block empty: 100000 rows x 64 x 8 114 / 152, x 64 x 16
// 220 / 156, x 127 x 8 191 / 156, 10^6 x 16 x 16 886 / 1500.
bool f64tc_pays(char op, bool split, int64_t m, int64_t n, int kc) {
    if (n < 16 || n > (1 << 25)) return false;
    if (op == 't' && n > 8192 && m * kc < 1000) return false;
    if (op == 'l' && n > 64 && !split) return true;
    if ((op == 'l' || split) && n <= 64) return n >= 24 && (kc >= 16 || (kc >= 8 && (n > 48 || m <= 32768)));
    if (kc >= 8) return true;
    return kc == 4 ? m * n >= 1ll << 22 && n > 64 : m * n >= 1ll << 24 && n >= 1024;
}

// Whether an unaligned product goes through the column classes, else through
// the element-wise kernel (a thread per row and one load in flight each, so
// it needs many rows; no inner dimension padded to 16).  Measured on GB300,
// element-wise / column classes in us:
//   binary32  10001 x 4099 x 5 663 / 35, 301 x 301 x 2 33 / 7; tall: 1000001 x
//             24 x 8 35 / 27, 200001 x 32 x 32 33 / 21, but 1000001 x 8 x 8
//             15 / 19, 200001 x 16 x 16 12.5 / 14.6, 200001 x 48 x 16 21 / 23
//             (too few row blocks to hide their ends).
//   binary64  3001 x 200 x 3 37 / 17, 10001 x 501 x 2 51 / 32, 20001 x 200 x 3
//             57 / 58, 200001 x 100 x 2 78 / 94 (bound by the FMA units).
bool shift_pays(int elem, int64_t m, int64_t n, int64_t k) {
    if (elem == 8) return n >= 256 || (n >= 64 && m < 16384);
    return !(n <= 64 && m >= (1 << 16) && k <= 16 && (n <= 8 || m * n < 10000000));
}

// One column chunk of binary64 TSM2R or TSM2L on the tensor cores
// (tsm2_f64tc.cu), or (op 't') of the transposed TSM2R with A read by rows.
// *ran = false: not done (no tensor map describes A, or the workspace cannot
// grow: no memory, or stream capture), the caller takes the FMA kernel.  Larger
// products run in slices: of rows, which keep 4.4 bytes each in the workspace,
// and of the inner dimension, each of whose indices keeps 576 (the sums of
// later slices are added in binary64).
tsm2_status gemm_f64tc(DeviceState *dev, char op, F64TCMode mode, const GemmArgs &g, cudaStream_t stream, bool *ran) {
    *ran = false;
    const int64_t inner = std::min(g.n, kDigitBytes / (int64_t)f64tc_digit_bytes(1 << 10) * (1 << 10));
    const int64_t rows = std::min(g.m, (int64_t)(1 << 14) * f64tc_rows(mode));
    const int64_t num_rb = (rows + f64tc_rows(mode) - 1) / f64tc_rows(mode);
    const int64_t ngroups = num_rb * ((inner + f64tc_step() - 1) / f64tc_step());
    int64_t grid = std::min<int64_t>(dev->sm_count, ngroups / 4);
    if (g_grid_override > 0) grid = std::min<int64_t>(g_grid_override, ngroups);
    if (t_grid_cap > 0 && grid > t_grid_cap) grid = t_grid_cap;
    if (grid < 1) grid = 1;
    auto up = [](size_t x) { return (x + 255) / 256 * 256; };
    const size_t digits = up(f64tc_digit_bytes(inner)), slots = up(f64tc_slot_bytes(grid)), fails = up(f64tc_fail_bytes(rows, mode));
    const size_t later = inner < g.n ? (size_t)rows * g.k * sizeof(double) : 0;
    Scratch scratch;
    tsm2_status st = workspace(stream, 0, digits + slots + fails + later, scratch);
    if (st != TSM2_SUCCESS) {
        (void)cudaGetLastError();  // (of the allocation)
        return TSM2_SUCCESS;
    }
    char *ws = static_cast<char *>(scratch.ws);
    double *sums = reinterpret_cast<double *>(ws + digits + slots + fails);
    t_last_config = mode == F64TCMode::Split ? "simple_f64_tc_kc16" : op == 't' ? "t_f64_tc_kc16" : op == 'r' ? "r_f64_tc_kc16" : g.n > 64 ? "lt_f64_tc_kc16" : "l_f64_tc_kc16";
    for (int64_t i = 0; i < g.m; i += rows)
        for (int64_t j = 0; j < g.n; j += inner) {
            F64TCLaunch L;
            std::memset(&L, 0, sizeof L);
            L.g = g;
            L.g.m = std::min(rows, g.m - i);
            L.g.n = std::min(inner, g.n - j);
            L.g.A = static_cast<const double *>(g.A) + (mode == F64TCMode::Transposed ? i * g.lda + j : i + j * g.lda);
            L.g.B = static_cast<const double *>(g.B) + j;
            double *C = static_cast<double *>(g.C) + i;
            L.g.C = j == 0 ? C : sums;
            L.g.ldc = j == 0 ? g.ldc : L.g.m;
            L.mode = mode;
            st = mode == F64TCMode::Split ? column_classes(&L.a, 8, L.g.A, L.g.m, L.g.n, g.lda)
                 : mode == F64TCMode::Transposed
                     ? encode_2d_ex(&L.a.map[0], CU_TENSOR_MAP_DATA_TYPE_FLOAT64, 8, L.g.A, L.g.n, L.g.m, g.lda,
                                    f64tc_step(), f64tc_rows(mode), CU_TENSOR_MAP_SWIZZLE_128B)
                     : encode_2d(&L.a.map[0], 8, L.g.A, L.g.m, L.g.n, g.lda, f64tc_rows(mode), f64tc_step());
            if (st != TSM2_SUCCESS) return TSM2_SUCCESS;
            L.digits = ws;
            L.slots = ws + digits;
            L.fails = ws + digits + slots;
            L.status = dev->status;
            L.wait_ns = g_wait_ns;
            const int64_t units = (L.g.m + f64tc_rows(mode) - 1) / f64tc_rows(mode) * ((L.g.n + f64tc_step() - 1) / f64tc_step());
            L.grid = (int)std::min(grid, units);
            L.blocks = t_grid_cap > 0 && t_grid_cap < dev->sm_count ? t_grid_cap : dev->sm_count;
            L.trace = (g_trace && g_trace_blocks >= grid) ? g_trace : nullptr;
            cudaError_t e = f64tc_launch(L, stream);
            if (e == cudaSuccess && j > 0) e = f64tc_add(L.g.m, g.k, sums, C, g.ldc, stream);
            if (e != cudaSuccess) return cuda_error(e, "binary64 tensor-core kernel launch");
        }
    *ran = true;
    return TSM2_SUCCESS;
}

tsm2_status gemm(const char *fn, char op, int elem, int64_t m, int64_t n, int64_t k, const void *A, int64_t lda,
                 const void *B, int64_t ldb, void *C, int64_t ldc, void *stream_v) {
    tsm2_status st = check_args(fn, m, n, k, A, lda, B, ldb, C, ldc, elem);
    if (st != TSM2_SUCCESS) return st;
    if (m == 0 || k == 0) {
        t_last_config = "empty";
        return TSM2_SUCCESS;
    }
    cudaStream_t stream = static_cast<cudaStream_t>(stream_v);
    if (n == 0) {
        t_last_config = "zero-fill";
        cudaError_t e = cudaMemset2DAsync(C, (size_t)ldc * elem, 0, (size_t)m * elem, (size_t)k, stream);
        return e == cudaSuccess ? TSM2_SUCCESS : cuda_error(e, "cudaMemset2DAsync");
    }
    DeviceState *dev = nullptr;
    st = device_state(&dev);
    if (st != TSM2_SUCCESS) return st;

    // TSM2L keeps B resident when n <= 64 and stages it with A otherwise
    // (whole row blocks either way).
    const bool staged_l = op == 'l' && n > 64;
    // The bulk-copy path needs 16-byte aligned bases and row strides, and
    // 32-bit tensor coordinates.  Resident B is read with ordinary loads, so
    // only A matters there.
    const bool a_ok = aligned16(A) && ((lda * elem) % 16 == 0) && m < (1ll << 31) - 4096 && n < (1ll << 31);
    const bool b_ok = (op == 'l' && !staged_l) || (aligned16(B) && ((ldb * elem) % 16 == 0));
    const bool use_stream = g_path != 1 && a_ok && b_ok;

    // Operands that one tensor map cannot describe go through column classes
    // (tsm2_shift.cu), unless the element-wise path is forced or the pointers
    // are not even multiples of the element size.
    const bool shift_ok = !use_stream && g_path != 1 &&
                          (((uintptr_t)A | (uintptr_t)B | (uintptr_t)C) & (uintptr_t)(elem - 1)) == 0 &&
                          m < (1ll << 31) - 4096 && n < (1ll << 31) - 64;
    const int kc_max = use_stream ? (op == 'l' ? 32 : 16) : shift_ok && elem == 4 ? 32 : simple_kc_max();
    if (elem == 8 && g_path != 2 && ((g_path != 1 && a_ok) || shift_ok) && f64s_pays(m, n, k, !a_ok)) {
        // (One kernel: the names begin with that of the FMA kernel whose call it is.)
        static const char *const names[2][7] = {
            {"r_f64_kc2_s_f64_tc", "r_f64_kc4_s_f64_tc", "r_f64_kc8_s_f64_tc", "r_f64_kc12_s_f64_tc",
             "r_f64_kc16_s_f64_tc", "r_f64_kc24_s_f64_tc", "r_f64_kc32_s_f64_tc"},
            {"l_f64_kc2_s_f64_tc", "l_f64_kc4_s_f64_tc", "l_f64_kc8_s_f64_tc", "l_f64_kc12_s_f64_tc",
             "l_f64_kc16_s_f64_tc", "l_f64_kc24_s_f64_tc", "l_f64_kc32_s_f64_tc"}};
        const int kc = kc_for((int)std::min<int64_t>(k, 32));
        const int w = kc == 2 ? 0 : kc == 4 ? 1 : kc == 8 ? 2 : kc == 12 ? 3 : kc == 16 ? 4 : kc == 24 ? 5 : 6;
        bool ran = false;
        st = product_f64s(dev, m, k, n, A, lda, B, 1, ldb, C, ldc, false, !a_ok, a_ok ? names[op == 'l'][w] : "simple_f64_s_tc",
                          stream, &ran);
        if (st != TSM2_SUCCESS || ran) return st;
    }
    for (int64_t c0 = 0; c0 < k; c0 += kc_max) {
        GemmArgs g;
        g.m = m;
        g.n = n;
        g.k = (int)((k - c0) < kc_max ? (k - c0) : kc_max);
        g.A = A;
        g.lda = lda;
        g.B = static_cast<const char *>(B) + (size_t)c0 * ldb * elem;
        g.ldb = ldb;
        g.C = static_cast<char *>(C) + (size_t)c0 * ldc * elem;
        g.ldc = ldc;
        cudaError_t e;
        if (elem == 8 && g_path != 2 && (use_stream || shift_ok) && f64tc_pays(op, !use_stream, m, n, kc_for(g.k))) {
            bool ran = true;
            for (int64_t c = 0; c < g.k && ran; c += f64tc_kc()) {
                GemmArgs h = g;
                h.k = (int)std::min<int64_t>(g.k - c, f64tc_kc());
                h.B = static_cast<const char *>(g.B) + (size_t)c * ldb * elem;
                h.C = static_cast<char *>(g.C) + (size_t)c * ldc * elem;
                st = gemm_f64tc(dev, op, use_stream ? F64TCMode::Plain : F64TCMode::Split, h, stream, &ran);
                if (st != TSM2_SUCCESS) return st;
            }
            if (ran) continue;
        }
        if (!use_stream) {
            if (shift_ok && shift_pays(elem, m, n, g.k)) {
                bool ran = false;
                st = gemm_shift(dev, elem, g, stream, &ran);
                if (st != TSM2_SUCCESS) return st;
                if (ran) continue;
            }
            t_last_config = elem == 8 ? "simple_f64" : "simple_f32";
            for (int64_t c = 0; c < g.k; c += simple_kc_max()) {
                GemmArgs h = g;
                h.k = (int)std::min<int64_t>(g.k - c, simple_kc_max());
                h.B = static_cast<const char *>(g.B) + (size_t)c * ldb * elem;
                h.C = static_cast<char *>(g.C) + (size_t)c * ldc * elem;
                e = simple_launch(elem, h, dev->status, stream);
                if (e != cudaSuccess) return cuda_error(e, "simple kernel launch");
            }
            continue;
        }
        int kc = kc_for(g.k);
        if (staged_l && kc < 4) kc = 4;  // staged-B TSM2L: C columns in groups of four
        const StreamShape *shape = stream_shape(elem, staged_l ? 't' : op, kc);
        if (op == 'l' && !staged_l) {
            // Tall A and wide C: the 8-rows-per-lane schedule (KC = 24, 32)
            // once every SM gets enough of its (larger) row blocks.  Measured
            // on GB300: KC = 24 wins from about 1.5 row blocks per SM (5-11%
            // at 2^18 .. 2^20 rows, a tie below), KC = 32 needs about 6.
            const StreamShape *wide = stream_shape(elem, 'w', kc);
            const int64_t min_rb_per_sm = kc == 24 ? 1 : 6;
            if (wide && (m + wide->BM - 1) / wide->BM >= min_rb_per_sm * (int64_t)dev->sm_count) shape = wide;
        }
        if (!shape) return set_error(TSM2_ERR_UNSUPPORTED, "%s: no kernel configuration for k chunk %d", fn, g.k);
        StreamLaunch L;
        std::memset(&L, 0, sizeof L);
        L.g = g;
        st = encode_2d(&L.mapA, elem, A, m, n, lda, shape->BOXM, shape->BNS);
        if (st != TSM2_SUCCESS) return st;
        if (!shape->b_resident) {
            st = encode_2d(&L.mapB, elem, g.B, n, g.k, ldb, shape->BNS, shape->KC);
            if (st != TSM2_SUCCESS) return st;
        }
        const int64_t num_rb = (m + shape->BM - 1) / shape->BM;
        const int64_t upr = (n + shape->BNS - 1) / shape->BNS;
        const bool whole = shape->gran_rows == 0;  // row blocks never split: no partial sums
        const int64_t ngroups = whole ? num_rb : num_rb * upr;
        int64_t grid = dev->sm_count;
        if (!whole) {
            // At least four stages per block so partial sums stay a small
            // fraction of the traffic.
            const int64_t cap = (num_rb * upr) / 4;
            if (cap < grid) grid = cap;
        }
        if (grid > ngroups) grid = ngroups;
        if (g_grid_override > 0) grid = g_grid_override < ngroups ? g_grid_override : ngroups;
        if (t_grid_cap > 0 && grid > t_grid_cap) grid = t_grid_cap;
        if (grid < 1) grid = 1;
        L.grid = (int)grid;
        Scratch scratch;
        if (!shape->b_resident && !whole) {
            const size_t slots = (size_t)(grid + num_rb) * shape->KC * shape->BM * elem;
            st = workspace(stream, (size_t)num_rb * sizeof(int), slots, scratch);
            if (st != TSM2_SUCCESS) return st;
        }
        L.ws = scratch.ws;
        L.counters = scratch.counters;
        if (shape->b_resident) {
            st = claim_counters(stream, &L.claims, scratch);
            if (st != TSM2_SUCCESS) return st;
        }
        L.status = dev->status;
        L.wait_ns = g_wait_ns;
        L.c_vec = aligned16(g.C) && ((ldc * elem) % 16 == 0);
        L.trace = (g_trace && g_trace_blocks >= grid) ? g_trace : nullptr;
        t_last_config = shape->name;
        e = stream_launch(shape, L, stream);
        if (e != cudaSuccess) return cuda_error(e, "stream kernel launch");
    }
    return TSM2_SUCCESS;
}

// ---- backward products ------------------------------------------------------

tsm2_status gemm_t(const char *fn, int elem, int64_t m, int64_t n, int64_t k, const void *A, int64_t lda,
                   const void *dC, int64_t lddc, void *dB, int64_t lddb, void *stream_v) {
    if (m < 0 || n < 0 || k < 0)
        return set_error(TSM2_ERR_INVALID_VALUE, "%s: negative dimension (m=%lld n=%lld k=%lld)", fn, (long long)m,
                         (long long)n, (long long)k);
    if (lda < (m > 1 ? m : 1)) return set_error(TSM2_ERR_INVALID_VALUE, "%s: lda=%lld < max(1,m)", fn, (long long)lda);
    if (lddc < (m > 1 ? m : 1))
        return set_error(TSM2_ERR_INVALID_VALUE, "%s: lddc=%lld < max(1,m)", fn, (long long)lddc);
    if (lddb < (n > 1 ? n : 1))
        return set_error(TSM2_ERR_INVALID_VALUE, "%s: lddb=%lld < max(1,n)", fn, (long long)lddb);
    if (n > 0 && k > 0 && dB == nullptr) return set_error(TSM2_ERR_INVALID_VALUE, "%s: dB is NULL", fn);
    if (m > 0 && n > 0 && k > 0 && (A == nullptr || dC == nullptr))
        return set_error(TSM2_ERR_INVALID_VALUE, "%s: A or dC is NULL", fn);
    if (n > 0 && k > 0 && m > 0) {
        const size_t ob = span_bytes(n, k, lddb, elem);
        if (ranges_overlap(dB, ob, A, span_bytes(m, n, lda, elem)) ||
            ranges_overlap(dB, ob, dC, span_bytes(m, k, lddc, elem)))
            return set_error(TSM2_ERR_INVALID_VALUE, "%s: dB overlaps A or dC", fn);
    }
    if (n == 0 || k == 0) {
        t_last_config = "empty";
        return TSM2_SUCCESS;
    }
    cudaStream_t stream = static_cast<cudaStream_t>(stream_v);
    if (m == 0) {
        t_last_config = "zero-fill";
        cudaError_t e = cudaMemset2DAsync(dB, (size_t)lddb * elem, 0, (size_t)n * elem, (size_t)k, stream);
        return e == cudaSuccess ? TSM2_SUCCESS : cuda_error(e, "cudaMemset2DAsync");
    }
    DeviceState *dev = nullptr;
    tsm2_status st = device_state(&dev);
    if (st != TSM2_SUCCESS) return st;
    const bool ok = g_path != 1 && aligned16(A) && aligned16(dC) && (lda * elem) % 16 == 0 &&
                    (lddc * elem) % 16 == 0 && m < (1ll << 31) - 4096 && n < (1ll << 31);
    for (int64_t c0 = 0; c0 < k; c0 += 16) {
        const int kk = (int)((k - c0) < 16 ? (k - c0) : 16);
        const void *dCc = static_cast<const char *>(dC) + (size_t)c0 * lddc * elem;
        void *dBc = static_cast<char *>(dB) + (size_t)c0 * lddb * elem;
        cudaError_t e;
        if (!ok) {
            t_last_config = elem == 8 ? "simple_t_f64" : "simple_t_f32";
            e = simple_t_launch(elem, m, n, kk, A, lda, dCc, lddc, dBc, lddb, stream);
            if (e != cudaSuccess) return cuda_error(e, "simple_t kernel launch");
            continue;
        }
        int kc = 2;
        while (kc < kk) kc *= 2;
        if (elem == 8 && g_path != 2 && f64tc_pays('t', false, n, m, kc)) {
            GemmArgs g;
            g.m = n;
            g.n = m;
            g.k = kk;
            g.A = A;
            g.lda = lda;
            g.B = dCc;
            g.ldb = lddc;
            g.C = dBc;
            g.ldc = lddb;
            bool ran = false;
            st = gemm_f64tc(dev, 't', F64TCMode::Transposed, g, stream, &ran);
            if (st != TSM2_SUCCESS) return st;
            if (ran) continue;
        }
        const TShape *shape = tsm2t_shape(elem, kc);
        if (!shape) return set_error(TSM2_ERR_UNSUPPORTED, "%s: no configuration for k chunk %d", fn, kk);
        TLaunch L;
        std::memset(&L, 0, sizeof L);
        L.m = m;
        L.n = n;
        L.k = kk;
        st = encode_2d(&L.mapA, elem, A, m, n, lda, shape->BOXM, shape->BNS);
        if (st != TSM2_SUCCESS) return st;
        st = encode_2d(&L.mapD, elem, dCc, m, kk, lddc, shape->BOXM, shape->KC);
        if (st != TSM2_SUCCESS) return st;
        const int64_t nrb = (m + shape->BM - 1) / shape->BM;
        const int64_t nch = (n + shape->BNS - 1) / shape->BNS;
        const int64_t nunits = nrb * nch;
        int64_t grid = dev->sm_count;
        if (nunits / 4 < grid) grid = nunits / 4;
        if (g_grid_override > 0) grid = g_grid_override;
        if (grid > nunits) grid = nunits;
        if (grid < 1) grid = 1;
        Scratch scratch;
        st = workspace(stream, (size_t)nch * sizeof(int), (size_t)(grid + nch) * shape->BNS * shape->KC * elem, scratch);
        if (st != TSM2_SUCCESS) return st;
        L.dB = dBc;
        L.lddb = lddb;
        L.ws = scratch.ws;
        L.counters = scratch.counters;
        L.status = dev->status;
        L.wait_ns = g_wait_ns;
        L.grid = (int)grid;
        t_last_config = shape->name;
        e = tsm2t_launch(shape, L, stream);
        if (e != cudaSuccess) return cuda_error(e, "transposed kernel launch");
    }
    return TSM2_SUCCESS;
}

tsm2_status rankk(const char *fn, int elem, int64_t m, int64_t n, int64_t k, const void *dC, int64_t lddc,
                  const void *B, int64_t ldb, void *dA, int64_t ldda, void *stream_v) {
    if (m < 0 || n < 0 || k < 0)
        return set_error(TSM2_ERR_INVALID_VALUE, "%s: negative dimension (m=%lld n=%lld k=%lld)", fn, (long long)m,
                         (long long)n, (long long)k);
    if (lddc < (m > 1 ? m : 1))
        return set_error(TSM2_ERR_INVALID_VALUE, "%s: lddc=%lld < max(1,m)", fn, (long long)lddc);
    if (ldb < (n > 1 ? n : 1)) return set_error(TSM2_ERR_INVALID_VALUE, "%s: ldb=%lld < max(1,n)", fn, (long long)ldb);
    if (ldda < (m > 1 ? m : 1))
        return set_error(TSM2_ERR_INVALID_VALUE, "%s: ldda=%lld < max(1,m)", fn, (long long)ldda);
    if (m > 0 && n > 0 && dA == nullptr) return set_error(TSM2_ERR_INVALID_VALUE, "%s: dA is NULL", fn);
    if (m > 0 && n > 0 && k > 0 && (dC == nullptr || B == nullptr))
        return set_error(TSM2_ERR_INVALID_VALUE, "%s: dC or B is NULL", fn);
    if (m > 0 && n > 0 && k > 0) {
        const size_t ob = span_bytes(m, n, ldda, elem);
        if (ranges_overlap(dA, ob, dC, span_bytes(m, k, lddc, elem)) ||
            ranges_overlap(dA, ob, B, span_bytes(n, k, ldb, elem)))
            return set_error(TSM2_ERR_INVALID_VALUE, "%s: dA overlaps dC or B", fn);
    }
    if (m == 0 || n == 0) {
        t_last_config = "empty";
        return TSM2_SUCCESS;
    }
    cudaStream_t stream = static_cast<cudaStream_t>(stream_v);
    if (k == 0) {
        t_last_config = "zero-fill";
        cudaError_t e = cudaMemset2DAsync(dA, (size_t)ldda * elem, 0, (size_t)m * elem, (size_t)n, stream);
        return e == cudaSuccess ? TSM2_SUCCESS : cuda_error(e, "cudaMemset2DAsync");
    }
    DeviceState *dev = nullptr;
    tsm2_status st = device_state(&dev);
    if (st != TSM2_SUCCESS) return st;
    if (elem == 8 && g_path != 1 && g_path != 2 && aligned16(dC) && lddc % 2 == 0 && f64s_pays_rankk(m, n, std::min<int64_t>(k, kF64SMaxK))) {
        bool ran = true;
        for (int64_t c0 = 0; c0 < k && ran; c0 += kF64SMaxK) {
            const int64_t kk = std::min<int64_t>(k - c0, kF64SMaxK);
            st = product_f64s(dev, m, n, kk, static_cast<const double *>(dC) + c0 * lddc, lddc,
                              static_cast<const double *>(B) + c0 * ldb, ldb, 1, dA, ldda, c0 > 0, false, "rankk_f64_tc",
                              stream, &ran);
            if (st != TSM2_SUCCESS) return st;
        }
        if (ran) return TSM2_SUCCESS;
    }
    const bool vec_ok = aligned16(dA) && (ldda * elem) % 16 == 0;
    t_last_config = elem == 8 ? "rankk_f64" : "rankk_f32";
    for (int64_t c0 = 0; c0 < k; c0 += 16) {
        const int kk = (int)((k - c0) < 16 ? (k - c0) : 16);
        cudaError_t e = rankk_launch(elem, m, n, kk, static_cast<const char *>(dC) + (size_t)c0 * lddc * elem, lddc,
                                     static_cast<const char *>(B) + (size_t)c0 * ldb * elem, ldb, dA, ldda, vec_ok,
                                     c0 > 0, dev->sm_count, stream);
        if (e != cudaSuccess) return cuda_error(e, "rank-k kernel launch");
    }
    return TSM2_SUCCESS;
}

// ---- bfloat16 A (tensor cores) -------------------------------------------------

tsm2_status gemm_bf16(int64_t m, int64_t n, int64_t k, const void *A_hi, const void *A_lo, int64_t lda,
                      const float *B, int64_t ldb, float *C, int64_t ldc, void *stream_v) {
    const char *fn = "tsm2r_bf16";
    if (m < 0 || n < 0 || k < 0)
        return set_error(TSM2_ERR_INVALID_VALUE, "%s: negative dimension (m=%lld n=%lld k=%lld)", fn, (long long)m,
                         (long long)n, (long long)k);
    if (lda < (m > 1 ? m : 1)) return set_error(TSM2_ERR_INVALID_VALUE, "%s: lda=%lld < max(1,m)", fn, (long long)lda);
    if (ldb < (n > 1 ? n : 1)) return set_error(TSM2_ERR_INVALID_VALUE, "%s: ldb=%lld < max(1,n)", fn, (long long)ldb);
    if (ldc < (m > 1 ? m : 1)) return set_error(TSM2_ERR_INVALID_VALUE, "%s: ldc=%lld < max(1,m)", fn, (long long)ldc);
    if (m > 0 && k > 0 && C == nullptr) return set_error(TSM2_ERR_INVALID_VALUE, "%s: C is NULL", fn);
    if (m > 0 && n > 0 && k > 0 && (A_hi == nullptr || B == nullptr))
        return set_error(TSM2_ERR_INVALID_VALUE, "%s: A_hi or B is NULL", fn);
    if (m > 0 && n > 0 && k > 0) {
        const size_t cb = span_bytes(m, k, ldc, 4);
        const size_t ab = span_bytes(m, n, lda, 2);
        if (ranges_overlap(C, cb, A_hi, ab) || ranges_overlap(C, cb, A_lo, ab) ||
            ranges_overlap(C, cb, B, span_bytes(n, k, ldb, 4)))
            return set_error(TSM2_ERR_INVALID_VALUE, "%s: C overlaps A_hi, A_lo or B", fn);
    }
    if (m == 0 || k == 0) {
        t_last_config = "empty";
        return TSM2_SUCCESS;
    }
    cudaStream_t stream = static_cast<cudaStream_t>(stream_v);
    if (n == 0) {
        t_last_config = "zero-fill";
        cudaError_t e = cudaMemset2DAsync(C, (size_t)ldc * 4, 0, (size_t)m * 4, (size_t)k, stream);
        return e == cudaSuccess ? TSM2_SUCCESS : cuda_error(e, "cudaMemset2DAsync");
    }
    DeviceState *dev = nullptr;
    tsm2_status st = device_state(&dev);
    if (st != TSM2_SUCCESS) return st;
    const bool ok = g_path != 1 && aligned16(A_hi) && (A_lo == nullptr || aligned16(A_lo)) && (lda * 2) % 16 == 0 &&
                    m < (1ll << 31) - 4096 && n < (1ll << 31);
    for (int64_t c0 = 0; c0 < k; c0 += 16) {
        const int kk = (int)((k - c0) < 16 ? (k - c0) : 16);
        const float *Bc = B + c0 * ldb;
        float *Cc = C + c0 * ldc;
        cudaError_t e;
        if (!ok) {
            t_last_config = "simple_bf16";
            e = bf16_simple_launch(m, n, kk, A_hi, A_lo, lda, Bc, ldb, Cc, ldc, stream);
            if (e != cudaSuccess) return cuda_error(e, "bf16 element-wise kernel launch");
            continue;
        }
        BF16Launch L;
        std::memset(&L, 0, sizeof L);
        L.m = m;
        L.n = n;
        L.k = kk;
        L.hilo = A_lo != nullptr;
        st = encode_2d_ex(&L.mapHi, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, A_hi, m, n, lda, 64, bf16_bk(L.hilo),
                          CU_TENSOR_MAP_SWIZZLE_128B);
        if (st != TSM2_SUCCESS) return st;
        if (L.hilo) {
            st = encode_2d_ex(&L.mapLo, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, A_lo, m, n, lda, 64, bf16_bk(L.hilo),
                              CU_TENSOR_MAP_SWIZZLE_128B);
            if (st != TSM2_SUCCESS) return st;
        }
        const int64_t num_rb = (m + bf16_bm() - 1) / bf16_bm();
        const int64_t upr = (n + bf16_bk(L.hilo) - 1) / bf16_bk(L.hilo);
        const int64_t ngroups = num_rb * upr;
        int64_t grid = dev->sm_count;
        if (ngroups / 4 < grid) grid = ngroups / 4;
        if (g_grid_override > 0) grid = g_grid_override;
        if (grid > ngroups) grid = ngroups;
        if (grid < 1) grid = 1;
        const size_t pieces = (bf16_bpieces_bytes(n, L.hilo) + 255) / 256 * 256;
        const size_t slots = (size_t)(grid + num_rb) * 16 * bf16_bm() * 4;
        Scratch scratch;
        st = workspace(stream, (size_t)num_rb * sizeof(int), pieces + slots, scratch);
        if (st != TSM2_SUCCESS) return st;
        e = bf16_prep_b(n, kk, Bc, ldb, scratch.ws, L.hilo, stream);
        if (e != cudaSuccess) return cuda_error(e, "bf16 B split kernel launch");
        L.bpieces = scratch.ws;
        L.ws = static_cast<char *>(scratch.ws) + pieces;
        L.counters = scratch.counters;
        L.C = Cc;
        L.ldc = ldc;
        L.status = dev->status;
        L.wait_ns = g_wait_ns;
        L.grid = (int)grid;
        t_last_config = L.hilo ? "tc_bf16_hilo" : "tc_bf16";
        e = bf16_launch(L, stream);
        if (e != cudaSuccess) return cuda_error(e, "bf16 tensor-core kernel launch");
    }
    return TSM2_SUCCESS;
}

// ---- batched problems ----------------------------------------------------------

}  // namespace
}  // namespace tsm2

struct tsm2_batch_plan_s {
    struct Cls {
        const tsm2::BatchClass *cls = nullptr;
        int slot = 0;             // slot of the class in the menu's kernel
        std::vector<tsm2::ProbDesc> host;
        int64_t ngroups = 0, nrb = 0;
        double bytes = 0;
        tsm2::ProbDesc *d_probs = nullptr;
        void *d_ws = nullptr;     // counters, then partial-sum slots
        size_t counter_bytes = 0;
        int grid = 1;             // blocks of the class in the concurrent mode
        cudaStream_t aux = nullptr;
        cudaEvent_t done = nullptr;
    };
    struct Zero {
        void *C;
        int64_t ldc, m, k;
    };
    int dev = 0;
    int sm_count = 0;
    int variant = 0;
    const tsm2::BatchMenu *menu = nullptr;
    int mode = TSM2_BATCH_SINGLE_LAUNCH;
    int single_grid = 0;             // blocks of the single launch
    std::vector<Cls> classes;
    std::vector<Zero> zeros;
    cudaEvent_t fork = nullptr;
    cudaGraphExec_t graph = nullptr;
    cudaStream_t capture = nullptr;  // private stream the graph is captured on
    double total_bytes = 0;
    tsm2::BatchBalance *d_bal = nullptr;  // adaptive TSM2L shares of the single launch
};

namespace tsm2 {
namespace {

// Live plans, so that a timeout can reset their arrival counters.
std::mutex g_plans_mu;
std::vector<tsm2_batch_plan_s *> g_plans;

void destroy_plan(tsm2_batch_plan_s *P) {
    if (!P) return;
    {
        std::lock_guard<std::mutex> lk(g_plans_mu);
        g_plans.erase(std::remove(g_plans.begin(), g_plans.end(), P), g_plans.end());
    }
    int cur = 0;
    cudaGetDevice(&cur);
    cudaSetDevice(P->dev);
    if (P->graph) cudaGraphExecDestroy(P->graph);
    for (auto &c : P->classes) {
        if (c.d_probs) cudaFree(c.d_probs);
        if (c.d_ws) cudaFree(c.d_ws);
        if (c.aux) cudaStreamDestroy(c.aux);
        if (c.done) cudaEventDestroy(c.done);
    }
    if (P->fork) cudaEventDestroy(P->fork);
    if (P->capture) cudaStreamDestroy(P->capture);
    if (P->d_bal) cudaFree(P->d_bal);
    cudaSetDevice(cur);
    delete P;
}

// Arrival counters of every live plan on device `dev` back to zero (after a
// launch that gave up, they may be left non-zero).
void reset_plan_counters(int dev) {
    std::lock_guard<std::mutex> lk(g_plans_mu);
    for (tsm2_batch_plan_s *P : g_plans)
        if (P->dev == dev) {
            for (auto &c : P->classes)
                if (c.d_ws) cudaMemset(c.d_ws, 0, c.counter_bytes);
            if (P->d_bal) cudaMemset(P->d_bal, 0, 4 * sizeof(int));  // epoch, done, bad
        }
}

void class_params(const tsm2_batch_plan_s::Cls &c, ClassParams &cp) {
    cp.probs = c.d_probs;
    cp.nprob = (int)c.host.size();
    cp.whole = c.cls->op == 'w' ? 1 : 0;
    cp.ngroups = c.ngroups;
    cp.counters = static_cast<int *>(c.d_ws);
    cp.ws = reinterpret_cast<float *>(static_cast<char *>(c.d_ws) + c.counter_bytes);
    cp.nrb = c.nrb;
}

// Adaptive TSM2L shares pay off when the TSM2L phase is long against the
// launch-to-launch noise of when blocks reach it.  Measured on GB300 (one
// launch, median of 15): the 512-problem batch (42.8 GB) 1.4-2.2% faster,
// its first 120 problems (9.3 GB) 0.4-1% slower, its first 40 (3.4 GB) 5%
// slower.  Plans below this size keep equal shares.
constexpr double kAdaptMinBytes = 16e9;

// One launch of the plan's batch kernel over the classes [lo, hi) (all
// other slots empty) on `grid` blocks; `adapt`: TSM2L shares from the plan's
// adaptive weights.
tsm2_status launch_classes(tsm2_batch_plan_s *P, int lo, int hi, int grid, cudaStream_t stream, bool adapt = false) {
    DeviceState *dev = nullptr;
    tsm2_status st = device_state(&dev);
    if (st != TSM2_SUCCESS) return st;
    BatchKParams kp;
    std::memset(&kp, 0, sizeof kp);
    for (int i = lo; i < hi; ++i) class_params(P->classes[i], kp.cls[P->classes[i].slot]);
    kp.status = dev->status;
    kp.wait_ns = g_wait_ns;
    kp.trace = (g_trace && g_trace_blocks >= grid) ? g_trace : nullptr;
    kp.bal = (adapt && g_balance != 1 && grid <= kBalanceMaxBlocks) ? P->d_bal : nullptr;
    const cudaError_t e = P->menu->launch(kp, grid < 1 ? 1 : grid, stream);
    return e == cudaSuccess ? TSM2_SUCCESS : cuda_error(e, "batch kernel launch");
}

int class_grid_alone(const tsm2_batch_plan_s *P, int i) {
    return (int)std::min<int64_t>(P->sm_count, P->classes[i].ngroups);
}

tsm2_status plan_execute(tsm2_batch_plan_s *P, cudaStream_t stream, int only) {
    cudaError_t e;
    const int nc = (int)P->classes.size();
    if (only >= 0) return launch_classes(P, only, only + 1, class_grid_alone(P, only), stream);
    for (const auto &z : P->zeros) {
        e = cudaMemset2DAsync(z.C, (size_t)z.ldc * 4, 0, (size_t)z.m * 4, (size_t)z.k, stream);
        if (e != cudaSuccess) return cuda_error(e, "cudaMemset2DAsync");
    }
    if (nc == 0) return TSM2_SUCCESS;
    if (P->mode == TSM2_BATCH_SINGLE_LAUNCH)
        return launch_classes(P, 0, nc, P->single_grid, stream, g_balance == 2 || P->total_bytes >= kAdaptMinBytes);
    if (P->mode == TSM2_BATCH_SERIAL) {
        for (int i = 0; i < nc; ++i) {
            tsm2_status s = launch_classes(P, i, i + 1, class_grid_alone(P, i), stream);
            if (s != TSM2_SUCCESS) return s;
        }
        return TSM2_SUCCESS;
    }
    // Concurrent: every class on its own SM share, forked onto the plan's
    // streams and joined back.
    if (nc > 1) {
        e = cudaEventRecord(P->fork, stream);
        if (e != cudaSuccess) return cuda_error(e, "cudaEventRecord");
    }
    for (int i = 0; i < nc; ++i) {
        auto &c = P->classes[i];
        cudaStream_t s = i == 0 ? stream : c.aux;
        if (i > 0) {
            e = cudaStreamWaitEvent(s, P->fork, 0);
            if (e != cudaSuccess) return cuda_error(e, "cudaStreamWaitEvent");
        }
        tsm2_status st = launch_classes(P, i, i + 1, c.grid, s);
        if (st != TSM2_SUCCESS) return st;
        if (i > 0) {
            e = cudaEventRecord(c.done, s);
            if (e != cudaSuccess) return cuda_error(e, "cudaEventRecord");
            e = cudaStreamWaitEvent(stream, c.done, 0);
            if (e != cudaSuccess) return cuda_error(e, "cudaStreamWaitEvent");
        }
    }
    return TSM2_SUCCESS;
}

// ---- allocation-free variant of the binary32 TSM2R bulk-copy path -----------
//
// Some callers cannot call cudaMalloc at all: a process whose device memory is
// entirely owned by another allocator (for example a framework's caching pool
// that has already reserved the free memory), or a latency-bound loop that
// must not pay cudaMalloc's cost and implicit synchronisation.  For them,
// tsm2r_s_noalloc keeps the partial sums of split row blocks and their
// arrival counters in this fixed, file-scope device array instead of the
// lazily allocated workspace.  Every GPU that loads the library holds these
// bytes until the process exits.

constexpr size_t kNoAllocScratchBytes = 16u << 20;     // 16 MiB
constexpr size_t kNoAllocCounterBytes = 64u << 10;     // first 64 KiB: arrival counters
static __device__ __align__(256) unsigned char g_noalloc_scratch[kNoAllocScratchBytes];

std::mutex g_noalloc_mu;
void *g_noalloc_ptr[64];  // device address of g_noalloc_scratch, per device

// Host code may not pass g_noalloc_scratch itself to a kernel: on the host
// that name is only a stand-in for the device array.  Its device address is
// looked up once per device, with that device current.
tsm2_status noalloc_scratch(void **out) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return cuda_error(e, "cudaGetDevice");
    if (dev < 0 || dev >= 64) return set_error(TSM2_ERR_UNSUPPORTED, "device ordinal %d out of range", dev);
    std::lock_guard<std::mutex> lk(g_noalloc_mu);
    if (!g_noalloc_ptr[dev]) {
        void *p = nullptr;
        e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
        if (e != cudaSuccess) return cuda_error(e, "cudaGetSymbolAddress(no-alloc scratch)");
        g_noalloc_ptr[dev] = p;
    }
    *out = g_noalloc_ptr[dev];
    return TSM2_SUCCESS;
}

tsm2_status gemm_r32_noalloc(int64_t m, int64_t n, int64_t k, const float *A, int64_t lda, const float *B,
                             int64_t ldb, float *C, int64_t ldc, void *stream_v) {
    const char *fn = "tsm2r_s_noalloc";
    const int elem = 4;
    tsm2_status st = check_args(fn, m, n, k, A, lda, B, ldb, C, ldc, elem);
    if (st != TSM2_SUCCESS) return st;
    if (m == 0 || k == 0) {
        t_last_config = "empty";
        return TSM2_SUCCESS;
    }
    cudaStream_t stream = static_cast<cudaStream_t>(stream_v);
    if (n == 0) {
        t_last_config = "zero-fill";
        cudaError_t e = cudaMemset2DAsync(C, (size_t)ldc * elem, 0, (size_t)m * elem, (size_t)k, stream);
        return e == cudaSuccess ? TSM2_SUCCESS : cuda_error(e, "cudaMemset2DAsync");
    }
    DeviceState *dev = nullptr;
    st = device_state(&dev);
    if (st != TSM2_SUCCESS) return st;
    const bool a_ok = aligned16(A) && ((lda * elem) % 16 == 0) && m < (1ll << 31) - 4096 && n < (1ll << 31);
    const bool b_ok = aligned16(B) && ((ldb * elem) % 16 == 0);
    const bool use_stream = g_path != 1 && a_ok && b_ok;
    void *scratch = nullptr;
    if (use_stream) {
        st = noalloc_scratch(&scratch);
        if (st != TSM2_SUCCESS) return st;
    }
    const int kc_max = use_stream ? 16 : simple_kc_max();
    for (int64_t c0 = 0; c0 < k; c0 += kc_max) {
        GemmArgs g;
        g.m = m;
        g.n = n;
        g.k = (int)((k - c0) < kc_max ? (k - c0) : kc_max);
        g.A = A;
        g.lda = lda;
        g.B = reinterpret_cast<const char *>(B) + (size_t)c0 * ldb * elem;
        g.ldb = ldb;
        g.C = reinterpret_cast<char *>(C) + (size_t)c0 * ldc * elem;
        g.ldc = ldc;
        cudaError_t e;
        if (!use_stream) {  // element-wise path: needs no scratch at all
            t_last_config = "simple_f32";
            e = simple_launch(elem, g, dev->status, stream);
            if (e != cudaSuccess) return cuda_error(e, "simple kernel launch");
            continue;
        }
        const int kc = kc_for(g.k);
        const StreamShape *shape = stream_shape(elem, 'r', kc);
        if (!shape) return set_error(TSM2_ERR_UNSUPPORTED, "%s: no kernel configuration for k chunk %d", fn, g.k);
        const int64_t num_rb = (m + shape->BM - 1) / shape->BM;
        const int64_t upr = (n + shape->BNS - 1) / shape->BNS;
        const int64_t ngroups = num_rb * upr;
        int64_t grid = dev->sm_count;
        const int64_t cap = ngroups / 4;
        if (cap < grid) grid = cap;
        if (g_grid_override > 0) grid = g_grid_override < ngroups ? g_grid_override : ngroups;
        if (grid > ngroups) grid = ngroups;
        if (grid < 1) grid = 1;
        const size_t counter_bytes = (size_t)num_rb * sizeof(int);
        // Partial-sum slots of split row blocks.
        const size_t slot_bytes = (size_t)(grid + num_rb) * shape->KC * shape->BM * elem;
        const size_t data_cap = kNoAllocScratchBytes - kNoAllocCounterBytes;
        if (counter_bytes > kNoAllocCounterBytes || slot_bytes > data_cap)
            return set_error(TSM2_ERR_UNSUPPORTED,
                             "%s: m=%lld n=%lld needs %zu bytes of counters and %zu bytes of partial sums; "
                             "the static scratch holds %zu and %zu; use tsm2r_s instead",
                             fn, (long long)m, (long long)n, counter_bytes, slot_bytes, kNoAllocCounterBytes,
                             data_cap);
        StreamLaunch L;
        std::memset(&L, 0, sizeof L);
        L.g = g;
        st = encode_2d(&L.mapA, elem, A, m, n, lda, shape->BOXM, shape->BNS);
        if (st != TSM2_SUCCESS) return st;
        st = encode_2d(&L.mapB, elem, g.B, n, g.k, ldb, shape->BNS, shape->KC);
        if (st != TSM2_SUCCESS) return st;
        // The array keeps whatever the previous call left; the arrival
        // counters must start at zero.
        e = cudaMemsetAsync(scratch, 0, counter_bytes, stream);
        if (e != cudaSuccess) return cuda_error(e, "cudaMemsetAsync(no-alloc counters)");
        L.grid = (int)grid;
        L.counters = static_cast<int *>(scratch);
        L.ws = static_cast<char *>(scratch) + kNoAllocCounterBytes;
        L.status = dev->status;
        L.wait_ns = g_wait_ns;
        L.c_vec = aligned16(g.C) && ((ldc * elem) % 16 == 0);
        t_last_config = shape->name;
        e = stream_launch(shape, L, stream);
        if (e != cudaSuccess) return cuda_error(e, "stream kernel launch");
    }
    return TSM2_SUCCESS;
}

// ---- TSM2X: choice between the TSM2R and TSM2L schedules --------------------
//
// TSM2R streams A in stages of 32 inner columns per row block of 256 (128)
// rows and splits the inner dimension between blocks; with few inner columns
// a row block is one or two stages long and the kernel is bound by latency
// and per-row-block overheads (the paper's observation for small inner
// dimensions, Sec. 3.2.1).  TSM2L owns whole, taller row blocks and keeps B
// on chip (or stages it, n > 64); it needs enough row blocks to occupy the
// GPU.  Largest n for which TSM2L was faster in a GB300 sweep over m in
// {15360, 2^18, 2^20, 2^22, 2^23}, n in {2, 4, ..., 1024}, k in {16, 32}:
//   binary32: m >= 2^17: n <= 256; shorter: n <= 64 (k <= 16), 128 (k > 16)
//   binary64: m >= 2^17: n <= 64 (k <= 16), 256 (k > 16); shorter: 32, 64.
int64_t tsm2x_l_max_n(int elem, int64_t m, int64_t k) {
    const bool tall = m >= (int64_t(1) << 17);
    const bool wide_c = k > 16;
    if (elem == 4) return tall ? 256 : (wide_c ? 128 : 64);
    return tall ? (wide_c ? 256 : 64) : (wide_c ? 64 : 32);
}

char tsm2x_schedule(int elem, int64_t m, int64_t n, int64_t k) {
    return n <= tsm2x_l_max_n(elem, m, k) ? 'l' : 'r';
}

// ---- host-resident operands: row-chunk pipeline ---------------------------
//
// A is streamed to the device in chunks of whole rows (a 2-D copy: mc rows of
// each of the n columns) into one of two staging slots.  Three streams run
// the stages: the copy-in stream fills slot (c & 1) with chunk c, the compute
// stream runs the device product on it, the copy-out stream returns its C
// rows.  Copy-in of chunk c+1 overlaps the product and copy-out of chunk c,
// and copy-in of chunk c+2 waits only for copy-out of chunk c (which itself
// followed the product), so the link stays busy in both directions.
//
// Page-locked buffers that the device can address are copied by SM kernels
// (tsm2_hostcopy.cu) on kCopyInSMs + up to kCopyOutSMs whole SMs, and the
// product kernels' grid is capped to the remaining SMs, so all three stages
// still run at once; other host memory goes through the copy engines.

constexpr int kCopyInSMs = 24;   // ~64 KB of loads in flight per SM covers the host link's latency
constexpr int kCopyOutSMs = 16;

// Device address of host memory at `p` when the current device can load and
// store it directly (page-locked and mapped), else nullptr.
void *device_view(const void *p) {
    if (g_host_copy != 0 || (reinterpret_cast<uintptr_t>(p) & 3)) return nullptr;  // copy kernels move 4-byte words
    cudaPointerAttributes a;
    if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
        cudaGetLastError();  // clear the error state the failed query left
        return nullptr;
    }
    if (a.type != cudaMemoryTypeHost || !a.devicePointer || !a.hostPointer) return nullptr;
    return static_cast<char *>(a.devicePointer) + (static_cast<const char *>(p) - static_cast<const char *>(a.hostPointer));
}

// Resets the calling thread's grid cap on scope exit.
struct GridCap {
    explicit GridCap(int cap) { t_grid_cap = cap; }
    ~GridCap() { t_grid_cap = 0; }
};

struct HostPipe {
    cudaStream_t in = nullptr, comp = nullptr, out = nullptr;
    cudaEvent_t entry = nullptr, b_ready = nullptr, done = nullptr;
    cudaEvent_t a_ready[2] = {}, c_ready[2] = {}, slot_free[2] = {};
    void *dA[2] = {}, *dC[2] = {}, *dB = nullptr;
    size_t a_bytes = 0, c_bytes = 0, b_bytes = 0;
    std::mutex mu;
};
std::mutex g_pipe_mu;
std::map<int, HostPipe *> g_pipes;

#ifndef TSM2_HOST_CHUNK_MB
#define TSM2_HOST_CHUNK_MB 256
#endif
#ifndef TSM2_HOST_MIN_SEGMENT_KB
#define TSM2_HOST_MIN_SEGMENT_KB 64
#endif
constexpr size_t kHostChunkBytes = (size_t)TSM2_HOST_CHUNK_MB << 20;        // target bytes of A per chunk
constexpr size_t kHostMinSegment = (size_t)TSM2_HOST_MIN_SEGMENT_KB << 10;  // least bytes per column piece

void pipe_free_buffers(HostPipe *P) {
    for (int i = 0; i < 2; ++i) {
        if (P->dA[i]) cudaFree(P->dA[i]);
        if (P->dC[i]) cudaFree(P->dC[i]);
        P->dA[i] = P->dC[i] = nullptr;
    }
    if (P->dB) cudaFree(P->dB);
    P->dB = nullptr;
    P->a_bytes = P->c_bytes = P->b_bytes = 0;
}

void pipe_destroy(HostPipe *P) {
    pipe_free_buffers(P);
    for (cudaStream_t s : {P->in, P->comp, P->out})
        if (s) cudaStreamDestroy(s);
    for (cudaEvent_t e : {P->entry, P->b_ready, P->done, P->a_ready[0], P->a_ready[1], P->c_ready[0], P->c_ready[1],
                          P->slot_free[0], P->slot_free[1]})
        if (e) cudaEventDestroy(e);
    delete P;
}

tsm2_status pipe_for_device(HostPipe **out) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return cuda_error(e, "cudaGetDevice");
    std::lock_guard<std::mutex> lk(g_pipe_mu);
    auto it = g_pipes.find(dev);
    if (it != g_pipes.end()) {
        *out = it->second;
        return TSM2_SUCCESS;
    }
    HostPipe *P = new HostPipe();
    for (cudaStream_t *s : {&P->in, &P->comp, &P->out})
        if (e == cudaSuccess) e = cudaStreamCreateWithFlags(s, cudaStreamNonBlocking);
    for (cudaEvent_t *ev : {&P->entry, &P->b_ready, &P->done, &P->a_ready[0], &P->a_ready[1], &P->c_ready[0],
                            &P->c_ready[1], &P->slot_free[0], &P->slot_free[1]})
        if (e == cudaSuccess) e = cudaEventCreateWithFlags(ev, cudaEventDisableTiming);
    if (e != cudaSuccess) {
        pipe_destroy(P);
        return cuda_error(e, "host pipeline set-up");
    }
    g_pipes[dev] = P;
    *out = P;
    return TSM2_SUCCESS;
}

// Grows a device buffer; the pipeline's streams are idle when this runs (the
// caller synchronises them first).
tsm2_status grow(void **p, size_t *have, size_t want) {
    if (*have >= want && *p) return TSM2_SUCCESS;
    if (*p) cudaFree(*p);
    *p = nullptr;
    *have = 0;
    cudaError_t e = cudaMalloc(p, want);
    if (e != cudaSuccess) {
        *p = nullptr;
        return cuda_error(e, "cudaMalloc(host pipeline staging)");
    }
    *have = want;
    return TSM2_SUCCESS;
}

tsm2_status gemm_host(const char *fn, char op, int elem, int64_t m, int64_t n, int64_t k, const void *hA, int64_t lda,
                      const void *hB, int64_t ldb, void *hC, int64_t ldc, void *stream_v) {
    tsm2_status st = check_args(fn, m, n, k, hA, lda, hB, ldb, hC, ldc, elem);
    if (st != TSM2_SUCCESS) return st;
    cudaStream_t stream = static_cast<cudaStream_t>(stream_v);
    cudaError_t e;
    if (m == 0 || k == 0) {
        t_last_config = "empty";
        return TSM2_SUCCESS;
    }
    if (n == 0) {  // C = 0 on the host, after the caller's pending work
        e = cudaStreamSynchronize(stream);
        if (e != cudaSuccess) return cuda_error(e, "cudaStreamSynchronize");
        for (int64_t c = 0; c < k; ++c) std::memset(static_cast<char *>(hC) + (size_t)(c * ldc) * elem, 0, (size_t)m * elem);
        t_last_config = "zero-fill";
        return TSM2_SUCCESS;
    }
    HostPipe *P = nullptr;
    st = pipe_for_device(&P);
    if (st != TSM2_SUCCESS) return st;
    std::lock_guard<std::mutex> lk(P->mu);

    // Rows per chunk: about kHostChunkBytes of A but column pieces of at
    // least kHostMinSegment bytes (a 2-D copy moves one piece per column),
    // a multiple of 256 rows (whole row blocks of every schedule); the
    // staging leading dimension is the chunk height rounded to 16 bytes.
    const int64_t vec = 16 / elem;
    int64_t mc = (int64_t)(kHostChunkBytes / ((size_t)n * elem));
    if (mc < (int64_t)(kHostMinSegment / elem)) mc = (int64_t)(kHostMinSegment / elem);
    mc = mc / 256 * 256;
    if (mc < 256) mc = 256;
    if (mc > m) mc = m;
    const int64_t ldd = (mc + vec - 1) / vec * vec;
    const int64_t ldbd = (n + vec - 1) / vec * vec;
    const size_t a_need = (size_t)ldd * n * elem, c_need = (size_t)ldd * k * elem, b_need = (size_t)ldbd * k * elem;
    if (P->a_bytes < a_need || P->c_bytes < c_need || P->b_bytes < b_need) {
        for (cudaStream_t s : {P->in, P->comp, P->out}) {
            e = cudaStreamSynchronize(s);
            if (e != cudaSuccess) return cuda_error(e, "cudaStreamSynchronize(host pipeline)");
        }
        size_t ah = P->a_bytes, ch = P->c_bytes;
        for (int i = 0; i < 2; ++i) {
            size_t a_have = ah, c_have = ch;
            if ((st = grow(&P->dA[i], &a_have, a_need)) != TSM2_SUCCESS) return st;
            if ((st = grow(&P->dC[i], &c_have, c_need)) != TSM2_SUCCESS) return st;
            if (i == 1) {
                P->a_bytes = a_have;
                P->c_bytes = c_have;
            }
        }
        if ((st = grow(&P->dB, &P->b_bytes, b_need)) != TSM2_SUCCESS) return st;
    }

    // SM copies where the device can address the host buffers (section
    // comment above); the product kernels get the SMs the copies leave.
    DeviceState *dev = nullptr;
    if ((st = device_state(&dev)) != TSM2_SUCCESS) return st;
    const void *vA = device_view(hA), *vB = device_view(hB);
    void *vC = device_view(hC);
    const int in_sms = vA ? kCopyInSMs : 0;
    int out_sms = 0;
    if (vC) {  // scaled to the bytes of C per byte of A, at least 2
        out_sms = (int)std::min<int64_t>(kCopyOutSMs, std::max<int64_t>(2, (kCopyOutSMs * k + n - 1) / n));
    }
    GridCap cap(in_sms + out_sms > 0 ? std::max(dev->sm_count - in_sms - out_sms, 1) : 0);
    static const char *const kCopyNames[8] = {"A:engine B:engine C:engine", "A:sm B:engine C:engine",
                                              "A:engine B:sm C:engine",     "A:sm B:sm C:engine",
                                              "A:engine B:engine C:sm",     "A:sm B:engine C:sm",
                                              "A:engine B:sm C:sm",         "A:sm B:sm C:sm"};
    t_last_host_copy = kCopyNames[(vA ? 1 : 0) | (vB ? 2 : 0) | (vC ? 4 : 0)];

    // Everything starts after the caller's pending work on `stream`.
    if ((e = cudaEventRecord(P->entry, stream)) != cudaSuccess) return cuda_error(e, "cudaEventRecord");
    for (cudaStream_t s : {P->in, P->comp, P->out})
        if ((e = cudaStreamWaitEvent(s, P->entry, 0)) != cudaSuccess) return cuda_error(e, "cudaStreamWaitEvent");
    if (vB) {
        e = sm_copy2d_launch(vB, ldb * elem, P->dB, ldbd * elem, n * elem, k, kCopyInSMs, P->in);
        if (e != cudaSuccess) return cuda_error(e, "host copy kernel (B)");
    } else {
        e = cudaMemcpy2DAsync(P->dB, (size_t)ldbd * elem, hB, (size_t)ldb * elem, (size_t)n * elem, (size_t)k,
                              cudaMemcpyHostToDevice, P->in);
        if (e != cudaSuccess) return cuda_error(e, "cudaMemcpy2DAsync(B)");
    }
    if ((e = cudaEventRecord(P->b_ready, P->in)) != cudaSuccess) return cuda_error(e, "cudaEventRecord");
    if ((e = cudaStreamWaitEvent(P->comp, P->b_ready, 0)) != cudaSuccess) return cuda_error(e, "cudaStreamWaitEvent");

    const char *config = "";
    int64_t chunk = 0;
    for (int64_t i0 = 0; i0 < m; i0 += mc, ++chunk) {
        const int slot = (int)(chunk & 1);
        const int64_t rows = (m - i0) < mc ? (m - i0) : mc;
        if (chunk >= 2 && (e = cudaStreamWaitEvent(P->in, P->slot_free[slot], 0)) != cudaSuccess)
            return cuda_error(e, "cudaStreamWaitEvent");
        if (vA) {
            e = sm_copy2d_launch(static_cast<const char *>(vA) + (size_t)i0 * elem, lda * elem, P->dA[slot],
                                 ldd * elem, rows * elem, n, in_sms, P->in);
            if (e != cudaSuccess) return cuda_error(e, "host copy kernel (A chunk)");
        } else {
            e = cudaMemcpy2DAsync(P->dA[slot], (size_t)ldd * elem, static_cast<const char *>(hA) + (size_t)i0 * elem,
                                  (size_t)lda * elem, (size_t)rows * elem, (size_t)n, cudaMemcpyHostToDevice, P->in);
            if (e != cudaSuccess) return cuda_error(e, "cudaMemcpy2DAsync(A chunk)");
        }
        if ((e = cudaEventRecord(P->a_ready[slot], P->in)) != cudaSuccess) return cuda_error(e, "cudaEventRecord");
        if ((e = cudaStreamWaitEvent(P->comp, P->a_ready[slot], 0)) != cudaSuccess)
            return cuda_error(e, "cudaStreamWaitEvent");
        st = gemm(fn, op, elem, rows, n, k, P->dA[slot], ldd, P->dB, ldbd, P->dC[slot], ldd, P->comp);
        if (st != TSM2_SUCCESS) return st;
        config = t_last_config;
        if ((e = cudaEventRecord(P->c_ready[slot], P->comp)) != cudaSuccess) return cuda_error(e, "cudaEventRecord");
        if ((e = cudaStreamWaitEvent(P->out, P->c_ready[slot], 0)) != cudaSuccess)
            return cuda_error(e, "cudaStreamWaitEvent");
        if (vC) {
            e = sm_copy2d_launch(P->dC[slot], ldd * elem, static_cast<char *>(vC) + (size_t)i0 * elem, ldc * elem,
                                 rows * elem, k, out_sms, P->out);
            if (e != cudaSuccess) return cuda_error(e, "host copy kernel (C chunk)");
        } else {
            e = cudaMemcpy2DAsync(static_cast<char *>(hC) + (size_t)i0 * elem, (size_t)ldc * elem, P->dC[slot],
                                  (size_t)ldd * elem, (size_t)rows * elem, (size_t)k, cudaMemcpyDeviceToHost, P->out);
            if (e != cudaSuccess) return cuda_error(e, "cudaMemcpy2DAsync(C chunk)");
        }
        if ((e = cudaEventRecord(P->slot_free[slot], P->out)) != cudaSuccess) return cuda_error(e, "cudaEventRecord");
    }
    // The caller's stream resumes once the last C rows are on the host.
    if ((e = cudaEventRecord(P->done, P->out)) != cudaSuccess) return cuda_error(e, "cudaEventRecord");
    if ((e = cudaStreamWaitEvent(stream, P->done, 0)) != cudaSuccess) return cuda_error(e, "cudaStreamWaitEvent");
    t_last_config = config;
    return TSM2_SUCCESS;
}

}  // namespace
}  // namespace tsm2

using namespace tsm2;

extern "C" {

tsm2_status tsm2r_d(int64_t m, int64_t n, int64_t k, const double *A, int64_t lda, const double *B, int64_t ldb,
                    double *C, int64_t ldc, void *stream) {
    return gemm("tsm2r_d", 'r', 8, m, n, k, A, lda, B, ldb, C, ldc, stream);
}

tsm2_status tsm2r_s(int64_t m, int64_t n, int64_t k, const float *A, int64_t lda, const float *B, int64_t ldb,
                    float *C, int64_t ldc, void *stream) {
    return gemm("tsm2r_s", 'r', 4, m, n, k, A, lda, B, ldb, C, ldc, stream);
}

tsm2_status tsm2l_d(int64_t m, int64_t n, int64_t k, const double *A, int64_t lda, const double *B, int64_t ldb,
                    double *C, int64_t ldc, void *stream) {
    return gemm("tsm2l_d", 'l', 8, m, n, k, A, lda, B, ldb, C, ldc, stream);
}

tsm2_status tsm2l_s(int64_t m, int64_t n, int64_t k, const float *A, int64_t lda, const float *B, int64_t ldb,
                    float *C, int64_t ldc, void *stream) {
    return gemm("tsm2l_s", 'l', 4, m, n, k, A, lda, B, ldb, C, ldc, stream);
}

const char *tsm2_get_last_error_string(void) { return t_last_error.c_str(); }

const char *tsm2_last_config(void) { return t_last_config; }

const char *tsm2_last_host_copy(void) { return t_last_host_copy; }

tsm2_status tsm2_get_device_status(void *stream) {
    cudaError_t e = cudaStreamSynchronize(static_cast<cudaStream_t>(stream));
    if (e != cudaSuccess) return cuda_error(e, "cudaStreamSynchronize");
    unsigned w = 0;
    e = cudaMemcpyFromSymbol(&w, g_status_word, sizeof w);
    if (e != cudaSuccess) return cuda_error(e, "cudaMemcpyFromSymbol(status)");
    if (w == 0) return TSM2_SUCCESS;
    const unsigned zero = 0;
    e = cudaMemcpyToSymbol(g_status_word, &zero, sizeof zero);
    if (e != cudaSuccess) return cuda_error(e, "cudaMemcpyToSymbol(status)");
    // An abandoned launch may leave arrival counters non-zero: clear them all
    // on this device (stream workspaces, graphs and batch plans).
    int dev = 0;
    cudaGetDevice(&dev);
    {
        std::lock_guard<std::mutex> lk(g_mu);
        for (auto &kv : g_ws) {
            if (kv.first.first != dev) continue;
            std::lock_guard<std::mutex> ws(kv.second.mu);
            if (kv.second.ptr) cudaMemset(kv.second.ptr, 0, kv.second.counter_bytes);
        }
    }
    {
        std::lock_guard<std::mutex> lk(g_graph_mu);
        for (auto &s : g_graph_scratch)
            if (s->dev == dev) cudaMemset(s->ptr, 0, s->counter_bytes);
    }
    reset_plan_counters(dev);
    cudaDeviceSynchronize();
    if (w & kStatusBounds)
        return set_error(TSM2_ERR_BOUNDS,
                         "debug build: a kernel computed an address outside its operand and skipped the access; the "
                         "output of that call is undefined");
    return set_error(TSM2_ERR_TIMEOUT, "a pipeline wait exceeded its bound; the output of that call is undefined");
}

int tsm2_debug_checks(void) { return kDebugChecks ? 1 : 0; }

void tsm2_shutdown(void) {
    int cur = 0;
    cudaGetDevice(&cur);
    {
        std::lock_guard<std::mutex> lk(g_pipe_mu);
        for (auto &kv : g_pipes) {
            cudaSetDevice(kv.first);
            for (cudaStream_t s : {kv.second->in, kv.second->comp, kv.second->out}) cudaStreamSynchronize(s);
            pipe_destroy(kv.second);
        }
        g_pipes.clear();
    }
    std::lock_guard<std::mutex> lk(g_mu);
    for (auto &kv : g_ws) {
        std::lock_guard<std::mutex> ws(kv.second.mu);
        if (!kv.second.ptr) continue;
        cudaSetDevice(kv.first.first);
        cudaFree(kv.second.ptr);
        kv.second.ptr = nullptr;
        kv.second.bytes = kv.second.counter_bytes = 0;
    }
    free_unused_graph_scratch();
    cudaSetDevice(cur);
}

tsm2_status tsm2x_s(int64_t m, int64_t n, int64_t k, const float *A, int64_t lda, const float *B, int64_t ldb, float *C,
                    int64_t ldc, void *stream) {
    return gemm("tsm2x_s", tsm2x_schedule(4, m, n, k), 4, m, n, k, A, lda, B, ldb, C, ldc, stream);
}

tsm2_status tsm2x_d(int64_t m, int64_t n, int64_t k, const double *A, int64_t lda, const double *B, int64_t ldb,
                    double *C, int64_t ldc, void *stream) {
    return gemm("tsm2x_d", tsm2x_schedule(8, m, n, k), 8, m, n, k, A, lda, B, ldb, C, ldc, stream);
}

char tsm2x_choice(int elem_bytes, int64_t m, int64_t n, int64_t k) {
    if ((elem_bytes != 4 && elem_bytes != 8) || m < 0 || n < 0 || k < 0) return 0;
    return tsm2x_schedule(elem_bytes, m, n, k);
}

tsm2_status tsm2r_s_host(int64_t m, int64_t n, int64_t k, const float *A, int64_t lda, const float *B, int64_t ldb,
                         float *C, int64_t ldc, void *stream) {
    return gemm_host("tsm2r_s_host", 'r', 4, m, n, k, A, lda, B, ldb, C, ldc, stream);
}

tsm2_status tsm2r_d_host(int64_t m, int64_t n, int64_t k, const double *A, int64_t lda, const double *B, int64_t ldb,
                         double *C, int64_t ldc, void *stream) {
    return gemm_host("tsm2r_d_host", 'r', 8, m, n, k, A, lda, B, ldb, C, ldc, stream);
}

tsm2_status tsm2l_s_host(int64_t m, int64_t n, int64_t k, const float *A, int64_t lda, const float *B, int64_t ldb,
                         float *C, int64_t ldc, void *stream) {
    return gemm_host("tsm2l_s_host", 'l', 4, m, n, k, A, lda, B, ldb, C, ldc, stream);
}

tsm2_status tsm2l_d_host(int64_t m, int64_t n, int64_t k, const double *A, int64_t lda, const double *B, int64_t ldb,
                         double *C, int64_t ldc, void *stream) {
    return gemm_host("tsm2l_d_host", 'l', 8, m, n, k, A, lda, B, ldb, C, ldc, stream);
}

tsm2_status tsm2r_t_d(int64_t m, int64_t n, int64_t k, const double *A, int64_t lda, const double *dC, int64_t lddc,
                      double *dB, int64_t lddb, void *stream) {
    return gemm_t("tsm2r_t_d", 8, m, n, k, A, lda, dC, lddc, dB, lddb, stream);
}

tsm2_status tsm2r_t_s(int64_t m, int64_t n, int64_t k, const float *A, int64_t lda, const float *dC, int64_t lddc,
                      float *dB, int64_t lddb, void *stream) {
    return gemm_t("tsm2r_t_s", 4, m, n, k, A, lda, dC, lddc, dB, lddb, stream);
}

tsm2_status tsm2_rankk_d(int64_t m, int64_t n, int64_t k, const double *dC, int64_t lddc, const double *B, int64_t ldb,
                         double *dA, int64_t ldda, void *stream) {
    return rankk("tsm2_rankk_d", 8, m, n, k, dC, lddc, B, ldb, dA, ldda, stream);
}

tsm2_status tsm2_rankk_s(int64_t m, int64_t n, int64_t k, const float *dC, int64_t lddc, const float *B, int64_t ldb,
                         float *dA, int64_t ldda, void *stream) {
    return rankk("tsm2_rankk_s", 4, m, n, k, dC, lddc, B, ldb, dA, ldda, stream);
}

tsm2_status tsm2r_bf16(int64_t m, int64_t n, int64_t k, const uint16_t *A_hi, const uint16_t *A_lo, int64_t lda,
                       const float *B, int64_t ldb, float *C, int64_t ldc, void *stream) {
    return gemm_bf16(m, n, k, A_hi, A_lo, lda, B, ldb, C, ldc, stream);
}

tsm2_status tsm2_split_bf16(int64_t rows, int64_t cols, const float *X, int64_t ldx, uint16_t *hi, uint16_t *lo,
                            int64_t ldh, void *stream) {
    if (rows < 0 || cols < 0) return set_error(TSM2_ERR_INVALID_VALUE, "tsm2_split_bf16: negative dimension");
    if (ldx < (rows > 1 ? rows : 1) || ldh < (rows > 1 ? rows : 1))
        return set_error(TSM2_ERR_INVALID_VALUE, "tsm2_split_bf16: leading dimension < max(1,rows)");
    if (rows == 0 || cols == 0) return TSM2_SUCCESS;
    if (!X || !hi) return set_error(TSM2_ERR_INVALID_VALUE, "tsm2_split_bf16: X or hi is NULL");
    DeviceState *dev = nullptr;
    tsm2_status st = device_state(&dev);
    if (st != TSM2_SUCCESS) return st;
    cudaError_t e = split_bf16_launch(rows, cols, X, ldx, hi, lo, ldh, dev->sm_count, static_cast<cudaStream_t>(stream));
    return e == cudaSuccess ? TSM2_SUCCESS : cuda_error(e, "split kernel launch");
}

tsm2_status tsm2_batch_plan_create_s(int nprob, const tsm2_problem_s *probs, int flags, tsm2_batch_plan_t *out) {
    if (!out) return set_error(TSM2_ERR_INVALID_VALUE, "tsm2_batch_plan_create_s: out is NULL");
    *out = nullptr;
    if (nprob < 0 || (nprob > 0 && !probs))
        return set_error(TSM2_ERR_INVALID_VALUE, "tsm2_batch_plan_create_s: bad problem list");
    const int variant = (flags >> 8) & 0xFF;
    if (variant >= batch_menu_count())
        return set_error(TSM2_ERR_INVALID_VALUE, "tsm2_batch_plan_create_s: tile variant %d out of [0, %d)", variant,
                         batch_menu_count());
    DeviceState *dev = nullptr;
    tsm2_status st = device_state(&dev);
    if (st != TSM2_SUCCESS) return st;
    tsm2_batch_plan_s *P = new tsm2_batch_plan_s();
    cudaGetDevice(&P->dev);
    P->sm_count = dev->sm_count;
    P->single_grid = dev->sm_count;
    P->variant = variant;
    P->menu = batch_menu(variant);
    const bool merge_r = (flags & TSM2_BATCH_MERGE_R) != 0;
    const bool merge_l = (flags & TSM2_BATCH_MERGE_L) != 0;
    // Class of a column chunk: the narrowest slot of its schedule that holds
    // kk columns (the widest with the merge flag).
    auto slot_for = [&](char op, int kk) -> int {
        int best = -1;
        for (int t = 0; t < P->menu->nslots; ++t) {
            const BatchClass *c = P->menu->slots[t];
            if (c->op != op || c->KC < kk) continue;
            const bool merge = op == 'r' ? merge_r : merge_l;
            if (best < 0 || (merge ? c->KC > P->menu->slots[best]->KC : c->KC < P->menu->slots[best]->KC)) best = t;
        }
        return best;
    };
    std::map<int, int> index;  // slot -> class
    for (int i = 0; i < nprob; ++i) {
        const tsm2_problem_s &q = probs[i];
        const char op = q.op == 'l' ? 'l' : (q.op == 'r' ? 'r' : 0);
        if (!op) {
            destroy_plan(P);
            return set_error(TSM2_ERR_INVALID_VALUE, "batch problem %d: op must be 'r' or 'l'", i);
        }
        st = check_args("tsm2_batch_plan_create_s", q.m, q.n, q.k, q.A, q.lda, q.B, q.ldb, q.C, q.ldc, 4);
        if (st != TSM2_SUCCESS) {
            destroy_plan(P);
            return st;
        }
        if (q.m == 0 || q.k == 0) continue;
        if (q.n == 0) {
            P->zeros.push_back({q.C, q.ldc, q.m, q.k});
            continue;
        }
        if (op == 'l' && (q.n > 64 || q.k > 64)) {
            destroy_plan(P);
            return set_error(TSM2_ERR_UNSUPPORTED, "batch problem %d: TSM2L needs n, k <= 64", i);
        }
        if (!aligned16(q.A) || (q.lda * 4) % 16 != 0 || q.m >= (1ll << 31) - 4096 || q.n >= (1ll << 31) ||
            (op == 'r' && (!aligned16(q.B) || (q.ldb * 4) % 16 != 0))) {
            destroy_plan(P);
            return set_error(TSM2_ERR_UNSUPPORTED,
                             "batch problem %d: batched operands need 16-byte aligned bases and leading dimensions", i);
        }
        const int kcmax = op == 'l' ? 32 : 16;
        for (int64_t c0 = 0; c0 < q.k; c0 += kcmax) {
            const int kk = (int)std::min<int64_t>(kcmax, q.k - c0);
            const int slot = slot_for(op == 'l' ? 'w' : 'r', kk);
            if (slot < 0) {
                destroy_plan(P);
                return set_error(TSM2_ERR_UNSUPPORTED, "batch problem %d: no class for k chunk %d", i, kk);
            }
            const BatchClass *cls = P->menu->slots[slot];
            auto it = index.find(slot);
            if (it == index.end()) {
                it = index.emplace(slot, (int)P->classes.size()).first;
                P->classes.emplace_back();
                P->classes.back().cls = cls;
                P->classes.back().slot = slot;
            }
            auto &C = P->classes[it->second];
            ProbDesc d;
            std::memset(&d, 0, sizeof d);
            const float *Bc = q.B + c0 * q.ldb;
            st = encode_2d(&d.mapA, 4, q.A, q.m, q.n, q.lda, cls->BOXM, cls->BNS);
            if (st == TSM2_SUCCESS && op == 'r') st = encode_2d(&d.mapB, 4, Bc, q.n, kk, q.ldb, cls->BNS, cls->KC);
            if (st != TSM2_SUCCESS) {
                destroy_plan(P);
                return st;
            }
            const int64_t num_rb = (q.m + cls->BM - 1) / cls->BM;
            const int64_t upr = (q.n + cls->BNS - 1) / cls->BNS;
            d.m = q.m;
            d.n = q.n;
            d.ldb = q.ldb;
            d.ldc = q.ldc;
            d.B = Bc;
            d.C = q.C + c0 * q.ldc;
            d.k = kk;
            d.upr = (int32_t)upr;
            d.gran = op == 'l' ? (int32_t)upr : 1;
            d.c_vec = aligned16(d.C) && (q.ldc * 4) % 16 == 0;
            d.group_begin = C.ngroups;
            d.rb_begin = C.nrb;
            C.ngroups += op == 'l' ? num_rb : num_rb * upr;
            C.nrb += num_rb;
            C.bytes += 4.0 * ((double)q.m * q.n + (double)q.n * kk + (double)q.m * kk);
            C.host.push_back(d);
        }
    }
    // Classes in menu order: the single launch walks them in this order.
    std::sort(P->classes.begin(), P->classes.end(),
              [](const tsm2_batch_plan_s::Cls &a, const tsm2_batch_plan_s::Cls &b) { return a.slot < b.slot; });
    cudaError_t e = cudaSuccess;
    for (auto &C : P->classes) {
        P->total_bytes += C.bytes;
        C.counter_bytes = ((size_t)C.nrb * sizeof(int) + 255) / 256 * 256;
        // Partial-sum slots for grids of up to one block per SM (TSM2R
        // classes split row blocks; TSM2L classes never do).
        const size_t slots = C.cls->op == 'r' ? (size_t)(P->sm_count + C.nrb) * C.cls->KC * C.cls->BM * 4 : 0;
        if ((e = cudaMalloc(&C.d_ws, C.counter_bytes + slots + 256)) != cudaSuccess) break;
        if ((e = cudaMalloc(&C.d_probs, C.host.size() * sizeof(ProbDesc))) != cudaSuccess) break;
        if ((e = cudaMemcpy(C.d_probs, C.host.data(), C.host.size() * sizeof(ProbDesc), cudaMemcpyHostToDevice)) !=
            cudaSuccess)
            break;
        if ((e = cudaMemset(C.d_ws, 0, C.counter_bytes)) != cudaSuccess) break;
        if ((e = cudaStreamCreateWithFlags(&C.aux, cudaStreamNonBlocking)) != cudaSuccess) break;
        if ((e = cudaEventCreateWithFlags(&C.done, cudaEventDisableTiming)) != cudaSuccess) break;
    }
    if (e == cudaSuccess) e = cudaEventCreateWithFlags(&P->fork, cudaEventDisableTiming);
    if (e == cudaSuccess) e = cudaStreamCreateWithFlags(&P->capture, cudaStreamNonBlocking);
    if (e == cudaSuccess) {
        // Even shares for the first single launch.
        std::vector<BatchBalance> init(1);
        std::memset(init.data(), 0, sizeof(BatchBalance));
        for (int b = 0; b < kBalanceMaxBlocks; ++b) init[0].w[0][b] = init[0].w[1][b] = 1.0f;
        e = cudaMalloc(&P->d_bal, sizeof(BatchBalance));
        if (e == cudaSuccess) e = cudaMemcpy(P->d_bal, init.data(), sizeof(BatchBalance), cudaMemcpyHostToDevice);
    }
    if (e != cudaSuccess) {
        destroy_plan(P);
        return cuda_error(e, "tsm2_batch_plan_create_s");
    }
    // Default SM shares of the concurrent mode: proportional to each class's
    // algorithmic bytes.
    const int nc = (int)P->classes.size();
    if (nc > 0) {
        int left = std::max(P->sm_count - nc, 0);
        double tot = 0;
        for (auto &C : P->classes) tot += C.bytes;
        for (auto &C : P->classes) {
            const int g = 1 + (int)((double)left * C.bytes / (tot > 0 ? tot : 1));
            C.grid = (int)std::min<int64_t>(g, C.ngroups);
        }
    }
    {
        std::lock_guard<std::mutex> lk(g_plans_mu);
        g_plans.push_back(P);
    }
    *out = P;
    return TSM2_SUCCESS;
}

tsm2_status tsm2_batch_plan_execute(tsm2_batch_plan_t plan, void *stream) {
    if (!plan) return set_error(TSM2_ERR_INVALID_VALUE, "tsm2_batch_plan_execute: NULL plan");
    return plan_execute(plan, static_cast<cudaStream_t>(stream), -1);
}

tsm2_status tsm2_batch_plan_execute_class(tsm2_batch_plan_t plan, int cls, void *stream) {
    if (!plan || cls < 0 || cls >= (int)plan->classes.size())
        return set_error(TSM2_ERR_INVALID_VALUE, "tsm2_batch_plan_execute_class: bad plan or class");
    return plan_execute(plan, static_cast<cudaStream_t>(stream), cls);
}

tsm2_status tsm2_batch_plan_graph_launch(tsm2_batch_plan_t plan, void *stream_v) {
    if (!plan) return set_error(TSM2_ERR_INVALID_VALUE, "tsm2_batch_plan_graph_launch: NULL plan");
    cudaStream_t stream = static_cast<cudaStream_t>(stream_v);
    cudaError_t e;
    if (!plan->graph) {
        // Captured once on the plan's own stream (the legacy default stream
        // cannot be captured); the executable graph then runs on any stream.
        e = cudaStreamBeginCapture(plan->capture, cudaStreamCaptureModeThreadLocal);
        if (e != cudaSuccess) return cuda_error(e, "cudaStreamBeginCapture");
        tsm2_status st = plan_execute(plan, plan->capture, -1);
        cudaGraph_t graph = nullptr;
        e = cudaStreamEndCapture(plan->capture, &graph);
        if (st != TSM2_SUCCESS) {
            if (graph) cudaGraphDestroy(graph);
            return st;
        }
        if (e != cudaSuccess) return cuda_error(e, "cudaStreamEndCapture");
        e = cudaGraphInstantiate(&plan->graph, graph, 0);
        cudaGraphDestroy(graph);
        if (e != cudaSuccess) {
            plan->graph = nullptr;
            return cuda_error(e, "cudaGraphInstantiate");
        }
    }
    e = cudaGraphLaunch(plan->graph, stream);
    return e == cudaSuccess ? TSM2_SUCCESS : cuda_error(e, "cudaGraphLaunch");
}

int tsm2_batch_plan_num_classes(tsm2_batch_plan_t plan) { return plan ? (int)plan->classes.size() : 0; }

tsm2_status tsm2_batch_plan_class_info(tsm2_batch_plan_t plan, int cls, const char **name, double *bytes, int *grid,
                                       int *nprob) {
    if (!plan || cls < 0 || cls >= (int)plan->classes.size())
        return set_error(TSM2_ERR_INVALID_VALUE, "tsm2_batch_plan_class_info: bad plan or class");
    const auto &c = plan->classes[cls];
    if (name) *name = c.cls->name;
    if (bytes) *bytes = c.bytes;
    if (grid) *grid = c.grid;
    if (nprob) *nprob = (int)c.host.size();
    return TSM2_SUCCESS;
}

static void drop_graph(tsm2_batch_plan_t plan) {
    if (plan->graph) {
        cudaGraphExecDestroy(plan->graph);
        plan->graph = nullptr;
    }
}

tsm2_status tsm2_batch_plan_set_grids(tsm2_batch_plan_t plan, int ncls, const int *grids) {
    if (!plan || ncls != (int)plan->classes.size() || (ncls > 0 && !grids))
        return set_error(TSM2_ERR_INVALID_VALUE, "tsm2_batch_plan_set_grids: bad arguments");
    for (int i = 0; i < ncls; ++i) {
        if (grids[i] < 1 || grids[i] > plan->sm_count)
            return set_error(TSM2_ERR_INVALID_VALUE, "tsm2_batch_plan_set_grids: grid %d out of [1, %d]", grids[i],
                             plan->sm_count);
    }
    for (int i = 0; i < ncls; ++i)
        plan->classes[i].grid = (int)std::min<int64_t>(grids[i], plan->classes[i].ngroups);
    drop_graph(plan);
    return TSM2_SUCCESS;
}

tsm2_status tsm2_batch_plan_set_serial(tsm2_batch_plan_t plan, int serial) {
    if (!plan) return set_error(TSM2_ERR_INVALID_VALUE, "tsm2_batch_plan_set_serial: NULL plan");
    return tsm2_batch_plan_set_mode(plan, serial ? TSM2_BATCH_SERIAL : TSM2_BATCH_CONCURRENT);
}

tsm2_status tsm2_batch_plan_set_mode(tsm2_batch_plan_t plan, int mode) {
    if (!plan) return set_error(TSM2_ERR_INVALID_VALUE, "tsm2_batch_plan_set_mode: NULL plan");
    if (mode != TSM2_BATCH_CONCURRENT && mode != TSM2_BATCH_SERIAL && mode != TSM2_BATCH_SINGLE_LAUNCH)
        return set_error(TSM2_ERR_INVALID_VALUE, "tsm2_batch_plan_set_mode: unknown mode %d", mode);
    if (plan->mode != mode) drop_graph(plan);
    plan->mode = mode;
    return TSM2_SUCCESS;
}

tsm2_status tsm2_batch_plan_set_single_grid(tsm2_batch_plan_t plan, int grid) {
    if (!plan || grid < 1 || grid > plan->sm_count)
        return set_error(TSM2_ERR_INVALID_VALUE, "tsm2_batch_plan_set_single_grid: bad plan or grid");
    if (plan->single_grid != grid) drop_graph(plan);
    plan->single_grid = grid;
    return TSM2_SUCCESS;
}

int tsm2_batch_plan_num_launches(tsm2_batch_plan_t plan) {
    if (!plan || plan->classes.empty()) return 0;
    return plan->mode == TSM2_BATCH_SINGLE_LAUNCH ? 1 : (int)plan->classes.size();
}

int tsm2_batch_num_variants(void) { return batch_menu_count(); }

tsm2_status tsm2_batch_variant_info(int variant, const char **name, int *stages, int *rows_per_lane,
                                    int *inner_per_warp) {
    const BatchMenu *m = (variant >= 0) ? batch_menu(variant) : nullptr;
    if (!m) return set_error(TSM2_ERR_INVALID_VALUE, "tsm2_batch_variant_info: variant %d out of range", variant);
    if (name) *name = m->name;
    if (stages) *stages = m->stages;
    if (rows_per_lane) *rows_per_lane = m->rows_per_lane;
    if (inner_per_warp) *inner_per_warp = m->inner_per_warp;
    return TSM2_SUCCESS;
}

void tsm2_batch_plan_destroy(tsm2_batch_plan_t plan) { destroy_plan(plan); }

void tsm2_set_wait_budget_ns(int64_t ns) { g_wait_ns = ns < 0 ? -1 : ns; }

void tsm2_set_path(int path) { g_path = path; }

void tsm2_set_grid(int blocks) { g_grid_override = blocks < 0 ? 0 : blocks; }

void tsm2_set_host_copy(int mode) { g_host_copy = mode == 1 ? 1 : 0; }

void tsm2_set_balance(int mode) { g_balance = (mode == 1 || mode == 2) ? mode : 0; }

void tsm2_set_trace(unsigned long long *device_words, int64_t blocks) {
    g_trace = device_words;
    g_trace_blocks = device_words ? blocks : 0;
}

tsm2_status tsm2r_s_noalloc(int64_t m, int64_t n, int64_t k, const float *A, int64_t lda, const float *B,
                            int64_t ldb, float *C, int64_t ldc, void *stream) {
    return gemm_r32_noalloc(m, n, k, A, lda, B, ldb, C, ldc, stream);
}

}  // extern "C"
