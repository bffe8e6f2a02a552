// TSM2R and TSM2L for operands with any alignment and leading dimensions
// (a matrix as a program happens to have it: odd sizes, no padding), through
// the bulk-copy engine.
//
// A tensor map wants a 16-byte aligned base and strides that are multiples of
// 16 bytes, which an odd leading dimension does not give.  But every P-th
// column (P = 4 in binary32, 2 in binary64) has a stride of P lda elements,
// a multiple of 16 bytes whatever lda is.  So A is read through P maps, one
// per class of columns j = q P + r, each starting at the 16-byte boundary at
// or below the class's first element: its rows then lie 0 .. P - 1 elements
// behind the map's.  (The elements before the first row belong to the column
// before, or to the same 16 bytes as the first element of A; they are copied
// and never used.)  A row block is BM - 4 rows (BM - 2 in binary64), so that
// it lies inside the BM elements that are copied in every class, and a lane
// reads its rows one by one from shared memory (32 lanes, 32 consecutive
// rows: no bank conflicts) at an offset per class.
//
// Everything else follows tsm2_stream.cu: outer products with A read once
// (Algorithm 2), a ring of stages filled by one producer lane, B rows stored
// row-major beside each stage by the three other producer warps and read by
// broadcast (Algorithm 3), a persistent grid.  Each warp owns 32 R rows and
// all inner columns, so no sums cross warps.  The inner dimension of every row
// block is cut into the same `splits` ranges (chosen by shift_splits), whose
// partial sums the last block to finish one of a row block adds in order: all
// rows are summed in the same order, as with the element-wise kernel.
//
// Bound by HBM where a row block has many stages (30719 x 20001 x 8: 367 us,
// 6.7 TB/s), else by the combine of the ranges and the launch.  Measured on
// GB300, element-wise kernel (one thread per row, one load in flight) / here,
// us: 10001 x 4099 x 5 660 / 35, x 16 880 / 46; TSM2L 300001 x 31 x 31 163 / 27.
//
// Every wait is bounded; on timeout the block records it, stops consuming,
// lets its copies land and exits.
#include "common.cuh"
#include "internal.h"
#include "shift.h"

#include <mutex>

namespace tsm2 {
namespace {

constexpr int kStep = kShiftStep;
constexpr int kWarps = 8;       // consumer warps
constexpr int kThreads = 384;   // + the producer warpgroup
constexpr int kBox = 256;       // elements per column of a box
constexpr int kMaxStages = 8;

template <typename T_, int KC_, int R_>
struct ShiftCfg {
    using T = T_;
    static constexpr int KC = KC_, R = R_;
    static constexpr int P = 16 / (int)sizeof(T);   // column classes
    static constexpr int Q = kStep / P;             // columns of a class per stage
    static constexpr int BM = kWarps * 32 * R;      // elements copied per column
    static constexpr int Rows = BM - P;             // rows per row block
    static constexpr int NB = BM / kBox;            // boxes per class
    static constexpr int AStage = kStep * BM;       // elements
    static constexpr int BStage = kStep * KC;
    static constexpr int StageBytes = (AStage + BStage) * (int)sizeof(T);
    static constexpr int Fit = (200 * 1024) / StageBytes;
    static constexpr int Stages = Fit < kMaxStages ? Fit : kMaxStages;
    static constexpr int Smem = Stages * StageBytes + 256 + 128;
    static constexpr size_t Slot = (size_t)KC * BM * sizeof(T);
    static_assert(BM % kBox == 0 && StageBytes % 128 == 0 && Stages >= 3, "stage geometry");
    static_assert((BStage * (int)sizeof(T)) % 128 == 0, "alignment of the next stage");
};

struct ShiftParams {
    ColumnClasses a;
    int64_t m, n;
    int k;
    const void *B;
    int64_t ldb;
    void *C;
    int64_t ldc;
    void *slots;     // one per range of a row block (splits > 1)
    int *counters;
    unsigned *status;
    int64_t wait_ns;
    int upr;         // stages per row block
    int splits;      // ranges per row block
    int items;       // ranges in total, range t of row block t / splits
};

template <class K>
__global__ void __launch_bounds__(kThreads, 1) shift_kernel(const __grid_constant__ ShiftParams p) {
    using T = typename K::T;
    extern __shared__ unsigned char smem_raw[];
    unsigned char *smem = smem_aligned<128>(smem_raw);
    uint64_t *full = reinterpret_cast<uint64_t *>(smem + K::Stages * K::StageBytes);
    uint64_t *empty = full + K::Stages;
    volatile int *flags = reinterpret_cast<volatile int *>(empty + K::Stages);  // [0] abort, [1] last arriver

    const int warp = threadIdx.x >> 5;
    const int lane = threadIdx.x & 31;
    const int G = gridDim.x, g = blockIdx.x;
    // The stages [first, last) of range t of its row block.
    auto first_of = [&](int t) { return (int)((int64_t)(t % p.splits) * p.upr / p.splits); };
    auto last_of = [&](int t) { return (int)((int64_t)(t % p.splits + 1) * p.upr / p.splits); };

    if (threadIdx.x == 0) {
        for (int s = 0; s < K::Stages; ++s) {
            mbar_init(&full[s], 2);  // the producer lane (and its bytes), a loader warp
            mbar_init(&empty[s], kWarps);
        }
        flags[0] = flags[1] = 0;
        fence_mbar_init();
    }
    __syncthreads();

    if (warp >= kWarps) {
        if (warp == kWarps && lane == 0) {
            // ---------------- producer ----------------
            for (int r = 0; r < K::P; ++r) prefetch_tensormap(&p.a.map[r]);
            const uint64_t policy = l2_policy_evict_first();
            int s = 0;
            uint32_t ph = 0, issued = 0, last_par = 0;
            for (int t = g; t < p.items && !flags[0]; t += G) {
                const int rb = t / p.splits, last = last_of(t);
                for (int kc = first_of(t); kc < last; ++kc) {
                    if (flags[0] || !mbar_wait_bounded(&empty[s], ph ^ 1u, p.wait_ns, flags)) {
                        flags[0] = 1;
                        atomicOr(p.status, kStatusTimeout);
                        break;
                    }
                    T *dst = reinterpret_cast<T *>(smem + s * K::StageBytes);
                    mbar_arrive_expect_tx(&full[s], K::AStage * (int)sizeof(T));
#pragma unroll
                    for (int r = 0; r < K::P; ++r)
#pragma unroll
                        for (int b = 0; b < K::NB; ++b)
                            // (A class without columns is copied from behind class 0's last: zeros.)
                            tma_load_2d_hint(dst + (r * K::NB + b) * K::Q * kBox, &p.a.map[r], rb * K::Rows + b * kBox,
                                             p.a.cols[r] ? kc * K::Q : p.a.cols[0], &full[s], policy);
                    issued |= 1u << s;
                    last_par = (last_par & ~(1u << s)) | (ph << s);
                    if (++s == K::Stages) { s = 0; ph ^= 1u; }
                }
            }
            for (int t = 0; t < K::Stages; ++t)
                if (issued & (1u << t)) (void)mbar_wait_bounded(&full[t], (last_par >> t) & 1u, 4000000000LL, nullptr);
        } else if (warp > kWarps) {
            // ---------------- loaders: B rows of every third stage, row-major ----------------
            const T *B = static_cast<const T *>(p.B);
            constexpr int N = (K::BStage + 31) / 32;
            const int mine = warp - kWarps - 1;
            int s = 0, turn = 0;
            uint32_t ph = 0;
            bool ok = true;
            for (int t = g; t < p.items && ok; t += G) {
                const int last = last_of(t);
                for (int kc = first_of(t); kc < last && ok; ++kc) {
                    if (turn == mine) {
                        ok = __all_sync(0xffffffffu,
                                        !flags[0] && mbar_wait_bounded(&empty[s], ph ^ 1u, p.wait_ns, flags));
                        if (!ok) {
                            if (lane == 0) {
                                flags[0] = 1;
                                atomicOr(p.status, kStatusTimeout);
                            }
                            break;
                        }
                        const int64_t j0 = (int64_t)kc * kStep;
                        T x[N];
#pragma unroll
                        for (int e = 0; e < N; ++e) {
                            const int q = e * 32 + lane, c = q / kStep;
                            const int64_t j = j0 + q % kStep;
                            x[e] = (c < p.k && j < p.n && dbg_in_bounds(j >= 0 && c >= 0, p.status)) ? __ldg(B + j + (int64_t)c * p.ldb) : T(0);
                        }
                        T *dst = reinterpret_cast<T *>(smem + s * K::StageBytes) + K::AStage;
#pragma unroll
                        for (int e = 0; e < N; ++e) {
                            const int q = e * 32 + lane;
                            if (q < K::BStage) dst[(q % kStep) * K::KC + q / kStep] = x[e];
                        }
                        __syncwarp();
                        if (lane == 0) mbar_arrive(&full[s]);
                    }
                    if (++turn == 3) turn = 0;
                    if (++s == K::Stages) { s = 0; ph ^= 1u; }
                }
            }
        }
        return;
    }

    // ---------------- consumers ----------------
    // Row i of the lane: 128-element spans of R x 32 rows per warp.
    auto row_of = [&](int i) { return warp * 32 * K::R + i * 32 + lane; };
    int off[K::P][K::R];
#pragma unroll
    for (int r = 0; r < K::P; ++r)
#pragma unroll
        for (int i = 0; i < K::R; ++i) {
            int x = row_of(i) + p.a.shift[r];
            if (x >= K::BM) x = K::BM - 1;  // (rows behind the row block: not stored)
            off[r][i] = (r * K::NB + x / kBox) * K::Q * kBox + x % kBox;
        }
    T acc[K::R][K::KC];
#pragma unroll
    for (int i = 0; i < K::R; ++i)
#pragma unroll
        for (int c = 0; c < K::KC; ++c) acc[i][c] = T(0);
    int s = 0;
    uint32_t ph = 0;
    bool aborted = false;
    T *C = static_cast<T *>(p.C);

    for (int item = g; item < p.items; item += G) {
        const int rb = item / p.splits, last_kc = last_of(item);
        for (int kc = first_of(item); kc < last_kc; ++kc) {
            if (!aborted) {
                const bool ok = __all_sync(0xffffffffu, !flags[0] && mbar_wait_bounded(&full[s], ph, p.wait_ns, flags));
                if (!ok) {
                    aborted = true;
                    if (lane == 0) {
                        flags[0] = 1;
                        atomicOr(p.status, kStatusTimeout);
                    }
                }
            }
            if (!aborted) {
                const T *a_st = reinterpret_cast<const T *>(smem + s * K::StageBytes);
                const T *b_st = a_st + K::AStage;
#pragma unroll
                for (int q = 0; q < K::Q; ++q)
#pragma unroll
                    for (int r = 0; r < K::P; ++r) {
                        T a[K::R];
#pragma unroll
                        for (int t = 0; t < K::R; ++t) a[t] = a_st[off[r][t] + q * kBox];
                        const T *b = b_st + (q * K::P + r) * K::KC;
                        if constexpr (sizeof(T) == 4) {
                            if constexpr (K::KC >= 4) {
#pragma unroll
                                for (int c = 0; c < K::KC; c += 4) {
                                    const float4 v = *reinterpret_cast<const float4 *>(b + c);
#pragma unroll
                                    for (int t = 0; t < K::R; ++t) {
                                        const float2 aa = make_float2(a[t], a[t]);
                                        const float2 x = __ffma2_rn(aa, make_float2(v.x, v.y), make_float2(acc[t][c], acc[t][c + 1]));
                                        const float2 y = __ffma2_rn(aa, make_float2(v.z, v.w), make_float2(acc[t][c + 2], acc[t][c + 3]));
                                        acc[t][c] = x.x;
                                        acc[t][c + 1] = x.y;
                                        acc[t][c + 2] = y.x;
                                        acc[t][c + 3] = y.y;
                                    }
                                }
                            } else {
                                const float2 v = *reinterpret_cast<const float2 *>(b);
#pragma unroll
                                for (int t = 0; t < K::R; ++t) {
                                    const float2 x = __ffma2_rn(make_float2(a[t], a[t]), v, make_float2(acc[t][0], acc[t][1]));
                                    acc[t][0] = x.x;
                                    acc[t][1] = x.y;
                                }
                            }
                        } else {
#pragma unroll
                            for (int c = 0; c < K::KC; c += 2) {
                                const double2 v = *reinterpret_cast<const double2 *>(b + c);
#pragma unroll
                                for (int t = 0; t < K::R; ++t) {
                                    acc[t][c] = fma(a[t], v.x, acc[t][c]);
                                    acc[t][c + 1] = fma(a[t], v.y, acc[t][c + 1]);
                                }
                            }
                        }
                    }
                __syncwarp();
                if (lane == 0) mbar_arrive(&empty[s]);
            }
            if (++s == K::Stages) { s = 0; ph ^= 1u; }
        }
        const int64_t row0 = (int64_t)rb * K::Rows;
        if (p.splits == 1) {
            if (!aborted)
#pragma unroll
                for (int t = 0; t < K::R; ++t) {
                    const int64_t row = row0 + row_of(t);
                    if (row_of(t) < K::Rows && row < p.m && dbg_in_bounds(row >= 0, p.status))
#pragma unroll
                        for (int c = 0; c < K::KC; ++c)
                            if (c < p.k) C[row + (int64_t)c * p.ldc] = acc[t][c];
                }
        } else {
            const int gA = rb * p.splits, gB = gA + p.splits - 1;
            const bool in = dbg_in_bounds(gA >= 0 && gB < p.items && item >= gA && item <= gB, p.status);
            auto piece = [&](int q) { return static_cast<T *>(p.slots) + (int64_t)q * (K::KC * K::BM); };
            T *slot = piece(item);
            if (in)
#pragma unroll
                for (int t = 0; t < K::R; ++t)
#pragma unroll
                    for (int c = 0; c < K::KC; ++c)
                        if (c < p.k) __stcg(slot + c * K::BM + row_of(t), acc[t][c]);
            __threadfence();
            named_bar_sync(1, kWarps * 32);
            if (threadIdx.x == 0) {
                int last = 0;
                if (!flags[0] && in) {
                    last = atomicAdd(&p.counters[rb], 1) == p.splits - 1;
                    if (last) p.counters[rb] = 0;
                }
                flags[1] = last;
            }
            named_bar_sync(1, kWarps * 32);
            if (flags[1]) {
                // The pieces in block order, several in flight.
                __threadfence();
                constexpr int U = 4, W = K::KC < 4 ? K::KC : 4;
#pragma unroll 1
                for (int c0 = 0; c0 < p.k; c0 += W) {
                    T sum[K::R][W];
#pragma unroll
                    for (int t = 0; t < K::R; ++t)
#pragma unroll
                        for (int c = 0; c < W; ++c) sum[t][c] = T(0);
#pragma unroll 1
                    for (int gp = gA; gp <= gB; gp += U) {
                        T x[U][K::R][W];
#pragma unroll
                        for (int u = 0; u < U; ++u) {
                            const T *src = piece(gp + u <= gB ? gp + u : gA);
#pragma unroll
                            for (int t = 0; t < K::R; ++t)
#pragma unroll
                                for (int c = 0; c < W; ++c)
                                    x[u][t][c] = gp + u <= gB && c0 + c < p.k
                                                     ? __ldcg(src + (c0 + c) * K::BM + row_of(t)) : T(0);
                        }
#pragma unroll
                        for (int u = 0; u < U; ++u)
#pragma unroll
                            for (int t = 0; t < K::R; ++t)
#pragma unroll
                                for (int c = 0; c < W; ++c)
                                    if (gp + u <= gB) sum[t][c] += x[u][t][c];
                    }
#pragma unroll
                    for (int t = 0; t < K::R; ++t) {
                        const int64_t row = row0 + row_of(t);
                        if (row_of(t) < K::Rows && row < p.m && dbg_in_bounds(row >= 0 && c0 >= 0, p.status))
#pragma unroll
                            for (int c = 0; c < W; ++c)
                                if (c0 + c < p.k) C[row + (int64_t)(c0 + c) * p.ldc] = sum[t][c];
                    }
                }
            }
            named_bar_sync(1, kWarps * 32);  // flags[1] is reused by the next piece
        }
#pragma unroll
        for (int t = 0; t < K::R; ++t)
#pragma unroll
            for (int c = 0; c < K::KC; ++c) acc[t][c] = T(0);
    }
}

template <class K>
cudaError_t launch_cfg(const ShiftLaunch &L, cudaStream_t stream) {
    static std::mutex mu;
    static uint64_t attr_done = 0;  // one bit per device
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    {
        std::lock_guard<std::mutex> lk(mu);
        if (dev >= 64 || !(attr_done & (1ull << dev))) {
            e = cudaFuncSetAttribute(shift_kernel<K>, cudaFuncAttributeMaxDynamicSharedMemorySize, K::Smem);
            if (e != cudaSuccess) return e;
            if (dev < 64) attr_done |= 1ull << dev;
        }
    }
    ShiftParams p;
    p.a = L.a;
    p.m = L.g.m;
    p.n = L.g.n;
    p.k = L.g.k;
    p.B = L.g.B;
    p.ldb = L.g.ldb;
    p.C = L.g.C;
    p.ldc = L.g.ldc;
    p.slots = L.slots;
    p.counters = L.counters;
    p.status = L.status;
    p.wait_ns = L.wait_ns;
    p.upr = (int)((L.g.n + kStep - 1) / kStep);
    p.splits = L.splits;
    p.items = (int)((L.g.m + K::Rows - 1) / K::Rows) * L.splits;
    shift_kernel<K><<<L.grid, kThreads, K::Smem, stream>>>(p);
    return cudaGetLastError();
}

struct Entry {
    ShiftShape shape;
    cudaError_t (*launch)(const ShiftLaunch &, cudaStream_t);
};
template <class K>
Entry entry(const char *name) {
    return Entry{ShiftShape{name, (int)sizeof(typename K::T), K::KC, K::R, K::Rows, K::Slot}, &launch_cfg<K>};
}
#define TSM2_SHIFT(T, N, KC, R) entry<ShiftCfg<T, KC, R>>("simple_shift_" N "_kc" #KC "_r" #R)
// Four rows per lane (binary64 and the wide chunks: two), or one where the
// problem has too few row blocks for the grid.
const Entry kEntries[] = {
    TSM2_SHIFT(float, "f32", 2, 4),  TSM2_SHIFT(float, "f32", 4, 4),  TSM2_SHIFT(float, "f32", 8, 4),
    TSM2_SHIFT(float, "f32", 16, 4), TSM2_SHIFT(float, "f32", 2, 1),  TSM2_SHIFT(float, "f32", 4, 1),
    TSM2_SHIFT(float, "f32", 8, 1),  TSM2_SHIFT(float, "f32", 16, 1), TSM2_SHIFT(double, "f64", 2, 2),
    TSM2_SHIFT(double, "f64", 4, 2), TSM2_SHIFT(double, "f64", 8, 2), TSM2_SHIFT(double, "f64", 16, 2),
    TSM2_SHIFT(float, "f32", 24, 2), TSM2_SHIFT(float, "f32", 32, 2), TSM2_SHIFT(float, "f32", 24, 1),
    TSM2_SHIFT(float, "f32", 32, 1),
    TSM2_SHIFT(double, "f64", 2, 1), TSM2_SHIFT(double, "f64", 4, 1), TSM2_SHIFT(double, "f64", 8, 1),
    TSM2_SHIFT(double, "f64", 16, 1),
};
#undef TSM2_SHIFT

}  // namespace

const ShiftShape *shift_shape(int elem, int kc, bool tall) {
    for (const Entry &e : kEntries)
        if (e.shape.elem == elem && e.shape.KC == kc && (e.shape.R > 1) == tall) return &e.shape;
    return nullptr;
}

size_t shift_slot_bytes(const ShiftShape *shape, int64_t num_rb, int splits) {
    return splits > 1 ? (size_t)(num_rb * splits) * shape->slot : 0;
}

// The cut of the inner dimension with the least estimated time, in stages: the
// rounds of `blocks` blocks over all ranges, each with its stages, the writing
// of its sums (a slot is KC / 16 of a stage, written and read) and the adding
// of a row block's ranges, which delays some block in every round (four
// columns of four slots at a time, 0.5 to 0.7 stages each).  On GB300 it gives
// 30719 x 20001 x 16 within 1% of the measured 458 / 426 / 440 / 475 / 518 us
// for 4 / 9 / 14 / 19 / 24 ranges.
int shift_splits(const ShiftShape *shape, int64_t num_rb, int64_t upr, int blocks) {
    int best = 1;
    double best_cost = 1e300;
    for (int s = 1; s <= 64 && s <= upr && (s == 1 || num_rb * s <= 8 * blocks); ++s) {
        const double rounds = (double)((num_rb * s + blocks - 1) / blocks);
        const double sums = s == 1 ? 0 : shape->KC / 8.0 + 1;
        const double add = s == 1 ? 0 : (s + 3) / 4 * ((shape->KC + 3) / 4) * (shape->R > 1 ? 0.7 : 0.5);
        const double cost = rounds * ((upr + s - 1) / s + sums + add);
        if (cost < best_cost) {
            best_cost = cost;
            best = s;
        }
    }
    return best;
}

cudaError_t shift_launch(const ShiftShape *shape, const ShiftLaunch &L, cudaStream_t stream) {
    for (const Entry &e : kEntries)
        if (&e.shape == shape) return e.launch(L, stream);
    return cudaErrorInvalidValue;
}

}  // namespace tsm2
