// Binary64 products with a short inner dimension on the tensor cores: C(M x N)
// = A(M x K) B(K x N), K <= 32 -- TSM2L (A tall, N small) and the rank-k
// update dA = dC B^T (N large).
//
// The numbers are those of tsm2_f64tc.cu: eight base-256 digits of A and B
// relative to a power-of-two scale per row of A and column of B, multiplied as
// binary16 integers, summed exactly in the binary32 accumulators and rounded
// once.  With so few products per output, two things differ.
//
//  * Ten weights s + t = 0 .. 9 are kept instead of eight, so that what is
//    dropped stays below 2^-72.7 alpha beta per product.
//  * An output is certified by flags of its row and column instead of by a
//    sum.  With the scale alpha the power of two at or below the largest
//    element, call an element cut if it is not zero and below 2^-9 of its scale
//    (only then does its fixed-point number lose bits), strong if at least 2^-4
//    and top if at least 1/2 of it.  If neither the row nor the column has a
//    cut element, every nonzero product is at least 2^-18 alpha beta and the
//    dropped pairs are below u / 2 of it (u = 2^-53).  If the column is strong
//    where the row is top, or the row where the column is, S = sum |a||b| is at
//    least 2^-5 alpha beta, and what the cut elements lose, at most
//    K 2^-59 alpha beta, is below K u / 2 S.  (Either way inside gamma_K S with
//    the final rounding.)  Otherwise the output is computed with binary64
//    FMAs, as are rows and columns with infinities, NaN or a scale outside
//    2^+-440.  (Of uniform inputs that is one output in 10^4 for K = 2 and none
//    from about K = 8.)
//
// Mapping.  One block per SM.  Four converter warps (a thread per row of a
// 128-row tile, or 126 of a tile by column classes where A is not aligned, A
// through a TMA ring) store the digits of a tile as the A
// operand in tensor memory; one MMA warp multiplies it by groups of 16 columns
// of B (digits from f64s_digits_kernel, resident in shared memory for N <= 64,
// else through a ring); 16 drainer warps, eight for each of the two
// accumulator buffers (160 columns: 10 weights x 16 columns of C), combine the
// ten sums of an output to a 96-bit integer, round it and store C.  The
// persistent grid splits tiles x column groups evenly.
//
// What bounds it: instructions, about 100 for an output and 30 for an element of
// A (the integer half-rate pipe 70 % busy, 0.65 of the issue slots; the tensor
// cores 12 to 22 %), where binary64 FMAs hold the FP64 pipe for 64 cycles per
// product and warp.  So padding columns are skipped, no output branches, and
// the loops stay rolled (the unrolled roles missed the instruction cache: 2^22
// x 32 x 32 2610 us).  Measured on GB300, us, FMA kernels / this: 2^20 x 32 x 32
// 1732 / 222 (2.4 TB/s of A and C), 24 x 24 1013 / 208, 16 x 16 455 / 114, 8 x 8
// 119 / 83; rank-k 4096^2 x 16 515 / 80, 10000^2 x 16 2688 / 450, 512^2 x 16
// 134 / 11.
//
// Every wait is bounded; TMEM is always released before the block exits.
#include "common.cuh"
#include "f64digits.cuh"
#include "f64s.h"
#include "internal.h"
#include "tcgen05.cuh"

#include <mutex>

namespace tsm2 {
namespace {

constexpr int kTile = 128;                 // rows = MMA M
constexpr int kStep = 16;                  // inner indices of a unit
constexpr int kMaxUnits = kF64SMaxK / kStep;
constexpr int kCols = 16;                  // C columns of a group
constexpr int kWeights = 10;
constexpr int kDCols = kWeights * kCols;   // accumulator columns
constexpr int kAUnit = kTile * kStep * 8;  // 16 KB
constexpr int kBHalf = kDCols * 32;        // operand G of 8 inner indices
constexpr int kBUnit = 2 * kBHalf;
constexpr int kARing = 6;
constexpr int kBRing = 4;                  // groups; also the most that stay resident
constexpr int kInfo = 8;                   // tiles whose row flags, groups whose column flags are kept
constexpr int kOperand = 2 * kDCols;       // first TMEM column of the A operand
constexpr int kHalfCols = 4 * 8;           // of 8 inner indices
constexpr int kOpRing = 6;                 // such
constexpr int kTmemCols = 512;
constexpr int kDrainers = 16;
constexpr int kWarpA = 24, kWarpMma = 25, kWarpB = 26;
constexpr int kThreads = 896;              // warps 0-15 drain, 16-23 convert, 24-26 issue, 27 idle
constexpr int kLaunchRegs = 72, kDrainerRegs = 80, kConverterRegs = 64, kIssuerRegs = 48;
constexpr float kUnit = 16777216.f;        // digits of A carry 2^-24
constexpr int kLowExp = 570, kHighExp = 1460;  // exponent fields of scales that every pair of is safe
static_assert(4 * kDrainerRegs + 2 * kConverterRegs + kIssuerRegs <= 7 * kLaunchRegs, "register split");
static_assert(kOperand + kOpRing * kHalfCols <= kTmemCols && kOpRing >= 2 * kMaxUnits, "TMEM columns");

struct RowInfo {
    int exp;          // exponent of alpha
    uint32_t strong;  // strong elements (zero rows: all)
    uint32_t top;     // top elements (zero rows: all)
    int flags;        // 1: has cut elements, 2: not finite or out of range
};
constexpr int kTail = 512;
constexpr int kOffB = kARing * kAUnit;
constexpr int kOffBar = kOffB + kBRing * kMaxUnits * kBUnit;
constexpr int kOffInfo = kOffBar + kTail;
constexpr int kOffCols = kOffInfo + kInfo * kTile * (int)sizeof(RowInfo);
constexpr int kSmem = kOffCols + kInfo * kCols * 16 + 1024;
static_assert(kSmem <= 227 * 1024 && kOffCols % 16 == 0 && kOffB % 1024 == 0 && kBUnit % 128 == 0, "shared memory");

__device__ __forceinline__ constexpr uint32_t idesc_n(int n) {
    return (1u << 4) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(kTile >> 4) << 24);
}

struct SParams {
    ColumnClasses a;            // map[0], or with column classes (shift.h) both
    int64_t M, N;
    int K;
    const double *A;
    int64_t lda;
    const double *B;
    int64_t bes, bcs;
    const unsigned char *bdig;  // [group][unit][half][kBHalf]
    const int4 *cinfo;          // per column: exponent of beta - 2128, strong, top, flags (1 cut, 2 special)
    double *C;
    int64_t ldc;
    int accumulate;
    unsigned *status;
    int64_t wait_ns;
    int groups;    // of 16 columns
    int total;     // tiles x groups
    int whole;     // blocks take whole tiles
    int resident;  // all groups stay in shared memory
    unsigned long long *trace;
    int w24, w16, w8, w0;  // 2^24, 2^16, 2^8, 1: opaque, so that they stay multipliers
};

// (Debug builds: see common.cuh.)
__device__ __forceinline__ bool dbg_output(const SParams &p, int64_t row, int64_t col) {
    return dbg_in_bounds(row >= 0 && row < p.M && col >= 0 && col < p.N, p.status);
}

// Flags of element i relative to exponent e.
__device__ __forceinline__ void flag(uint32_t hi, uint32_t lo, int e, int i, uint32_t &strong, uint32_t &top, bool &cut) {
    const int d = e - exp_field(hi);
    strong |= (uint32_t)(d <= 4) << i;
    top |= (uint32_t)(d <= 1) << i;
    cut |= d > 9 && ((hi << 1) | lo) != 0u;
}
// The exponent and flags of a row or column; emax: its largest exponent field.
__device__ __forceinline__ RowInfo finish_flags(int emax, bool zero, uint32_t strong, uint32_t top, bool cut) {
    RowInfo r;
    const bool special = !zero && (emax < kLowExp || emax > kHighExp);
    r.exp = zero || special ? 1023 : emax;
    r.flags = (int)cut | (int)special << 1;
    r.strong = zero ? ~0u : strong;
    r.top = zero ? ~0u : top;
    return r;
}

// One thread per column and four inner indices: the column's scale and flags,
// and its part of G (tsm2_f64tc.cu): [group][unit][half][N group of 8][4 inner
// indices][8 columns][4 inner indices][digit v - 2, digit v], N group
// 2 v + (column % 16) / 8, v = 0 .. 9 (digits 8 and 9 are zero).
__global__ void __launch_bounds__(128) f64s_digits_kernel(int64_t N, int K, const double *__restrict__ B, int64_t bes,
                                                          int64_t bcs, unsigned char *out, int4 *cinfo, int units) {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int c = threadIdx.x & 15, quads = units * 4;
    const int64_t group = blockIdx.x;
    const int64_t col = group * kCols + c;
    int emax = 0;
    bool any = false;
    for (int j = 0; j < K; ++j) {
        const long long v = col < N ? __double_as_longlong(__ldg(B + j * bes + col * bcs)) & 0x7fffffffffffffffll : 0;
        emax = max(emax, (int)(v >> 52));
        any |= v != 0;
    }
    const bool special = any && (emax < kLowExp || emax > kHighExp);
    const int e = !any || special ? 1023 : emax;
    const uint32_t key = scale_key(e);
    if (threadIdx.x < 16) {
        uint32_t strong = 0, top = 0;
        bool cut = false;
        for (int j = 0; j < K; ++j) {
            const double b = col < N ? __ldg(B + j * bes + col * bcs) : 0.0;
            flag((uint32_t)__double2hiint(b), (uint32_t)__double2loint(b), e, j, strong, top, cut);
        }
        const RowInfo r = finish_flags(emax, !any, strong, top, cut);
        cinfo[col] = make_int4(r.exp - 2128, (int)r.strong, (int)r.top, r.flags);
    }
    for (int q = threadIdx.x >> 4; q < quads; q += 8) {
        uint64_t x[4];
        bool neg[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int j = q * 4 + i;
            const double b = (j < K && col < N) ? __ldg(B + j * bes + col * bcs) : 0.0;
            const uint32_t hi = (uint32_t)__double2hiint(b);
            x[i] = fixed_point(hi, (uint32_t)__double2loint(b), key) + 0x8080808080808080ull;
            neg[i] = hi >> 31;
        }
        unsigned char *o = out + (group * units * 2 + (q >> 1)) * kBHalf + (q & 1) * 128 + (c >> 3) * 256 + (c & 7) * 16;
#pragma unroll
        for (int v = 0; v < kWeights; ++v) {
            uint32_t g[4];
#pragma unroll
            for (int i = 0; i < 4; ++i)
                g[i] = (v < 8 ? digit_b(x[i], neg[i], v) << 16 : 0u) | (v >= 2 ? digit_b(x[i], neg[i], v - 2) : 0u);
            *reinterpret_cast<uint4 *>(o + v * 512) = make_uint4(g[0], g[1], g[2], g[3]);
        }
    }
}

// |x2:x1:x0| 2^s, rounded, where x2 is not zero in the fast path: the slow one
// is for every other sum.
__device__ __noinline__ double combine_small(uint32_t x0, uint32_t x1, uint32_t x2, uint32_t neg, int s) {
    uint32_t c = 0;
    if (neg) {  // x is the complement of the sum; the magnitude is one more
        c = ++x0 == 0;
        x1 += c;
        c = c && x1 == 0;
        x2 += c;
    }
    uint32_t a = x2, b = x1, d = x0;
    int e = s + 95;
    if (a == 0) { a = b; b = d; d = 0; e -= 32; }
    if (a == 0) { a = b; b = 0; e -= 32; }
    if (a == 0) return 0.0;
    const int z = __clz((int)a);
    uint64_t m = (uint64_t)__funnelshift_l(b, a, z) << 32 | __funnelshift_l(d, b, z);
    m = (m >> 11) + (m >> 10 & 1u);
    m += (uint64_t)(uint32_t)(e - z + 1022) << 52;
    return __longlong_as_double((long long)(m | (uint64_t)(neg & 0x80000000u) << 32));
}

// Two floats plus two others in one instruction.
__device__ __forceinline__ void add2(uint32_t a0, uint32_t a1, float b, int &r0, int &r1) {
    asm("{\n\t.reg .b64 x, y;\n\tmov.b64 x, {%2, %3};\n\tmov.b64 y, {%4, %4};\n\tadd.rn.f32x2 x, x, y;\n\t"
        "mov.b64 {%0, %1}, x;\n\t}"
        : "=r"(r0), "=r"(r1)
        : "r"(a0), "r"(a1), "f"(b));
}

// The sums of the ten weights of an output, as integers, of which the first
// kBiased<U> carry 0x3f400000, combined to a 96-bit integer, rounded (halves
// away from zero) and scaled by 2^s.  Written for the ALU pipe, half the rate
// of the FMA pipe: wide multiply-adds take the bias off and put the sums
// together.  mul: 2^24, 2^16, 2^8, 1 in registers, so that they stay
// multipliers.  Sums below 2^64 units are left to another call (few), so that
// what is done for each output has no branches.
template <int U>
constexpr int kBiased = U == 1 ? kWeights : 5;
template <int U, bool kAny>
__device__ __forceinline__ double combine(const int (&b)[kWeights], int s, const int (&mul)[4], bool &few) {
    constexpr int64_t kBias = 0x3f400000;
    // Weights 6-9 and 2-5; 2^48 makes the first positive.
    constexpr int64_t kLow = (U == 1 ? -kBias * 0x1010101 : 0) + (1ll << 48);
    constexpr int64_t kMid = -kBias * (U == 1 ? 0x1010101 : 0x1010100) - (1ll << 16);
    int64_t low = kLow, mid = kMid;
#pragma unroll
    for (int w = 0; w < 4; ++w) {
        low = mad_wide(b[6 + w], mul[w], low);
        mid = mad_wide(b[2 + w], mul[w], mid);
    }
    uint32_t x0 = (uint32_t)low, x1, x2;
    const uint32_t top = (uint32_t)(b[0] * mul[2] + b[1]) - (uint32_t)(kBias * 257);
    asm("{\n\tadd.cc.u32 %0, %2, %3;\n\taddc.u32 %1, %4, %5;\n\t}"
        : "=&r"(x1), "=r"(x2)
        : "r"((uint32_t)mid), "r"((uint32_t)(low >> 32)), "r"((uint32_t)(mid >> 32)), "r"(top));
    // The magnitude, one unit (2^-82 alpha beta) less where negative: that
    // matters only for sums of few bits.
    const uint32_t neg = (uint32_t)((int32_t)x2 >> 31);
    x0 ^= neg;
    x1 ^= neg;
    x2 ^= neg;
    if (kAny) {
        if (x2 == 0) return combine_small(x0, x1, x2, neg, s);
    } else {
        few = x2 == 0;
    }
    // x2 < 2^30: 53 bits from its first, at bit 10 of two words.
    const int z = __clz((int)x2) - 1;
    const uint32_t h = __funnelshift_l(x1, x2, z), l = __funnelshift_l(x0, x1, z);
    uint32_t rl, rh;
    asm("{\n\tadd.cc.u32 %0, %2, %4;\n\taddc.u32 %1, %3, 0;\n\t}" : "=&r"(rl), "=r"(rh) : "r"(l), "r"(h), "r"(0x200u));
    const uint32_t lo = __funnelshift_r(rl, rh, 10), hi = (rh >> 10) + ((uint32_t)(s + 94 + 1022 - z) << 20);
    return __hiloint2double((int)(hi | (neg & 0x80000000u)), (int)lo);
}

template <int U>
__device__ __noinline__ double combine_any(int b0, int b1, int b2, int b3, int b4, int b5, int b6, int b7, int b8, int b9, int s) {
    const int b[kWeights] = {b0, b1, b2, b3, b4, b5, b6, b7, b8, b9}, mul[4] = {1 << 24, 1 << 16, 1 << 8, 1};
    bool few;
    return combine<U, true>(b, s, mul, few);
}

// The output by binary64 FMAs.
__device__ __forceinline__ void fma_store(const SParams &p, int64_t row, int64_t col) {
    double out = 0.0;
    if (!dbg_output(p, row, col)) return;
#pragma unroll 1
    for (int j0 = 0; j0 < p.K; j0 += 8) {  // (eight at a time: their loads overlap)
        double a[8], b[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int j = min(j0 + i, p.K - 1);
            a[i] = __ldg(p.A + row + j * p.lda);
            b[i] = __ldg(p.B + j * p.bes + col * p.bcs);
        }
#pragma unroll
        for (int i = 0; i < 8; ++i)
            if (j0 + i < p.K) out = fma(a[i], b[i], out);
    }
    double *dst = p.C + row + col * p.ldc;
    *dst = p.accumulate ? *dst + out : out;
}

// Those of a warp's rows row0 .. row0 + 31 in columns col0 + i, bits i of each
// lane's `bad`: an output per lane, wherever it is.  (With every lane at its own
// row a warp took as many turns as its worst row has, two rows in 32 as long as
// all of them: 2^20 x 32 x 32 with one large row of B 2049 us, 1733 by the FMA
// kernel, here 590.)
__device__ __noinline__ void fma_outputs(const SParams &p, int64_t row0, int64_t col0, uint32_t bad) {
    const int lane = threadIdx.x & 31;
    int upto = __popc(bad);  // outputs of the lanes up to this one
#pragma unroll
    for (int o = 1; o < 32; o *= 2) {
        const int x = __shfl_up_sync(0xffffffffu, upto, o);
        if (lane >= o) upto += x;
    }
    const int total = __shfl_sync(0xffffffffu, upto, 31);
    for (int t = lane; t - lane < total; t += 32) {
        int l = 0;  // the lane that output t is of
#pragma unroll
        for (int o = 16; o >= 1; o /= 2)
            if (__shfl_sync(0xffffffffu, upto, l + o - 1) <= t) l += o;
        l = min(l, 31);
        uint32_t bits = __shfl_sync(0xffffffffu, bad, l);
        const int first = __shfl_sync(0xffffffffu, upto, l) - __popc(bits);
        if (t >= total) continue;
        for (int i = first; i < t; ++i) bits &= bits - 1u;
        fma_store(p, row0 + l, col0 + __ffs(bits) - 1);
    }
}

// The segments (tile, column groups g0 .. g1) of a block: a range of tile x
// group in order, or whole tiles in turn.
struct Walk {
    int pos, end, skip, groups;
    int tile, g0, g1;
    __device__ __forceinline__ Walk(const SParams &p, int g, int G);
    __device__ __forceinline__ bool next() {
        if (pos >= end) return false;
        tile = pos / groups;
        g0 = pos - tile * groups;
        g1 = min(groups, g0 + (end - pos));
        pos += g1 - g0;
        pos = end - pos > skip ? pos + skip : end;
        return true;
    }
};
__device__ __forceinline__ Walk::Walk(const SParams &p, int g, int G) {
    groups = p.groups;
    if (p.whole) {
        pos = g * groups;
        end = p.total;
        skip = (G - 1) * groups;
    } else {
        pos = (int)((int64_t)p.total * g / G);
        end = (int)((int64_t)p.total * (g + 1) / G);
        skip = 0;
    }
}

template <int U, bool Acc, bool Split>
__global__ void __launch_bounds__(kThreads, 1) f64s_kernel(const __grid_constant__ SParams p) {
    extern __shared__ unsigned char smem_raw[];
    unsigned char *smem = smem_aligned<1024>(smem_raw);
    uint64_t *afull = reinterpret_cast<uint64_t *>(smem + kOffBar);  // [kARing] A unit landed
    uint64_t *aempty = afull + kARing;                               // [kARing] converted
    uint64_t *bfull = aempty + kARing;                               // [kBRing] B group landed
    uint64_t *bempty = bfull + kBRing;                               // [kBRing] its MMAs done
    uint64_t *opfull = bempty + kBRing;                              // [kOpRing] A operand half stored
    uint64_t *opdone = opfull + kOpRing;                             // [kOpRing] its MMAs done
    uint64_t *dfull = opdone + kOpRing;                                    // [2] sums of a group ready
    uint64_t *dfree = dfull + 2;                                     // [2] read by the drainers
    uint64_t *info = dfree + 2;                                      // [kInfo] row flags of a tile written
    uint64_t *fin = info + kInfo;
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(fin + 1);
    volatile int *flags = reinterpret_cast<volatile int *>(tmem_slot + 2);  // [0] abort
    volatile RowInfo *rows = reinterpret_cast<volatile RowInfo *>(smem + kOffInfo);

    const int warp = threadIdx.x >> 5;
    const int lane = threadIdx.x & 31;
    const int G = gridDim.x, g = blockIdx.x;
    const int halves = (p.K + 7) / 8;
    constexpr int kRowsT = Split ? kTile - 2 : kTile;  // rows of a tile

    if (threadIdx.x == 0) {
        for (int s = 0; s < kARing; ++s) {
            mbar_init(&afull[s], 1);
            mbar_init(&aempty[s], 4);
        }
        for (int s = 0; s < kBRing; ++s) {
            mbar_init(&bfull[s], 1);
            mbar_init(&bempty[s], 1);
        }
        for (int s = 0; s < kOpRing; ++s) {
            mbar_init(&opfull[s], 4);
            mbar_init(&opdone[s], 1);
        }
        for (int s = 0; s < 2; ++s) {
            mbar_init(&dfull[s], 2);
            mbar_init(&dfree[s], kDrainers / 2);
        }
        for (int s = 0; s < kInfo; ++s) mbar_init(&info[s], 4);
        mbar_init(fin, 1);
        flags[0] = 0;
        if (p.trace) {
            p.trace[4 * g] = globaltimer_ns();
            p.trace[4 * g + 3] = (unsigned long long)((int64_t)p.total * (g + 1) / G - (int64_t)p.total * g / G);
        }
        fence_mbar_init();
    }
    if (warp == kWarpMma) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                     "r"(kTmemCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *reinterpret_cast<volatile uint32_t *>(tmem_slot);

    auto give_up = [&]() {
        flags[0] = 1;
        atomicOr(p.status, kStatusTimeout);
    };
    // Waits of whole warps, with one result for all lanes.
    auto wait = [&](uint64_t *bar, uint32_t parity) {
        bool ok = p.wait_ns >= 0 && mbar_try_wait(bar, parity);
        if (__all_sync(0xffffffffu, ok)) return true;
        ok = __all_sync(0xffffffffu, mbar_wait_bounded(bar, parity, p.wait_ns, flags));
        if (!ok && lane == 0) give_up();
        return ok;
    };

    if (warp >= kWarpA) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kIssuerRegs));
        if (warp == kWarpA && lane == 0) {
            // ---------------- A units ----------------
            prefetch_tensormap(&p.a.map[0]);
            const uint64_t policy = l2_policy_evict_first();
            int s = 0;
            uint32_t ph = 0, issued = 0, last_par = 0;
            Walk walk(p, g, G);
            while (!flags[0] && walk.next())
                for (int u = 0; u < U; ++u) {
                    if (flags[0] || !mbar_wait_bounded(&aempty[s], ph ^ 1u, p.wait_ns, flags)) {
                        give_up();
                        break;
                    }
                    mbar_arrive_expect_tx(&afull[s], kAUnit);
                    if (Split) {
#pragma unroll
                        for (int c = 0; c < 2; ++c)
                            tma_load_2d_hint(smem + s * kAUnit + c * (kAUnit / 2), &p.a.map[c], walk.tile * kRowsT,
                                             u * (kStep / 2), &afull[s], policy);
                    } else {
                        tma_load_2d_hint(smem + s * kAUnit, &p.a.map[0], walk.tile * kRowsT, u * kStep, &afull[s], policy);
                    }
                    issued |= 1u << s;
                    last_par = (last_par & ~(1u << s)) | (ph << s);
                    if (++s == kARing) { s = 0; ph ^= 1u; }
                }
            for (int t = 0; t < kARing; ++t)
                if (issued & (1u << t)) (void)mbar_wait_bounded(&afull[t], (last_par >> t) & 1u, 4000000000LL, nullptr);
        } else if (warp == kWarpB && lane == 0) {
            // ---------------- B groups ----------------
            asm volatile("griddepcontrol.wait;" ::: "memory");
            int s = 0;
            uint32_t ph = 0, issued = 0, last_par = 0;
            const uint32_t bytes = (uint32_t)(halves * kBHalf);
            int cslot = 0;
            auto copy = [&](int group) {
                if (!dbg_in_bounds(group >= 0 && group < p.groups, p.status) || flags[0] || !mbar_wait_bounded(&bempty[s], ph ^ 1u, p.wait_ns, flags)) {
                    give_up();
                    return;
                }
                mbar_arrive_expect_tx(&bfull[s], bytes + kCols * 16);
                bulk_g2s(smem + kOffB + s * U * kBUnit, p.bdig + (size_t)group * U * kBUnit, bytes, &bfull[s]);
                // (Its column flags, to the next of kInfo places; with B
                // resident to the group's own.  The drainers are done with the
                // group of kInfo = 2 kBRing groups ago when this slot is free:
                // its MMAs came after those that waited for them.)
                bulk_g2s(smem + kOffCols + cslot * kCols * 16, p.cinfo + (size_t)group * kCols, kCols * 16, &bfull[s]);
                if (++cslot == kInfo) cslot = 0;
                issued |= 1u << s;
                last_par = (last_par & ~(1u << s)) | (ph << s);
                if (++s == kBRing) { s = 0; ph ^= 1u; }
            };
            if (p.resident) {
                for (int q = 0; q < p.groups; ++q) copy(q);
            } else {
                Walk walk(p, g, G);
                while (!flags[0] && walk.next())
                    for (int q = walk.g0; q < walk.g1 && !flags[0]; ++q) copy(q);
            }
            for (int t = 0; t < kBRing; ++t)
                if (issued & (1u << t)) (void)mbar_wait_bounded(&bfull[t], (last_par >> t) & 1u, 4000000000LL, nullptr);
        } else if (warp == kWarpMma) {
            // ---------------- MMA issuer (a converged warp: elect_one) ----------------
            int s = 0, q = 0, tile = 0;
            uint32_t ph = 0;
            bool ok = true;
            Walk walk(p, g, G);
            for (; ok && walk.next(); ++tile) {
                const int op = tile * halves;
                for (int h = 0; h < halves && ok; ++h) ok = wait(&opfull[(op + h) % kOpRing], (uint32_t)((op + h) / kOpRing) & 1u);
                for (int group = walk.g0; group < walk.g1 && ok; ++group, ++q) {
                    const int slot = p.resident ? group : s;
                    ok = wait(&bfull[slot], p.resident ? 0u : ph) &&
                         (q < 2 || wait(&dfree[q & 1], (uint32_t)((q >> 1) - 1) & 1u));
                    if (!ok) break;
                    tc_fence_after();
                    const uint64_t bd = sdesc(smem_u32(smem + kOffB + slot * U * kBUnit), 128, 256, 0);
                    const uint32_t d = tmem + (uint32_t)((q & 1) * kDCols);
                    if (elect_one()) {
#pragma unroll
                        for (int h = 0; h < 2 * U; ++h) {
                            if (h >= halves) break;
                            const uint64_t b = bd + h * (kBHalf >> 4);
                            const int slot_a = (op + h) % kOpRing;
                            const uint32_t ah = tmem + (uint32_t)(kOperand + slot_a * kHalfCols);
                            umma_f16_ts(d, ah, b, idesc_n(10 * kCols), h > 0);
                            umma_f16_ts(d + 1 * kCols, ah + 8, b, idesc_n(9 * kCols), 1u);
                            umma_f16_ts(d + 4 * kCols, ah + 16, b, idesc_n(6 * kCols), 1u);
                            umma_f16_ts(d + 5 * kCols, ah + 24, b, idesc_n(5 * kCols), 1u);
                            if (group == walk.g1 - 1) umma_commit(&opdone[slot_a]);
                        }
                        umma_commit(&dfull[q & 1]);
                        if (!p.resident) umma_commit(&bempty[slot]);
                    }
                    __syncwarp();
                    // (With the tensor core's arrival, one of this thread, that
                    // hands on the column flags, which it has waited for.)
                    if (lane == 0) mbar_arrive(&dfull[q & 1]);
                    if (!p.resident && ++s == kBRing) { s = 0; ph ^= 1u; }
                }
            }
            // Every MMA of this warp has completed before TMEM is freed.
            if (elect_one()) umma_commit(fin);
            (void)mbar_wait_bounded(fin, 0, 4000000000LL, nullptr);
        }
    } else if (warp >= kDrainers) {
        // ---------------- converters: four warps for the even tiles, four for the odd; a thread per row --------
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kConverterRegs));
        const int r = threadIdx.x & (kTile - 1), set = (warp - kDrainers) >> 2;
        const uint32_t tA = tmem + ((uint32_t)((warp & 3) * 32) << 16) + kOperand;
        // With column classes: even and odd columns, rows behind by their shifts
        // (the last threads have no row).
        const int at0 = Split ? min(r + p.a.shift[0], kTile - 1) : r, at1 = Split ? min(r + p.a.shift[1], kTile - 1) : r;
        auto at = [&](int j) {
            return Split ? ((j & 1) * (kStep / 2) + (j >> 1)) * kTile + ((j & 1) ? at1 : at0) : j * kTile + r;
        };
        int tile = 0;
        bool ok = true;
        Walk walk(p, g, G);
        for (; ok && walk.next(); ++tile) {
            if ((tile & 1) != set) continue;
            // The largest exponent of the row.
            float mx = 0.f;
            uint32_t low = 0;
#pragma unroll 1
            for (int u = 0; u < U; ++u) {
                const int unit = tile * U + u;
                ok = ok && wait(&afull[unit % kARing], (uint32_t)(unit / kARing) & 1u);
                if (!ok) break;
                const uint2 *src = reinterpret_cast<const uint2 *>(smem + unit % kARing * kAUnit);
#pragma unroll
                for (int j = 0; j < kStep; ++j) {
                    const uint2 v = src[at(j)];
                    float d;
                    asm("max.NaN.f32 %0, %1, %2;" : "=f"(d) : "f"(fabsf(__uint_as_float(v.y))), "f"(mx));
                    mx = d;
                    low |= v.x;
                }
            }
            if (!ok) break;
            if (p.trace && tile == 0 && r == 0) p.trace[4 * g + 1] = globaltimer_ns();
            const bool zero = __float_as_int(mx) == 0 && low == 0;
            const int emax = __float_as_int(mx) >> 20;  // (2047 for patterns that are NaN in binary32)
            const bool special = !zero && (emax < kLowExp || emax > kHighExp);
            const int e = zero || special ? 1023 : emax;
            const uint32_t key = scale_key(e);
            uint32_t strong = 0, top = 0;
            bool cut = false;
#pragma unroll 1
            for (int h = 0; h < 2 * U; ++h) {
                const int unit = tile * U + h / 2;
                if (h < halves && ok) {
                    const uint2 *src = reinterpret_cast<const uint2 *>(smem + unit % kARing * kAUnit) +
                                       h % 2 * (Split ? 4 * kTile : 8 * kTile);
                    uint32_t w[8][4], strong8 = 0, top8 = 0;
#pragma unroll
                    for (int j = 0; j < 8; ++j) {
                        const uint2 v = src[at(j)];
                        flag(v.y, v.x, e, j, strong8, top8, cut);
                        digits(fixed_point(v.y, v.x, key), v.y, w[j]);
                    }
                    strong |= strong8 << (h * 8);
                    top |= top8 << (h * 8);
                    const int op = tile * halves + h, slot = op % kOpRing;
                    ok = op < kOpRing || wait(&opdone[slot], (uint32_t)(op / kOpRing - 1) & 1u);
                    if (ok) {
                        tc_fence_after();
#pragma unroll
                        for (int t = 0; t < 4; ++t)
                            tmem_st8(tA + slot * kHalfCols + t * 8, w[0][t], w[1][t], w[2][t], w[3][t], w[4][t],
                                     w[5][t], w[6][t], w[7][t]);
                        if (h < halves - 1) {
                            tmem_st_wait();
                            tc_fence_before();
                            __syncwarp();
                            if (lane == 0) mbar_arrive(&opfull[slot]);
                        }
                    }
                }
                if (h % 2 == 1) {
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&aempty[unit % kARing]);
                }
            }
            if (!ok) break;
            const RowInfo f = finish_flags(emax, zero, strong, top, cut);
            volatile RowInfo &out = rows[(tile % kInfo) * kTile + r];
            out.exp = f.exp;
            out.strong = f.strong;
            out.top = f.top;
            out.flags = f.flags;
            tmem_st_wait();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) {
                mbar_arrive(&info[tile % kInfo]);
                mbar_arrive(&opfull[(tile * halves + halves - 1) % kOpRing]);
            }
        }
    } else {
        // ---------------- drainers ----------------
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kDrainerRegs));
        const int dbuf = warp >> 3, c0 = (warp >> 2 & 1) * 8, r = (warp & 3) * 32 + lane;
        const uint32_t tD = tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)(dbuf * kDCols + c0);
        const int mul[4] = {p.w24, p.w16, p.w8, p.w0};
        auto put = [&](double *dst, double out) {
            if (Acc) out += *dst;
            __stcs(dst, out);
        };
        int q = 0, tile = 0;
        bool ok = true;
        Walk walk(p, g, G);
        for (; ok && walk.next(); ++tile) {
            const int64_t row = (int64_t)walk.tile * kRowsT + r;
            RowInfo me;
            bool have = false;
            for (int group = walk.g0; group < walk.g1; ++group, ++q) {
                if ((q & 1) != dbuf) continue;
                if (!have) {
                    ok = wait(&info[tile % kInfo], (uint32_t)(tile / kInfo) & 1u);
                    if (!ok) break;
                    const volatile RowInfo &in = rows[(tile % kInfo) * kTile + r];
                    me.exp = in.exp;
                    me.strong = in.strong;
                    me.top = in.top;
                    me.flags = in.flags;
                    have = true;
                }
                ok = wait(&dfull[dbuf], (uint32_t)(q >> 1) & 1u);
                if (!ok) break;
                tc_fence_after();
                const int4 *cols = reinterpret_cast<const int4 *>(smem + kOffCols) + (p.resident ? group : q % kInfo) * kCols + c0;
                if (!dbg_in_bounds(group >= 0 && group < p.groups, p.status)) break;
                const int64_t col0 = (int64_t)group * kCols + c0;
                const int live = r < kRowsT && row < p.M ? (int)min((int64_t)8, p.N - col0) : 0;
                double *dst = p.C + row + col0 * p.ldc;
                uint32_t bad = 0;
                // (Not unrolled, as the converters' loops: the code of the
                // roles together stays within the instruction cache.)
#pragma unroll 1
                for (int b = 0; b < 2; ++b) {
                    if (col0 + b * 4 >= p.N) {  // (only padding)
                        if (b == 0) {
                            tc_fence_before();
                            __syncwarp();
                            if (lane == 0) mbar_arrive(&dfree[dbuf]);
                        }
                        break;
                    }
                    const bool last = b == 1 || col0 + 4 >= p.N;
                    uint32_t v[kWeights][4];
#pragma unroll
                    for (int w = 0; w < kWeights; ++w) tmem_ld4(tD + w * kCols + b * 4, v[w]);
                    tmem_ld_wait();
                    if (last) {
                        tc_fence_before();
                        __syncwarp();
                        if (lane == 0) mbar_arrive(&dfree[dbuf]);
                    }
                    uint32_t small = 0;
#pragma unroll
                    for (int c = 0; c < 4; ++c) {
                        int x[kWeights];
#pragma unroll
                        for (int w = 0; w < kWeights; ++w) {
                            // (|sum| < 2^22 2^-24: adding 0.75 leaves an integer.)
                            if (w < kBiased<U>) {
                                if ((c & 1) == 0) {
                                    int x0, x1;
                                    add2(v[w][c], v[w][c + 1], 0.75f, x0, x1);
                                    v[w][c] = (uint32_t)x0;
                                    v[w][c + 1] = (uint32_t)x1;
                                }
                                x[w] = (int)v[w][c];
                            } else {
                                x[w] = __float2int_rn(__uint_as_float(v[w][c]) * kUnit);
                            }
                        }
                        const int4 ci = cols[b * 4 + c];
                        bool few;
                        const double out = combine<U, false>(x, me.exp + ci.x, mul, few);
                        const int fl = me.flags | ci.w;
                        const bool fail = (((uint32_t)ci.y & me.top) == 0 && (me.strong & (uint32_t)ci.z) == 0 && fl != 0) || fl > 1;
                        if (fail) bad |= 1u << (b * 4 + c);
                        if (few) small |= 1u << c;
                        if (b * 4 + c < live && !fail && !few && dbg_output(p, row, col0 + b * 4 + c)) put(dst + c * p.ldc, out);
                    }
                    if (__any_sync(0xffffffffu, small != 0)) {
#pragma unroll
                        for (int c = 0; c < 4; ++c)
                            if (b * 4 + c < live && (small & ~(bad >> (b * 4))) >> c & 1u && dbg_output(p, row, col0 + b * 4 + c)) {
                                int x[kWeights];
#pragma unroll
                                for (int w = 0; w < kWeights; ++w)
                                    x[w] = w < kBiased<U> ? (int)v[w][c] : __float2int_rn(__uint_as_float(v[w][c]) * kUnit);
                                put(dst + c * p.ldc, combine_any<U>(x[0], x[1], x[2], x[3], x[4], x[5], x[6], x[7], x[8],
                                                                    x[9], me.exp + cols[b * 4 + c].x));
                            }
                    }
                    dst += 4 * p.ldc;
                }
                // What was not certified, by binary64 FMAs.
                if (__any_sync(0xffffffffu, bad != 0)) fma_outputs(p, row - lane, col0, live > 0 ? bad & ((1u << live) - 1u) : 0u);
            }
        }
    }
    // Everyone (including idle lanes) meets here before the TMEM is freed.
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (p.trace && threadIdx.x == 0) p.trace[4 * g + 2] = globaltimer_ns();
    if (warp == kWarpMma)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols) : "memory");
}

template <int U, bool Acc, bool Split>
cudaError_t launch_units(const SParams &p, int grid, cudaStream_t stream) {
    static std::mutex mu;
    static uint64_t attr_done = 0;  // one bit per device
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    {
        std::lock_guard<std::mutex> lk(mu);
        if (dev >= 64 || !(attr_done & (1ull << dev))) {
            e = cudaFuncSetAttribute(f64s_kernel<U, Acc, Split>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmem);
            if (e != cudaSuccess) return e;
            if (dev < 64) attr_done |= 1ull << dev;
        }
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = kSmem;
    cfg.stream = stream;
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, f64s_kernel<U, Acc, Split>, p);
}

}  // namespace

int f64s_tile() { return kTile; }
int f64s_rows(bool split) { return split ? kTile - 2 : kTile; }
int f64s_cols() { return kCols; }
int f64s_step() { return kStep; }

size_t f64s_digit_bytes(int64_t N, int K) {
    const int64_t groups = (N + kCols - 1) / kCols, units = (K + kStep - 1) / kStep;
    return (size_t)groups * ((size_t)units * kBUnit + kCols * sizeof(int4));
}

cudaError_t f64s_launch(const F64SLaunch &L, cudaStream_t stream) {
    SParams p;
    p.a = L.a;
    p.M = L.M;
    p.N = L.N;
    p.K = L.K;
    p.A = L.A;
    p.lda = L.lda;
    p.B = L.B;
    p.bes = L.bes;
    p.bcs = L.bcs;
    const int units = (L.K + kStep - 1) / kStep;
    p.groups = (int)((L.N + kCols - 1) / kCols);
    unsigned char *bdig = static_cast<unsigned char *>(L.digits);
    int4 *cinfo = reinterpret_cast<int4 *>(bdig + (size_t)p.groups * units * kBUnit);
    p.bdig = bdig;
    p.cinfo = cinfo;
    p.C = L.C;
    p.ldc = L.ldc;
    p.accumulate = L.accumulate;
    p.status = L.status;
    p.wait_ns = L.wait_ns;
    p.w24 = 1 << 24;
    p.w16 = 1 << 16;
    p.w8 = 1 << 8;
    p.w0 = 1;
    // A block's part: as many tile x group pairs as another's, in order, so
    // that it converts few tiles more than once -- or, with several tiles for a
    // block and little B, whole tiles in turn, so that neighbours read
    // neighbouring rows.
    const int rows = f64s_rows(L.split);
    const int64_t tiles = (L.M + rows - 1) / rows;
    p.resident = p.groups <= kBRing;
    p.total = (int)(tiles * p.groups);
    p.whole = p.resident && tiles >= 8 * (int64_t)L.blocks;
    const int grid = (int)(p.total < L.blocks ? p.total : L.blocks);
    p.trace = L.trace && L.trace_blocks >= grid ? L.trace : nullptr;
    f64s_digits_kernel<<<(unsigned)p.groups, 128, 0, stream>>>(L.N, L.K, L.B, L.bes, L.bcs, bdig, cinfo, units);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    if (L.split)
        return units == 1 ? launch_units<1, false, true>(p, grid, stream) : launch_units<2, false, true>(p, grid, stream);
    if (L.accumulate)
        return units == 1 ? launch_units<1, true, false>(p, grid, stream) : launch_units<2, true, false>(p, grid, stream);
    return units == 1 ? launch_units<1, false, false>(p, grid, stream) : launch_units<2, false, false>(p, grid, stream);
}

}  // namespace tsm2
