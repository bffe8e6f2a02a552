// Binary64 TSM2R on the tensor cores: C(m x k) = A(m x n) B(n x k), exact
// fixed-point digits of A and B multiplied as binary16 integers.  Also with A
// of any alignment (column classes, shift.h) and transposed (dB = A^T dC: the
// rows are then columns of A in memory, read as swizzled lines of 128 bytes).
//
// Why.  GB300 has two binary64 FMA units per SM and cycle (1.25 TFLOP/s), so
// the outer-product kernel (tsm2_stream.cu) is bound by them from k = 2 on:
// at k = 16 it streams A at 5% of HBM.  The tensor cores multiply binary16
// 2000 times faster, and products and sums of small integers are exact in
// their binary32 accumulators.  So the product is taken over integer digits
// (the error-free splitting of Ozaki, Ogita, Oishi and Rump, 2012), with the
// digits of A made on the fly from the streamed tile: A is read once.
//
// Numbers.  Row i of A has a power-of-two scale alpha_i, column c of B a
// scale beta_c.  |a| / alpha is cut to a fixed-point number X < 2^62 (one
// unit is 2^-61 alpha, all |a| < 2 alpha).  The digits A_s of a are the eight
// bytes of X, most significant first, each with the sign of a; those of b,
// B_t, are made from the same number but lie in -128..127 (128 is added to
// every byte and taken off each digit).  Then
//     sum_j a_ij b_jc = alpha beta 2^-122 sum_{s,t} 2^(8 (14 - s - t)) sum_j A_s B_t.
// All pairs of digits s + t <= 7 are multiplied (36 of 64).  The pairs with
// the same s + t share one accumulator, exactly: at most 8 pairs x 64 inner
// indices x 255 x 128 < 2^24.  After 64 inner indices the eight accumulators
// go into a 96-bit integer (H 2^32 + L) in registers, which is exact, so the
// summation order does not matter; one rounding to binary64 ends the sum.
// A digit of A needs no conversion: the binary16 bit pattern 0x00bb is the
// subnormal bb 2^-24, and 0x80bb its negative, so one byte select per pair
// of digits makes the operand.  (Digits of A in -128..127 would allow 128
// inner indices, but take twice the converters' instructions.)
//
// Error.  Cutting a and b: 2^-59 alpha beta per product; dropped pairs
// (s + t >= 8): at most 14 * 2^-60 alpha beta.  Together at most 2^-56
// alpha beta per product that is not zero.  Where S = sum |a||b| is at least
// alpha beta / 2, the error is at most n u / 4 S (u = 2^-53) before the final
// rounding, where it is at least alpha beta / 7 and eight products are not zero
// 7/8 n u S, of which the rounding adds no more than the rest: inside the
// gamma_n bound of the binary64 FMA chain; for values of similar size it is
// far smaller (about 2^-60 alpha beta sqrt(n)).  (In a piece of l of the n inner
// indices l / n of that alpha beta / 7 is enough: the pieces' errors add up to
// the same.)  That is checked for every
// output of every piece of a row block, on the terms of S from the first on
// until they suffice (about 8 of uniform or normally distributed values; with
// alpha beta / 2 alone the latter took 32, and 4096^2 x 16 107 us instead of
// 91, 2^20 x 64 x 64 3300 instead of 1900).  Outputs that do not reach it --
// rows or columns with zeros or very uneven magnitudes where they meet,
// infinities, NaN, scales near the ends of the exponent range -- are computed
// again with binary64 FMAs by a kernel behind this one (settle), so every input
// has the same bound and the IEEE results for special values, and the time
// depends on the values (figures at settle).
//
// The scale of a row is four times the power of two above the first 16
// elements that are not all zero.  When a later element does not fit, the accumulators of the
// block are drained, the row takes the larger scale and its integer sum is
// shifted right (at most 2^-66 alpha beta per change).
//
// Mapping.  One block per SM: 8 converter warps, 8 drainer warps, two MMA
// warps and a producer warp each for A and B.  A stage is 256 rows x 16 inner
// columns of A (32 KB) and the digits of 16 rows of B (8 KB, prepared by
// f64_digits_kernel); A has a ring of six, free again as soon as the
// converters have read it, B one of three, held until the MMAs are done.  Every
// converter thread owns one row: it reads its 16 elements from shared memory
// (consecutive lanes, consecutive rows: no bank
// conflicts), makes the digits and stores them as the A operand in tensor
// memory (one lane = one row); shared memory carries A twice (written by TMA,
// read once) instead of four times as with an A operand there.  A packed pair
// holds digits s and s + 2 of one element (two bytes of a word that are
// already 16 bits apart, so nothing is interleaved): the 16 K slots of an MMA
// are 8 elements x 2 digits, and the B operand G has in N column (v, c) digit
// v of B for the slots of digit s and digit v - 2 for those of digit s + 2,
// so that both land in accumulator s + v.  The same G serves the digit pairs
// (0,2), (1,3), (4,6) and (5,7): it meets them at accumulator columns 0, 1, 4
// and 5 with N = 128, 112, 64 and 48.  The two halves of the row block (128
// rows each) have their own accumulators (128 columns), two operand buffers
// (64 columns each), MMA warp and drainers, so tensor memory is full, and
// they drain at different times.  The drainers hold the integer sums, add the
// accumulators to them (128 columns, each a conversion to an integer and a
// wide multiply-add, every 64 inner indices) and end the row blocks, while
// the converters go on.  Converter warp w and drainer warp w share 32 rows
// (TMEM lanes) and nothing else: the converter posts a task (which MMAs to
// wait for, the rows' scales, the end of a row block) at the end of every
// chunk of 64 inner indices and when one of its rows needs a larger scale; in
// that case the drainer also clears the 32 lanes, and the accumulation goes
// on for the other warps.  Row blocks split between blocks (stream-K, as in
// tsm2_stream.cu) meet as integers in the workspace, added by a third kernel.
//
// Measured (GB300): 20480^2 x 16 10754 us with binary64 FMAs, 785 us here
// (A at 4.3 TB/s, 63% of the copy rate); 4096^2 x 16
// 457 / 61, 1024^2 x 8 43 / 25.  What bounds it: instruction issue and latency
// of the converters (1320 warp instructions per scheduler and stage, 0.55
// issued per cycle; ALU pipe 52%, tensor cores 29% busy); small products: the
// three launches and the combine of split row blocks.
//
// Every wait is bounded; TMEM is always released before the block exits.
#include "common.cuh"
#include "f64digits.cuh"
#include "f64tc.h"
#include "internal.h"
#include "tcgen05.cuh"

#include <cooperative_groups.h>

#include <mutex>

namespace tsm2 {
namespace {

constexpr int kRows = 256;                   // rows per row block (less kClasses with column classes)
constexpr int kClasses = 2;                  // column classes of an unaligned A (shift.h)
constexpr int kHalf = 128;                   // rows per warpgroup = MMA M
constexpr int kStep = 16;                    // inner columns per stage = MMA K
constexpr int kDig = 8;                      // digits per number
constexpr int kKC = 16;                      // C columns per pass
constexpr int kAStage = kRows * kStep * 8;   // 32 KB
constexpr int kG = kDig * kKC * 32;          // 4096: G for 8 inner indices (16 slots)
constexpr int kBStage = 2 * kG;
constexpr int kARing = 6, kBRing = 3;         // stages
constexpr int kRingBytes = kARing * kAStage + kBRing * kBStage;
constexpr int kChunk = 4;                    // stages per drain: 64 inner indices keep the sums below 2^24
constexpr int kDCols = kDig * kKC;           // accumulator columns per warpgroup
constexpr int kAHalf = 4 * 8;                // operand columns of 8 inner indices: 4 digit pairs
constexpr int kABuf = 2 * kAHalf;            // of a stage
constexpr int kACols = 2 * kABuf;            // two buffers
constexpr int kTmemCols = 512;
constexpr int kThreads = 640;                // warps 0-7 convert, 8-15 drain, 16 and 19 producers of A and B, 17-18 MMA issuers
constexpr int kConverterRegs = 88, kDrainerRegs = 128, kIssuerRegs = 48;  // of 640 x 96 at launch
constexpr int kHeadroom = 2;                 // bits above the first elements of a row
constexpr float kUnit = 16777216.f;          // digits of A carry 2^-24
constexpr float kCertify = 0.51f;            // S in units of alpha beta (a half, and the rounding of its sum)
constexpr float kCertifyDense = 0.146f;      // with eight products that are not zero (a seventh), of a whole row
constexpr int kScan = 4096;                  // inner indices that a drainer looks at for that
constexpr int kZeroCol = -1;                 // scale of a column of zeros
constexpr int kFailCount = 16;               // (index in bexp) strips listed
constexpr int kShort = 64;                   // inner indices that the drainers settle themselves
constexpr int kSettleCols = 4;               // columns of a block that adds pieces
constexpr int kSettleWarps = 8;
constexpr int kSettlePerSM = 4;              // blocks that settle
constexpr int kSettleHalf = kKC / 2;         // columns that one of them takes
constexpr int kSettleUnits = 4096;           // parts of sums in the workspace
constexpr int kLaunchRegs = 96;
static_assert(kConverterRegs <= kLaunchRegs && kIssuerRegs <= kLaunchRegs && kDrainerRegs >= kLaunchRegs &&
                  2 * kConverterRegs + 2 * kDrainerRegs + kIssuerRegs <= 5 * kLaunchRegs,
              "register split");
static_assert(2 * (kDCols + kACols) <= kTmemCols, "TMEM columns");
// Shared memory behind the stages: barriers and flags, then one task per
// converter warp.
struct Task {
    int stage;       // stage whose MMAs end the sums
    int clear;       // clear the lanes afterwards (a scale changes inside a chunk)
    int rb;          // end of a piece of row block rb (-1: not an end): stages kc0 .. kc1 - 1,
    int kc0, kc1;
    int whole;       // all of the row block
    int last;        // no more tasks
    int pad;
    int exp[32];     // exponent of alpha, per row, and kNonzero if the row of the piece is not zeros
};
constexpr int kNonzero = 1 << 12;
constexpr int kTail = 512;
constexpr int kSmem = kRingBytes + kTail + 8 * (int)sizeof(Task) + 8 * 512 + 1024;
static_assert(kSmem <= 227 * 1024 && sizeof(Task) % 16 == 0, "shared memory");

// Partial sums of one piece of a row block: its rows' words, and H, L per
// column and row.  The word of a row: columns that the sums do not certify
// (bits 0-15), exponent of alpha (from bit 16).
constexpr size_t kSlotBytes = (size_t)kRows * 4 + (size_t)2 * kKC * kRows * 8;

// kind::f16, D f32, A and B binary16, both K-major, M = 128, N = n.
__device__ __forceinline__ constexpr uint32_t idesc_n(int n) {
    return (1u << 4) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(kHalf >> 4) << 24);
}

struct FParams {
    ColumnClasses a;            // map[0], or with column classes both
    int64_t m, n;
    int rows;                   // rows per row block
    int k;
    const double *A;            // element (row, j) at A[row rs + j cs]
    int64_t rs, cs;
    const double *B;
    int64_t ldb;
    const unsigned char *bdig;  // [stage][kBStage]
    int *bexp;                  // [16] exponent field of beta_c (kZeroCol, or 2047: not finite), then kFailCount
    const float *brel;          // [inner index][16] |b| / beta, cut (zero where bexp is not a scale)
    double *C;
    int64_t ldc;
    unsigned char *slots;       // 2 per block: a piece that starts inside a row block, one that starts with it
    // Strips of 32 rows that hold outputs which are not certified.
    uint32_t *fail_words;       // [row] words of the rows of whole row blocks
    int *fail_listed;           // [strip] set by the first piece that lists it
    int *fail_arrived;          // [strip][half of the columns] parts of its sums done
    int *fail_list;
    double *fail_sums;          // [kSettleUnits][kSettleHalf][32]
    bool here;                  // whole row blocks are settled by the drainers (n <= kShort)
    unsigned *status;
    int64_t wait_ns;
    int64_t upr;                // stages per row block
    int64_t ngroups;            // stages in total
    bool merge;                 // the last stage of a row block is no piece of its own (cut_at)
    unsigned long long *trace;  // optional: 4 words per block (start, first data, end, stages)
    int w24, w16, w8, w0;       // 2^24, 2^16, 2^8, 1: opaque, so that they stay multipliers
};

// (Debug builds: see common.cuh.)
__device__ __forceinline__ bool dbg_output(const FParams &p, int64_t row, int c) {
    return dbg_in_bounds(row >= 0 && row < p.m && c >= 0 && c < p.k, p.status);
}
__device__ __forceinline__ bool dbg_strip(const FParams &p, int64_t strip) {
    return dbg_in_bounds(strip >= 0 && strip < p.ngroups / p.upr * (kRows / 32), p.status);
}

// First stage of block g of G.  A last stage of fewer than eight inner indices
// goes with the one before (merge): too few products to certify, it would have
// its rows settled (40000 x 100 x 8: 54 us with, 67 without).
__host__ __device__ __forceinline__ int64_t cut_at(const FParams &p, int64_t g, int64_t G) {
    const int64_t c = g * p.ngroups / G;
    return p.merge && (uint32_t)c % (uint32_t)p.upr == (uint32_t)p.upr - 1u ? c + 1 : c;
}
// The same, its second division out of line: in it, the product kernel takes 789
// us for 20480^2 x 16 instead of 779.
__device__ __noinline__ int64_t behind_short(int64_t c, uint32_t upr) { return (uint32_t)c % upr == upr - 1u ? c + 1 : c; }
// The block that stage x is of.
__device__ __forceinline__ int64_t owner_f(const FParams &p, int64_t x, int64_t G) {
    const int64_t g = ((x + 1) * G + p.ngroups - 1) / p.ngroups - 1;
    return p.merge && cut_at(p, g, G) > x ? g - 1 : g;
}

__device__ __forceinline__ constexpr uint32_t limit_of(int e) { return (uint32_t)e << 20 | 0xfffffu; }

// max(|a|, |b|, |c|) of the high words of binary64 numbers, compared as
// binary32 (the same order; NaN patterns, magnitudes of 2^1017 and more, give
// a NaN, which as an integer is above every scale).
__device__ __forceinline__ float max_abs3(uint32_t a, uint32_t b, float c) {
    float d;
    asm("max.NaN.f32 %0, %1, %2, %3;"
        : "=f"(d)
        : "f"(fabsf(__uint_as_float(a))), "f"(fabsf(__uint_as_float(b))), "f"(c));
    return d;
}

// |x| / 2^(e - 1023) for the high word of a binary64 |x| < 2^(e - 1022), cut
// to 21 bits.
__device__ __forceinline__ float relative(uint32_t hi, int e) {
    const int x = exp_field(hi) - e + 127;
    return x <= 0 ? 0.f : __int_as_float(x << 23 | (int)((hi & 0xfffffu) << 3));
}

// ---- digits of B ------------------------------------------------------------
//
// One cluster of blocks per column, each with a part of it: the column's
// largest exponent, then its part of G in the layout of the MMA B operand
// (K-major, no swizzle: 8 x 16-byte core matrices): [8 inner indices][N group
// of 8][4 inner indices][8 columns][4 inner indices][digit v - 2, digit v], N
// group 2 v + c / 8.  Columns k..15 are zeros.  Bound by latency (n x 16
// numbers); eight blocks per column instead of one took it from 22 to 5 us at
// n = 10240, and the product kernel starts beside it.
constexpr int kDigitBlocks = 8;
__global__ void __cluster_dims__(kDigitBlocks, 1, 1) __launch_bounds__(256)
f64_digits_kernel(int64_t n, int k, const double *__restrict__ B, int64_t ldb, unsigned char *out, int *bexp,
                  float *brel, int64_t nsteps, int *zero, int64_t nzero) {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    __shared__ int part[2];  // largest exponent, any nonzero: of this block
    namespace cg = cooperative_groups;
    cg::cluster_group cluster = cg::this_cluster();
    const int c = blockIdx.y;
    const double *col = B + (int64_t)c * ldb;
    const int tid = blockIdx.x * blockDim.x + threadIdx.x, nthreads = kDigitBlocks * blockDim.x;
    for (int64_t i = c * nthreads + tid; i < nzero; i += kKC * nthreads) zero[i] = 0;
    if (threadIdx.x < 2) part[threadIdx.x] = 0;
    __syncthreads();
    // Four inner indices at a time; the first four stay in registers.
    auto quad = [&](int64_t q, double (&v)[4]) {
#pragma unroll
        for (int e = 0; e < 4; ++e) v[e] = (c < k && q * 4 + e < n) ? __ldg(col + q * 4 + e) : 0.0;
    };
    double keep[4];
    quad(tid, keep);
    int emax = 0, any = 0;
    for (int64_t q = tid; q * 4 < n && c < k; q += nthreads) {
        double v[4];
        if (q == tid) {
#pragma unroll
            for (int e = 0; e < 4; ++e) v[e] = keep[e];
        } else {
            quad(q, v);
        }
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const long long x = __double_as_longlong(v[e]) & 0x7fffffffffffffffll;
            emax = max(emax, (int)(x >> 52));
            any |= x != 0;
        }
    }
    emax = __reduce_max_sync(0xffffffffu, emax);
    any = __any_sync(0xffffffffu, any);
    if ((threadIdx.x & 31) == 0) {
        atomicMax(&part[0], emax);
        atomicOr(&part[1], any);
    }
    cluster.sync();
    emax = kMinExp;
    any = 0;
#pragma unroll
    for (int b = 0; b < kDigitBlocks; ++b) {
        const int *other = cluster.map_shared_rank(part, b);
        emax = max(emax, other[0]);
        any |= other[1];
    }
    cluster.barrier_arrive();  // (waited for at the end: no block leaves while others read its part)
    if (tid == 0) bexp[c] = any ? emax : kZeroCol;
    if (tid == 0 && c == 0) bexp[kFailCount] = 0;
    const uint32_t key = scale_key(emax);
    unsigned char *dst = out + (c >> 3) * 256 + (c & 7) * 16;
    for (int64_t q = tid; q < 4 * nsteps; q += nthreads) {
        if (q != tid) quad(q, keep);
        uint64_t x[4];
        bool neg[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const double b = keep[e];
            const uint32_t hi = (uint32_t)__double2hiint(b);
            x[e] = fixed_point(hi, (uint32_t)__double2loint(b), key) + 0x8080808080808080ull;
            neg[e] = hi >> 31;
            brel[(q * 4 + e) * kKC + c] = emax < 2047 ? relative(hi, emax) : 0.f;
        }
        unsigned char *o = dst + (q >> 1) * kG + (q & 1) * 128;
#pragma unroll
        for (int v = 0; v < kDig; ++v) {
            uint32_t g[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) g[e] = digit_b(x[e], neg[e], v) << 16 | (v >= 2 ? digit_b(x[e], neg[e], v - 2) : 0u);
            *reinterpret_cast<uint4 *>(o + v * 512) = make_uint4(g[0], g[1], g[2], g[3]);
        }
    }
    cluster.barrier_wait();
}

// ---- sums -------------------------------------------------------------------

// (H 2^32 + L) >> shift (arithmetic, rounding down), shift >= 0.
__device__ __forceinline__ void shift_sum(int64_t &H, int64_t &L, int shift) {
    if (shift > 95) H = L = shift = 0;  // |H 2^32 + L| < 2^95: less than one unit is left
    while (shift > 0) {
        const int s = shift < 24 ? shift : 24;
        const int64_t h = H >> s;
        L = (L >> s) + (((H - (h << s)) << 32) >> s);
        H = h;
        shift -= s;
    }
}

// The same sum with 0 <= L < 2^32: sums of many (16384 drains, 2^20 inner
// indices, at most add 2^62 to L).
__device__ __forceinline__ void carry_sum(int64_t &H, int64_t &L) {
    H += L >> 32;
    L &= 0xffffffffll;
}

// Exponent of the unit of H 2^32 + L; false: outside the safe range.
__device__ __forceinline__ bool unit_exp(int ea, int eb, int &s) {
    s = ea + eb - 2112;
    return s >= -1000 && s <= 900;
}

// The first eight inner indices of a piece, loaded ahead: the high words of
// the lane's row, and its four of the 8 x 16 |b| / beta.
constexpr int kFirst = 8;
struct First {
    uint32_t a[kFirst];
    float4 b;
};
__device__ __forceinline__ void load_first(const FParams &p, int64_t row, int64_t j0, int64_t j1, First &f) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int u = 0; u < kFirst; ++u)
        f.a[u] = row < p.m && j0 + u < j1 && dbg_in_bounds(row >= 0 && j0 >= 0 && j0 + u < p.n, p.status)
                     ? __ldg(reinterpret_cast<const uint32_t *>(p.A + row * p.rs + (j0 + u) * p.cs) + 1) : 0u;
    f.b = j0 < j1 && dbg_in_bounds(j0 >= 0 && j0 + kFirst <= p.upr * kStep, p.status) ? __ldcg(reinterpret_cast<const float4 *>(p.brel + j0 * kKC) + lane) : make_float4(0.f, 0.f, 0.f, 0.f);
}

// Columns c (bits) for which sum_j |a_j||b_jc| over inner indices [j0, j1) of
// the lane's row is large enough (see above): the terms are added, eight inner
// indices at a time, until every lane of the warp has all its columns or the
// limit is reached (what is left then is f64_combine_kernel's: the
// pipeline stands still here).  eb:
// bexp[lane % 16]; buf: 512 bytes of the warp, so that a round loads each
// |b| / beta once (16 broadcast loads from L2 for each inner index took 2 us).
__device__ __forceinline__ uint32_t certify(const FParams &p, bool active, int64_t row, int64_t j0, int64_t j1, int E,
                                            int eb, float dense_sum, First &first, float4 *buf) {
    const int lane = threadIdx.x & 31;
    float S[kKC];
    uint32_t sure = 0, dense = 0xffffu;
#pragma unroll
    for (int c = 0; c < kKC; ++c) S[c] = 0.f;
    const uint32_t need = __ballot_sync(0xffffffffu, lane < p.k && eb != kZeroCol && eb < 2047);
    const int64_t end = min(j1, j0 + kScan);
    for (int64_t j = j0; j < end && __any_sync(0xffffffffu, active && (need & ~sure) != 0); j += kFirst) {
        if (j > j0) load_first(p, row, j, j1, first);
        __syncwarp();
        buf[lane] = first.b;
        __syncwarp();
#pragma unroll
        for (int u = 0; u < kFirst; ++u) {
            const float a = relative(first.a[u], E);
            if (j == j0 && first.a[u] << 1 == 0) dense = 0;
#pragma unroll
            for (int q = 0; q < kKC / 4; ++q) {
                const float4 x = buf[u * (kKC / 4) + q];
                S[4 * q] += a * x.x;
                S[4 * q + 1] += a * x.y;
                S[4 * q + 2] += a * x.z;
                S[4 * q + 3] += a * x.w;
            }
        }
#pragma unroll
        for (int c = 0; c < kKC; ++c) sure |= (uint32_t)(S[c] >= kCertify) << c;
        if (!__any_sync(0xffffffffu, active && (need & ~sure) != 0)) break;
        if (j == j0) {
            // The columns whose first eight elements are not zero: a lane
            // looks at four of one column.
            bool all = true;
#pragma unroll
            for (int u = 0; u < kFirst / 2; ++u)
                all = all && reinterpret_cast<const float *>(buf)[((lane >> 4) * (kFirst / 2) + u) * kKC + (lane & 15)] > 0.f;
            const uint32_t cols = __ballot_sync(0xffffffffu, all);
            dense &= cols & (cols >> 16);
        }
#pragma unroll
        for (int c = 0; c < kKC; ++c) sure |= (uint32_t)(S[c] >= dense_sum) << c & dense;
    }
    return sure;
}

// Short rows (all of the inner dimension, kShort at most) settled where they are:
// a kernel behind this one costs 2.5 us, of 16.5 for 15360 x 64 x 8, and with
// parts this short is slower (2^20 x 64 x 16 with 10% of A not zero 3550 us, here
// 3190).  Many rows of the warp: every lane its own; few: one after the other,
// the inner indices across the lanes.
__device__ __forceinline__ void settle_short(const FParams &p, int64_t row, uint32_t mask) {
    const int lane = threadIdx.x & 31;
    __syncwarp();  // (C holds the sums of the lanes' rows: another lane may write over them)
    uint32_t rows = __ballot_sync(0xffffffffu, mask != 0);
    if (__popc(rows) >= 8) {
        double acc[kKC] = {};
#pragma unroll 2
        for (int64_t j = 0; j < p.n; ++j) {
            const double a = mask ? __ldg(p.A + row * p.rs + j * p.cs) : 0.0;
#pragma unroll
            for (int c = 0; c < kKC; ++c)
                if (c < p.k) acc[c] = fma(a, __ldg(p.B + j + c * p.ldb), acc[c]);
        }
#pragma unroll
        for (int c = 0; c < kKC; ++c)
            if (mask >> c & 1u && dbg_output(p, row, c)) p.C[row + c * p.ldc] = acc[c];
        return;
    }
    for (; rows; rows &= rows - 1) {
        const int l = __ffs(rows) - 1;
        const int64_t r = __shfl_sync(0xffffffffu, row, l);
        const uint32_t bits = __shfl_sync(0xffffffffu, mask, l);
        double x[kShort / 32];
#pragma unroll
        for (int v = 0; v < kShort / 32; ++v)
            x[v] = lane + 32 * v < p.n ? __ldg(p.A + r * p.rs + (lane + 32 * v) * p.cs) : 0.0;
#pragma unroll 4
        for (int c = 0; c < p.k; ++c) {
            double s = 0.0;
#pragma unroll
            for (int v = 0; v < kShort / 32; ++v)
                if (lane + 32 * v < p.n) s = fma(x[v], __ldg(p.B + lane + 32 * v + c * p.ldb), s);
#pragma unroll
            for (int o = 16; o >= 1; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
            if (lane == 0 && bits >> c & 1u && dbg_output(p, r, c)) p.C[r + c * p.ldc] = s;
        }
    }
}

// The end of a piece of a row block: stores C, or leaves the sums in the
// workspace for f64_combine_kernel, and lists its strips of 32 rows that have
// outputs which are not certified.
__device__ __forceinline__ void finish(const FParams &p, const int64_t (&H)[kKC], const int64_t (&L)[kKC], int E, bool zero,
                                       int rb, int r, bool whole, int kc0, int kc1, int64_t g, int eb, First &first,
                                       float4 *buf) {
    const int64_t row = (int64_t)rb * p.rows + r;
    const bool live = r < p.rows && row < p.m;
    const int64_t j0 = (int64_t)kc0 * kStep, j1 = min((int64_t)kc1 * kStep, p.n);
    // The sums first, certified or not: their registers are free for the rest.
    unsigned char *slot = p.slots + (size_t)(2 * g + (kc0 == 0 ? 1 : 0)) * kSlotBytes;
    long long *sh = reinterpret_cast<long long *>(slot + kRows * 4) + r;
#pragma unroll
    for (int c = 0; c < kKC; ++c) {
        const int e = __shfl_sync(0xffffffffu, eb, c);
        if (!live || c >= p.k || !dbg_output(p, row, c) || !dbg_in_bounds(g >= 0 && g < gridDim.x && r < kRows, p.status)) continue;
        if (whole) {
            int ue;
            unit_exp(E, e, ue);
            p.C[row + (int64_t)c * p.ldc] = to_double(H[c], L[c], ue);
        } else {
            __stcg(sh + c * kRows, (long long)H[c]);
            __stcg(sh + (kKC + c) * kRows, (long long)L[c]);
        }
    }
    const float dense_sum = whole ? kCertifyDense : kCertifyDense * (float)(j1 - j0) / (float)p.n;
    const uint32_t sure = certify(p, live && E < 2047 && E > kMinExp, row, j0, j1, E, eb, dense_sum, first, buf);
    uint32_t mask = 0;
#pragma unroll
    for (int c = 0; c < kKC; ++c) {
        const int e = __shfl_sync(0xffffffffu, eb, c);
        int ue;
        const bool range = unit_exp(E, e, ue);
        const bool ok = E < 2047 && e < 2047 && (e == kZeroCol || zero || ((sure >> c) & 1u && range));
        if (live && c < p.k && !ok) mask |= 1u << c;
    }
    if (live && !whole && dbg_in_bounds(g >= 0 && g < gridDim.x && r < kRows, p.status))
        __stcg(reinterpret_cast<uint32_t *>(slot) + r, mask | (uint32_t)E << 16);
    if (p.here && whole) {
        if (__any_sync(0xffffffffu, mask != 0)) settle_short(p, row, mask);
    } else if (__any_sync(0xffffffffu, mask != 0)) {
        const int strip = rb * (kRows / 32) + r / 32;
        if (whole && dbg_strip(p, strip)) __stcg(p.fail_words + (int64_t)rb * kRows + r, mask);
        if (r % 32 == 0 && dbg_strip(p, strip) && atomicExch(p.fail_listed + strip, 1) == 0) {
            const int at = atomicAdd(p.bexp + kFailCount, 1);
            if (dbg_strip(p, at)) __stcg(p.fail_list + at, strip);
        }
    }
}

// ---- behind the product kernel -------------------------------------------------

// The blocks of row block rb, and its pieces' slots (the first piece starts with
// the row block, the others inside it).
struct Pieces {
    int64_t gA, gB;
    __device__ __forceinline__ Pieces(const FParams &p, int64_t rb, int64_t G)
        : gA(owner_f(p, rb * p.upr, G)), gB(owner_f(p, rb * p.upr + p.upr - 1, G)) {}
    __device__ __forceinline__ int count() const { return (int)(gB - gA) + 1; }
    __device__ __forceinline__ unsigned char *slot(const FParams &p, int i) const {
        return p.slots + (size_t)(2 * (gA + i) + (i == 0 ? 1 : 0)) * kSlotBytes;
    }
    __device__ __forceinline__ uint32_t word(const FParams &p, int i, int r) const {
        return __ldcg(reinterpret_cast<const uint32_t *>(slot(p, i)) + r);
    }
};

// The pieces of 32 rows of four columns of a row block that is cut, added in
// block order, as integers at their largest scale (exact unless a scale
// changed); a warp takes every eighth piece.
struct Combine {
    uint32_t words[kSettleWarps][32];
    long long h[kSettleWarps][kSettleCols][32], l[kSettleWarps][kSettleCols][32];
};
__device__ __forceinline__ void combine(const FParams &p, Combine &sh, int64_t G, int by_cut, int block) {
    const int strip = block % (kRows / 32), z = block / (kRows / 32);
    const int groups = (p.k + kSettleCols - 1) / kSettleCols, c0 = z % groups * kSettleCols;
    int64_t rb = z / groups;
    if (by_cut) {
        // Few cuts: the row block that cut rb + 1 is in, if that is its first.
        const int64_t first = cut_at(p, rb, G), cut = cut_at(p, rb + 1, G);
        rb = cut / p.upr;
        if (cut == rb * p.upr || first > rb * p.upr) return;
    }
    const Pieces pieces(p, rb, G);
    const int P = pieces.count();
    if (P == 1 || !dbg_in_bounds(pieces.gA >= 0 && pieces.gB < G && rb < p.ngroups / p.upr, p.status)) return;
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31, r = strip * 32 + lane;
    const int64_t row = rb * p.rows + r;
    const bool live = r < p.rows && row < p.m;
    // The sums of the first two are on their way before the scale is known.
    constexpr int kEarly = 2;
    long long h0[kEarly][kSettleCols], l0[kEarly][kSettleCols];
    uint32_t x0[kEarly];
    auto load = [&](int i, long long (&h)[kSettleCols], long long (&l)[kSettleCols]) {
        const long long *at = reinterpret_cast<const long long *>(pieces.slot(p, i) + kRows * 4) + (size_t)c0 * kRows + r;
#pragma unroll
        for (int c = 0; c < kSettleCols; ++c) {
            const bool in = live && i < P && c0 + c < p.k;
            h[c] = in ? __ldcg(at + c * kRows) : 0;
            l[c] = in ? __ldcg(at + (kKC + c) * kRows) : 0;
        }
    };
    int em = 0;
    uint32_t mask = 0;
#pragma unroll
    for (int q = 0; q < kEarly; ++q) x0[q] = live && w + q * kSettleWarps < P ? pieces.word(p, w + q * kSettleWarps, r) : 0u;
#pragma unroll
    for (int q = 0; q < kEarly; ++q)
        if (q * kSettleWarps < P) load(w + q * kSettleWarps, h0[q], l0[q]);
#pragma unroll
    for (int q = 0; q < kEarly; ++q) {
        em = max(em, (int)(x0[q] >> 16));
        mask |= x0[q] & 0xffffu;
    }
    for (int i = w + kEarly * kSettleWarps; i < P; i += kSettleWarps) {
        const uint32_t x = live ? pieces.word(p, i, r) : 0u;
        em = max(em, (int)(x >> 16));
        mask |= x & 0xffffu;
    }
    sh.words[w][lane] = mask | (uint32_t)em << 16;
    __syncthreads();
    em = 0;
    mask = 0;
#pragma unroll
    for (int v = 0; v < kSettleWarps; ++v) {
        em = max(em, (int)(sh.words[v][lane] >> 16));
        mask |= sh.words[v][lane] & 0xffffu;
    }
    int64_t hs[kSettleCols] = {}, ls[kSettleCols] = {};
    auto add = [&](int e, const long long (&h)[kSettleCols], const long long (&l)[kSettleCols]) {
#pragma unroll
        for (int c = 0; c < kSettleCols; ++c) {
            int64_t x = h[c], y = l[c];
            shift_sum(x, y, em - e);
            carry_sum(x, y);
            hs[c] += x;
            ls[c] += y;
        }
    };
#pragma unroll
    for (int q = 0; q < kEarly; ++q)
        if (q * kSettleWarps < P) add((int)(x0[q] >> 16), h0[q], l0[q]);
#pragma unroll 1
    for (int i = w + kEarly * kSettleWarps; i < P; i += kSettleWarps) {
        const int e = live ? (int)(pieces.word(p, i, r) >> 16) : 0;
        load(i, h0[0], l0[0]);
        add(e, h0[0], l0[0]);
    }
#pragma unroll
    for (int c = 0; c < kSettleCols; ++c) {
        sh.h[w][c][lane] = (long long)hs[c];
        sh.l[w][c][lane] = (long long)ls[c];
    }
    __syncthreads();
    if (w >= kSettleCols || !live || c0 + w >= p.k || (mask >> (c0 + w) & 1u) || !dbg_output(p, row, c0 + w)) return;
    int64_t h = 0, l = 0;
#pragma unroll
    for (int v = 0; v < kSettleWarps; ++v) {
        h += sh.h[v][w][lane];
        l += sh.l[v][w][lane];
    }
    int ue;
    const bool in = unit_exp(em, __ldcg(p.bexp + c0 + w), ue);
    p.C[row + (int64_t)(c0 + w) * p.ldc] = (h | l) == 0 || !in ? 0.0 : to_double(h, l, ue);
}

// Outputs that are not certified, by binary64 FMAs, without those of a zero
// where B is finite.  The strips listed are cut into parts of their inner
// dimension, as many as keep all blocks busy; the last block done with a strip
// adds its parts in order.  A block takes eight columns of a part; its warps
// share the inner indices, eight at a time, their lanes the rows (consecutive
// in memory), or with an A read by rows the other way round.
//
// The FP64 units bound it where all outputs are listed (about the time of the
// FMA kernels, on top of the product kernel's), the reading of A where A is
// mostly zeros.  Measured (GB300, us; FMA kernels / by the product kernel's
// drainers / here): 4096^2 x 16 dense 457 / 61 / 61, banded 457 / 880 / 228,
// identity 457 / 912 / 224, 1% not zero 457 / 1105 / 435, large diagonal 457 /
// 743 / 732; x 4 dense 122 / 60 / 59, banded 122 / 600 / 180, large diagonal 122 /
// 647 / 292; 20480^2 x 16 dense 10754 / 785 / 785, banded 10754 / 21547 / 3310.
struct SettleShared {
    double d[kSettleWarps][kSettleHalf][32];
    double b[kSettleWarps][8][kSettleHalf];  // of the warp's eight inner indices
    int last;
};
// (In integers: a comparison of binary64 numbers is the FP64 units' work.)
__device__ __forceinline__ bool nonzero(double x) { return __double_as_longlong(x) << 1 != 0; }
// acc += x b.  Instantiated for the columns there are: FMAs behind a test of
// their number are done all the same and dropped.
template <int N>
__device__ __forceinline__ void fma_columns(double (&acc)[kSettleHalf], double x, const double (&b)[kSettleHalf]) {
#pragma unroll
    for (int c = 0; c < N; ++c) acc[c] = fma(x, b[c], acc[c]);
}
// Inner indices j0 .. j1 - 1 of up to N columns from B on, into sh.d.  Row
// `lane` of the strip starts at a (null: none), its elements cs apart.
template <int N>
__device__ __forceinline__ void settle_rows(const FParams &p, SettleShared &sh, const double *a, const double *B, int cols,
                                            int64_t j0, int64_t j1, bool special) {
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    double acc[kSettleHalf] = {};
    const int bc = lane >> 2, bj = (lane & 3) * 2;
    const double *b = B + (int64_t)(bc < cols ? bc : 0) * p.ldb + bj;
    double (*tile)[kSettleHalf] = sh.b[w];
    for (int64_t j = j0 + w * 8; j < j1; j += kSettleWarps * 8) {
        double x[8];
        const double b0 = j + bj < j1 ? __ldg(b + j) : 0.0, b1 = j + bj + 1 < j1 ? __ldg(b + j + 1) : 0.0;
#pragma unroll
        for (int v = 0; v < 8; ++v) x[v] = a && j + v < j1 ? __ldg(a + (j + v) * p.cs) : 0.0;
        __syncwarp();
        tile[bj][bc] = b0;
        tile[bj + 1][bc] = b1;
        __syncwarp();
#pragma unroll
        for (int v = 0; v < 8; ++v)
            if (special || __any_sync(0xffffffffu, nonzero(x[v]))) fma_columns<N>(acc, x[v], tile[v]);
    }
#pragma unroll
    for (int c = 0; c < kSettleHalf; ++c) sh.d[w][c][lane] = acc[c];
}
// The same with the inner indices across the lanes: rows `rows` from a on, rs apart.
template <int N>
__device__ __forceinline__ void settle_lines(const FParams &p, SettleShared &sh, const double *A, uint32_t rows, const double *B,
                                             int cols, int64_t j0, int64_t j1, bool special) {
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
#pragma unroll
    for (int c = 0; c < kSettleHalf; ++c) sh.d[w][c][lane] = 0.0;
    __syncwarp();
    for (int t = w; t < 32; t += kSettleWarps) {
        if (!(rows >> t & 1u)) continue;
        double acc[kSettleHalf] = {};
        const double *a = A + t * p.rs;
        for (int64_t j = j0 + lane; j - lane < j1; j += 4 * 32) {
            double x[4];
#pragma unroll
            for (int v = 0; v < 4; ++v) x[v] = j + v * 32 < j1 ? __ldg(a + (j + v * 32) * p.cs) : 0.0;
#pragma unroll
            for (int v = 0; v < 4; ++v) {
                if (!special && !__any_sync(0xffffffffu, nonzero(x[v]))) continue;
                const double *from = B + (j + v * 32 < j1 ? j + v * 32 : 0);
                double b[kSettleHalf];
#pragma unroll
                for (int c = 0; c < N; ++c) b[c] = __ldg(from + (c < cols ? c : 0) * p.ldb);
                if (j + v * 32 < j1) fma_columns<N>(acc, x[v], b);
            }
        }
#pragma unroll
        for (int c = 0; c < N; ++c) {
#pragma unroll
            for (int o = 16; o >= 1; o >>= 1) acc[c] += __shfl_xor_sync(0xffffffffu, acc[c], o);
            if (lane == 0) sh.d[w][c][t] = acc[c];
        }
    }
}
__device__ __forceinline__ void settle(const FParams &p, SettleShared &sh, int64_t G, int block, int blocks) {
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t count = __ldcg(p.bexp + kFailCount);
    const int eb = __ldcg(p.bexp + (lane & 15));
    if (count == 0) return;
    const int halves = (p.k + kSettleHalf - 1) / kSettleHalf;
    // Parts: as short as 64 inner indices for few strips, else what ends soonest
    // (a part costs about as much again as 64 inner indices).
    const int64_t sets = count * halves, most = (p.n + 63) / 64;
    int64_t parts = min(most, blocks / sets);
    if (parts < 32) {
        const uint32_t x = lane + 1, total = (uint32_t)sets * x;
        const bool can = x == 1 || (total <= kSettleUnits && x <= most);
        const uint32_t cost = can ? (total + blocks - 1) / blocks * ((uint32_t)p.n / x + 64) : ~0u;
        parts = __ffs(__ballot_sync(0xffffffffu, cost == __reduce_min_sync(0xffffffffu, cost)));
    }
    const int64_t len = ((p.n + parts - 1) / parts + 63) / 64 * 64;
    parts = (p.n + len - 1) / len;
    const bool special = __any_sync(0xffffffffu, lane < p.k && eb == 2047);
    const int64_t units = sets * parts;
    auto strip_of = [&](int64_t u) { return u < units ? __ldcg(p.fail_list + u / parts / halves) : 0; };
    int next = strip_of(block);
    for (int64_t u = block; u < units; u += blocks) {
        const int64_t at = u / parts, part = u - at * parts;
        const int half = (int)(at % halves), strip = next;
        next = strip_of(u + blocks);
        if (!dbg_strip(p, strip) || !dbg_in_bounds(parts == 1 || (u >= 0 && u < kSettleUnits), p.status)) break;
        const int c0 = half * kSettleHalf, cols = min(kSettleHalf, p.k - c0);
        const int64_t rb = strip / (kRows / 32), row0 = rb * p.rows + strip % (kRows / 32) * 32;
        const int r = strip % (kRows / 32) * 32 + lane;
        // The outputs to settle of row `lane`.
        const Pieces pieces(p, rb, G);
        const bool live = r < p.rows && row0 + lane < p.m;
        const uint32_t alone = live && pieces.count() == 1 ? __ldcg(p.fail_words + rb * kRows + r) : 0u;
        auto wanted = [&]() {
            uint32_t mask = alone;
            if (live && pieces.count() > 1) {
#pragma unroll 8
                for (int i = 0; i < pieces.count(); ++i) mask |= pieces.word(p, i, r);
            }
            return mask >> c0 & 0xffu;
        };
        const int64_t j0 = part * len, j1 = min(p.n, j0 + len);
        // (Columns beyond the last one read the first.)
        const double *B = p.B + (int64_t)c0 * p.ldb;
        if (p.rs == 1) {
            const double *a = row0 + lane < p.m ? p.A + row0 + lane : nullptr;
            if (cols <= 2) settle_rows<2>(p, sh, a, B, cols, j0, j1, special);
            else if (cols <= 4) settle_rows<4>(p, sh, a, B, cols, j0, j1, special);
            else settle_rows<8>(p, sh, a, B, cols, j0, j1, special);
        } else {
            const double *A = p.A + row0 * p.rs;
            const uint32_t rows = __ballot_sync(0xffffffffu, wanted() != 0);
            if (cols <= 2) settle_lines<2>(p, sh, A, rows, B, cols, j0, j1, special);
            else if (cols <= 4) settle_lines<4>(p, sh, A, rows, B, cols, j0, j1, special);
            else settle_lines<8>(p, sh, A, rows, B, cols, j0, j1, special);
        }
        __syncthreads();
        // Thread: column w of row `lane`.
        double out = 0.0;
#pragma unroll
        for (int v = 0; v < kSettleWarps; ++v) out += sh.d[v][w][lane];
        bool store = true;
        if (parts > 1) {
            if (dbg_in_bounds(u < kSettleUnits, p.status)) __stcg(p.fail_sums + (u * kSettleHalf + w) * 32 + lane, out);
            __threadfence();
            __syncthreads();
            if (threadIdx.x == 0) sh.last = atomicAdd(p.fail_arrived + strip * 2 + half, 1) == parts - 1;
            __syncthreads();
            store = sh.last;
            if (store) {
                __threadfence();
                out = 0.0;
                const double *from = p.fail_sums + ((u - part) * kSettleHalf + w) * 32 + lane;
#pragma unroll 16
                for (int i = 0; i < (int)parts; ++i) out += __ldcg(from + i * kSettleHalf * 32);
            }
        }
        if (store && (wanted() >> w & 1u) && dbg_output(p, row0 + lane, c0 + w)) p.C[row0 + lane + (int64_t)(c0 + w) * p.ldc] = out;
        __syncthreads();
    }
}

// One launch for both, started beside the product kernel (griddepcontrol).
// (Added by the product kernel's last warp to arrive, pieces took 18 us of a
// 1024^2 product and 21 us of a 4096^2 one, few warps waiting for one another's
// loads in two levels; here 3 to 5 us.  The outputs that are not certified were
// the product kernel's drainers' work, eight warps that held up their pipeline
// and could make its bounded waits run out.)
__global__ void __launch_bounds__(32 * kSettleWarps, kSettlePerSM) f64_combine_kernel(const __grid_constant__ FParams p,
                                                                                   int64_t G, int by_cut, int add) {
    __shared__ union { Combine combine; SettleShared settle; } sh;
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if ((int)blockIdx.x < add) combine(p, sh.combine, G, by_cut, blockIdx.x);
    else settle(p, sh.settle, G, blockIdx.x - add, gridDim.x - add);
}

template <F64TCMode MODE>
__global__ void __launch_bounds__(kThreads, 1) f64tc_kernel(const __grid_constant__ FParams p) {
    constexpr bool SPLIT = MODE == F64TCMode::Split;
    extern __shared__ unsigned char smem_raw[];
    unsigned char *smem = smem_aligned<1024>(smem_raw);
    uint64_t *full = reinterpret_cast<uint64_t *>(smem + kRingBytes);        // [kARing] A landed
    uint64_t *empty = full + kARing;                                         // [kARing] read by the converters
    uint64_t *bfull = empty + kARing;                                        // [kBRing] B landed
    uint64_t *bempty = bfull + kBRing;                                       // [kBRing] MMAs of both halves done
    uint64_t *afull = bempty + kBRing;                                       // [2 wg + buffer] operand in TMEM
    uint64_t *adone = afull + 4;                                             // [2 wg + buffer] its MMAs done
    uint64_t *dfree = adone + 4;                                             // [wg] accumulators drained
    uint64_t *posted = dfree + 2;                                            // [8] task posted
    uint64_t *taken = posted + 8;                                            // [8] task done
    uint64_t *fin = taken + 8;                                               // [wg] all MMAs done
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(fin + 2);
    volatile int *flags = reinterpret_cast<volatile int *>(tmem_slot + 2);   // [0] abort
    volatile int *accum = flags + 2;                                         // [2 wg + buffer] its MMAs accumulate
    volatile Task *tasks = reinterpret_cast<volatile Task *>(smem + kRingBytes + kTail);
    float4 *firsts = reinterpret_cast<float4 *>(smem + kRingBytes + kTail + 8 * sizeof(Task));  // [8][32]

    const int warp = threadIdx.x >> 5;
    const int lane = threadIdx.x & 31;
    const int64_t G = gridDim.x, g = blockIdx.x;
    int64_t u_begin = g * p.ngroups / G, u_end = (g + 1) * p.ngroups / G;  // cut_at
    if (p.merge) {
        u_begin = behind_short(u_begin, (uint32_t)p.upr);
        u_end = behind_short(u_end, (uint32_t)p.upr);
    }
    const int nunits = (int)(u_end - u_begin);
    const int upr = (int)p.upr;
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

    if (threadIdx.x == 0) {
        for (int s = 0; s < kARing; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 8);
        }
        for (int s = 0; s < kBRing; ++s) {
            mbar_init(&bfull[s], 1);
            mbar_init(&bempty[s], 2);
        }
        for (int w = 0; w < 4; ++w) {
            mbar_init(&afull[w], 4);
            mbar_init(&adone[w], 1);
        }
        for (int w = 0; w < 2; ++w) {
            mbar_init(&dfree[w], 4);
            mbar_init(&fin[w], 1);
        }
        for (int w = 0; w < 8; ++w) {
            mbar_init(&posted[w], 1);
            mbar_init(&taken[w], 1);
        }
        flags[0] = 0;
        if (p.trace) {
            p.trace[4 * g] = globaltimer_ns();
            p.trace[4 * g + 3] = (unsigned long long)nunits;
        }
        fence_mbar_init();
    }
    if (warp == 17) {
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

    if (warp >= 16) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kIssuerRegs));
        if (warp == 16 || warp == 19) {
            // ---------------- producers: A, B ----------------
            if (lane == 0) {
                const bool isA = warp == 16;
                const int ring = isA ? kARing : kBRing;
                uint64_t *fl = isA ? full : bfull, *em = isA ? empty : bempty;
                if (isA) prefetch_tensormap(&p.a.map[0]);
                else asm volatile("griddepcontrol.wait;" ::: "memory");  // the digits of B
                const uint64_t policy = l2_policy_evict_first();
                int s = 0;
                uint32_t ph = 0, issued = 0, last_par = 0;
                int rb = (int)(u_begin / p.upr);
                int kc = (int)(u_begin - (int64_t)rb * p.upr);
                for (int i = 0; i < nunits; ++i) {
                    if (flags[0]) break;
                    if (!mbar_wait_bounded(&em[s], ph ^ 1u, p.wait_ns, flags)) {
                        give_up();
                        break;
                    }
                    if (isA) {
                        mbar_arrive_expect_tx(&fl[s], kAStage);
                        if constexpr (SPLIT) {
#pragma unroll
                            for (int c = 0; c < kClasses; ++c)
                                tma_load_2d_hint(smem + s * kAStage + c * (kAStage / kClasses), &p.a.map[c],
                                                 rb * (kRows - kClasses), kc * (kStep / kClasses), &fl[s], policy);
                        } else if constexpr (MODE == F64TCMode::Transposed) {
                            tma_load_2d_hint(smem + s * kAStage, &p.a.map[0], kc * kStep, rb * kRows, &fl[s], policy);
                        } else {
                            tma_load_2d_hint(smem + s * kAStage, &p.a.map[0], rb * kRows, kc * kStep, &fl[s], policy);
                        }
                    } else {
                        mbar_arrive_expect_tx(&fl[s], kBStage);
                        bulk_g2s(smem + kARing * kAStage + s * kBStage, p.bdig + (size_t)kc * kBStage, kBStage, &fl[s]);
                    }
                    issued |= 1u << s;
                    last_par = (last_par & ~(1u << s)) | (ph << s);
                    if (++s == ring) { s = 0; ph ^= 1u; }
                    if (++kc == upr) { kc = 0; ++rb; }
                }
                for (int t = 0; t < ring; ++t)
                    if (issued & (1u << t)) (void)mbar_wait_bounded(&fl[t], (last_par >> t) & 1u, 4000000000LL, nullptr);
            }
        } else {
            // ---------------- MMA issuers, one for each half of the rows ----------------
            // (converged warps: elect_one)
            const int w = warp - 17;
            const uint32_t d = tmem + (uint32_t)(w * kDCols);
            int s = 0;
            uint32_t ph = 0;
            uint32_t chunks = 0;  // chunks started
            bool ok = true;
            for (int i = 0; i < nunits && ok; ++i) {
                const uint64_t bd = sdesc(smem_u32(smem + kARing * kAStage + s * kBStage), 128, 256, 0);
                const int q = 2 * w + (i & 1);
                ok = wait(&bfull[s], ph) && wait(&afull[q], (uint32_t)(i >> 1) & 1u);
                if (!ok) break;
                const uint32_t acc = (uint32_t)accum[q];
                if (!acc) {
                    // A new chunk: the drainers have read the last one.
                    if (chunks > 0) ok = wait(&dfree[w], (chunks - 1) & 1u);
                    if (!ok) break;
                    ++chunks;
                }
                tc_fence_after();
                const uint32_t a = tmem + (uint32_t)(2 * kDCols + q * kABuf);
                if (elect_one()) {
#pragma unroll
                    for (int h = 0; h < 2; ++h) {  // 8 inner indices
                        const uint64_t b = bd + h * (kG >> 4);
                        const uint32_t ah = a + h * kAHalf;
                        umma_f16_ts(d, ah, b, idesc_n(8 * kKC), h == 0 ? acc : 1u);
                        umma_f16_ts(d + 1 * kKC, ah + 8, b, idesc_n(7 * kKC), 1u);
                        umma_f16_ts(d + 4 * kKC, ah + 16, b, idesc_n(4 * kKC), 1u);
                        umma_f16_ts(d + 5 * kKC, ah + 24, b, idesc_n(3 * kKC), 1u);
                    }
                    umma_commit(&adone[q]);
                    umma_commit(&bempty[s]);
                }
                __syncwarp();
                if (++s == kBRing) { s = 0; ph ^= 1u; }
            }
            // Every MMA of this warp has completed before TMEM is freed.
            if (elect_one()) umma_commit(&fin[w]);
            (void)mbar_wait_bounded(&fin[w], 0, 4000000000LL, nullptr);
        }
    } else if (warp >= 8) {
        // ---------------- drainers ----------------
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kDrainerRegs));
        const int w = warp - 8, wg = w >> 2;
        const uint32_t tD = tmem + ((uint32_t)((w & 3) * 32) << 16) + (uint32_t)(wg * kDCols);
        const volatile Task &task = tasks[w];
        int64_t H[kKC], L[kKC];
        int E = kMinExp;
#pragma unroll
        for (int c = 0; c < kKC; ++c) H[c] = L[c] = 0;
        asm volatile("griddepcontrol.wait;" ::: "memory");  // bexp, brel
        const int eb = __ldcg(p.bexp + (lane & 15));
        for (uint32_t t = 0; nunits > 0; ++t) {
            if (!wait(&posted[w], t & 1u)) break;
            const int stage = task.stage, clear = task.clear, rb = task.rb, kc0 = task.kc0, kc1 = task.kc1;
            const bool whole = task.whole, last = task.last;
            const int e = task.exp[lane] & (kNonzero - 1);
            First first;
            if (rb >= 0) load_first(p, (int64_t)rb * p.rows + w * 32 + lane, (int64_t)kc0 * kStep,
                                    min((int64_t)kc1 * kStep, p.n), first);
            // (The MMAs complete in order.)
            if (!wait(&adone[2 * wg + (stage & 1)], (uint32_t)(stage >> 1) & 1u)) break;
            tc_fence_after();
            if (e > E) {
#pragma unroll
                for (int c = 0; c < kKC; ++c) shift_sum(H[c], L[c], e - E);
                E = e;
            }
            // Column group d: the sums of the digit pairs s + t = d.  They carry
            // 2^-24.  |sum| < 2^22 for d <= 2 (the leading digits are at most 63
            // and 64), so there the addition of 0.75 leaves the integer in the
            // low bits; the others, up to 2^24, need the conversion.
            const int mul[4] = {p.w24, p.w16, p.w8, p.w0};
            uint32_t v[48];
            auto group = [&](int d, const uint32_t *x) {
#pragma unroll
                for (int c = 0; c < kKC; ++c) {
                    const float f = __uint_as_float(x[c]);
                    const int q = d <= 2 ? __float_as_int(f + 0.75f) - 0x3f400000 : __float2int_rn(f * kUnit);
                    if (d < 4) H[c] = mad_wide(q, mul[d], H[c]);
                    else L[c] = mad_wide(q, mul[d - 4], L[c]);
                }
            };
            tmem_ld32(tD, v);
            tmem_ld16(tD + 2 * kKC, v + 32);
            tmem_ld_wait();
            group(0, v);
            group(1, v + 16);
            group(2, v + 32);
            tmem_ld32(tD + 3 * kKC, v);
            tmem_ld16(tD + 5 * kKC, v + 32);
            tmem_ld_wait();
            group(3, v);
            group(4, v + 16);
            group(5, v + 32);
            tmem_ld32(tD + 6 * kKC, v);
            tmem_ld_wait();
            // The accumulators are free.
            if (clear) {
#pragma unroll
                for (int d = 0; d < kDCols; d += 8) tmem_st8_zero(tD + d);
                tmem_st_wait();
            }
            tc_fence_before();
            __syncwarp();
            if (!clear && lane == 0) mbar_arrive(&dfree[wg]);
            group(6, v);
            group(7, v + 16);
            if ((t & 16383u) == 16383u) {
#pragma unroll
                for (int c = 0; c < kKC; ++c) carry_sum(H[c], L[c]);
            }
            if (rb >= 0) {
                finish(p, H, L, E, !(task.exp[lane] & kNonzero), rb, w * 32 + lane, whole, kc0, kc1, g, eb, first, firsts + w * 32);
#pragma unroll
                for (int c = 0; c < kKC; ++c) H[c] = L[c] = 0;
                E = kMinExp;
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(&taken[w]);
            if (last) break;
        }
    } else {
        // ---------------- converters: warps 0-3 rows 0..127, warps 4-7 rows 128..255 ----------------
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kConverterRegs));
        const int wg = warp >> 2;
        const int r = threadIdx.x;  // row within the row block
        const uint32_t tA = tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)(2 * kDCols + wg * kACols);
        volatile Task &task = tasks[warp];
        // The scale, as the largest high word that fits: exponent of alpha << 20 |
        // 0xfffff (limit_of(2047): the row holds an infinity or a NaN; 0: the row
        // of the piece is zeros so far, and with it its sums at any scale).
        uint32_t limit = 0;
        int s = 0;
        uint32_t ph = 0;
        int cnt = 0;         // stages in the accumulators
        // The halves of the row block drain in turn: the second starts with half a chunk.
        int chunk = wg == 0 ? kChunk : kChunk / 2;
        uint32_t ntask = 0;  // tasks posted
        int rb = (int)(u_begin / p.upr);
        int kc = (int)(u_begin - (int64_t)rb * p.upr);
        int kc_first = kc;

        // The MMAs of stage i (buffer i & 1) have completed.
        auto wait_done = [&](int i) {
            if (i < 0) return true;
            const bool ok = wait(&adone[2 * wg + (i & 1)], (uint32_t)(i >> 1) & 1u);
            tc_fence_after();
            return ok;
        };
        // The operand of stage i is stored: hand it to the MMA warp.
        auto hand_over = [&](int i) {
            tmem_st_wait();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&afull[2 * wg + (i & 1)]);
        };
        auto post = [&](int stage, int clear, int end_rb, int kc1, int whole, int last) {
            if (ntask > 0 && !wait(&taken[warp], (ntask - 1) & 1u)) return false;
            if (lane == 0) {
                task.stage = stage;
                task.clear = clear;
                task.rb = end_rb;
                task.kc0 = kc_first;
                task.kc1 = kc1;
                task.whole = whole;
                task.last = last;
            }
            task.exp[lane] = limit ? (int)(limit >> 20) | kNonzero : kMinExp;
            __syncwarp();
            if (lane == 0) mbar_arrive(&posted[warp]);
            ++ntask;
            return true;
        };
        // With column classes: even and odd columns, rows behind by their shifts
        // (the last threads have no row).
        const int at0 = SPLIT ? min(r + p.a.shift[0], kRows - 1) : 0, at1 = SPLIT ? min(r + p.a.shift[1], kRows - 1) : 0;
        uint32_t hi[kStep], lo[kStep];
        auto load = [&]() {
            if constexpr (MODE == F64TCMode::Transposed) {
                // Row r is a line of 128 bytes, its 16-byte pieces swizzled.
                const uint4 *line = reinterpret_cast<const uint4 *>(smem + s * kAStage + r * (kStep * 8));
#pragma unroll
                for (int j = 0; j < kStep; j += 2) {
                    const uint4 v = line[(j >> 1) ^ (r & 7)];
                    lo[j] = v.x;
                    hi[j] = v.y;
                    lo[j + 1] = v.z;
                    hi[j + 1] = v.w;
                }
                return;
            }
            const uint2 *src = reinterpret_cast<const uint2 *>(smem + s * kAStage);
#pragma unroll
            for (int j = 0; j < kStep; ++j) {
                const uint2 v = SPLIT ? src[((j & 1) * (kStep / kClasses) + (j >> 1)) * kRows + ((j & 1) ? at1 : at0)]
                                      : src[j * kRows + r];
                lo[j] = v.x;
                hi[j] = v.y;
            }
        };
        bool ok = nunits == 0 || wait(&full[s], ph);
        if (p.trace && threadIdx.x == 0) p.trace[4 * g + 1] = globaltimer_ns();
        if (ok && nunits > 0) load();
        bool pending = false;  // the operand of stage i - 1 is not handed over yet
        for (int i = 0; i < nunits && ok; ++i) {
            float mx = 0.f;
#pragma unroll
            for (int j = 0; j < kStep; j += 2) mx = max_abs3(hi[j], hi[j + 1], mx);
            // Above the limit, or (one comparison for both) zeros, which are looked
            // at here, where the elements are in registers: read again one by one
            // at the end of the piece, one row of zeros in 256 took a product of
            // 20480^2 x 16 from 784 to 6156 us.
            const uint32_t most = __float_as_uint(mx);
            if (__any_sync(0xffffffffu, most - 1u >= limit)) {
                bool grow = most > limit;
                if (limit == 0u && !grow) {
                    uint32_t low = 0;
#pragma unroll
                    for (int j = 0; j < kStep; ++j) low |= lo[j];
                    grow = low != 0u;
                }
                if (__any_sync(0xffffffffu, grow && limit != 0u)) {
                    // A row needs a larger scale: first its sums so far.
                    if (pending) hand_over(i - 1);
                    pending = false;
                    if (cnt > 0) {
                        ok = post(i - 1, 1, -1, 0, 0, 0) && wait(&taken[warp], (ntask - 1) & 1u);
                        if (!ok) break;
                    }
                }
                if (grow) {
                    int em = kMinExp - kHeadroom;
#pragma unroll
                    for (int j = 0; j < kStep; ++j) em = max(em, exp_field(hi[j]));
                    limit = em == 2047 || limit == limit_of(2047) ? limit_of(2047)
                                                                  : max(limit, limit_of(min(em + kHeadroom, 2046)));
                }
            }
            const uint32_t key = 2 * max(limit, limit_of(kMinExp)) + 1;  // scale_key
            const uint32_t ta = tA + (i & 1) * kABuf;
            const bool last = i == nunits - 1;
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                uint32_t w[8][4];
#pragma unroll
                for (int j = 0; j < 8; ++j) digits(fixed_point(hi[h * 8 + j], lo[h * 8 + j], key), hi[h * 8 + j], w[j]);
                if (h == 0) {
                    if (pending) hand_over(i - 1);
                    ok = wait_done(i - 2);
                    if (!ok) break;
                } else {
                    // The stage is read (the digits hold its values); the next
                    // one's elements are on their way while these are stored.
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&empty[s]);
                    if (++s == kARing) { s = 0; ph ^= 1u; }
                    if (!last) {
                        ok = wait(&full[s], ph);
                        if (!ok) break;
                        load();
                    }
                }
#pragma unroll
                for (int t = 0; t < 4; ++t)
                    tmem_st8(ta + h * kAHalf + t * 8, w[0][t], w[1][t], w[2][t], w[3][t], w[4][t], w[5][t], w[6][t], w[7][t]);
            }
            if (!ok) break;
            if (r == wg * kHalf) accum[2 * wg + (i & 1)] = cnt > 0;
            pending = true;
            ++cnt;
            const bool rb_end = kc == upr - 1;
            if (cnt == chunk || rb_end || last) {
                hand_over(i);
                pending = false;
                const bool end = rb_end || last;
                ok = post(i, 0, end ? rb : -1, kc + 1, kc_first == 0 && rb_end, last);
                if (!ok) break;
                cnt = 0;
                chunk = kChunk;
                if (end) {
                    limit = 0;
                    kc_first = rb_end ? 0 : kc + 1;
                }
            }
            if (++kc == upr) { kc = 0; ++rb; }
        }
    }
    // Everyone (including idle lanes) meets here before the TMEM is freed.
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (p.trace && threadIdx.x == 0) p.trace[4 * g + 2] = globaltimer_ns();
    if (warp == 17)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols) : "memory");
}

// C += X (m x k without padding).
__global__ void __launch_bounds__(256) f64_add_kernel(int64_t m, int64_t total, const double *X, double *C, int64_t ldc) {
    const int64_t t = (int64_t)blockIdx.x * 256 + threadIdx.x;
    if (t < total) C[t % m + t / m * ldc] += X[t];
}

}  // namespace

int f64tc_rows(F64TCMode mode) { return mode == F64TCMode::Split ? kRows - kClasses : kRows; }
int f64tc_step() { return kStep; }
int f64tc_kc() { return kKC; }
size_t f64tc_digit_bytes(int64_t n) {
    return 256 + (size_t)((n + kStep - 1) / kStep) * (kBStage + kStep * kKC * sizeof(float));
}
size_t f64tc_slot_bytes(int64_t grid) { return (size_t)(2 * grid) * kSlotBytes; }
size_t f64tc_fail_bytes(int64_t m, F64TCMode mode) {
    const int64_t num_rb = (m + f64tc_rows(mode) - 1) / f64tc_rows(mode);
    return (size_t)kSettleUnits * kSettleHalf * 32 * 8 + (size_t)num_rb * (kRows + 4 * (kRows / 32)) * 4;
}

template <F64TCMode MODE>
cudaError_t f64tc_set_smem() {
    static std::mutex mu;
    static uint64_t attr_done = 0;  // one bit per device
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    std::lock_guard<std::mutex> lk(mu);
    if (dev >= 64 || !(attr_done & (1ull << dev))) {
        e = cudaFuncSetAttribute(f64tc_kernel<MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmem);
        if (e != cudaSuccess) return e;
        if (dev < 64) attr_done |= 1ull << dev;
    }
    return cudaSuccess;
}

cudaError_t f64tc_launch(const F64TCLaunch &L, cudaStream_t stream) {
    using M = F64TCMode;
    cudaError_t e = L.mode == M::Split ? f64tc_set_smem<M::Split>()
                    : L.mode == M::Transposed ? f64tc_set_smem<M::Transposed>() : f64tc_set_smem<M::Plain>();
    if (e != cudaSuccess) return e;
    const int64_t nsteps = (L.g.n + kStep - 1) / kStep;
    int *bexp = static_cast<int *>(L.digits);
    unsigned char *bdig = static_cast<unsigned char *>(L.digits) + 256;
    float *brel = reinterpret_cast<float *>(bdig + nsteps * kBStage);
    const int64_t num_rb = (L.g.m + f64tc_rows(L.mode) - 1) / f64tc_rows(L.mode), strips = num_rb * (kRows / 32);
    FParams p;
    p.fail_sums = static_cast<double *>(L.fails);
    p.fail_words = reinterpret_cast<uint32_t *>(p.fail_sums + (size_t)kSettleUnits * kSettleHalf * 32);
    p.fail_listed = reinterpret_cast<int *>(p.fail_words + num_rb * kRows);
    p.fail_arrived = p.fail_listed + strips;
    p.fail_list = p.fail_arrived + 2 * strips;
    f64_digits_kernel<<<dim3(kDigitBlocks, kKC), 256, 0, stream>>>(L.g.n, L.g.k, static_cast<const double *>(L.g.B),
                                                                   L.g.ldb, bdig, bexp, brel, nsteps, p.fail_listed,
                                                                   3 * strips);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    p.a = L.a;
    p.rows = f64tc_rows(L.mode);
    p.m = L.g.m;
    p.n = L.g.n;
    p.k = L.g.k;
    p.A = static_cast<const double *>(L.g.A);
    p.rs = L.mode == M::Transposed ? L.g.lda : 1;
    p.cs = L.mode == M::Transposed ? 1 : L.g.lda;
    p.B = static_cast<const double *>(L.g.B);
    p.ldb = L.g.ldb;
    p.bdig = bdig;
    p.bexp = bexp;
    p.brel = brel;
    p.C = static_cast<double *>(L.g.C);
    p.ldc = L.g.ldc;
    p.slots = static_cast<unsigned char *>(L.slots);
    p.status = L.status;
    // (The waits for B include the digits kernel, about 0.5 ns an inner index.  A
    // griddepcontrol.wait before them cost the product 1.4%.)
    p.wait_ns = L.wait_ns > 0 ? L.wait_ns + 16 * L.g.n : L.wait_ns;
    p.upr = nsteps;
    p.ngroups = num_rb * nsteps;
    p.merge = nsteps > 1 && L.g.n % kStep != 0 && L.g.n % kStep < kFirst;
    p.trace = L.trace;
    p.w24 = 1 << 24;
    p.w16 = 1 << 16;
    p.w8 = 1 << 8;
    p.w0 = 1;
    bool cut = false;
    for (int64_t c = 1; c < L.grid; ++c) cut |= cut_at(p, c, L.grid) % p.upr != 0;
    p.here = L.g.n <= kShort;
    // The product starts beside the digits kernel (griddepcontrol): its first
    // stages of A are on their way when the digits are done.
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)L.grid);
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = kSmem;
    cfg.stream = stream;
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    e = L.mode == M::Split ? cudaLaunchKernelEx(&cfg, f64tc_kernel<M::Split>, p)
        : L.mode == M::Transposed ? cudaLaunchKernelEx(&cfg, f64tc_kernel<M::Transposed>, p)
                                  : cudaLaunchKernelEx(&cfg, f64tc_kernel<M::Plain>, p);
    if (e != cudaSuccess) return e;
    if (p.here && !cut) return e;
    // Blocks that add the pieces of the row blocks that are cut, then those that
    // settle what is not certified.
    const bool by_cut = num_rb >= L.grid;
    const int64_t add = !cut ? 0 : (by_cut ? L.grid - 1 : num_rb) * (kRows / 32) * ((p.k + kSettleCols - 1) / kSettleCols);
    cfg.gridDim = dim3((unsigned)(add + (p.here ? 1 : kSettlePerSM) * L.blocks));
    cfg.blockDim = dim3(32 * kSettleWarps);
    cfg.dynamicSmemBytes = 0;
    return cudaLaunchKernelEx(&cfg, f64_combine_kernel, p, (int64_t)L.grid, (int)by_cut, (int)add);
}

cudaError_t f64tc_add(int64_t m, int k, const double *X, double *C, int64_t ldc, cudaStream_t stream) {
    f64_add_kernel<<<(unsigned)((m * k + 255) / 256), 256, 0, stream>>>(m, m * k, X, C, ldc);
    return cudaGetLastError();
}

}  // namespace tsm2
