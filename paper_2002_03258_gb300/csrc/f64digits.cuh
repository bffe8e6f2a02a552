// Integer digits of binary64 numbers and exact sums of their products, shared
// by the binary64 tensor-core kernels (tsm2_f64tc.cu describes the method).
#pragma once

#include "common.cuh"

#include <cuda_fp16.h>

namespace tsm2 {

__device__ __forceinline__ int exp_field(uint32_t hi) { return (int)((hi >> 20) & 0x7ffu); }

// |x| 2^61 / alpha cut to an integer: byte 7 - s is digit s of |x|.  key =
// scale_key(exponent field of alpha), so that (key - 2 hi) >> 21 is the
// exponent of alpha minus that of x (not negative; 64 or more shifts
// everything out: zeros and subnormals have exponent field 0 and alpha at
// least kMinExp).
__device__ __forceinline__ uint64_t fixed_point(uint32_t hi, uint32_t lo, uint32_t key) {
    const uint32_t d = (key - 2u * hi) >> 21;
    const uint32_t h = (__funnelshift_l(lo, hi, 9) & 0x1fffffffu) | 0x20000000u;
    uint64_t x = (uint64_t)h << 32 | (lo << 9);
    asm("shr.u64 %0, %0, %1;" : "+l"(x) : "r"(d));
    return x;
}
__device__ __forceinline__ uint32_t scale_key(int e) { return ((uint32_t)e << 21) + 0x1fffffu; }
constexpr int kMinExp = 64;  // scales below 2^(64-1023) are not used

// The digits of one element of A as packed binary16 (times 2^-24), low half
// digit s + 2, high half digit s: out[0..3] for s = 0, 1, 4, 5.
__device__ __forceinline__ void digits(uint64_t x, uint32_t hi, uint32_t (&out)[4]) {
    const uint32_t h = (uint32_t)(x >> 32), l = (uint32_t)x, sign = hi & 0x80000000u;
    out[0] = __byte_perm(h, sign, 0x7371);
    out[1] = __byte_perm(h, sign, 0x7270);
    out[2] = __byte_perm(l, sign, 0x7371);
    out[3] = __byte_perm(l, sign, 0x7270);
}

// Digit t of an element of B as binary16 bits: -128..127 times the sign.  x =
// fixed_point + 0x8080808080808080.
__device__ __forceinline__ uint32_t digit_b(uint64_t x, bool neg, int t) {
    const int d = (int)((x >> (8 * (7 - t))) & 0xffu) - 128;
    return (uint32_t)__half_as_ushort(__int2half_rn(neg ? -d : d));
}

__device__ __forceinline__ int64_t mad_wide(int a, int b, int64_t c) {
    int64_t d;
    asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(d) : "r"(a), "r"(b), "l"(c));
    return d;
}

// (H 2^32 + L) 2^s rounded to nearest even; s such that the result is neither
// subnormal nor too large.  In integers: with two binary64 operations per SM
// and cycle, a conversion by them (two I2D, an FMA and a product) holds the
// pipe for 320 cycles per warp, this takes about 40 instructions.
__device__ __forceinline__ double to_double(int64_t H, int64_t L, int s) {
    int64_t hi = H + (L >> 32);
    uint32_t lo = (uint32_t)L;
    const bool neg = hi < 0;
    if (neg) {
        hi = ~hi + (lo == 0u ? 1 : 0);
        lo = 0u - lo;
    }
    uint64_t top = (uint64_t)hi, rest = (uint64_t)lo << 32;
    if (top == 0) {  // below 2^32
        top = rest;
        rest = 0;
        s -= 64;
    }
    if (top == 0) return 0.0;
    const int z = __clzll((long long)top);
    top = (top << z) | (rest >> 1 >> (63 - z));
    rest <<= z;
    // 53 bits, the first of them 2^(95 - z + s).
    const uint32_t cut = (uint32_t)top & 0x7ffu;
    uint64_t bits = (top >> 11) + ((uint64_t)(95 - z + s + 1022) << 52);
    if (cut > 0x400u || (cut == 0x400u && (rest != 0 || (bits & 1u)))) ++bits;
    return __longlong_as_double((long long)(bits | (uint64_t)neg << 63));
}

}  // namespace tsm2
