// intfp.cuh -- IEEE binary64 operations evaluated with integer instructions.
//
// GB300 executes FP64 at 2 fused multiply-adds per clock per SM, 64 times
// slower than its integer pipes; the FP64 window kernels are bound by that
// pipe.  The functions here give, for the operands they accept, exactly the
// IEEE binary64 result (round to nearest, ties to even) that the FP64
// instruction would give, using integer instructions only; for the operands
// they refuse (zeros, subnormal, infinite or NaN inputs, results that would
// overflow or fall below the normal range) they return false and the caller
// issues the FP64 instruction.  Compiled for the host as well, so that
// tests/test_intfp.py checks them against the CPU's binary64 arithmetic.
#pragma once

#include <stdint.h>
#include <string.h>

#if defined(__CUDACC__)
#define PIC_HD __host__ __device__ __forceinline__
#else
#define PIC_HD inline
#endif

namespace pic {

PIC_HD uint64_t lf_bits(double x) {
#if defined(__CUDA_ARCH__)
    return (uint64_t)__double_as_longlong(x);
#else
    uint64_t b;
    memcpy(&b, &x, 8);
    return b;
#endif
}

PIC_HD double lf_double(uint64_t b) {
#if defined(__CUDA_ARCH__)
    return __longlong_as_double((long long)b);
#else
    double x;
    memcpy(&x, &b, 8);
    return x;
#endif
}

// position of the leading one bit (x > 0)
PIC_HD int lf_msb(uint64_t x) {
#if defined(__CUDA_ARCH__)
    return 63 - __clzll((long long)x);
#else
    return 63 - __builtin_clzll(x);
#endif
}

// high 64 bits of the 128-bit product a b
PIC_HD uint64_t lf_mulhi(uint64_t a, uint64_t b) {
#if defined(__CUDA_ARCH__)
    return __umul64hi(a, b);
#else
    return (uint64_t)(((unsigned __int128)a * b) >> 64);
#endif
}

// x * y rounded to nearest even.  The product of the significands shifted up
// to 64 bits has its leading bit at 127 or 126 of 128; the upper word keeps 53
// bits, the bits below them round, and the lower word only says whether
// anything lies below those.  No branch: `out` is always written, and holds
// the product where the result is true, so that several products can be
// interleaved and tested together.  (With a branch for the carry and one per
// check, the four products of a Lawson sweep cost FP64 windows of 10^6 particles
// 0.35 ms more of 8.8.)
PIC_HD bool imul64(double x, double y, double& out) {
    const uint64_t M52 = (1ull << 52) - 1;
    const uint64_t bx = lf_bits(x), by = lf_bits(y);
    const int ex = (int)((bx >> 52) & 0x7ff), ey = (int)((by >> 52) & 0x7ff);
    const uint64_t mx = ((bx & M52) | (1ull << 52)) << 11, my = ((by & M52) | (1ull << 52)) << 11;
    const uint64_t lo = mx * my, hi = lf_mulhi(mx, my);
    const int top = (int)(hi >> 63);
    const int sh = 10 + top;                           // bits of hi below the kept 53
    const uint32_t rem = (uint32_t)hi & ((1u << sh) - 1u), half = 1u << (sh - 1);
    const uint64_t q = hi >> sh;
    const uint32_t odd = ((uint32_t)q | (lo != 0ull ? 1u : 0u)) & 1u;  // a half rounds up when odd or not exact
    const uint32_t up = rem + odd > half ? 1u : 0u;
    const int e = ex + ey - 1023 + top;                // biased exponent (before a carry of the rounding)
    // q carries its leading bit into the exponent field, and a carry too
    out = lf_double(((bx ^ by) & (1ull << 63)) | (((uint64_t)(uint32_t)(e - 1) << 52) + q + up));
    return (uint32_t)(ex - 1) < 0x7feu & (uint32_t)(ey - 1) < 0x7feu & (uint32_t)(e - 1) < 0x7fdu;
}

}  // namespace pic
