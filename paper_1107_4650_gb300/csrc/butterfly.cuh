// The sum and the difference of the same two FP64 operands: every sweep of the scheme is built from such pairs
// (u = a + b and w = a - b, then a' = u + w' and b' = u - w').
//
// FP64 is bound by the FP64 pipe on GB300 (rated two instructions an SM and clock, 1/64 of the FP32 rate), so the
// pair is split over two pipes.  Of a + b and a - b one adds the operands' magnitudes (where their signs agree, the
// sum) and the other subtracts them.  The subtraction, which may cancel any number of bits, stays on the FP64 pipe;
// the magnitude sum needs no leading-zero search (its leading bit is the larger operand's or the one above) and is
// formed from the operands' bits in integer arithmetic, rounded to nearest, ties to even: the value the FP64 add
// gives, bit for bit (IEEE 754's definition of addition; zeros, subnormals, overflow and infinities included), so
// nothing downstream can tell which pipe did it.
// Measured, clocks an SM and warp at 1.92 GHz with four pairs a thread in flight: the pair alone 37.7, split 24.8 (the
// integer side's); with one FP64 multiply-add beside each pair, the 2-D step's ratio, 56.2 and 38.2.  The 2-D step at
// 2048^2: 9.6 -> 13.9 G point-steps/s, the FP64 pipe then 80 % busy.
#pragma once

#include <stdint.h>
#ifdef __CUDACC__
#include <cuda_runtime.h>
#define DIRAC_HD __host__ __device__ __forceinline__
#else
#define DIRAC_HD static inline
#endif

namespace dirac {

// |x| + |y| with x's sign, as bits.  The larger mantissa's leading bit sits at bit 62 with ten guard bits below; the
// smaller one is shifted down by the exponents' difference, its lost bits jammed into bit 0; the sum's leading bit is
// bit 62 or 63 (or lower for subnormals), so the rounding position is bit 10 or 11.
DIRAC_HD uint64_t magnitude_sum_bits(uint64_t x, uint64_t y) {
    const uint32_t xh = (uint32_t)(x >> 32), xl = (uint32_t)x, yh = (uint32_t)(y >> 32), yl = (uint32_t)y;
    const uint32_t xa = xh & 0x7fffffffu, ya = yh & 0x7fffffffu;
    // The larger magnitude by all 63 bits: with equal high words the order matters to an infinity and a NaN alone (the NaN is
    // the larger).  By a subtraction with borrow: FP64 2048^2 303 us a step, 580 by a comparison of 64-bit integers, 303 by
    // one of the high words, which took such a NaN for the smaller.
    int borrow;
#ifdef __CUDA_ARCH__
    asm("{\n\t.reg .u32 t;\n\tsub.cc.u32 t, %1, %2;\n\tsubc.u32 %0, %3, %4;\n\t}" : "=r"(borrow) : "r"(xl), "r"(yl), "r"(xa), "r"(ya));
#else
    borrow = -(((uint64_t)xa << 32 | xl) < ((uint64_t)ya << 32 | yl));
#endif
    const bool sw = borrow < 0;
    const uint32_t bh = sw ? ya : xa, bl = sw ? yl : xl, sh = sw ? xa : ya, sl = sw ? xl : yl;
    // exponents less one, zero for subnormals too: high word - (e << 20) is the mantissa with its hidden bit
    const int be = (int)(bh >> 20) - 1 > 0 ? (int)(bh >> 20) - 1 : 0, se = (int)(sh >> 20) - 1 > 0 ? (int)(sh >> 20) - 1 : 0;
    const uint32_t d = (uint32_t)(be - se);
    const uint64_t B = ((uint64_t)(bh - ((uint32_t)be << 20)) << 32 | bl) << 10;
    const uint64_t S = ((uint64_t)(sh - ((uint32_t)se << 20)) << 32 | sl) << 10;
    uint64_t T, L;
#ifdef __CUDA_ARCH__
    // PTX shifts clamp: 64 places or more leave zero
    asm("shr.u64 %0, %1, %2;" : "=l"(T) : "l"(S), "r"(d));
    asm("shl.b64 %0, %1, %2;" : "=l"(L) : "l"(T), "r"(d));
#else
    T = d < 64 ? S >> d : 0;
    L = d < 64 ? T << d : 0;
#endif
    uint64_t U = B + T;
    U |= (L != S) ? 1u : 0u;
    const uint32_t c = (uint32_t)(U >> 63), q = 10 + c;
    const uint32_t lsb = (uint32_t)(U >> q) & 1u;
    U += lsb + (511u + 512u * c);
    U >>= q;
    const uint32_t rh = (uint32_t)(U >> 32) + (((uint32_t)be + c) << 20);
    const bool over = rh >= 0x7ff00000u;  // overflow, or an infinity or NaN operand (the larger one)
    const uint32_t oh = over ? (bh > 0x7ff00000u ? bh : 0x7ff00000u) : rh, ol = over ? (bh >= 0x7ff00000u ? bl : 0u) : (uint32_t)U;
    return ((uint64_t)(oh | (xh & 0x80000000u)) << 32) | ol;
}

#ifdef __CUDACC__
// s = a + b and d = a - b
__device__ __forceinline__ void butterfly(double a, double b, double &s, double &d) {
    const int ah = __double2hiint(a), bh = __double2hiint(b);
    // b with the sign that makes a + b a subtraction of magnitudes
    const double nb = __hiloint2double((bh & 0x7fffffff) | (~ah & (int)0x80000000), __double2loint(b));
    const double low = __dadd_rn(a, nb);
    const double high =
        __longlong_as_double((long long)magnitude_sum_bits((uint64_t)__double_as_longlong(a), (uint64_t)__double_as_longlong(b)));
    const bool agree = (ah ^ bh) >= 0;
    s = agree ? high : low;
    d = agree ? low : high;
}
#endif

}  // namespace dirac
