// FP64 products on the integer pipe.  GB300's FP64 pipe takes a warp's multiplication 64 cycles
// (2 lanes a cycle and SM); the same product in 32-bit pieces takes about 52 cycles of the integer
// pipes, which run beside it: a loop of products with five of eight moved ran 2.3 times as fast
// (33 against 76 cycles a product).  It pays in kernels that are bound by the FP64 pipe, have warps
// to spare and little code; it does not in the persistent evaluation, which is bound by latency and
// instruction fetch as well (2,000 buses x 512: 416 us, and 461 with 29 of a branch's 46 products
// moved).
#pragma once

#include <cuda_runtime.h>

#include <cstdint>

namespace exago {

// x y, correctly rounded, for x and y in mul_window.  Two 53-bit significands (y's moved up to bit
// 63) make a 117-bit product in four 32 x 32 -> 64 multiply-adds; its upper 64 bits hold 52 or 53
// significant ones, which are aligned, rounded to nearest even by the lower half's carry, and given
// the sum of the exponents: the bits a multiplication gives.
__device__ __forceinline__ double int_mul(double x, double y) {
    const uint32_t xl = (uint32_t)__double2loint(x), xh = (uint32_t)__double2hiint(x);
    const uint32_t yl = (uint32_t)__double2loint(y), yh = (uint32_t)__double2hiint(y);
    const uint32_t mx = (xh & 0xfffff) | 0x100000, my = (yh & 0xfffff) | 0x100000;
    const uint32_t y1 = __funnelshift_l(yl, my, 11), y0 = yl << 11;
    const uint64_t p0 = (uint64_t)xl * y0;
    const uint64_t p1 = (uint64_t)mx * y0 + (p0 >> 32);
    const uint64_t p2 = (uint64_t)xl * y1 + (uint32_t)p1;
    uint64_t hi = (uint64_t)mx * y1 + (p1 >> 32) + (p2 >> 32);
    uint64_t lo = (p2 << 32) | (uint32_t)p0;
    uint32_t e = (xh & 0x7ff00000) + (yh & 0x7ff00000) - (1023u << 20);
    if (!(hi >> 52)) {   // 52 bits: the leading one would have added 1 to the exponent field
        hi = (hi << 1) | (lo >> 63);
        lo <<= 1;
        e -= 1u << 20;
    }
    // round to nearest even: the carry out of lo + 0x7fff.. + (lowest kept bit)
    const uint64_t t = lo + 0x7fffffffffffffffull, t2 = t + (hi & 1);
    hi += (uint64_t)(t < lo) + (uint64_t)(t2 < t);
    const uint32_t oh = ((uint32_t)(hi >> 32) + e) | ((xh ^ yh) & 0x80000000u);
    return __hiloint2double((int)oh, (int)(uint32_t)hi);
}

// Whether |x| lies in [2^-255, 2^257): operands whose product neither overflows nor becomes
// subnormal (zero, infinities and NaNs lie outside).
__device__ __forceinline__ bool mul_window(double x) {
    return ((uint32_t)__double2hiint(x) << 1) - (768u << 21) < (512u << 21);
}

__device__ __forceinline__ bool is_zero(double x) {
    return (((uint32_t)__double2hiint(x) << 1) | (uint32_t)__double2loint(x)) == 0;
}

// x y, correctly rounded, for x and y in mul_window or zero: what int_mul gives, or a zero of the
// product's sign.
__device__ __forceinline__ double int_mul_zero(double x, double y) {
    const double p = int_mul(x, y);
    const int sign = (__double2hiint(x) ^ __double2hiint(y)) & (int)0x80000000;
    return is_zero(x) || is_zero(y) ? __hiloint2double(sign, 0) : p;
}

// How an item multiplies.  INT: products whose operands are ordinary values (voltages, flows and
// their derivatives, never multipliers or sin th) go to the integer pipe; need() notes an operand
// outside the window, and the item is then computed again with INT = false.  Operands that are exactly
// zero in ordinary states (of a lossless branch without an angle across it the conductance terms)
// are noted by need_or_zero() and multiplied by or_zero(): computed twice, they took every warp that
// held one such branch through both paths.
template <bool INT>
struct Mul {
    bool ok = true;
    __device__ __forceinline__ double operator()(double x, double y) const {
        return INT ? int_mul(x, y) : x * y;
    }
    __device__ __forceinline__ double or_zero(double x, double y) const {
        return INT ? int_mul_zero(x, y) : x * y;
    }
    __device__ __forceinline__ void need(double x) {
        if (INT) ok = ok && mul_window(x);
    }
    __device__ __forceinline__ void need_or_zero(double x) {
        if (INT) ok = ok && (mul_window(x) || is_zero(x));
    }
};

}  // namespace exago
