// tt_soft64.cuh -- binary64 products on the integer pipes (sm_103a).
//
// GB300 issues FP64 at 2 lanes per SM per clock (a warp's DMUL holds its
// sub-partition's FP64 unit for 64 cycles whatever lanes are active), while the
// integer pipes take 64 lanes per SM per clock and stood idle: the FP64 tracer
// kept the FP64 unit busy 87 % of cycles and issued in 8 % of them.  40 % of its
// FP64 instructions are multiplications, and the 106-bit product of two 53-bit
// significands is four 32 x 32 -> 64 bit multiply-adds and ~17 integer
// instructions around them, rounded to nearest even exactly as DMUL rounds:
// 9.8 cycles per warp and SM against DMUL's 16 (19.4 against 9.8 at one clock in
// a chain of products), beside the FP64 unit instead of on it.
#pragma once

#include <cuda_runtime.h>

namespace tt {

// a * b for a and b normal and a product well inside the normal range; any
// other operands give a wrong value (never a fault), which the callers' range
// checks below catch.
__device__ __forceinline__ double soft_mul64(double a, double b) {
    typedef unsigned long long u64;
    const unsigned al = __double2loint(a), ah = __double2hiint(a);
    const unsigned bl = __double2loint(b), bh = __double2hiint(b);
    const unsigned am = (ah & 0xfffffu) | 0x100000u, bm = (bh & 0xfffffu) | 0x100000u;
    // the product as w3 2^64 + lo(w2) 2^32 + lo(w0), w3 in [2^40, 2^42)
    const u64 w0 = (u64)al * bl;
    const u64 w1 = (u64)am * bl + (w0 >> 32);
    const u64 w2 = (u64)al * bm + w1;
    const u64 w3 = (u64)am * bm + (w2 >> 32);
    const unsigned z = (unsigned)w2, t = (unsigned)w0, l3 = (unsigned)w3, h3 = (unsigned)(w3 >> 32);
    // the upper 53 bits: shift by 20, or by 21 when the significands' product is >= 2
    const unsigned sh = (h3 >> 9) + 20u;
    const unsigned ml = __funnelshift_r(z, l3, sh), mh = __funnelshift_r(l3, h3, sh);
    // round to nearest even: the bits shifted out, left-justified, carry out of
    // rem + 0x7fffffff + (odd or sticky)
    const unsigned rem = __funnelshift_r(0u, z, sh);
    const unsigned up = min((ml & 1u) | t, 1u) + 0x7fffffffu;
    // sign and exponent: each high word minus its significand is its sign and
    // exponent, and the sums of the signs wrap; mh holds the leading bit
    const unsigned e = (ah + bh - (1042u << 20)) - am - bm + (sh << 20);
    unsigned lo, hi;
    asm("{\n\t"
        ".reg .u32 d;\n\t"
        "add.cc.u32 d, %2, %3;\n\t"
        "addc.cc.u32 %0, %4, 0;\n\t"
        "addc.u32 %1, %5, %6;\n\t"
        "}"
        : "=r"(lo), "=r"(hi)
        : "r"(rem), "r"(up), "r"(ml), "r"(mh), "r"(e));
    return __hiloint2double((int)hi, (int)lo);
}

// How a block of FP64 arithmetic forms its products.
//   mul(a, b)  the product
//   chk(a, b)  the product, whose magnitude is to lie in 2^-100 .. 2^100
//   see(x)     x, which is to lie there
// With FpMul all three are plain FP64.  With IntMul products are formed on the
// integer pipes and `bad` collects what lies outside (zeros, infinities, NaNs,
// subnormals included): when ok() is false at the end the block's results are
// discarded and the caller runs it with FpMul, so results are the same bit for
// bit either way.  A checked product is reliable when one factor is known to be
// normal and within 2^+-700: the exponent field of a product with a zero,
// subnormal, infinite or NaN factor then falls outside the window.
struct FpMul {
    __device__ __forceinline__ double mul(double a, double b) { return a * b; }
    __device__ __forceinline__ double chk(double a, double b) { return a * b; }
    __device__ __forceinline__ void see(double) {}
};

struct IntMul {
    unsigned bad = 0;
    __device__ __forceinline__ double mul(double a, double b) { return soft_mul64(a, b); }
    __device__ __forceinline__ double chk(double a, double b) {
        const double p = soft_mul64(a, b);
        see(p);
        return p;
    }
    // the exponent field (twice the high word drops the sign) relative to 2^-100
    __device__ __forceinline__ void see(double x) {
        const unsigned hi = (unsigned)__double2hiint(x);
        bad = max(bad, hi + hi - ((1023u - 100u) << 21));
    }
    __device__ __forceinline__ bool ok() const { return bad < (200u << 21); }
};

}  // namespace tt
