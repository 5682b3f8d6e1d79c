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

// The significand of a normal double as an integer in [2^52, 2^53) (2^53 for a
// result rounded up to the next binade).
struct Sig53 {
    unsigned m, l;          // the high 21 (22) and the low 32 bits
};

__device__ __forceinline__ Sig53 sig53(double x) {
    return Sig53{((unsigned)__double2hiint(x) & 0xfffffu) | 0x100000u, (unsigned)__double2loint(x)};
}

// |x| in units of its LSB / 2^10
__device__ __forceinline__ unsigned long long frame64(double x) {
    const Sig53 a = sig53(x);
    return (((unsigned long long)a.m << 32) | a.l) << 10;
}

// the double a 2^-53, a in [2^52, 2^53]
__device__ __forceinline__ double near_one(Sig53 a) {
    return __hiloint2double((int)(a.m - 0x100000u + (1022u << 20)), (int)a.l);
}

// |c| - |a b|, rounded to nearest even, for |a b| < |c| / 16 and a result whose
// LSB L is known: its significand.  c64 = |c| / (L / 2^10); the product's upper 64
// bits, P = a b / 2^42, are 2^n times that unit.  ~26 integer instructions: 12
// cycles per warp and SM against 16 of the FP64 unit.
__device__ __forceinline__ Sig53 soft_sub_from(unsigned long long c64, Sig53 a, Sig53 b, unsigned n) {
    typedef unsigned long long u64;
    const u64 w0 = (u64)a.l * b.l;
    const u64 w1 = (u64)a.m * b.l + (w0 >> 32);
    const u64 w2 = (u64)a.l * b.m + w1;
    const u64 w3 = (u64)a.m * b.m + (w2 >> 32);
    const unsigned z = (unsigned)w2, t = (unsigned)w0;
    // the product's upper 64 bits, in units of 2^n of the result's frame
    const u64 p = (w3 << 22) | (z >> 10);
    const unsigned rest = (z << 22) | t;
    u64 q, back;            // (these shifts give 0 for n >= 64)
    asm("shr.u64 %0, %1, %2;" : "=l"(q) : "l"(p), "r"(n));
    asm("shl.b64 %0, %1, %2;" : "=l"(back) : "l"(q), "r"(n));
    const u64 lost = back ^ p;
    const unsigned sticky = min((unsigned)lost | (unsigned)(lost >> 32) | rest, 1u);
    const u64 r = c64 - q - sticky;
    const unsigned rl = (unsigned)r, rh = (unsigned)(r >> 32);
    const unsigned ml = __funnelshift_r(rl, rh, 10), mh = rh >> 10;
    const unsigned up = ((ml & 1u) | sticky) + 0x7fffffffu;
    Sig53 o;
    asm("{\n\t"
        ".reg .u32 d;\n\t"
        "add.cc.u32 d, %2, %3;\n\t"
        "addc.cc.u32 %0, %4, 0;\n\t"
        "addc.u32 %1, %5, 0;\n\t"
        "}"
        : "=r"(o.l), "=r"(o.m)
        : "r"(rl << 22), "r"(up), "r"(ml), "r"(mh));
    return o;
}

// (double)x for a finite x, on the integer pipes: a conversion takes an FP64 slot
// like a multiply-add (predicated off too, so no branch around one may be short
// enough to be predicated).  x below 2^-60 goes through x 2^64, so that subnormals
// are normal on the way.
__device__ __forceinline__ double int_to_double(float x) {
    const bool small = fabsf(x) < 0x1p-60f;
    const unsigned u = __float_as_uint(small ? x * 0x1p64f : x);
    const unsigned bias = small ? (896u - 64u) << 20 : 896u << 20;
    const unsigned hi = (((u >> 3) & 0x0fffffffu) + bias) | (u & 0x80000000u);
    return __hiloint2double((int)(x == 0.0f ? u : hi), (int)(u << 29));
}

// Whether int_to_float does not take x: not zero, and outside the normal floats.
__device__ __forceinline__ bool float_odd(double x) {
    const unsigned hi = (unsigned)__double2hiint(x);
    return (hi & 0x7ff00000u) - (897u << 20) >= (254u << 20) && ((hi << 1) | (unsigned)__double2loint(x)) != 0u;
}

// (float)x for an x that is not odd, on the integer pipes.
__device__ __forceinline__ float int_to_float(double x) {
    const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
    // 23 bits of the significand below 9 of the exponent, rounded to nearest even
    const unsigned a = __funnelshift_l(lo, hi, 3) - (384u << 23);
    const unsigned up = (a & 1u) + 0x7fffffffu;
    unsigned r;
    asm("{\n\t"
        ".reg .u32 d;\n\t"
        "add.cc.u32 d, %1, %2;\n\t"
        "addc.u32 %0, %3, 0;\n\t"
        "}"
        : "=r"(r)
        : "r"(lo << 3), "r"(up), "r"(a));
    return __uint_as_float(((hi << 1) == 0u ? 0u : r) | (hi & 0x80000000u));
}

// How a block of FP64 arithmetic forms its products.
//   mul(a, b)  the product
//   chk(a, b)  the product, whose magnitude is to lie in 2^-100 .. 2^100
//   see(x)     x, which is to lie there
//   must(b)    b is to hold
// With FpMul all three are plain FP64.  With IntMul products are formed on the
// integer pipes and `bad` collects what lies outside (zeros, infinities, NaNs,
// subnormals included): when ok() is false at the end the block's results are
// discarded and the caller runs it with FpMul, so results are the same bit for
// bit either way.  A checked product is reliable when one factor is known to be
// normal and within 2^+-700: the exponent field of a product with a zero,
// subnormal, infinite or NaN factor then falls outside the window.
//   neg(x)     -x
//   mulz(a, b) the product where a may be zero
//   chkw(a, b) the same, whose magnitude is to be zero or in 2^-400 .. 2^400
//   chkz(a, b) the same where b may be zero too
//   chkm(a, b) the product, whose magnitude is to lie in 2^-200 .. 2^200
//   seew(x)    x, which is to be zero or in 2^-400 .. 2^400
//   rest(a, b) the product of an a that seew has taken and a constant
// p_phi, p_theta and what follows from them are zero or tiny in earnest (the column
// alpha = 0 of an image, the equatorial plane, a metric without spin), for whole
// rays: they take the wide forms, since one lane that fails its checks at every
// attempt, or one ray in 20 at each, makes whole warps run both kinds of attempt (a
// 97 x 61 table image of odd width, with such a column, 220 ms; 127 with the wide
// forms, 138 with plain attempts alone; without spin 56, 33.5 and 36.7; 65536
// equatorial rays 18.0, 9.3 and 17.3 ms).
struct FpMul {
    static constexpr bool kInt = false;
    __device__ __forceinline__ double neg(double x) { return -x; }
    __device__ __forceinline__ double mulz(double a, double b) { return a * b; }
    __device__ __forceinline__ double chkw(double a, double b) { return a * b; }
    __device__ __forceinline__ double chkz(double a, double b) { return a * b; }
    __device__ __forceinline__ double chkm(double a, double b) { return a * b; }
    __device__ __forceinline__ double rest(double a, double b) { return a * b; }
    __device__ __forceinline__ void seew(double) {}
    __device__ __forceinline__ double mul(double a, double b) { return a * b; }
    __device__ __forceinline__ double chk(double a, double b) { return a * b; }
    __device__ __forceinline__ void see(double) {}
    __device__ __forceinline__ void must(bool) {}
};

struct IntMul {
    static constexpr bool kInt = true;
    // (the sign bit of a product that integer instructions made: as a floating-point
    // negation it was a DADD)
    __device__ __forceinline__ double neg(double x) {
        return __hiloint2double(__double2hiint(x) ^ 0x80000000, __double2loint(x));
    }
    unsigned bad = 0;
    static __device__ __forceinline__ bool is_zero(double x) {
        return ((__double2hiint(x) << 1) | __double2loint(x)) == 0;
    }
    static __device__ __forceinline__ double zero_of(double a, double b) {
        return __hiloint2double((__double2hiint(a) ^ __double2hiint(b)) & 0x80000000, 0);
    }
    // the exponent field relative to 2^-400, in the units of see()'s bound
    __device__ __forceinline__ void wide(unsigned hi) { bad = max(bad, (hi + hi - ((1023u - 400u) << 21)) >> 2); }
    __device__ __forceinline__ double mulz(double a, double b) {
        const bool zero = is_zero(a);
        const double p = soft_mul64(a, b);
        see(zero ? 1.0 : p);
        return zero ? zero_of(a, b) : p;
    }
    __device__ __forceinline__ double chkw(double a, double b) {
        const bool zero = is_zero(a);
        const double p = soft_mul64(a, b);
        wide(zero ? 1023u << 20 : (unsigned)__double2hiint(p));
        return zero ? zero_of(a, b) : p;
    }
    __device__ __forceinline__ double chkz(double a, double b) {
        const bool zero = is_zero(a) || is_zero(b);
        const double p = soft_mul64(a, b);
        wide(zero ? 1023u << 20 : (unsigned)__double2hiint(p));
        return zero ? zero_of(a, b) : p;
    }
    __device__ __forceinline__ double chkm(double a, double b) {
        const double p = soft_mul64(a, b);
        const unsigned hi = (unsigned)__double2hiint(p);
        bad = max(bad, (hi + hi - ((1023u - 200u) << 21)) >> 1);
        return p;
    }
    __device__ __forceinline__ void seew(double x) { wide(is_zero(x) ? 1023u << 20 : (unsigned)__double2hiint(x)); }
    __device__ __forceinline__ double rest(double a, double b) {
        const double p = soft_mul64(a, b);
        return is_zero(a) ? zero_of(a, b) : p;
    }
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
    __device__ __forceinline__ void must(bool b) { bad = b ? bad : ~0u; }
    __device__ __forceinline__ bool ok() const { return bad < (200u << 21); }
};

}  // namespace tt
