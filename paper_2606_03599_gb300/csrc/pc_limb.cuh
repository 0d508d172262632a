// Sums of complex products of a few FP64 values on the integer pipe, for the tall-skinny products of
// the outer loop.
//
// GB300 runs 2 FP64 FMAs per clock and SM but 64 multiply-adds of 32 x 32 + 64 bits, so a group of
// products is formed in block floating point: the group's values become 57-bit integers in units set
// by their largest exponent, split into a high limb (28 bits) and a low limb (29 bits); a real product
// is three multiply-adds (high x high and the two mixed ones; low x low, below 2^-56 of the largest
// product, is left out) and the sum of up to 16 of them is exact.  It is turned into a double once per
// group, where an FP64 chain rounds every product.
#pragma once

#include <stdint.h>
#include <math.h>
#include <string.h>

#include "pc_complex.cuh"

namespace pc {

struct Limb {
    int hi, lo;  // hi 2^29 + lo, both with the value's sign
};
struct LimbC {
    Limb re, im;
};
struct LimbAcc {
    int64_t hi, mid;  // hi 2^58 + mid 2^29
};

// biased exponents a group may have (all others: FP64); the sum of two stays inside FP64's range
constexpr int kLimbLow = 600, kLimbHigh = 1450;

PC_HD int64_t limb_bits(double v) {
#if defined(__CUDA_ARCH__)
    return __double_as_longlong(v);
#else
    int64_t b;
    memcpy(&b, &v, 8);
    return b;
#endif
}
// the larger of m and the magnitude bits of v's high words
PC_HD int limb_top(double2 v, int m) {
    const int a = (int)(limb_bits(v.x) >> 32) & 0x7fffffff, b = (int)(limb_bits(v.y) >> 32) & 0x7fffffff;
    m = a > m ? a : m;
    return b > m ? b : m;
}
// v in units of 2^(E - 1079), E >= v's biased exponent and >= 64
PC_HD Limb limb_of(double v, int E) {
    const int64_t b = limb_bits(v);
    const int h = (int)(b >> 32);
    int sh = E - ((h >> 20) & 0x7ff);
    sh = sh > 63 ? 63 : sh;
    const uint64_t m = ((((uint64_t)b & 0xfffffffffffffULL) | 0x10000000000000ULL) << 4) >> sh;
    const int s = h >> 31;
    Limb r;
    r.hi = ((int)(m >> 29) ^ s) - s;
    r.lo = ((int)((uint32_t)m & 0x1fffffffu) ^ s) - s;
    return r;
}
PC_HD LimbC limb_of(double2 v, int E) {
    LimbC r;
    r.re = limb_of(v.x, E);
    r.im = limb_of(v.y, E);
    return r;
}
PC_HD void limb_mad(int64_t& acc, int a, int b) {
#if defined(__CUDA_ARCH__)
    asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(acc) : "r"(a), "r"(b));
#else
    acc += (int64_t)a * b;
#endif
}
PC_HD void limb_mac(LimbAcc& c, Limb a, Limb b) {
    limb_mad(c.hi, a.hi, b.hi);
    limb_mad(c.mid, a.hi, b.lo);
    limb_mad(c.mid, a.lo, b.hi);
}
PC_HD Limb limb_neg(Limb a) {
    a.hi = -a.hi;
    a.lo = -a.lo;
    return a;
}
// The accumulated sum of products of values with group exponents Ea and Eb.
PC_HD double limb_sum(LimbAcc c, int Ea, int Eb) {
    const int64_t t = c.hi * 4 + ((c.mid + (1 << 26)) >> 27);  // units of 2^56 products
    const double d = (double)t;
#if defined(__CUDA_ARCH__)
    return t == 0 ? 0.0 : __hiloint2double(__double2hiint(d) + (Ea + Eb - 2102) * (1 << 20), __double2loint(d));
#else
    return ldexp(d, Ea + Eb - 2102);
#endif
}

}  // namespace pc
