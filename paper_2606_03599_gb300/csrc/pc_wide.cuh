// FP64 values on the integer pipe: a 64-bit integer and a binary exponent for every real number.
//
// GB300 issues 2 FP64 lanes per clock and SM, but 64 lanes of 64-bit integer addition and 64 of
// 32 x 32 + 64 bit multiply-add (measured: add.s64 63.9, mad.wide.s32 63.7, fma.f64 2.0), so FP64
// operations written out in integers still run several times as fast as the FP64 instructions.
//
// A number is m 2^u (m, u integers).  Nothing shares an exponent with anything it is not added to, and a sum
// is taken in units of its largest term, so every operation here rounds at 2^-57 or less of its
// largest operand, where FP64 rounds its result at 2^-53:
//   normalise   |m| in [2^61, 2^62), the form that products take
//   product     top 64 bits of the 124-bit product from three 32 x 32 bit ones (the low x low part, below
//               one unit, is left out): at least 2^58 units, off by at most two
//   sum         terms shifted down to the largest unit
// Zero has the unit kWideZero, below any other, so it never decides the unit of a sum.
#pragma once

#include <math.h>
#include <stdint.h>
#include <string.h>

#include "pc_complex.cuh"

namespace pc {

constexpr int kWideZero = -16000;    // unit of zero; fits 16 bits, as all units of finite FP64 data do
constexpr int kWideSpecial = 16384;  // unit that marks infinities and NaN

struct WideHalf {
    int hi, lo;  // m = hi 2^32 + lo, lo signed
};
struct WideEntry {  // a normalised factor: (hi 2^32 + lo) 2^u
    int hi, lo, u, pad;
};

PC_HD int imax(int a, int b) { return a > b ? a : b; }
PC_HD int imin(int a, int b) { return a < b ? a : b; }

PC_HD int64_t wide_bits(double v) {
#if defined(__CUDA_ARCH__)
    return __double_as_longlong(v);
#else
    int64_t b;
    memcpy(&b, &v, 8);
    return b;
#endif
}

// v >> s for any s >= 0.  In PTX on the device, whose shifts saturate: a shift beyond 63 leaves the sign.
PC_HD int64_t wide_shr(int64_t v, int s) {
#if defined(__CUDA_ARCH__)
    int64_t r;
    asm("shr.s64 %0, %1, %2;" : "=l"(r) : "l"(v), "r"(s));
    return r;
#else
    return v >> (s > 63 ? 63 : s);
#endif
}

PC_HD int wide_clz(uint32_t v) {
#if defined(__CUDA_ARCH__)
    return __clz((int)v);
#else
    return v ? __builtin_clz(v) : 32;
#endif
}

// m 2^u normalised; zero (and -1, all that a shift leaves of a small negative number) gets kWideZero.  One
// search in the high word, of which the GPU does 16 per clock and SM; below 2^32 the number moves up first.
PC_HD int64_t wide_norm(int64_t m, int& u) {
    int h = (int)(m >> 32);
    uint32_t f = (uint32_t)(h ^ (h >> 31));
    if (f == 0) {
        m = (int64_t)((uint64_t)m << 31);
        u -= 31;
        h = (int)(m >> 32);
        f = (uint32_t)(h ^ (h >> 31));
        if (f == 0) {
            u = kWideZero;
            return 0;
        }
    }
    const int s = wide_clz(f) - 1;  // 0..30: leading bit to position 62
    u += 1 - s;
    return (int64_t)((uint64_t)m << s) >> 1;
}

PC_HD WideHalf wide_split(int64_t m) {
    WideHalf h;
    h.hi = (int)((m + 0x80000000LL) >> 32);
    h.lo = (int)(uint32_t)m;
    return h;
}

// acc + a b.  In PTX on the device: written in C++ the compiler loses sight of the operands being
// 32 bits wide and multiplies 64 x 64.
PC_HD void wide_mad(int64_t& acc, int a, int b) {
#if defined(__CUDA_ARCH__)
    asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(acc) : "r"(a), "r"(b));
#else
    acc += (int64_t)a * b;
#endif
}

// The product of two normalised numbers in units of 2^64: below 2^60.
PC_HD int64_t wide_mul(WideHalf a, WideHalf b) {
    int64_t mid = 0x80000000LL, hi = 0;
    wide_mad(mid, a.hi, b.lo);
    wide_mad(mid, a.lo, b.hi);
    wide_mad(hi, a.hi, b.hi);
    wide_mad(hi, (int)(mid >> 32), 1);
    return hi;
}
PC_HD int64_t wide_mul(WideHalf a, const WideEntry& b) {
    WideHalf h;
    h.hi = b.hi;
    h.lo = b.lo;
    return wide_mul(a, h);
}

// A finite double with `lead` (3..10) bits below its last: |m| < 2^(53 + lead).  Infinities and NaN give
// some m and the unit kWideSpecial.
PC_HD int64_t wide_from_double(double v, int lead, int& u) {
    const int64_t b = wide_bits(v);
    const int hi = (int)(b >> 32), e = (hi >> 20) & 0x7ff;
    const uint64_t m = ((uint64_t)(uint32_t)((hi & 0xfffff) | (e != 0 ? 0x100000 : 0)) << 32 | (uint32_t)b) << lead;
    const int64_t s = hi >> 31;
    u = m == 0 ? kWideZero : e == 0x7ff ? kWideSpecial : imax(e, 1) - 1075 - lead;
    return ((int64_t)m ^ s) - s;
}

// A double as a factor of products.
PC_HD WideEntry wide_entry(double v) {
    int u;
    int64_t m = wide_from_double(v, 9, u);  // normalised unless subnormal
    if (m != 0 && u <= 1 - 1075 - 9) m = wide_norm(m, u);
    const WideHalf h = wide_split(m);
    WideEntry e;
    e.hi = h.hi;
    e.lo = h.lo;
    e.u = u;
    e.pad = 0;
    return e;
}

// Rows of a 3 x 3 table of normalised numbers through the lattice mixing M: out[m] = sum_s M[s][m] in[s], or
// (rows) out[s] = sum_m M[s][m] in[m]; one column of the table, below 3 2^60.
PC_HD void wide_mix3(const WideEntry* M, int64_t* V, int* U, bool rows) {
    WideHalf v[3];
    int u[3];
#pragma unroll
    for (int s = 0; s < 3; ++s) {
        v[s] = wide_split(V[s]);
        u[s] = U[s];
    }
#pragma unroll
    for (int m = 0; m < 3; ++m) {
        int64_t p[3];
        int pu[3], top = 2 * kWideZero;
#pragma unroll
        for (int s = 0; s < 3; ++s) {
            const WideEntry& w = M[rows ? m * 3 + s : s * 3 + m];
            p[s] = wide_mul(v[s], w);
            pu[s] = u[s] + w.u;
            top = imax(top, pu[s]);
        }
        U[m] = top + 64;
        V[m] = wide_shr(p[0], top - pu[0]) + wide_shr(p[1], top - pu[1]) + wide_shr(p[2], top - pu[2]);
    }
}

// Strain (xx, yy, zz, yz, xz, xy) of one part of a node: normalised halves and units.  load(a, x, u) gives component
// a's values, 2^59 at most, at the four backward neighbours and at the node itself, and their units.
template <bool CUBIC, typename Load>
PC_HD void wide_strain(const WideEntry* mix, const Load& load, WideHalf* e, int* eu) {
    int64_t H[3][3];
    int hu[3][3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        int64_t x[5];
        int u[5];
        load(a, x, u);
        const int U = imax(imax(imax(u[0], u[1]), imax(u[2], u[3])), u[4]);
#pragma unroll
        for (int l = 0; l < 5; ++l) x[l] = wide_shr(x[l], U - u[l]);
        const int64_t p = x[0] + x[1], q = x[2] + x[3];
        H[0][a] = p + q - 4 * x[4];  // 8 2^59 at most
        H[1][a] = p - q;
        H[2][a] = (x[0] - x[1]) + (x[2] - x[3]);
#pragma unroll
        for (int s = 0; s < 3; ++s) hu[s][a] = U;
        if (!CUBIC) {
            int64_t V[3] = {H[0][a], H[1][a], H[2][a]};
            int W[3] = {U, U, U};
#pragma unroll
            for (int s = 0; s < 3; ++s) V[s] = wide_norm(V[s], W[s]);
            wide_mix3(mix, V, W, false);
#pragma unroll
            for (int s = 0; s < 3; ++s) {
                H[s][a] = V[s];
                hu[s][a] = W[s];
            }
        }
    }
#pragma unroll
    for (int p = 0; p < 3; ++p) {
        const int a = p == 0 ? 1 : 0, b = p == 2 ? 1 : 2;
        eu[p] = hu[p][p];
        e[p] = wide_split(wide_norm(H[p][p], eu[p]));
        // a difference that vanishes (a uniform component) leaves the other's bits alone
        const int ua = H[b][a] == 0 ? kWideZero : hu[b][a], ub = H[a][b] == 0 ? kWideZero : hu[a][b];
        eu[3 + p] = imax(ua, ub);
        const int64_t sum = wide_shr(H[b][a], eu[3 + p] - ua) + wide_shr(H[a][b], eu[3 + p] - ub);
        e[3 + p] = wide_split(wide_norm(sum, eu[3 + p]));
    }
}

// Factors of sums of complex products (Gram products of pc_blas.cu).
struct WideC {
    WideHalf re, im;
};
constexpr int kWideLow = 600, kWideHigh = 1450;  // biased exponents of a group's largest value: its sum stays in
                                                 // FP64's normal range; all others go to FP64
// the larger of m and the magnitude bits of v's high words
PC_HD int wide_top(double2 v, int m) {
    m = imax(m, (int)(wide_bits(v.x) >> 32) & 0x7fffffff);
    return imax(m, (int)(wide_bits(v.y) >> 32) & 0x7fffffff);
}
// A double of such a group as a factor; subnormal values count as zero.
PC_HD WideHalf wide_factor(double v, int& u) {
    const int64_t b = wide_bits(v);
    const int hi = (int)(b >> 32), e = (hi >> 20) & 0x7ff;
    const int64_t m = (int64_t)(((uint64_t)b & 0xfffffffffffffULL) | 0x10000000000000ULL) << 9;
    const int64_t s = hi >> 31;
    WideHalf h = wide_split((m ^ s) - s);
    u = e - 1084;
    if (e == 0) {
        h.hi = h.lo = 0;
        u = kWideZero;
    }
    return h;
}
PC_HD WideC wide_factor(double2 v, int& ur, int& ui) {
    WideC r;
    r.re = wide_factor(v.x, ur);
    r.im = wide_factor(v.y, ui);
    return r;
}
// p >> s to nearest, s >= 1.
PC_HD int64_t wide_shr_near(int64_t p, int s) { return (wide_shr(p, s - 1) + 1) >> 1; }
// The unit wide_factor gives a double.
PC_HD int wide_unit(double v) {
    const int e = (int)(wide_bits(v) >> 52) & 0x7ff;
    return e == 0 ? kWideZero : e - 1084;
}
// A sum of up to 16 products (eight complex ones): m 2^(u + 64).  u is found from the products' units first
// (wide_reach for each pair), three bits above the largest, so that the sum stays below 2^61.
struct WideSum {
    int64_t m;
    int u;
};
PC_HD WideSum wide_sum0() {
    WideSum s;
    s.m = 0;
    s.u = 2 * kWideZero;
    return s;
}
PC_HD void wide_reach(WideSum& s, int ua, int ub, int uc, int ud) { s.u = imax(s.u, imax(ua + ub, uc + ud) + 3); }
// s + a b + c d, or (SUB) s + a b - c d.  Shifts round to nearest, and one of the products is taken away, so that
// halves rounded up cancel in the mean.  A product changes sign as 64 bits: a
// factor's low half can be -2^31, whose negative has no 32 bits.
template <bool SUB>
PC_HD void wide_mac2(WideSum& s, WideHalf a, int ua, WideHalf b, int ub, WideHalf c, int uc, WideHalf d, int ud) {
    const int64_t p = wide_mul(c, d);
    s.m += wide_shr_near(wide_mul(a, b), s.u - ua - ub) - wide_shr_near(SUB ? p : -p, s.u - uc - ud);
}

// m 2^u to the nearest double (results below the normal range round twice).
PC_HD double wide_to_double(int64_t m, int u) {
    const double d = (double)m;
#if defined(__CUDA_ARCH__)
    const int hi = __double2hiint(d), e = (hi >> 20) & 0x7ff;
    // the scale goes into the exponent field
    if ((unsigned)(e + u - 1) < 2046u) return m == 0 ? 0.0 : __hiloint2double(hi + u * (1 << 20), __double2loint(d));
#endif
    return m == 0 ? 0.0 : ldexp(d, u);
}

PC_HD double wide_to_double(WideSum s) { return wide_to_double(s.m, s.u + 64); }

}  // namespace pc
