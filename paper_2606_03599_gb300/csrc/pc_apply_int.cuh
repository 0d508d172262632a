// Complex128 stencil apply on the integer pipe: y = (A - shift M) x with every FP64 operand of the
// stencil held as a 64-bit integer and one binary exponent per node.
//
// GB300 issues 2 FP64 lanes per clock and SM, but 64 lanes of 64-bit integer addition and 64 of
// 32 x 32 + 64 bit multiply-add (measured: add.s64 63.9, mad.wide.s32 63.7, fma.f64 2.0).  The
// stencil is additions and products with constants, so it is done in block floating point: a node's
// six reals are integers below 2^56 in units of 2^(E - 1078), E the largest biased exponent among
// them (FP64 values with an exponent within 3 of E keep every bit).  Sums are exact; a product with
// a stiffness entry is 3 multiply-adds of 32-bit halves (the low x low part, below 2^-2 units, is
// left out) and rounds once per output.  The rounding of a flux is a few units of 2^-57 of the
// largest strain its node's values allow, where FP64 rounds the same sums at 2^-53 of them.
//
// Bounds (units of the node's exponent): x < 2^56, the sums H < 2^59 and strain < 2^60, stiffness
// rows sum to less than 2^62 so that a stress is below 2^58 after the division by 2^64 (general
// lattice: mixed sums < 2^59, stresses < 2^60 and their mixing < 0.98 2^59), fluxes < 2^59.6 and an output
// below 2^62.2 (2^60.6 and 0.98 2^63).  Accumulated products: high parts < 2^58, middle parts < 2^62.4.
//
// The operator, the layouts and the flux regions are those of pc_apply_tile.cuh.  A full-space
// vector is treated as its four parity blocks with strided addresses (the blocks do not couple), so
// one geometry serves both layouts.
//
// The tile and its march are pc_apply_cells.cuh's: each cell is one thread (two in small launches, see
// FixApply), which stages x of its column (asynchronous copy, Bloch phase if wrapped, conversion), forms
// the fluxes of its column when the plane's parity needs them, and, among the first TX x TY, finishes the
// outputs.
//
// Measured (one GB300, N = 48, 64 block vectors, shift on): 0.212 ms against 0.667 ms of the two-pass
// FP64 kernels; N = 60 FCC sub-pixel material, four blocks: 0.086 against 0.195 ms; N = 64 nodewise
// material, full space: 0.090 against 0.146 ms.  Bound by the instruction stream (half the issue slots
// at 16 warps per SM); DRAM moves 143 MB per launch at N = 48, close to the 170 MB of x and y.
//
// Values outside the exponent range (infinities, NaN, below 2^-823 or above 2^877) mark their node;
// a column is handed to FP64 (slow_column) from the first output that depends on a marked node.
#pragma once

#include <math.h>
#include <stdint.h>
#include <string.h>

#include "pc_apply_cells.cuh"
#include "pc_apply_tile.cuh"  // PC_IDX
#include "pc_complex.cuh"
#include "pc_internal.h"

#if defined(__CUDACC__)
#define PC_FIX_COLD __noinline__
#else
#define PC_FIX_COLD
#endif

namespace pc {

constexpr int kFixSpecial = 1 << 14;  // exponent of a node that FP64 has to handle
constexpr int kFixLow = 200, kFixHigh = 1900;  // biased exponents the integer path takes

struct FixHalf {
    int hi, lo;  // c = hi 2^32 + lo, lo signed
};

struct FixParams {
    StencilParams<double> P;  // FP64 tables: density, slow_column
    FixHalf c[2][21];         // phase tables; MATK 1: C_0 and C_1 - C_0
    FixHalf mix[9];           // lattice mixing (general lattices)
    int coff[2];              // exponent a product with c[p] adds
    int moff;                 // and the two lattice mixings together
    int nthr;
};

PC_HD FixHalf fix_split(int64_t v) {
    FixHalf h;
    h.hi = (int)((v + 0x80000000LL) >> 32);
    h.lo = (int)(uint32_t)v;
    return h;
}
PC_HD int fix_upper(int p, int r) { return p <= r ? p * 6 - p * (p - 1) / 2 + (r - p) : r * 6 - r * (r - 1) / 2 + (p - r); }

// Tables of one launch; false when a scale is out of the exponent range the kernel allows for.
inline bool make_fix_params(FixParams& F, const StencilParams<double>& P, bool cubic, int matkind) {
    F.P = P;
    memset(F.c, 0, sizeof(F.c));
    memset(F.mix, 0, sizeof(F.mix));
    F.coff[0] = F.coff[1] = F.moff = 0;
    if (matkind != 2) {
        double rs[2];
        for (int p = 0; p < 2; ++p) {
            rs[p] = 0.0;
            for (int i = 0; i < 6; ++i) {
                double s = 0.0;
                for (int j = 0; j < 6; ++j) s += fabs(P.C[p][i * 6 + j]);
                rs[p] = fmax(rs[p], s);
            }
        }
        if (matkind == 1) rs[0] = rs[1] = fmax(rs[0], rs[1]);
        int k[2];
        for (int p = 0; p < 2; ++p) {
            int ex = 0;
            if (!isfinite(rs[p])) return false;
            if (rs[p] > 0) frexp(rs[p], &ex);
            k[p] = (matkind == 1 ? 61 : 62) - ex;  // row sums of |c| below 2^62 (2^61: C_1 - C_0)
            F.coff[p] = 64 - k[p];
        }
        for (int i = 0; i < 6; ++i)
            for (int j = i; j < 6; ++j) {
                const int64_t a = llrint(ldexp(P.C[0][i * 6 + j], k[0]));
                const int64_t b = llrint(ldexp(P.C[1][i * 6 + j], k[1]));
                F.c[0][fix_upper(i, j)] = fix_split(a);
                F.c[1][fix_upper(i, j)] = fix_split(matkind == 1 ? b - a : b);
            }
    }
    if (!cubic) {
        double ms = 0.0;
        for (int i = 0; i < 3; ++i) {
            ms = fmax(ms, fabs(P.Mmix[i]) + fabs(P.Mmix[3 + i]) + fabs(P.Mmix[6 + i]));
            ms = fmax(ms, fabs(P.Mmix[3 * i]) + fabs(P.Mmix[3 * i + 1]) + fabs(P.Mmix[3 * i + 2]));
        }
        int ex = 0;
        if (!isfinite(ms)) return false;
        // sums below 0.98 2^62: the outputs, below 16 x 0.98 2^59, stay clear of the sign bit
        if (ms > 0 && frexp(ms, &ex) > 0.98) ++ex;
        F.moff = 2 * (64 - (62 - ex)) - 5;  // both mixings, less the bits their shifts keep
        for (int e = 0; e < 9; ++e) F.mix[e] = fix_split(llrint(ldexp(P.Mmix[e], 62 - ex)));
    }
    for (int p = 0; p < 2; ++p)
        if (F.coff[p] + F.moff > 100 || F.coff[p] + F.moff < -100) return false;
    return true;
}

PC_HD longlong2 fix_ashr2(longlong2 v, int s) {
    longlong2 r;
    r.x = v.x >> s;
    r.y = v.y >> s;
    return r;
}
PC_HD int imax(int a, int b) { return a > b ? a : b; }
PC_HD int imin(int a, int b) { return a < b ? a : b; }

PC_HD int64_t fix_bits(double v) {
#if defined(__CUDA_ARCH__)
    return __double_as_longlong(v);
#else
    int64_t b;
    memcpy(&b, &v, 8);
    return b;
#endif
}
PC_HD double fix_from_bits(int64_t b) {
#if defined(__CUDA_ARCH__)
    return __longlong_as_double(b);
#else
    double v;
    memcpy(&v, &b, 8);
    return v;
#endif
}
PC_HD int fix_clz64(uint64_t v) {
#if defined(__CUDA_ARCH__)
    return __clzll((long long)v);
#else
    return __builtin_clzll(v);
#endif
}

// v as an integer below 2^up (up in 53..63) in units of 2^(E - 1022 - up); base = E, or 64 for E = 0
// (all values of the node zero).  Bits below the unit are dropped.
PC_HD int64_t fix_from_double(double v, int base, int lead) {
    const int64_t b = fix_bits(v);
    const int hi = (int)(b >> 32);
    const int e = (hi >> 20) & 0x7ff;
    const uint64_t m = (((uint64_t)b & 0xfffffffffffffULL) | 0x10000000000000ULL) << lead;
    const int64_t s = hi >> 31;
    return ((int64_t)(m >> imin(base - e, 63)) ^ s) - s;
}
// largest |high word| of a complex number
PC_HD int fix_high(double2 v, int m) {
    m = imax(m, (int)(fix_bits(v.x) >> 32) & 0x7fffffff);
    return imax(m, (int)(fix_bits(v.y) >> 32) & 0x7fffffff);
}
// v 2^(E - 1078), rounded to nearest
PC_HD double fix_to_double(int64_t v, int E) {
#if defined(__CUDA_ARCH__)
    // one conversion on the FP64 pipe, which has room, instead of twenty integer instructions; the
    // scale goes into the exponent field
    const double d = __ll2double_rn(v);
    return v == 0 ? 0.0 : __hiloint2double(__double2hiint(d) + (E - 1078) * (1 << 20), __double2loint(d));
#else
    const int64_t s = v >> 63;
    const uint64_t mag = (uint64_t)((v ^ s) - s);
    if (mag == 0) return 0.0;
    const int lz = fix_clz64(mag);
    const uint64_t n = mag << lz;
    const uint64_t r = (n >> 11) + ((n >> 10) & 1);
    const uint64_t bits = ((uint64_t)(E + 7 - lz) << 52) + r;
    return fix_from_bits((int64_t)(bits | ((uint64_t)s & 0x8000000000000000ULL)));
#endif
}

// acc + a b.  In PTX on the device: written in C++ the compiler loses sight of the operands being
// 32 bits wide and multiplies 64 x 64.
PC_HD void fix_mad(int64_t& acc, int a, int b) {
#if defined(__CUDA_ARCH__)
    asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(acc) : "r"(a), "r"(b));
#else
    acc += (int64_t)a * b;
#endif
}
// hi 2^64 + mid 2^32 accumulates e c for signed halves
PC_HD void fix_mac(int64_t& hi, int64_t& mid, FixHalf e, FixHalf c) {
    fix_mad(hi, e.hi, c.hi);
    fix_mad(mid, e.hi, c.lo);
    fix_mad(mid, e.lo, c.hi);
}
// the accumulated product over 2^(64 - s), rounded (s in 0..8)
PC_HD int64_t fix_sum(int64_t hi, int64_t mid, int s) { return (hi << s) + ((mid + (0x80000000LL >> s)) >> (32 - s)); }

// theta in [0, 1] as an integer in units of 2^-62
PC_HD int64_t fix_theta(float t) {
#if defined(__CUDA_ARCH__)
    const uint32_t b = __float_as_uint(t);
#else
    uint32_t b;
    memcpy(&b, &t, 4);
#endif
    const int e = (int)(b >> 23);
    if (e == 0) return 0;
    const uint64_t m = (uint64_t)((b & 0x7fffffu) | 0x800000u) << 39;
    return (int64_t)(m >> imin(127 - e, 63));
}

// MATK: 0 = phase ids, 1 = inclusion fraction, 2 = nodewise material (as SplitApply).
// NP: parts (real, imaginary) of a cell in one thread; they meet in the Bloch phase and in the shared
// exponent only.  NP = 2 runs fewer instructions and is the form of launches that fill the GPU (N = 48, 64
// block vectors: 212 us, 267 us with NP = 1).  NP = 1, two adjacent lanes per cell, halves a thread's chain
// of dependent instructions: the form of launches with at most one CTA per SM, which wait for that chain
// (N = 8, one block vector: 14.3 us, 18.4 us with NP = 2).  The results are the same.
template <bool CUBIC, int MATK, int NP>
struct FixApply {
    struct Shared {
        int64_t* xs;  // [3 slots][3][kCells][2]
        int64_t* fs;  // [12][kCells][2]: F_l of component c at l * 3 + c
        double* raw;  // [3][kCells][2]: the next plane of x, as read
        double2* ph;  // [27] Bloch phases of the wraps (wa, wb, wk)
        FixHalf* c;   // [2][21]
        int* xe;      // [3][kCells]
        int* fe;      // [kCells]
    };
    static constexpr int kRow = 2 * kCells;  // stride of one component's array
    static constexpr size_t shared_bytes() {
        return (size_t)kCells * (16 * (9 + 12 + 3) + 4 * 4) + 16 * 27 + sizeof(FixHalf) * 42;
    }
    static PC_HD void carve(Shared& sh, unsigned char* p) {
        sh.xs = reinterpret_cast<int64_t*>(p);
        sh.fs = sh.xs + 9 * kRow;
        sh.raw = reinterpret_cast<double*>(sh.fs + 12 * kRow);
        sh.ph = reinterpret_cast<double2*>(sh.raw + 3 * kRow);
        sh.c = reinterpret_cast<FixHalf*>(sh.ph + 27);
        sh.xe = reinterpret_cast<int*>(sh.c + 42);
        sh.fe = sh.xe + 3 * kCells;
    }

    struct Ctx {
        const FixParams* F;
        const CellGeom* G;
        const double (*kph)[2];
        const double2* x;
        double2* y;
        const void* mat;
        double shift;
        bool dot;
        int a0, b0, k0, tz, p12, p13;
    };
    struct Regs : CellMap {
        int half;                // NP = 1: 0 real, 1 imaginary
        PC_HD int part() const { return NP == 1 ? half : 0; }
        int mprev, mcur, mnext;  // material of planes kf - 1, kf, kf + 1 (id, or the float's bits)
        int64_t pv[3][NP], cv[3][NP];  // y(kf - 1) and y(kf) so far
        int pe, ce;
        int ks;  // first output plane left to slow_column
        double xo[3][NP];
        double dot;
    };

    static PC_HD int wrap1(int v, int n, int& w) { return cell_wrap(v, n, w); }

    // Combine over the two parts of a cell (NP = 1: the neighbouring lane's, which takes every branch alike).
#if defined(__CUDA_ARCH__)
    static __device__ unsigned pair() { return 3u << (threadIdx.x & 30); }
#endif
    static PC_HD int pair_max(int v) {
#if defined(__CUDA_ARCH__)
        if (NP == 1) v = imax(v, __shfl_xor_sync(pair(), v, 1));
#endif
        return v;
    }
    static PC_HD int pair_or(int v) {
#if defined(__CUDA_ARCH__)
        if (NP == 1) v |= __shfl_xor_sync(pair(), v, 1);
#endif
        return v;
    }

    // a cell's parts: one 16-byte access, or 8 bytes of it
    static PC_HD void get(const int64_t* p, int64_t* v) {
        if (NP == 2) {
            const longlong2 t = *reinterpret_cast<const longlong2*>(p);
            v[0] = t.x;
            v[NP - 1] = t.y;
        } else {
            v[0] = *p;
        }
    }
    static PC_HD void put(int64_t* p, const int64_t* v) {
        if (NP == 2) {
            longlong2 t;
            t.x = v[0];
            t.y = v[NP - 1];
            *reinterpret_cast<longlong2*>(p) = t;
        } else {
            *p = v[0];
        }
    }
    static PC_HD void get(const double* p, double* v) {
        if (NP == 2) {
            const double2 t = *reinterpret_cast<const double2*>(p);
            v[0] = t.x;
            v[NP - 1] = t.y;
        } else {
            v[0] = *p;
        }
    }

    static PC_HD void init(const Ctx& c, int cell, int part, Regs& r) {
        cell_init(*c.G, c.a0, c.b0, c.p12, c.p13, cell, r);
        if (NP == 1) r.half = part;
        r.pe = r.ce = 0;
        r.ks = 1 << 30;
#pragma unroll
        for (int a = 0; a < 3; ++a)
#pragma unroll
            for (int i = 0; i < NP; ++i) {
                r.pv[a][i] = r.cv[a][i] = 0;
                r.xo[a][i] = 0.0;
            }
        r.dot = 0.0;
        r.mprev = r.mcur = r.mnext = 0;
    }

    static PC_HD void load_tables(const Ctx& c, Shared& sh, int tid, int nthr) {
        for (int i = tid; i < 42; i += nthr) sh.c[i] = c.F->c[i / 21][i % 21];
        for (int i = tid; i < 27; i += nthr) {
            const int w[3] = {i % 3 - 1, (i / 3) % 3 - 1, i / 9 - 1};
            double2 e = cmk(1.0, 0.0);
            for (int l = 0; l < 3; ++l)
                if (w[l] != 0) e = cmul(e, cmk(c.kph[l][0], w[l] < 0 ? -c.kph[l][1] : c.kph[l][1]));
            sh.ph[i] = e;
        }
    }

    // Start the copy of plane kp (parity Q) of x into the staging cells (one read by its own threads only).
    template <int Q>
    static PC_HD void stage(const Ctx& c, Shared& sh, const Regs& r, int cell, int kp) {
        const CellGeom& G = *c.G;
        int wk;
        const int k = wrap1(kp, G.Z, wk);
        const int at = k * G.plane + r.off[Q];
        PC_IDX(at, G.vstr);
        PC_IDX(cell, G.ncell);
        const double2* s = c.x + at;
        double* d = sh.raw + 2 * cell + r.part();
#pragma unroll
        for (int a = 0; a < 3; ++a) {
#if defined(__CUDA_ARCH__)
            const uint32_t to = (uint32_t)__cvta_generic_to_shared(d + a * kRow);
            const double* from = reinterpret_cast<const double*>(s + (int64_t)a * G.vstr) + r.part();
            if (NP == 2) asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(to), "l"(from) : "memory");
            else asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(to), "l"(from) : "memory");
#else
            const double* from = reinterpret_cast<const double*>(s + (int64_t)a * G.vstr);
            for (int i = 0; i < NP; ++i) d[a * kRow + i] = from[i];
#endif
        }
    }

    // Plane kp from the staging cells into slot sl: phase, exponent, integers.
    template <int Q>
    static PC_HD void convert(const Ctx& c, Shared& sh, const Regs& r, int cell, int kp, int sl) {
        const CellGeom& G = *c.G;
        int wk;
        wrap1(kp, G.Z, wk);
        const int w = r.wab[Q] + 9 * (wk + 1);
        double v[3][NP];
        const double* d = sh.raw + 2 * cell + r.part();
#pragma unroll
        for (int a = 0; a < 3; ++a) get(d + a * kRow, v[a]);
        if (w != 13) {
            const double2 ph = sh.ph[w];
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                if (NP == 2) {
                    const double2 z = cmul(cmk(v[a][0], v[a][NP - 1]), ph);
                    v[a][0] = z.x;
                    v[a][NP - 1] = z.y;
                } else {
#if defined(__CUDA_ARCH__)
                    const double o = __shfl_xor_sync(pair(), v[a][0], 1);
                    const double m = r.part() ? o * ph.y : v[a][0] * ph.x;  // as cmul rounds
                    v[a][0] = fma(r.part() ? v[a][0] : -o, r.part() ? ph.x : ph.y, m);
#endif
                }
            }
        }
        int top = 0;
#pragma unroll
        for (int a = 0; a < 3; ++a)
#pragma unroll
            for (int i = 0; i < NP; ++i) top = imax(top, (int)(fix_bits(v[a][i]) >> 32) & 0x7fffffff);
        int E = pair_max(top) >> 20, base = E;
        if (E < kFixLow || E > kFixHigh) {
            int64_t any = 0;
#pragma unroll
            for (int a = 0; a < 3; ++a)
#pragma unroll
                for (int i = 0; i < NP; ++i) any |= fix_bits(v[a][i]) & 0x7fffffffffffffffLL;
            base = 64;
            E = pair_or(any != 0) ? kFixSpecial : 0;
        }
        int64_t* xs = sh.xs + sl * 3 * kRow + 2 * r.own[Q] + r.part();
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            int64_t o[NP];
#pragma unroll
            for (int i = 0; i < NP; ++i) o[i] = E == 0 ? 0 : fix_from_double(v[a][i], base, 3);
            put(xs + a * kRow, o);
        }
        sh.xe[sl * kCells + r.own[Q]] = E;
    }

    template <int Q>
    static PC_HD int read_mat(const Ctx& c, const Regs& r, int kp) {
        if (MATK == 2) return 0;
        const CellGeom& G = *c.G;
        int wk;
        const int k = wrap1(kp, G.Z, wk);
        const int at = k * G.plane + r.off[Q];
        PC_IDX(at, G.vstr);
        if (MATK == 0) return static_cast<const uint8_t*>(c.mat)[at];
#if defined(__CUDA_ARCH__)
        return __float_as_int(static_cast<const float*>(c.mat)[at]);
#else
        int b;
        memcpy(&b, static_cast<const float*>(c.mat) + at, 4);
        return b;
#endif
    }
    static PC_HD float mat_theta(int b) {
#if defined(__CUDA_ARCH__)
        return __int_as_float(b);
#else
        float f;
        memcpy(&f, &b, 4);
        return f;
#endif
    }

    template <bool ORTHO>
    static PC_HD void stress(const FixHalf* C, const FixHalf (*e)[NP], int64_t (*t)[NP]) {
#pragma unroll
        for (int p = 0; p < 6; ++p) {
            int64_t h[NP], m[NP];
#pragma unroll
            for (int i = 0; i < NP; ++i) h[i] = m[i] = 0;
#pragma unroll
            for (int u = 0; u < 6; ++u) {
                if (ORTHO && !((p < 3 && u < 3) || p == u)) continue;
                const FixHalf cc = C[fix_upper(p, u)];
#pragma unroll
                for (int i = 0; i < NP; ++i) fix_mac(h[i], m[i], e[u][i], cc);
            }
#pragma unroll
            for (int i = 0; i < NP; ++i) t[p][i] = fix_sum(h[i], m[i], CUBIC ? 0 : 2);
        }
    }

    // Fluxes of plane kf (parity Q) at the thread's column; -4 P_0 into y(kf).  sm, sc, sp: slots of planes
    // kf - 1, kf, kf + 1.
    template <int Q>
    static PC_HD void flux(const Ctx& c, Shared& sh, Regs& r, int kf, int sm, int sc, int sp) {
        const CellGeom& G = *c.G;
        constexpr int n = kCells;
        if (!((r.flags >> Q) & 1)) return;
        const int n0 = r.nb[Q] & 0xffff, n1 = r.nb[Q] >> 16, own = r.own[Q];
        PC_IDX(n0, G.ncell);
        PC_IDX(n1, G.ncell);
        const int eo = sh.xe[sc * n + own];
        const int e0 = sh.xe[sm * n + n0], e1 = sh.xe[sp * n + n0], e2 = sh.xe[sm * n + n1], e3 = sh.xe[sp * n + n1];
        const int E = imax(imax(imax(e0, e1), imax(e2, e3)), eo);
        if (E >= kFixSpecial) {
            sh.fe[own] = kFixSpecial;
            r.ce = kFixSpecial;
            return;
        }
        const int s0 = imin(E - e0, 63), s1 = imin(E - e1, 63), s2 = imin(E - e2, 63), s3 = imin(E - e3, 63),
                  so = imin(E - eo, 63);
        const int64_t *p0 = sh.xs + sm * 3 * kRow + 2 * n0 + r.part(), *p1 = sh.xs + sp * 3 * kRow + 2 * n0 + r.part(),
                      *p2 = sh.xs + sm * 3 * kRow + 2 * n1 + r.part(), *p3 = sh.xs + sp * 3 * kRow + 2 * n1 + r.part(),
                      *po = sh.xs + sc * 3 * kRow + 2 * own + r.part();
        int64_t H[3][3][NP];
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            int64_t x0[NP], x1[NP], x2[NP], x3[NP], xo[NP];
            get(p0 + a * kRow, x0);
            get(p1 + a * kRow, x1);
            get(p2 + a * kRow, x2);
            get(p3 + a * kRow, x3);
            get(po + a * kRow, xo);
            int64_t u[NP], v[NP];
#pragma unroll
            for (int i = 0; i < NP; ++i) {
                x0[i] >>= s0;
                x1[i] >>= s1;
            }
#pragma unroll
            for (int i = 0; i < NP; ++i) {
                x2[i] >>= s2;
                x3[i] >>= s3;
            }
#pragma unroll
            for (int i = 0; i < NP; ++i) {
                xo[i] >>= so;
                u[i] = x0[i] + x1[i];
                v[i] = x2[i] + x3[i];
            }
#pragma unroll
            for (int i = 0; i < NP; ++i) H[0][a][i] = u[i] + v[i] - 4 * xo[i];
#pragma unroll
            for (int i = 0; i < NP; ++i) H[1][a][i] = u[i] - v[i];
#pragma unroll
            for (int i = 0; i < NP; ++i) H[2][a][i] = (x0[i] - x1[i]) + (x2[i] - x3[i]);
        }
        int up = 0;
        if (!CUBIC || MATK != 0) {
            // more roundings follow than in the plain case: scale the sums up to their bound first
            int top = 0;
#pragma unroll
            for (int m = 0; m < 3; ++m)
#pragma unroll
                for (int a = 0; a < 3; ++a)
#pragma unroll
                    for (int i = 0; i < NP; ++i) top |= (int)((H[m][a][i] ^ (H[m][a][i] >> 63)) >> 32);
            up = fix_clz64((uint64_t)(uint32_t)pair_or(top) | 1) - 32 - 5;
#pragma unroll
            for (int m = 0; m < 3; ++m)
#pragma unroll
                for (int a = 0; a < 3; ++a)
#pragma unroll
                    for (int i = 0; i < NP; ++i) H[m][a][i] <<= up;
        }
        if (!CUBIC) mix3(c, H, false);
        // strain halves: xx, yy, zz, yz, xz, xy
        FixHalf e[6][NP];
#pragma unroll
        for (int p = 0; p < 3; ++p) {
            const int u = p == 0 ? 1 : 0, v = p == 2 ? 1 : 2;
#pragma unroll
            for (int i = 0; i < NP; ++i) e[p][i] = fix_split(H[p][p][i]);
#pragma unroll
            for (int i = 0; i < NP; ++i) e[3 + p][i] = fix_split(H[v][u][i] + H[u][v][i]);
        }
        int64_t t[6][NP];
        int fe = E - up + c.F->moff;
        if (MATK == 0) {
            const int ph = r.mcur != 0 ? 1 : 0;
            const FixHalf* C = sh.c + 21 * ph;
            fe += ph ? c.F->coff[1] : c.F->coff[0];
            // every node of the warp orthotropic: normal block and shear diagonal only
            if (warp_all(c.F->P.ortho[ph] != 0)) stress<true>(C, e, t);
            else stress<false>(C, e, t);
        } else {
            int64_t h[6][NP], m[6][NP];
#pragma unroll
            for (int p = 0; p < 6; ++p)
#pragma unroll
                for (int i = 0; i < NP; ++i) h[p][i] = m[p][i] = 0;
            int row[6] = {0, 0, 0, 0, 0, 0};  // row sums of |c| / 2^32
            FixHalf th = {0, 0};
            const double* md = nullptr;
            int base = 64;
            bool empty = false;  // a void: zero fluxes, whatever x is
            if (MATK == 1) {
                th = fix_split(fix_theta(mat_theta(r.mcur)));
                fe += c.F->coff[0];
            } else {
                int wk;
                const int at = wrap1(kf, G.Z, wk) * G.plane + r.off[Q];
                md = static_cast<const double*>(c.mat) + at;
                int top = 0;
#pragma unroll
                for (int u = 0; u < 21; ++u) top = imax(top, (int)(fix_bits(md[(int64_t)u * G.vstr]) >> 32) & 0x7fffffff);
                base = top >> 20;  // entries below 2^59: row sums below 2^62
                fe += base - 1017;
                if (base == 0) {
                    int64_t any = 0;
#pragma unroll
                    for (int u = 0; u < 21; ++u) any |= fix_bits(md[(int64_t)u * G.vstr]);
                    empty = (any & 0x7fffffffffffffffLL) == 0;
                    base = empty ? 1000 : 0;
                }
                if (base < 950 || base > 1100) {  // tables far outside hat units
                    sh.fe[own] = kFixSpecial;
                    r.ce = kFixSpecial;
                    return;
                }
            }
#pragma unroll
            for (int p = 0; p < 6; ++p)
#pragma unroll
                for (int u = p; u < 6; ++u) {
                    FixHalf cc;
                    if (MATK == 1) {  // c = C_0 + theta (C_1 - C_0)
                        int64_t hh = 0, mm = 1LL << 29;
                        const FixHalf d = sh.c[21 + fix_upper(p, u)], z = sh.c[fix_upper(p, u)];
                        fix_mac(hh, mm, th, d);
                        cc = fix_split((int64_t)z.hi * 0x100000000LL + z.lo + hh * 4 + (mm >> 30));
                    } else {
                        cc = fix_split(fix_from_double(md[(int64_t)fix_upper(p, u) * G.vstr], base, 6));
                    }
                    const int ab = cc.hi < 0 ? -cc.hi : cc.hi;
                    row[p] += ab;
                    if (u != p) row[u] += ab;
#pragma unroll
                    for (int i = 0; i < NP; ++i) {
                        fix_mac(h[p][i], m[p][i], e[u][i], cc);
                        if (u != p) fix_mac(h[u][i], m[u][i], e[p][i], cc);
                    }
                }
            // the node's own row sums are below the bound the scale allows for: keep that many more bits
            const int top = imax(imax(imax(row[0], row[1]), imax(row[2], row[3])), imax(row[4], row[5])) + 6;
            int sh2 = (top < (1 << 24) ? 6 : top < (1 << 25) ? 5 : top < (1 << 26) ? 4 : top < (1 << 27) ? 3
                       : top < (1 << 28) ? 2 : top < (1 << 29) ? 1 : 0);
            fe = empty ? 0 : fe - sh2;
            sh2 += CUBIC ? 0 : 2;
#pragma unroll
            for (int p = 0; p < 6; ++p)
#pragma unroll
                for (int i = 0; i < NP; ++i) t[p][i] = fix_sum(h[p][i], m[p][i], sh2);
        }
        if (E == 0) fe = 0;  // zero fluxes
        sh.fe[own] = fe;
        // P_s (s, component)
        int64_t Ps[3][3][NP];
#pragma unroll
        for (int i = 0; i < NP; ++i) {
            Ps[0][0][i] = t[0][i];
            Ps[1][1][i] = t[1][i];
            Ps[2][2][i] = t[2][i];
            Ps[0][1][i] = Ps[1][0][i] = t[5][i];
            Ps[0][2][i] = Ps[2][0][i] = t[4][i];
            Ps[1][2][i] = Ps[2][1][i] = t[3][i];
        }
        if (!CUBIC) mix3(c, Ps, true);
        int64_t* f = sh.fs + 2 * own + r.part();
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            int64_t u[NP], v[NP], g[NP];
#pragma unroll
            for (int i = 0; i < NP; ++i) {
                u[i] = Ps[0][a][i] + Ps[1][a][i];
                v[i] = Ps[0][a][i] - Ps[1][a][i];
            }
#pragma unroll
            for (int l = 0; l < 4; ++l) {
#pragma unroll
                for (int i = 0; i < NP; ++i) g[i] = (l < 2 ? u[i] : v[i]) + (l & 1 ? -Ps[2][a][i] : Ps[2][a][i]);
                put(f + (l * 3 + a) * kRow, g);
            }
        }
        if (r.flags & 4) {
            const int m = imax(r.ce, fe);
            const int sa = imin(m - r.ce, 63), sf = imin(m - fe, 63);
#pragma unroll
            for (int a = 0; a < 3; ++a)
#pragma unroll
                for (int i = 0; i < NP; ++i) r.cv[a][i] = (r.cv[a][i] >> sa) - 4 * (Ps[0][a][i] >> sf);
            r.ce = m;
        }
    }

    // Rows of a 3 x 3 table through the lattice mixing: out[m] = sum_s Mmix[s][m] in[s], or (rows)
    // out[s] = sum_m Mmix[s][m] in[m].
    static PC_HD void mix3(const Ctx& c, int64_t (*V)[3][NP], bool rows) {
#pragma unroll
        for (int a = 0; a < 3; ++a)
#pragma unroll
            for (int i = 0; i < NP; ++i) {
                FixHalf v[3];
#pragma unroll
                for (int s = 0; s < 3; ++s) v[s] = fix_split(V[s][a][i]);
#pragma unroll
                for (int m = 0; m < 3; ++m) {
                    int64_t h = 0, md = 0;
#pragma unroll
                    for (int s = 0; s < 3; ++s) fix_mac(h, md, v[s], c.F->mix[rows ? m * 3 + s : s * 3 + m]);
                    V[m][a][i] = fix_sum(h, md, rows ? 1 : 2);
                }
            }
    }

    // The node's own x of plane kf - 1, for the shift term and the inner product.
    template <int Q>
    static PC_HD void load_own(const Ctx& c, Regs& r, int kf) {
        const int k = kf - 1;
        if (!(r.flags & 4) || k < c.k0) return;
        const int at = k * c.G->plane + r.off[1 - Q];
        PC_IDX(at, c.G->vstr);
        const double2* s = c.x + at;
#pragma unroll
        for (int a = 0; a < 3; ++a) get(reinterpret_cast<const double*>(s + (int64_t)a * c.G->vstr) + r.part(), r.xo[a]);
    }

    // Outputs y(kf - 1); y(kf) moves on; y(kf + 1) starts with F_1, F_3 of plane kf.
    template <int Q>
    static PC_HD void gather(const Ctx& c, Shared& sh, Regs& r, int kf) {
        const CellGeom& G = *c.G;
        if (!(r.flags & 4)) return;
        const int k = kf - 1;  // planes kf - 1 and kf + 1 share the offsets
        const int c0 = r.gn[1 - Q] & 0xffff, c1 = r.gn[1 - Q] >> 16;
        PC_IDX(c0, G.ncell);
        PC_IDX(c1, G.ncell);
        const int f0 = sh.fe[c0], f1 = sh.fe[c1];
        const int64_t *a0 = sh.fs + 2 * c0 + r.part(), *a1 = sh.fs + 2 * c1 + r.part();
        if (k >= c.k0) {
            const int at = k * G.plane + r.off[1 - Q];
            const int E = imax(r.pe, imax(f0, f1));
            if (E >= kFixSpecial && r.ks > k) r.ks = k;
            if (k < r.ks) {
                const double sr = c.shift * density(c, r.mprev, at);
                const int sa = imin(E - r.pe, 63), s0 = imin(E - f0, 63), s1 = imin(E - f1, 63);
#pragma unroll
                for (int a = 0; a < 3; ++a) {
                    int64_t g0[NP], g1[NP];
                    double w[NP];
                    get(a0 + a * kRow, g0);
                    get(a1 + (6 + a) * kRow, g1);
#pragma unroll
                    for (int i = 0; i < NP; ++i) {
                        w[i] = fix_to_double((r.pv[a][i] >> sa) + (g0[i] >> s0) + (g1[i] >> s1), E);
                        w[i] = fma(-sr, r.xo[a][i], w[i]);
                    }
                    double2* y = c.y + at + (int64_t)a * G.vstr;
                    if (NP == 2) *y = cmk(w[0], w[NP - 1]);
                    else reinterpret_cast<double*>(y)[r.part()] = w[0];
                    if (c.dot) {
#pragma unroll
                        for (int i = 0; i < NP; ++i) r.dot = fma(r.xo[a][i], w[i], r.dot);
                    }
                }
            }
        }
        const int E = imax(f0, f1);
        r.pe = r.ce;
        r.ce = E;
        const int s0 = imin(E - f0, 63), s1 = imin(E - f1, 63);
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            int64_t g0[NP], g1[NP];
            get(a0 + (3 + a) * kRow, g0);
            get(a1 + (9 + a) * kRow, g1);
#pragma unroll
            for (int i = 0; i < NP; ++i) {
                r.pv[a][i] = r.cv[a][i];
                r.cv[a][i] = (g0[i] >> s0) + (g1[i] >> s1);
            }
        }
    }

    static PC_HD double density(const Ctx& c, int m, int at) {
        const StencilParams<double>& P = c.F->P;
        if (MATK == 0) return P.rho[m != 0 ? 1 : 0];
        if (MATK == 1) return P.rho[0] + (double)mat_theta(m) * (P.rho[1] - P.rho[0]);
        return static_cast<const double*>(c.mat)[21LL * c.G->vstr + at];
    }

    static PC_HD void next_mat(Regs& r) {
        r.mprev = r.mcur;
        r.mcur = r.mnext;
    }

    // Fluxes at node (a, b, k) of the block in FP64 (coordinates inside the grid).
    static __host__ __device__ void slow_flux(const Ctx& c, int a, int b, int k, double2 (*Fo)[3]) {
        const CellGeom& G = *c.G;
        const StencilParams<double>& P = c.F->P;
        auto addr = [&](int aa, int bb, int kk) -> int64_t {
            const int i0 = (kk + c.p13) & 1, j0 = (kk + c.p12 + c.p13) & 1;
            return (int64_t)kk * G.plane + (G.full ? (2 * aa + i0) + (int64_t)G.N * (2 * bb + j0) : aa + (int64_t)G.X * bb);
        };
        const int64_t at = addr(a, b, k);
        const int i0 = (k + c.p13) & 1, j0 = (k + c.p12 + c.p13) & 1;
        double2 H[3][3];
        for (int al = 0; al < 3; ++al) {
            double2 nv[4];
            for (int l = 0; l < 4; ++l) {
                const int s2 = (l < 2) ? 1 : -1, s3 = (l & 1) ? -1 : 1;
                int w[3];
                const int na = wrap1(a + i0 - 1, G.X, w[0]), nbb = wrap1(b + j0 - ((s2 + 1) >> 1), G.Y, w[1]),
                          nk = wrap1(k - s3, G.Z, w[2]);
                nv[l] = c.x[(int64_t)al * G.vstr + addr(na, nbb, nk)];
                if (w[0] | w[1] | w[2]) {
                    double2 ph = cmk(1.0, 0.0);
                    for (int d = 0; d < 3; ++d)
                        if (w[d] != 0) ph = cmul(ph, cmk(c.kph[d][0], w[d] < 0 ? -c.kph[d][1] : c.kph[d][1]));
                    nv[l] = cmul(nv[l], ph);
                }
            }
            const double2 u = cadd(nv[0], nv[1]), v = cadd(nv[2], nv[3]);
            H[0][al] = cfma(-4.0, c.x[(int64_t)al * G.vstr + at], cadd(u, v));
            H[1][al] = csub(u, v);
            H[2][al] = cadd(csub(nv[0], nv[1]), csub(nv[2], nv[3]));
        }
        double2 Gm[3][3];
        for (int m = 0; m < 3; ++m)
            for (int al = 0; al < 3; ++al) {
                if (CUBIC) {
                    Gm[m][al] = H[m][al];
                } else {
                    double2 acc = cscale(P.Mmix[m], H[0][al]);
                    acc = cfma(P.Mmix[3 + m], H[1][al], acc);
                    Gm[m][al] = cfma(P.Mmix[6 + m], H[2][al], acc);
                }
            }
        const double2 e[6] = {Gm[0][0], Gm[1][1], Gm[2][2], cadd(Gm[2][1], Gm[1][2]), cadd(Gm[2][0], Gm[0][2]),
                              cadd(Gm[1][0], Gm[0][1])};
        double2 t[6];
        int ph = 0;
        double th = 0.0;
        if (MATK == 0) ph = static_cast<const uint8_t*>(c.mat)[at] != 0 ? 1 : 0;
        if (MATK == 1) th = (double)static_cast<const float*>(c.mat)[at];
        for (int p = 0; p < 6; ++p) {
            double2 acc = czero(0.0);
            bool first = true;
            for (int u = 0; u < 6; ++u) {
                double cc;
                if (MATK == 0) {
                    if (P.ortho[ph] && !((p < 3 && u < 3) || p == u)) continue;  // structural zeros
                    cc = P.C[ph][p * 6 + u];
                } else if (MATK == 1) {
                    cc = P.C[0][p * 6 + u] + th * (P.C[1][p * 6 + u] - P.C[0][p * 6 + u]);
                } else {
                    cc = static_cast<const double*>(c.mat)[(int64_t)fix_upper(p, u) * G.vstr + at];
                }
                acc = first ? cscale(cc, e[u]) : cfma(cc, e[u], acc);
                first = false;
            }
            t[p] = acc;
        }
        const double2 S[3][3] = {{t[0], t[5], t[4]}, {t[5], t[1], t[3]}, {t[4], t[3], t[2]}};
        for (int al = 0; al < 3; ++al) {
            double2 Pm[3];
            for (int s = 0; s < 3; ++s) {
                if (CUBIC) {
                    Pm[s] = S[al][s];
                } else {
                    double2 acc = cscale(P.Mmix[s * 3], S[al][0]);
                    acc = cfma(P.Mmix[s * 3 + 1], S[al][1], acc);
                    Pm[s] = cfma(P.Mmix[s * 3 + 2], S[al][2], acc);
                }
            }
            const double2 u = cadd(Pm[0], Pm[1]), v = csub(Pm[0], Pm[1]);
            Fo[0][al] = cadd(u, Pm[2]);
            Fo[1][al] = csub(u, Pm[2]);
            Fo[2][al] = cadd(v, Pm[2]);
            Fo[3][al] = csub(v, Pm[2]);
            Fo[4][al] = Pm[0];
        }
    }

    // Outputs of the thread's column from plane k to the end of the chunk in FP64, from x itself:
    // the first node whose values leave the integer path's range hands its column over.  Rare, so
    // its speed does not matter; after the march and not inlined, so that it costs the march no
    // registers.  Returns the column's part of Re<x, y>.
    static __host__ __device__ PC_FIX_COLD double slow_column(const Ctx& c, int k, int off0, int off1) {
        const CellGeom& G = *c.G;
        double dot = 0.0;
        for (; k < c.k0 + c.tz; ++k) {
            const int off = (k & 1) ? off1 : off0;
            const int i0 = (k + c.p13) & 1, j0 = (k + c.p12 + c.p13) & 1;
            const int a = G.full ? (off % G.N - i0) >> 1 : off % G.X, b = G.full ? (off / G.N - j0) >> 1 : off / G.X;
            const int64_t at = (int64_t)k * G.plane + off;
            PC_IDX(at, G.vstr);
            double2 F[5][3], own[3], g[4][3];
            slow_flux(c, a, b, k, F);
            for (int al = 0; al < 3; ++al) own[al] = F[4][al];
            for (int l = 0; l < 4; ++l) {
                const int s2 = (l < 2) ? 1 : -1, s3 = (l & 1) ? -1 : 1;
                int w[3];
                const int na = wrap1(a + i0, G.X, w[0]), nb = wrap1(b + j0 + ((s2 - 1) >> 1), G.Y, w[1]),
                          nk = wrap1(k + s3, G.Z, w[2]);
                slow_flux(c, na, nb, nk, F);
                double2 ph = cmk(1.0, 0.0);
                for (int d = 0; d < 3; ++d)
                    if (w[d] != 0) ph = cmul(ph, cmk(c.kph[d][0], w[d] < 0 ? -c.kph[d][1] : c.kph[d][1]));
                for (int al = 0; al < 3; ++al) g[l][al] = (w[0] | w[1] | w[2]) ? cmul(F[l][al], ph) : F[l][al];
            }
            double rho;
            if (MATK == 0) rho = c.F->P.rho[static_cast<const uint8_t*>(c.mat)[at] != 0 ? 1 : 0];
            else if (MATK == 1)
                rho = c.F->P.rho[0] + (double)static_cast<const float*>(c.mat)[at] * (c.F->P.rho[1] - c.F->P.rho[0]);
            else rho = static_cast<const double*>(c.mat)[21LL * G.vstr + at];
            for (int al = 0; al < 3; ++al) {
                const double2 xv = c.x[(int64_t)al * G.vstr + at];
                double2 w = cfma(-4.0, own[al], cadd(cadd(g[0][al], g[1][al]), cadd(g[2][al], g[3][al])));
                w = cfma(-(c.shift * rho), xv, w);
                c.y[(int64_t)al * G.vstr + at] = w;
                dot = cdotre(xv, w, dot);
            }
        }
        return dot;
    }
};

}  // namespace pc
