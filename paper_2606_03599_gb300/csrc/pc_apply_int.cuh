// Complex128 stencil apply on the integer pipe: y = (A - shift M) x with the FP64 operations of the stencil
// done on 64-bit integers with an exponent each (pc_wide.cuh).
//
// GB300 issues 2 FP64 lanes per clock and SM and 64 of 64-bit integer additions, so even written out as
// alignment, addition and normalisation an FP64 operation costs a fraction of its instruction.  Real and
// imaginary parts, components, strains, stresses and stiffness entries all keep exponents of their own: what
// is not added never shares a unit, so a small part, a small component or a soft phase is as accurate next to
// a large one as in FP64.  Errors, against FP64's 2^-53 of the result of every operation:
//   x           53 bits and 6 below them; the five values of a difference sum (one component, one part) are cut
//               at 2^-59 of the largest, and the sums themselves are exact
//   strain      normal exact, shear cut at 2^-59 of the larger component's x; a difference that vanishes
//               does not count (a uniform component leaves the other's bits alone)
//   stress      products at 2^-57, their sums cut at 2^-58 of the largest product
//   flux        stresses cut at 2^-54 to 2^-57 of the largest, their sums exact
//   output      sums of fluxes of one unit exact (others cut at that of the largest), one rounding to FP64, the
//               shift term by an FMA
// Against extended precision the result is 5e-17 off on broad-band vectors (FP64: 1.1e-16) and 3e-16 on long
// waves at N = 48 (FP64: 2e-15).  One exponent shared by a node's six reals took two thirds of the time and left
// 1e-13 of a transverse wave along an axis in steel, 1e-9 in a gel, 2e-8 of a strain next to a uniform
// displacement 1e8 times as large.
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
// Measured (one GB300, shift on, against the two-pass FP64 kernels): N = 48, 64 block vectors, one phase fully
// anisotropic 0.353 / 0.667 ms, both isotropic 0.286 ms; N = 60 FCC sub-pixel material, four blocks 0.137 / 0.195 ms; N = 64 nodewise
// material, full space 0.157 / 0.146 ms, which is why nodewise materials take it only where the autotuner finds
// it faster.  Bound by the integer instruction stream (16 warps per SM): a product and its place in a sum are ten
// instructions, half of them at half rate.  (Nine products instead of 36 in warps whose nodes are orthotropic pay
// for phase ids; for fractions and nodewise tables the second copy of the loop cost more than it saved: 169 and
// 144 us.)
//
// Infinities, NaN and nodes whose values are all below 2^-943 (their products with the Bloch phase round as
// subnormals, and FP64's order of operations counts) mark their node; a column is handed to FP64 (slow_column)
// from the first output that depends on a marked node.
#pragma once

#include <math.h>
#include <stdint.h>
#include <string.h>

#include "pc_apply_cells.cuh"
#include "pc_apply_tile.cuh"  // PC_IDX
#include "pc_complex.cuh"
#include "pc_internal.h"
#include "pc_wide.cuh"

#if defined(__CUDACC__)
#define PC_FIX_COLD __noinline__
#else
#define PC_FIX_COLD
#endif

namespace pc {

struct FixParams {
    StencilParams<double> P;  // FP64 tables: density, slow_column
    WideEntry c[2][21];       // MATK 0: phase tables
    double c0[21], dc[21];    // MATK 1: C_0 and C_1 - C_0
    WideEntry mix[9];         // lattice mixing (general lattices)
};

PC_HD int fix_upper(int p, int r) { return p <= r ? p * 6 - p * (p - 1) / 2 + (r - p) : r * 6 - r * (r - 1) / 2 + (p - r); }

// Tables of one launch; false when an entry is not finite.
inline bool make_fix_params(FixParams& F, const StencilParams<double>& P, bool cubic, int matkind) {
    memset(&F, 0, sizeof(F));
    F.P = P;
    bool ok = true;
    if (matkind != 2)
        for (int i = 0; i < 6; ++i)
            for (int j = i; j < 6; ++j) {
                const int q = fix_upper(i, j);
                for (int p = 0; p < 2; ++p) {
                    ok = ok && isfinite(P.C[p][i * 6 + j]);
                    F.c[p][q] = wide_entry(P.C[p][i * 6 + j]);
                }
                F.c0[q] = P.C[0][i * 6 + j];
                F.dc[q] = P.C[1][i * 6 + j] - P.C[0][i * 6 + j];
                ok = ok && isfinite(F.dc[q]);
            }
    if (!cubic)
        for (int e = 0; e < 9; ++e) {
            ok = ok && isfinite(P.Mmix[e]);
            F.mix[e] = wide_entry(P.Mmix[e]);
        }
    return ok;
}

// MATK: 0 = phase ids, 1 = inclusion fraction, 2 = nodewise material (as SplitApply).
// NP: parts (real, imaginary) of a cell in one thread; they meet in the Bloch phase only.  NP = 2 computes
// addresses and node-dependent stiffness once for both and is the form of launches that fill the GPU (N = 48, 64
// block vectors: 340 us, 379 us with NP = 1 in the same run).  NP = 1, two adjacent lanes per cell, halves a
// thread's chain of dependent instructions: the form of small launches, which wait for that chain (N = 8, one block
// vector: 16.6 us, 24.8 us with NP = 2).  The results are the same.
template <bool CUBIC, int MATK, int NP>
struct FixApply {
    struct Shared {
        int64_t* xs;   // [2 parts][3 slots][3][kCells]
        int64_t* fs;   // [12][2][kCells]: F_l of component c at l * 3 + c, in units of 2^fe
        double* raw;   // [3][kCells][2]: the next plane of x, as read
        double2* ph;   // [27] Bloch phases of the wraps (wa, wb, wk)
        WideEntry* c;  // [2][21]
        int* xe;       // [3 slots][3][kCells]: units of the two parts, 16 bits each
        int* fe;       // [3][kCells]
    };
    static constexpr int kRow = 2 * kCells;  // stride of one component's two arrays
    static constexpr size_t shared_bytes() {
        return (size_t)kCells * (16 * (9 + 12 + 3) + 4 * (9 + 3)) + 16 * 27 + sizeof(WideEntry) * 42;
    }
    static PC_HD void carve(Shared& sh, unsigned char* p) {
        sh.xs = reinterpret_cast<int64_t*>(p);
        sh.fs = sh.xs + 9 * kRow;
        sh.raw = reinterpret_cast<double*>(sh.fs + 12 * kRow);
        sh.ph = reinterpret_cast<double2*>(sh.raw + 3 * kRow);
        sh.c = reinterpret_cast<WideEntry*>(sh.ph + 27);
        sh.xe = reinterpret_cast<int*>(sh.c + 42);
        sh.fe = sh.xe + 9 * kCells;
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
        int64_t pv[3][NP], cv[3][NP];  // y(kf - 1) and y(kf) so far, with their units
        int pe[3][NP], ce[3][NP];
        int ks;  // first output plane left to slow_column
        double xo[3][NP];
        double dot;
    };

    static PC_HD int wrap1(int v, int n, int& w) { return cell_wrap(v, n, w); }

    // OR over the two parts of a cell (NP = 1: the neighbouring lane's, which takes every branch alike).
#if defined(__CUDA_ARCH__)
    static __device__ unsigned pair() { return 3u << (threadIdx.x & 30); }
#endif
    static PC_HD int pair_or(int v) {
#if defined(__CUDA_ARCH__)
        if (NP == 1) v |= __shfl_xor_sync(pair(), v, 1);
#endif
        return v;
    }

    // a cell's parts of x as read: one 16-byte access, or 8 bytes of it
    static PC_HD void get(const double* p, double* v) {
        if (NP == 2) {
            const double2 t = *reinterpret_cast<const double2*>(p);
            v[0] = t.x;
            v[NP - 1] = t.y;
        } else {
            v[0] = *p;
        }
    }
    static PC_HD int unit_of(const int* p, int part) { return reinterpret_cast<const int16_t*>(p)[part]; }

    // a cell's units: both, or the part's own 16 bits
    static PC_HD void get_units(const int* p, int part, int* u) {
        if (NP == 2) {
            const int w = *p;
            u[0] = (int16_t)w;
            u[NP - 1] = w >> 16;
        } else {
            u[0] = reinterpret_cast<const int16_t*>(p)[part];
        }
    }
    static PC_HD void put_units(int* p, int part, const int* u) {
        if (NP == 2) *p = (int)((uint32_t)u[NP - 1] << 16 | ((uint32_t)u[0] & 0xffffu));
        else reinterpret_cast<int16_t*>(p)[part] = (int16_t)u[0];
    }

    static PC_HD void init(const Ctx& c, int cell, int part, Regs& r) {
        cell_init(*c.G, c.a0, c.b0, c.p12, c.p13, cell, r);
        if (NP == 1) r.half = part;
        r.ks = 1 << 30;
#pragma unroll
        for (int a = 0; a < 3; ++a)
#pragma unroll
            for (int i = 0; i < NP; ++i) {
                r.pv[a][i] = r.cv[a][i] = 0;
                r.pe[a][i] = r.ce[a][i] = kWideZero;
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
        int64_t o[3][NP];
        int u[3][NP];
        int has = 0;  // 1: infinities or NaN, 2: values of 2^-943 or more, 4: values other than zero
#pragma unroll
        for (int a = 0; a < 3; ++a)
#pragma unroll
            for (int i = 0; i < NP; ++i) {
                o[a][i] = wide_from_double(v[a][i], 6, u[a][i]);
                has |= u[a][i] == kWideSpecial ? 1 : u[a][i] >= 80 - 1075 - 6 ? 2 : u[a][i] == kWideZero ? 0 : 4;
            }
        has = pair_or(has);
        if (has == 4 || (has & 1)) {  // all of the node's units: its readers look at one component
#pragma unroll
            for (int a = 0; a < 3; ++a)
#pragma unroll
                for (int i = 0; i < NP; ++i) u[a][i] = kWideSpecial;
        }
        int64_t* xs = sh.xs + (r.part() * 9 + sl * 3) * kCells + r.own[Q];
        int* xe = sh.xe + sl * 3 * kCells + r.own[Q];
#pragma unroll
        for (int a = 0; a < 3; ++a) {
#pragma unroll
            for (int i = 0; i < NP; ++i) xs[(a + 9 * i) * kCells] = o[a][i];
            put_units(xe + a * kCells, r.part(), u[a]);
        }
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

    // t = C e of one part with the phase table C; t in units of 2^tu, a product below 2^60.
    template <bool ORTHO>
    static PC_HD void stress(const WideEntry* C, const WideHalf* e, const int* eu, int64_t* t, int* tu) {
#pragma unroll
        for (int p = 0; p < 6; ++p) {
            if (ORTHO && p >= 3) {
                const WideEntry cc = C[fix_upper(p, p)];
                t[p] = wide_mul(e[p], cc);
                tu[p] = eu[p] + cc.u + 64;
                continue;
            }
            constexpr int n = ORTHO ? 3 : 6;
            int64_t m[n];
            int u[n], U = 2 * kWideZero;
#pragma unroll
            for (int v = 0; v < n; ++v) {
                const WideEntry cc = C[fix_upper(p, v)];
                m[v] = wide_mul(e[v], cc);
                u[v] = eu[v] + cc.u;
                U = imax(U, u[v]);
            }
            t[p] = 0;
#pragma unroll
            for (int v = 0; v < n; ++v) t[p] += wide_shr(m[v], U - u[v]);
            tu[p] = U + 64;
        }
    }

    // Strain of one part from the staged planes.  at: the cells of the four neighbours and of the node itself,
    // slot * 3 * kCells + cell.
    static PC_HD void strain(const Ctx& c, const Shared& sh, const int (&at)[5], int part, WideHalf* e, int* eu) {
        wide_strain<CUBIC>(
            c.F->mix,
            [&](int a, int64_t* x, int* u) {
#pragma unroll
                for (int l = 0; l < 5; ++l) {
                    u[l] = unit_of(sh.xe + at[l] + a * kCells, part);
                    x[l] = sh.xs[at[l] + (a + 9 * part) * kCells];
                }
            },
            e, eu);
    }

    // Fluxes of one part from its stresses; -4 P_0 into y(kf).  Stresses are cut `pad` bits below their unit, so that
    // four fluxes and 4 P_0 sum to less than 2^63: rows of one product and of three (cubic lattice, orthotropic: 32
    // products, pad 3), of six (96, pad 4), or mixed (48, pad 3).
    static PC_HD void spread(const Ctx& c, Shared& sh, Regs& r, int own, int i, int part, int64_t* t, int* tu, int pad) {
        if (!CUBIC) {
#pragma unroll
            for (int p = 0; p < 6; ++p) t[p] = wide_norm(t[p], tu[p]);
            pad = 3;
        }
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            constexpr int voigt[3][3] = {{0, 5, 4}, {5, 1, 3}, {4, 3, 2}};
            int64_t P[3] = {t[voigt[a][0]], t[voigt[a][1]], t[voigt[a][2]]};
            int u[3] = {tu[voigt[a][0]], tu[voigt[a][1]], tu[voigt[a][2]]};
            if (!CUBIC) wide_mix3(c.F->mix, P, u, true);
            const int fu = imax(imax(u[0], u[1]), u[2]) + pad;
#pragma unroll
            for (int s = 0; s < 3; ++s) P[s] = wide_shr(P[s], fu - u[s]);
            const int64_t g = P[0] + P[1], h = P[0] - P[1];
            int64_t* f = sh.fs + a * kRow + part * kCells + own;
            f[0] = g + P[2];
            f[3 * kRow] = g - P[2];
            f[6 * kRow] = h + P[2];
            f[9 * kRow] = h - P[2];
            reinterpret_cast<int16_t*>(sh.fe + a * kCells + own)[part] = (int16_t)fu;
            if (r.flags & 4) {
                const int m = imax(r.ce[a][i], fu);
                r.cv[a][i] = wide_shr(r.cv[a][i], m - r.ce[a][i]) - 4 * wide_shr(P[0], m - fu);
                r.ce[a][i] = m;
            }
        }
    }

    // Stiffness entry (p, v) of a node with its own: blended in FP64 as the FP64 kernels do, or its table's.
    static PC_HD WideEntry node_entry(const Ctx& c, float theta, const double* md, int q) {
        if (MATK == 1) return wide_entry(fma((double)theta, c.F->dc[q], c.F->c0[q]));
        return wide_entry(md[(int64_t)q * c.G->vstr]);
    }

    // Fluxes of plane kf (parity Q) at the thread's column.  sm, sc, sp: slots of planes kf - 1, kf, kf + 1.
    // The parts one after the other: together they spill.
    template <int Q>
    static PC_HD void flux(const Ctx& c, Shared& sh, Regs& r, int kf, int sm, int sc, int sp) {
        const CellGeom& G = *c.G;
        constexpr int n = kCells;
        if (!((r.flags >> Q) & 1)) return;
        const int own = r.own[Q], part = r.part(), n0 = r.nb[Q] & 0xffff, n1 = r.nb[Q] >> 16;
        PC_IDX(n0, G.ncell);
        PC_IDX(n1, G.ncell);
        const int at[5] = {sm * 3 * n + n0, sp * 3 * n + n0, sm * 3 * n + n1, sp * 3 * n + n1, sc * 3 * n + own};
        {
            int U = 0;
#pragma unroll
            for (int l = 0; l < 5; ++l) U = imax(U, unit_of(sh.xe + at[l], part));
            if (U >= kWideSpecial) {
#pragma unroll
                for (int i = 0; i < NP; ++i) reinterpret_cast<int16_t*>(sh.fe + own)[part + i] = kWideSpecial;
                r.ce[0][0] = kWideSpecial;
                return;
            }
        }
        if (MATK == 0) {
            const int ph = r.mcur != 0 ? 1 : 0;
            const WideEntry* C = sh.c + 21 * ph;
            // every node of the warp orthotropic: normal block and shear diagonal only (the same bits as with the zeros)
            const bool ortho = warp_all(c.F->P.ortho[ph] != 0);
            const int pad = c.F->P.ortho[ph] != 0 ? 3 : 4;
            // a loop, with y(kf) of the part at hand in the first place: unrolled, the parts' instructions are
            // interleaved and their registers spill
#pragma unroll 1
            for (int i = 0; i < NP; ++i) {
                WideHalf e[6];
                int64_t t[6];
                int eu[6], tu[6];
                strain(c, sh, at, part + i, e, eu);
                if (ortho) stress<true>(C, e, eu, t, tu);
                else stress<false>(C, e, eu, t, tu);
                spread(c, sh, r, own, 0, part + i, t, tu, pad);
                if (NP == 2) {
#pragma unroll
                    for (int a = 0; a < 3; ++a) {
                        const int64_t v = r.cv[a][0];
                        const int u = r.ce[a][0];
                        r.cv[a][0] = r.cv[a][NP - 1];
                        r.ce[a][0] = r.ce[a][NP - 1];
                        r.cv[a][NP - 1] = v;
                        r.ce[a][NP - 1] = u;
                    }
                }
            }
            return;
        }
        WideHalf e[NP][6];
        int64_t t[NP][6];
        int eu[NP][6], tu[NP][6];
#pragma unroll
        for (int i = 0; i < NP; ++i) {
            strain(c, sh, at, part + i, e[i], eu[i]);
#pragma unroll
            for (int p = 0; p < 6; ++p) {
                t[i][p] = 0;
                tu[i][p] = 2 * kWideZero;
            }
        }
        const double* md = nullptr;
        if (MATK == 2) {
            int wk;
            md = static_cast<const double*>(c.mat) + wrap1(kf, G.Z, wk) * G.plane + r.off[Q];
        }
        const float theta = MATK == 1 ? mat_theta(r.mcur) : 0.f;
        auto add = [&](int i, int p, int64_t m, int u) {
            const int U = imax(tu[i][p], u);
            t[i][p] = wide_shr(t[i][p], U - tu[i][p]) + wide_shr(m, U - u);
            tu[i][p] = U;
        };
#pragma unroll
        for (int p = 0; p < 6; ++p)
#pragma unroll
            for (int v = p; v < 6; ++v) {
                const WideEntry cc = node_entry(c, theta, md, fix_upper(p, v));
#pragma unroll
                for (int i = 0; i < NP; ++i) {
                    add(i, p, wide_mul(e[i][v], cc), eu[i][v] + cc.u);
                    if (v != p) add(i, v, wide_mul(e[i][p], cc), eu[i][p] + cc.u);
                }
            }
#pragma unroll
        for (int i = 0; i < NP; ++i) {
#pragma unroll
            for (int p = 0; p < 6; ++p) tu[i][p] += 64;
            spread(c, sh, r, own, i, part + i, t[i], tu[i], 4);
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
        const int64_t *a0 = sh.fs + r.part() * kCells + c0, *a1 = sh.fs + r.part() * kCells + c1;
        int f0[3][NP], f1[3][NP];
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            get_units(sh.fe + a * kCells + c0, r.part(), f0[a]);
            get_units(sh.fe + a * kCells + c1, r.part(), f1[a]);
        }
        if (k >= c.k0) {
            const int at = k * G.plane + r.off[1 - Q];
            if (imax(r.pe[0][0], imax(f0[0][0], f1[0][0])) >= kWideSpecial && r.ks > k) r.ks = k;
            if (k < r.ks) {
                const double sr = c.shift * density(c, r.mprev, at);
#pragma unroll
                for (int a = 0; a < 3; ++a) {
                    double w[NP];
#pragma unroll
                    for (int i = 0; i < NP; ++i) {
                        const int E = imax(r.pe[a][i], imax(f0[a][i], f1[a][i]));
                        w[i] = wide_to_double(wide_shr(r.pv[a][i], E - r.pe[a][i]) + 
                                                  wide_shr(a0[a * kRow + i * kCells], E - f0[a][i]) +
                                                  wide_shr(a1[(6 + a) * kRow + i * kCells], E - f1[a][i]),
                                              E);
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
#pragma unroll
        for (int a = 0; a < 3; ++a) {
#pragma unroll
            for (int i = 0; i < NP; ++i) {
                const int E = imax(f0[a][i], f1[a][i]);
                r.pv[a][i] = r.cv[a][i];
                r.pe[a][i] = r.ce[a][i];
                r.cv[a][i] = wide_shr(a0[(3 + a) * kRow + i * kCells], E - f0[a][i]) +
                             wide_shr(a1[(9 + a) * kRow + i * kCells], E - f1[a][i]);
                r.ce[a][i] = E;
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
