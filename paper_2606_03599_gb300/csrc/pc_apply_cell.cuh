// Complex64 stencil apply with one cell per thread (tiles and march of pc_apply_cells.cuh), every layout
// and even grid size.
//
// Bound: memory (49 bytes per node) as an ideal, in fact the latencies of shared memory and of the two
// barriers per plane.  The plane-pipelined kernel keeps two flux rows and their neighbour sets in a
// thread's registers (167 of them, one CTA of 11 warps per SM); here a thread has one node's fluxes and
// reads its neighbours from shared memory, so 80 registers and 48 KB serve a CTA of 256 threads and three
// of them share an SM.  (Four CTAs at 64 registers spill and run no faster.)  The halo columns cost a third
// more threads.  A cell's three components lie in one 16-byte and one 8-byte word: a third fewer shared
// accesses than three 8-byte words.
//
// Measured (one GB300, this kernel against the plane-pipelined one, or the TMA tile kernel for the full
// space): N = 48, 64 block vectors 51 / 84 us; N = 60, 64: 120 / 203 us; N = 128, 8: 102 / 110 us; N = 48,
// one block vector 11 / 30 us; N = 96, full space 32 / 80 us.
//
// A plane's x goes straight from global memory to its ring slot (asynchronous copies that arrive on the
// slot's mbarrier); a wrapped cell's thread multiplies its three values by the Bloch phase in place.
#pragma once

#include <string.h>

#include "pc_apply_cells.cuh"
#include "pc_apply_pipe.cuh"
#include "pc_internal.h"

namespace pc {

template <bool CUBIC, int MATK>
struct CellApply {
    using C = float2;
    static constexpr int NS = 4;  // ring: planes kf - 1, kf, kf + 1 and the one in flight
    // a cell's three components: one 16-byte and one 8-byte access
    struct Shared {
        float4* x4;  // [NS][kCells]: components 0 and 1 of x
        C* x2;       // [NS][kCells]: component 2
        float4* f4;  // [4][kCells]: F_l
        C* f2;
        C* ph;       // [27] Bloch phases of the wraps
    };
    static constexpr size_t shared_bytes() { return sizeof(C) * ((size_t)kCells * (3 * NS + 12) + 28); }
    static PC_HD void carve(Shared& sh, float4* p) {
        sh.x4 = p;
        sh.f4 = sh.x4 + NS * kCells;
        sh.x2 = reinterpret_cast<C*>(sh.f4 + 4 * kCells);
        sh.f2 = sh.x2 + NS * kCells;
        sh.ph = sh.f2 + 4 * kCells;
    }
    static PC_HD void get3(const float4* p4, const C* p2, C* v) {
        const float4 u = *p4;
        v[0] = cmk(u.x, u.y);
        v[1] = cmk(u.z, u.w);
        v[2] = *p2;
    }
    static PC_HD void put3(float4* p4, C* p2, const C* v) {
        *p4 = make_float4(v[0].x, v[0].y, v[1].x, v[1].y);
        *p2 = v[2];
    }
    struct Ctx {
        const StencilParams<float>* P;
        const CellGeom* G;
        const float (*kph)[2];
        const C* x;
        C* y;
        const void* mat;
        float shift;
        bool dot;
        int a0, b0, k0, tz, p12, p13;
    };
    struct Regs : CellMap {
        int mcur, mnext;  // material of planes kf, kf + 1 (phase id, or the fraction's bits)
        C pv[3], cv[3];     // y(kf - 1) and y(kf) so far
        float dot;
    };

    static PC_HD void init(const Ctx& c, int tid, Regs& r) {
        cell_init(*c.G, c.a0, c.b0, c.p12, c.p13, tid, r);
        r.mcur = r.mnext = 0;
        r.dot = 0.f;
        for (int a = 0; a < 3; ++a) r.pv[a] = r.cv[a] = czero(0.f);
    }

    static PC_HD void load_tables(const Ctx& c, Shared& sh, int tid, int nthr) {
        for (int i = tid; i < 27; i += nthr) {
            const int w[3] = {i % 3 - 1, (i / 3) % 3 - 1, i / 9 - 1};
            C e = cmk(1.f, 0.f);
            for (int l = 0; l < 3; ++l)
                if (w[l] != 0) e = cmul(e, cmk(c.kph[l][0], w[l] < 0 ? -c.kph[l][1] : c.kph[l][1]));
            sh.ph[i] = e;
        }
    }

    // Q: parity of plane kp
    template <int Q>
    static PC_HD int node_at(const Ctx& c, const Regs& r, int kp) {
        int wk;
        const int at = cell_wrap(kp, c.G->Z, wk) * c.G->plane + r.off[Q];
        PC_IDX(at, c.G->vstr);
        return at;
    }

    // Start the copy of plane kp of x into the thread's cell of slot sl.
    template <int Q>
    static PC_HD void stage(const Ctx& c, Shared& sh, const Regs& r, int kp, int sl) {
        const CellGeom& G = *c.G;
        const C* s = c.x + node_at<Q>(c, r, kp);
        const int at = sl * kCells + r.own[Q];
        C* const d[3] = {reinterpret_cast<C*>(sh.x4 + at), reinterpret_cast<C*>(sh.x4 + at) + 1, sh.x2 + at};
        PC_IDX(r.own[Q], G.ncell);
#pragma unroll
        for (int a = 0; a < 3; ++a) {
#if defined(__CUDA_ARCH__)
            asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"((uint32_t)__cvta_generic_to_shared(d[a])),
                         "l"(s + (int64_t)a * G.vstr)
                         : "memory");
#else
            *d[a] = s[(int64_t)a * G.vstr];
#endif
        }
    }

    // The arrived plane kp of slot sl: Bloch phase of a wrapped cell, by its own thread.
    template <int Q>
    static PC_HD void settle(const Ctx& c, Shared& sh, const Regs& r, int kp, int sl) {
        const CellGeom& G = *c.G;
        int wk;
        cell_wrap(kp, G.Z, wk);
        const int w = r.wab[Q] + 9 * (wk + 1);
        if (w == 13) return;
        const int at = sl * kCells + r.own[Q];
        const C ph = sh.ph[w];
        C v[3];
        get3(sh.x4 + at, sh.x2 + at, v);
#pragma unroll
        for (int a = 0; a < 3; ++a) v[a] = cmul(v[a], ph);
        put3(sh.x4 + at, sh.x2 + at, v);
    }

    template <int Q>
    static PC_HD int read_mat(const Ctx& c, const Regs& r, int kp) {
        const int at = node_at<Q>(c, r, kp);
        if (MATK == 0) return static_cast<const uint8_t*>(c.mat)[at];
        return static_cast<const int*>(c.mat)[at];
    }
    static PC_HD float mat_value(int m) {
        if (MATK == 0) return (float)m;
#if defined(__CUDA_ARCH__)
        return __int_as_float(m);
#else
        float f;
        memcpy(&f, &m, 4);
        return f;
#endif
    }

    // Fluxes of plane kf (parity Q) at the thread's column; local and shift terms into y(kf).  sm, sc, sp:
    // slots of planes kf - 1, kf, kf + 1.
    template <int Q>
    static PC_HD void flux(const Ctx& c, Shared& sh, Regs& r, int sm, int sc, int sp) {
        const CellGeom& G = *c.G;
        const StencilParams<float>& P = *c.P;
        constexpr int n = kCells;
        if (!((r.flags >> Q) & 1)) return;
        const int c0 = r.nb[Q] & 0xffff, c1 = r.nb[Q] >> 16;
        PC_IDX(c0, G.ncell);
        PC_IDX(c1, G.ncell);
        const int am = sm * n, ac = sc * n + r.own[Q], ap = sp * n;
        C n0[3], n1[3], n2[3], n3[3], xo[3], F[4][3], loc[3];
        get3(sh.x4 + am + c0, sh.x2 + am + c0, n0);
        get3(sh.x4 + ap + c0, sh.x2 + ap + c0, n1);
        get3(sh.x4 + am + c1, sh.x2 + am + c1, n2);
        get3(sh.x4 + ap + c1, sh.x2 + ap + c1, n3);
        get3(sh.x4 + ac, sh.x2 + ac, xo);
        // differences first (own value zero from there on): sums of neighbours around 2 x would round away
        // what is left after the own value is taken off (error against 64 bits 1.1e-7, not 4e-7)
        C zero[3];
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            n0[a] = csub(n0[a], xo[a]);
            n1[a] = csub(n1[a], xo[a]);
            n2[a] = csub(n2[a], xo[a]);
            n3[a] = csub(n3[a], xo[a]);
            zero[a] = czero(0.f);
        }
        const float mv = mat_value(r.mcur);
        PipeTile<CUBIC, MATK>::flux_node(P, mv, n0, n1, n2, n3, zero, F, loc);
#pragma unroll
        for (int l = 0; l < 4; ++l) put3(sh.f4 + l * n + r.own[Q], sh.f2 + l * n + r.own[Q], F[l]);
        if (r.flags & 4) {
            const float rho = (MATK == 0) ? (r.mcur != 0 ? P.rho[1] : P.rho[0]) : P.rho[0] + mv * (P.rho[1] - P.rho[0]);
            const float sr = -c.shift * rho;
#pragma unroll
            for (int a = 0; a < 3; ++a) r.cv[a] = cfma(sr, xo[a], csub(r.cv[a], loc[a]));
        }
    }

    // Step kf of parity Q: outputs y(kf - 1) (own x from slot sm for the inner product); y(kf + 1) starts with F_1, F_3.
    template <int Q>
    static PC_HD void gather(const Ctx& c, Shared& sh, Regs& r, int kf, int sm) {
        const CellGeom& G = *c.G;
        if (!(r.flags & 4)) return;
        constexpr int n = kCells;
        const int k = kf - 1;  // planes kf - 1 and kf + 1 share the offsets
        const int c0 = r.gn[1 - Q] & 0xffff, c1 = r.gn[1 - Q] >> 16;
        PC_IDX(c0, G.ncell);
        PC_IDX(c1, G.ncell);
        const float4 *a4 = sh.f4 + c0, *b4 = sh.f4 + c1;
        const C *a2 = sh.f2 + c0, *b2 = sh.f2 + c1;
        C u[3], v[3];
        if (k >= c.k0) {
            C* y = c.y + node_at<1 - Q>(c, r, k);
            get3(a4, a2, u);
            get3(b4 + 2 * n, b2 + 2 * n, v);
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                r.pv[a] = cadd(r.pv[a], cadd(u[a], v[a]));
                y[(int64_t)a * G.vstr] = r.pv[a];
            }
            if (c.dot) {
                get3(sh.x4 + sm * n + r.own[1 - Q], sh.x2 + sm * n + r.own[1 - Q], u);
#pragma unroll
                for (int a = 0; a < 3; ++a) r.dot = cdotre(u[a], r.pv[a], r.dot);
            }
        }
        get3(a4 + n, a2 + n, u);
        get3(b4 + 3 * n, b2 + 3 * n, v);
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            r.pv[a] = r.cv[a];
            r.cv[a] = cadd(u[a], v[a]);
        }
    }
};

}  // namespace pc
