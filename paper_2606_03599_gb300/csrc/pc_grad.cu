// Adjoint (Hellmann-Feynman) kernel: gradients of eigenvalues with respect to the
// nodewise stiffness and density.
//
// For an eigenpair A x = lambda M x with x^H M x = 1 and A = B C B^H (Eq.
// discrete_GEP_main), a change dC, dM of the nodewise material moves the
// eigenvalue by d lambda = x^H (B dC B^H - lambda dM) x = sum_i e_i^H dC_i e_i -
// lambda sum_i rho'_i |x(i)|^2 with e = B^H x the Voigt strain at node i.  Per
// node and per independent entry of the symmetric 6x6 stiffness (upper
// triangle, Voigt order [11,22,33,23,13,12]):
//     d lambda / d C_i[p][q] = Re(conj(e_p) e_q) * (2 if p != q else 1),
//     d lambda / d rho_i      = -lambda sum_alpha |x_alpha(i)|^2.
// The strain is evaluated exactly as in the apply kernel (Bloch-phased backward
// body-diagonal differences, reconstruction, lattice mixing, engineering shear).
//
// The work is FP64 arithmetic in form (about 220 operations per node and vector, 1.63 ms for 12
// vectors on 64^3 nodes when done so) against 48 bytes read, so it runs on the integer pipe like the
// apply (pc_apply_int.cuh): the five values a component's differences need become integers
// with one exponent, sums are exact, and the strain, scaled by sqrt(|w|), is split into limbs
// (pc_limb.cuh) whose products are summed over the vectors in integers; the running sums carry one
// exponent per node and turn into doubles once, after up to 32 vectors.  A node with values outside the exponent range is left to FP64.
//
// Measured (one GB300, N = 64 full space, 12 vectors): 0.44 ms, where the FP64 form took 1.63 ms; bound by
// the integer instructions, half of them the conversion of a node's 15 values (196 MB of DRAM traffic
// would take 0.03 ms).
#include <algorithm>
#include <cmath>
#include <cstdlib>

#include "pc_apply_int.cuh"
#include "pc_limb.cuh"
#include "pc_solver.h"

namespace pc {

namespace {

struct FixHalf {
    int hi, lo;  // c = hi 2^32 + lo, lo signed
};

PC_HD FixHalf fix_split(int64_t v) {
    FixHalf h;
    h.hi = (int)((v + 0x80000000LL) >> 32);
    h.lo = (int)(uint32_t)v;
    return h;
}
PC_HD longlong2 fix_ashr2(longlong2 v, int s) {
    longlong2 r;
    r.x = v.x >> s;
    r.y = v.y >> s;
    return r;
}
PC_HD int64_t fix_bits(double v) {
#if defined(__CUDA_ARCH__)
    return __double_as_longlong(v);
#else
    int64_t b;
    memcpy(&b, &v, 8);
    return b;
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

constexpr int kGradVecs = 32;  // vectors per launch: their limb products sum to less than 2^62
constexpr int kGradThreads = 128;
constexpr int kGradLow = 720;  // least biased exponent of the integer path: squares stay above FP64's smallest

struct GradVec {
    FixHalf s;     // sqrt(|w| scaleC) (times the lattice factor on a cubic lattice) = s 2^(ex - 62)
    int ex, neg;   // neg: w < 0
    double wC, wR; // w scaleC, -w lambda scaleR
};
struct GradParams {
    double Mmix[9];  // (A_hat^-1)_{s m} / (4 h_s)
    double ph[3][2];
    FixHalf mix[9], pi[3][2];  // the same in units of 2^(mex - 62) and 2^-62
    int mex;
    int X, Y, Z, N;  // quarter-grid extents
    int full, block;
    int plane, vstr;  // nodes per plane and component of the layout
    int nvec, all_slow;  // all_slow: a weight's scale is outside the exponents the sums allow for
    GradVec v[kGradVecs];
};

__device__ __forceinline__ int wrapg(int v, int n, int& w) {
    w = v < 0 ? -1 : (v >= n ? 1 : 0);
    return v - w * n;
}

// One node: block, quarter-grid coordinates, offset in its vector, backward neighbours and their wraps.
struct GradNode {
    int at, nb[4], wrap[4];  // wrap: (wa + 1) + 3 (wb + 1) + 9 (wk + 1), 13 = inside
};
__device__ __forceinline__ GradNode grad_node(const GradParams& P, int blk, int a, int b, int k) {
    GradNode r;
    const int p12 = blk >> 1, p13 = blk & 1;
    auto addr = [&](int aa, int bb, int kk) {
        const int i0 = (kk + p13) & 1, j0 = (kk + p12 + p13) & 1;
        return kk * P.plane + (P.full ? (2 * aa + i0) + P.N * (2 * bb + j0) : aa + P.X * bb);
    };
    r.at = addr(a, b, k);
    const int i0 = (k + p13) & 1, j0 = (k + p12 + p13) & 1;
#pragma unroll
    for (int l = 0; l < 4; ++l) {
        const int s2 = (l < 2) ? 1 : -1, s3 = (l & 1) ? -1 : 1;
        int wa, wb, wk;
        const int aa = wrapg(a + i0 - 1, P.X, wa), bb = wrapg(b + j0 - ((s2 + 1) >> 1), P.Y, wb), kk = wrapg(k - s3, P.Z, wk);
        r.nb[l] = addr(aa, bb, kk);
        r.wrap[l] = (wa + 1) + 3 * (wb + 1) + 9 * (wk + 1);
    }
    return r;
}

__device__ __forceinline__ double2 grad_phase(const GradParams& P, int wrap) {
    double2 e = make_double2(1.0, 0.0);
    const int w[3] = {wrap % 3 - 1, (wrap / 3) % 3 - 1, wrap / 9 - 1};
    for (int s = 0; s < 3; ++s)
        if (w[s] != 0) e = cmul(e, make_double2(P.ph[s][0], w[s] < 0 ? -P.ph[s][1] : P.ph[s][1]));
    return e;
}

// A node in FP64, added to the outputs: values the integer path does not take.  Never inlined (rare).
__device__ __noinline__ void grad_slow(const GradParams& P, const double2* __restrict__ X, const GradNode nd, int64_t l,
                                       double* __restrict__ dC, double* __restrict__ drho, int64_t n_full) {
    const int64_t m = P.vstr;
    double g21[21];
    for (int q = 0; q < 21; ++q) g21[q] = 0.0;
    double gr = 0.0;
    for (int v = 0; v < P.nvec; ++v) {
        const double2* x = X + (int64_t)v * 3 * m;
        double2 H[3][3];
        double xx = 0.0;
        for (int al = 0; al < 3; ++al) {
            const double2 x0 = x[al * m + nd.at];
            xx += x0.x * x0.x + x0.y * x0.y;
            double2 g[4];
            for (int ll = 0; ll < 4; ++ll) {
                double2 nv = x[al * m + nd.nb[ll]];
                if (nd.wrap[ll] != 13) nv = cmul(grad_phase(P, nd.wrap[ll]), nv);
                g[ll] = csub(nv, x0);
            }
            const double2 u = cadd(g[0], g[1]), vv = cadd(g[2], g[3]);
            H[0][al] = cadd(u, vv);
            H[1][al] = csub(u, vv);
            H[2][al] = cadd(csub(g[0], g[1]), csub(g[2], g[3]));
        }
        double2 G[3][3];  // G[m][alpha] = sum_s Mmix_{s m} H_{s alpha}  (the hat strain is i G)
        for (int mm = 0; mm < 3; ++mm)
            for (int al = 0; al < 3; ++al) {
                double2 acc = cscale(P.Mmix[0 * 3 + mm], H[0][al]);
                acc = cfma(P.Mmix[1 * 3 + mm], H[1][al], acc);
                G[mm][al] = cfma(P.Mmix[2 * 3 + mm], H[2][al], acc);
            }
        const double2 e[6] = {G[0][0], G[1][1], G[2][2], cadd(G[2][1], G[1][2]), cadd(G[2][0], G[0][2]),
                              cadd(G[1][0], G[0][1])};
        int q = 0;
        for (int p = 0; p < 6; ++p)
            for (int r = p; r < 6; ++r, ++q) {
                const double re = e[p].x * e[r].x + e[p].y * e[r].y;
                g21[q] += P.v[v].wC * (p == r ? re : 2.0 * re);
            }
        gr += P.v[v].wR * xx;
    }
    for (int q = 0; q < 21; ++q) dC[(int64_t)q * n_full + l] += g21[q];
    drho[l] += gr;
}

// One thread per node; loops over the vectors, so that each output entry has a single writer (no
// atomics, deterministic).  blockIdx.y: parity block of a full-space layout.
// Bounds: x < 2^57, phased values below sqrt(2) of it, sums H scaled up to 2^61, strain < 2^62 and as
// much after the products with s; limbs of 28 and 29 bits, so a vector adds at most 2^57 to a high sum
// and 2^58 to a middle one.
template <bool CUBIC>
__global__ void __launch_bounds__(kGradThreads, 3)
    eig_grad_kernel(const __grid_constant__ GradParams P, const double2* __restrict__ X, double* __restrict__ dC,
                    double* __restrict__ drho, int64_t n_full) {
    const int blk = P.full ? (int)blockIdx.y : P.block;
    const uint32_t nodes = (uint32_t)P.X * P.Y * P.Z;
    const uint32_t t = blockIdx.x * kGradThreads + threadIdx.x;
    if (t >= nodes) return;
    int a, b, k;
    split3(t, P.X, P.Y, a, b, k);
    const GradNode nd = grad_node(P, blk, a, b, k);
    int64_t l;  // full-grid index
    {
        const int p12 = blk >> 1, p13 = blk & 1;
        l = (2 * a + ((k + p13) & 1)) + (int64_t)P.N * ((2 * b + ((k + p12 + p13) & 1)) + (int64_t)P.N * k);
    }
    bool slow = P.all_slow != 0;
    double gr = 0.0;
    int64_t hi[21], mid[21];
#pragma unroll
    for (int q = 0; q < 21; ++q) hi[q] = mid[q] = 0;
    int A = -100000;  // exponent of the limbs' unit
    for (int v = 0; v < P.nvec; ++v) {
        const GradVec& V = P.v[v];
        const double2* __restrict__ x = X + (int64_t)v * 3 * P.vstr;
        longlong2 H[3][3];
        int E[3], any = 0;
        double xx = 0.0;
        bool bad = false;
#pragma unroll
        for (int al = 0; al < 3; ++al) {
            const double2* xc = x + (int64_t)al * P.vstr;
            double2 xv[5];
#pragma unroll
            for (int ll = 0; ll < 4; ++ll) xv[ll] = xc[nd.nb[ll]];
            xv[4] = xc[nd.at];
            int top = 0;
#pragma unroll
            for (int ll = 0; ll < 5; ++ll) top = fix_high(xv[ll], top);
            xx = cdotre(xv[4], xv[4], xx);
            E[al] = top >> 20;
            if (E[al] < kGradLow || E[al] > kLimbHigh) {
                // a component of zeros counts as such; anything else goes to FP64
                int64_t low = 0;
#pragma unroll
                for (int ll = 0; ll < 5; ++ll) low |= fix_bits(xv[ll].x) | fix_bits(xv[ll].y);
                bad = bad || (low & 0x7fffffffffffffffLL) != 0;
                E[al] = kGradLow;
            }
            longlong2 n[5];
#pragma unroll
            for (int ll = 0; ll < 5; ++ll) {
                n[ll].x = fix_from_double(xv[ll].x, E[al], 4);
                n[ll].y = fix_from_double(xv[ll].y, E[al], 4);
            }
#pragma unroll
            for (int ll = 0; ll < 4; ++ll) {
                int w = nd.wrap[ll];
                if (w != 13) {
#pragma unroll 1
                    for (int d = 0; d < 3; ++d) {
                        const int wd = w % 3 - 1;
                        w /= 3;
                        if (wd == 0) continue;
                        const FixHalf c = P.pi[d][0], sn = P.pi[d][1];
                        FixHalf sp, sm;
                        sp.hi = wd < 0 ? -sn.hi : sn.hi;
                        sp.lo = wd < 0 ? -sn.lo : sn.lo;
                        sm.hi = -sp.hi;
                        sm.lo = -sp.lo;
                        const FixHalf zx = fix_split(n[ll].x), zy = fix_split(n[ll].y);
                        int64_t hx = 0, mx = 0, hy = 0, my = 0;
                        fix_mac(hx, mx, zx, c);
                        fix_mac(hx, mx, zy, sm);
                        fix_mac(hy, my, zy, c);
                        fix_mac(hy, my, zx, sp);
                        n[ll].x = fix_sum(hx, mx, 2);
                        n[ll].y = fix_sum(hy, my, 2);
                    }
                }
            }
            const int64_t ux = n[0].x + n[1].x, uy = n[0].y + n[1].y, vx = n[2].x + n[3].x, vy = n[2].y + n[3].y;
            H[0][al].x = ux + vx - 4 * n[4].x;
            H[0][al].y = uy + vy - 4 * n[4].y;
            H[1][al].x = ux - vx;
            H[1][al].y = uy - vy;
            H[2][al].x = (n[0].x - n[1].x) + (n[2].x - n[3].x);
            H[2][al].y = (n[0].y - n[1].y) + (n[2].y - n[3].y);
            any |= top;
        }
        gr = fma(V.wR, xx, gr);
        slow = slow || bad;
        if (!bad && any != 0 && V.wC != 0.0) {
            const int Em = imax(imax(E[0], E[1]), E[2]);
            int bits = 0;
#pragma unroll
            for (int al = 0; al < 3; ++al) {
                const int d = imin(Em - E[al], 63);
#pragma unroll
                for (int s = 0; s < 3; ++s) {
                    H[s][al] = fix_ashr2(H[s][al], d);
                    bits |= (int)((H[s][al].x ^ (H[s][al].x >> 63)) >> 32) | (int)((H[s][al].y ^ (H[s][al].y >> 63)) >> 32);
                }
            }
            const int up = __clz(bits | 1) - 3;
#pragma unroll
            for (int s = 0; s < 3; ++s)
#pragma unroll
                for (int al = 0; al < 3; ++al) {
                    H[s][al].x <<= up;
                    H[s][al].y <<= up;
                }
            int u = Em - 1079 - up + V.ex;  // exponent of the strain's unit
            if (!CUBIC) {
                u += P.mex;
#pragma unroll
                for (int al = 0; al < 3; ++al) {
                    FixHalf hx[3], hy[3];
#pragma unroll
                    for (int s = 0; s < 3; ++s) {
                        hx[s] = fix_split(H[s][al].x);
                        hy[s] = fix_split(H[s][al].y);
                    }
#pragma unroll
                    for (int m = 0; m < 3; ++m) {
                        int64_t px = 0, qx = 0, py = 0, qy = 0;
#pragma unroll
                        for (int s = 0; s < 3; ++s) {
                            fix_mac(px, qx, hx[s], P.mix[s * 3 + m]);
                            fix_mac(py, qy, hy[s], P.mix[s * 3 + m]);
                        }
                        H[m][al].x = fix_sum(px, qx, 2);
                        H[m][al].y = fix_sum(py, qy, 2);
                    }
                }
            }
            longlong2 e[6];
            e[0] = H[0][0];
            e[1] = H[1][1];
            e[2] = H[2][2];
            e[3] = make_longlong2(H[2][1].x + H[1][2].x, H[2][1].y + H[1][2].y);
            e[4] = make_longlong2(H[2][0].x + H[0][2].x, H[2][0].y + H[0][2].y);
            e[5] = make_longlong2(H[1][0].x + H[0][1].x, H[1][0].y + H[0][1].y);
            bits = 0;
#pragma unroll
            for (int p = 0; p < 6; ++p) {
                const FixHalf ex = fix_split(e[p].x), ey = fix_split(e[p].y);
                int64_t h = 0, m = 0;
                fix_mac(h, m, ex, V.s);
                e[p].x = fix_sum(h, m, 2);
                h = m = 0;
                fix_mac(h, m, ey, V.s);
                e[p].y = fix_sum(h, m, 2);
                bits |= (int)((e[p].x ^ (e[p].x >> 63)) >> 32) | (int)((e[p].y ^ (e[p].y >> 63)) >> 32);
            }
            // common unit of the running sums: a larger strain scales them down
            const int need = u + imax(0, 7 - __clz(bits | 1));  // 57 bits: seven leading bits clear
            if (need > A) {
                const int d = imin(2 * (need - A), 63);
                if (d > 0 && A > -100000) {
#pragma unroll
                    for (int q = 0; q < 21; ++q) {
                        hi[q] >>= d;
                        mid[q] >>= d;
                    }
                }
                A = need;
            }
            const int sh = imin(A - u, 63);
            Limb lx[6], ly[6];
#pragma unroll
            for (int p = 0; p < 6; ++p) {
                const int64_t px = e[p].x >> sh, py = e[p].y >> sh;
                lx[p].hi = (int)((px + (1 << 28)) >> 29);
                lx[p].lo = ((int)px << 3) >> 3;
                ly[p].hi = (int)((py + (1 << 28)) >> 29);
                ly[p].lo = ((int)py << 3) >> 3;
            }
            const int sg = V.neg ? -1 : 0;
            int q = 0;
#pragma unroll
            for (int p = 0; p < 6; ++p) {
                Limb fx, fy;
                fx.hi = (lx[p].hi ^ sg) - sg;
                fx.lo = (lx[p].lo ^ sg) - sg;
                fy.hi = (ly[p].hi ^ sg) - sg;
                fy.lo = (ly[p].lo ^ sg) - sg;
#pragma unroll
                for (int r = p; r < 6; ++r, ++q) {
                    limb_mad(hi[q], fx.hi, lx[r].hi);
                    limb_mad(hi[q], fy.hi, ly[r].hi);
                    limb_mad(mid[q], fx.hi, lx[r].lo);
                    limb_mad(mid[q], fx.lo, lx[r].hi);
                    limb_mad(mid[q], fy.hi, ly[r].lo);
                    limb_mad(mid[q], fy.lo, ly[r].hi);
                }
            }
        }
        // the middle sums hold eight vectors: their upper part moves on
        if ((v & 7) == 7)
#pragma unroll
            for (int q = 0; q < 21; ++q) {
                hi[q] += mid[q] >> 29;
                mid[q] &= (1 << 29) - 1;
            }
    }
    if (slow) {
        grad_slow(P, X, nd, l, dC, drho, n_full);
        return;
    }
    int q = 0;
#pragma unroll
    for (int p = 0; p < 6; ++p)
#pragma unroll
        for (int r = p; r < 6; ++r, ++q) {
            const int64_t tt = hi[q] + ((mid[q] + (1 << 28)) >> 29);  // units of 2^(2 A + 58)
            const double d = __ll2double_rn(tt);
            if (tt != 0)
                dC[(int64_t)q * n_full + l] += __hiloint2double(
                    __double2hiint(d) + (2 * A + 58 + (p == r ? 0 : 1)) * (1 << 20), __double2loint(d));
        }
    drho[l] += gr;
}

}  // namespace

}  // namespace pc

using namespace pc;

extern "C" int pc_eig_grad(pc_grid* g, int block, int nvec, const void* X, const double* lambdas, const double* weights,
                           double* dC, double* drho, void* stream) {
    if (!g || (!X && nvec > 0) || !lambdas || !weights || !dC || !drho)
        return fail(PC_EINVAL, "pc_eig_grad: null argument");
    if (block < -1 || block > 3) return fail(PC_EINVAL, "pc_eig_grad: block must be -1..3");
    if (nvec < 0 || nvec > 4096) return fail(PC_EINVAL, "pc_eig_grad: nvec must be in 0..4096");
    if (!g->k.set) return fail(PC_ESTATE, "pc_eig_grad: call pc_set_k (or pc_eigs) first");
    if (nvec == 0) return PC_OK;
    for (int v = 0; v < nvec; ++v)
        if (!std::isfinite(lambdas[v]) || !std::isfinite(weights[v]))
            return fail(PC_EINVAL, "pc_eig_grad: non-finite eigenvalue or weight");
    const double q = g->N / 4.0;
    const double scaleC = 1.0 / (g->rho0 * g->L * g->L), scaleR = 1.0 / g->rho0;
    cudaStream_t s = (cudaStream_t)stream;
    for (int base = 0; base < nvec; base += kGradVecs) {
        GradParams P;
        P.nvec = std::min(nvec - base, kGradVecs);
        P.all_slow = 0;
        double ms = 0.0;
        for (int e = 0; e < 9; ++e) P.Mmix[e] = g->Ainv[e] * q;
        for (int i = 0; i < 3; ++i)
            ms = std::fmax(ms, std::fabs(P.Mmix[i]) + std::fabs(P.Mmix[3 + i]) + std::fabs(P.Mmix[6 + i]));
        std::frexp(ms, &P.mex);
        for (int e = 0; e < 9; ++e) P.mix[e] = fix_split(std::llrint(std::ldexp(P.Mmix[e], 62 - P.mex)));
        for (int l = 0; l < 3; ++l) {
            P.ph[l][0] = std::cos(g->k.phi[l]);
            P.ph[l][1] = std::sin(g->k.phi[l]);
            for (int c = 0; c < 2; ++c) P.pi[l][c] = fix_split(std::llrint(std::ldexp(P.ph[l][c], 62)));
        }
        P.N = g->N;
        P.full = block < 0 ? 1 : 0;
        P.block = block < 0 ? 0 : block;
        P.X = g->X;
        P.Y = g->Y;
        P.Z = g->Z;
        P.plane = P.full ? g->N * g->N : g->X * g->Y;
        P.vstr = P.plane * g->Z;
        for (int v = 0; v < P.nvec; ++v) {
            const double w = weights[base + v];
            GradVec& V = P.v[v];
            // extended precision: the root's rounding would enter every product twice
            const long double sq = sqrtl((long double)std::fabs(w) / ((long double)g->rho0 * g->L * g->L)) *
                                   (g->cubic ? (long double)q : 1.0L);
            V.neg = w < 0 ? 1 : 0;
            V.ex = 0;
            if (sq > 0) frexpl(sq, &V.ex);
            if (std::abs(V.ex) + std::abs(P.mex) > 60) P.all_slow = 1;
            V.s = fix_split(llrintl(ldexpl(sq, 62 - V.ex)));
            V.wC = w * scaleC;
            V.wR = -w * lambdas[base + v] * scaleR;
        }
        const int64_t nodes = (int64_t)P.X * P.Y * P.Z;
        const dim3 grid((unsigned)((nodes + kGradThreads - 1) / kGradThreads), P.full ? 4 : 1);
        const double2* Xb = static_cast<const double2*>(X) + (int64_t)base * 3 * P.vstr;
        if (g->cubic) eig_grad_kernel<true><<<grid, kGradThreads, 0, s>>>(P, Xb, dC, drho, g->n);
        else eig_grad_kernel<false><<<grid, kGradThreads, 0, s>>>(P, Xb, dC, drho, g->n);
        note_launch();
        PC_CUDA_TRY(cudaGetLastError());
    }
    return PC_OK;
}
