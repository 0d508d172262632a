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
// apply (pc_wide.cuh): real and imaginary parts, components, strains and each of the 21 sums have exponents of
// their own, so that a small strain's products are as accurate next to a large one's as in FP64.  The strain is
// scaled by sqrt(|w|) and normalised, its products are summed over up to 32 vectors in integers and turn into
// doubles once.  A node with infinities or NaN is left to FP64.
//
// Measured (one GB300, FP64 form / this one): N = 64 full space, 12 vectors 1.63 / 0.95 ms, one vector 0.183 / 0.143
// ms; N = 8, 12 vectors 138 / 85 us.  Bound by the integer instructions, about 1700 per node, vector and part (196 MB
// of DRAM traffic would take 0.03 ms).  (One exponent for a node's strains and sums took 0.44 ms and left nothing
// of a strain's square 1e-8 below another's.)
#include <algorithm>
#include <cmath>
#include <cstdlib>

#include "pc_complex.cuh"
#include "pc_solver.h"
#include "pc_wide.cuh"

namespace pc {

namespace {

constexpr int kGradVecs = 32;  // vectors per launch: the 64 products of their parts, four bits down, sum to 2^62 at most
constexpr int kGradThreads = 128;

struct GradVec {
    WideEntry s;    // sqrt(|w| scaleC) (times the lattice factor on a cubic lattice)
    int neg;        // w < 0
    double wC, wR;  // w scaleC, -w lambda scaleR
};
struct GradParams {
    double Mmix[9];  // (A_hat^-1)_{s m} / (4 h_s)
    double ph[3][2];
    WideEntry mix[9], phase[27][2];  // the same; cos and sin of every wrap's phase
    int X, Y, Z, N;                  // quarter-grid extents
    int full, block;
    int plane, vstr;  // nodes per plane and component of the layout
    int nvec;
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

__host__ __device__ __forceinline__ double2 grad_phase(const GradParams& P, int wrap) {
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

// Two adjacent lanes per node, one for the real parts and one for the imaginary ones, which meet in the wraps'
// phases only (one lane for both: N = 24, 12 vectors 165 us instead of 121, N = 64 0.84 ms).  They loop over the vectors and
// their sums are added at the end, so that each output entry has a single writer (no atomics, deterministic).
// blockIdx.y: parity block of a full-space layout.
template <bool CUBIC>
__global__ void __launch_bounds__(kGradThreads, 4)
    eig_grad_kernel(const __grid_constant__ GradParams P, const double2* __restrict__ X, double* __restrict__ dC,
                    double* __restrict__ drho, int64_t n_full) {
    __shared__ WideEntry phase[27][2];
    for (int i = threadIdx.x; i < 54; i += kGradThreads) phase[i >> 1][i & 1] = P.phase[i >> 1][i & 1];
    __syncthreads();
    const int blk = P.full ? (int)blockIdx.y : P.block;
    const uint32_t nodes = (uint32_t)P.X * P.Y * P.Z;
    const uint32_t t = (blockIdx.x * kGradThreads + threadIdx.x) >> 1;
    const int part = threadIdx.x & 1;
    if (t >= nodes) return;
    int a, b, k;
    split3(t, P.X, P.Y, a, b, k);
    const GradNode nd = grad_node(P, blk, a, b, k);
    int64_t l;  // full-grid index
    {
        const int p12 = blk >> 1, p13 = blk & 1;
        l = (2 * a + ((k + p13) & 1)) + (int64_t)P.N * ((2 * b + ((k + p12 + p13) & 1)) + (int64_t)P.N * k);
    }
    bool slow = false;
    double gr = 0.0;
    int64_t g[21];
    int gu[21];
#pragma unroll
    for (int q = 0; q < 21; ++q) {
        g[q] = 0;
        gu[q] = 2 * kWideZero;
    }
    for (int v = 0; v < P.nvec; ++v) {
        const GradVec& V = P.v[v];
        const double2* __restrict__ x = X + (int64_t)v * 3 * P.vstr;
        double xx = 0.0;
#pragma unroll
        for (int al = 0; al < 3; ++al) {
            const double2 xo = x[(int64_t)al * P.vstr + nd.at];
            xx = cdotre(xo, xo, xx);  // both parts in both lanes
        }
        gr = fma(V.wR, xx, gr);
        WideHalf f[6], h[6];
        int fu[6];
        wide_strain<CUBIC>(
            P.mix,
            [&](int al, int64_t* m, int* u) {
                const double2* xc = x + (int64_t)al * P.vstr;
#pragma unroll
                for (int ll = 0; ll < 5; ++ll) {
                    const double2 z = xc[ll < 4 ? nd.nb[ll] : nd.at];
                    m[ll] = wide_from_double(part ? z.y : z.x, 6, u[ll]);
                    slow = slow || u[ll] == kWideSpecial;
                    if (ll < 4 && nd.wrap[ll] != 13) {  // times the phase, the other part's share included
                        const WideEntry p = wide_entry(part ? z.y : z.x), o = wide_entry(part ? z.x : z.y);
                        const WideEntry c = phase[nd.wrap[ll]][0], sn = phase[nd.wrap[ll]][1];
                        const WideHalf ph = {p.hi, p.lo}, oh = {o.hi, o.lo};
                        const int u1 = p.u + c.u, u2 = o.u + sn.u, U = imax(u1, u2) + 2;
                        const int64_t m1 = wide_shr(wide_mul(ph, c), U - u1), m2 = wide_shr(wide_mul(oh, sn), U - u2);
                        slow = slow || o.u == kWideSpecial;
                        m[ll] = part ? m1 + m2 : m1 - m2;
                        u[ll] = U + 64;
                    }
                }
            },
            f, fu);
        // a shift rounds down: the real parts' products are added, the imaginary parts' taken away with the
        // sign turned (as 64 bits: a low half of -2^31 has no negative), so that the roundings of a square cancel
        const int64_t turn = (V.neg != 0) != (part != 0) ? -1 : 0;
#pragma unroll
        for (int p = 0; p < 6; ++p) {
            fu[p] += V.s.u + 64;
            const int64_t m = wide_norm(wide_mul(f[p], V.s), fu[p]);
            f[p] = wide_split(m);
            h[p] = wide_split((m ^ turn) - turn);
        }
        int q = 0;
#pragma unroll
        for (int p = 0; p < 6; ++p) {
#pragma unroll
            for (int r = p; r < 6; ++r, ++q) {
                const int u = fu[p] + fu[r] + 4, U = imax(gu[q], u);
                const int64_t m = wide_shr(wide_mul(h[p], f[r]), U - u + 4), s = wide_shr(g[q], U - gu[q]);
                g[q] = part ? s - m : s + m;
                gu[q] = U;
            }
        }
    }
    // the two lanes of a node take every branch alike
    const unsigned pair = 3u << (threadIdx.x & 30);
    slow = __shfl_xor_sync(pair, (int)slow, 1) != 0 || slow;
#pragma unroll
    for (int q = 0; q < 21; ++q) {
        const int64_t o = __shfl_xor_sync(pair, g[q], 1);
        const int ou = __shfl_xor_sync(pair, gu[q], 1), U = imax(gu[q], ou);
        g[q] = wide_shr(g[q], U - gu[q]) + wide_shr(o, U - ou);
        gu[q] = U;
    }
    if (part != 0) return;
    if (slow) {
        grad_slow(P, X, nd, l, dC, drho, n_full);
        return;
    }
    int q = 0;
#pragma unroll
    for (int p = 0; p < 6; ++p)
#pragma unroll
        for (int r = p; r < 6; ++r, ++q)
            if (g[q] != 0) dC[(int64_t)q * n_full + l] += wide_to_double(g[q], gu[q] + 64 + (p == r ? 0 : 1));
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
        for (int e = 0; e < 9; ++e) {
            P.Mmix[e] = g->Ainv[e] * q;
            P.mix[e] = wide_entry(P.Mmix[e]);
        }
        for (int l = 0; l < 3; ++l) {
            P.ph[l][0] = std::cos(g->k.phi[l]);
            P.ph[l][1] = std::sin(g->k.phi[l]);
        }
        for (int w = 0; w < 27; ++w) {
            const double2 e = grad_phase(P, w);
            P.phase[w][0] = wide_entry(e.x);
            P.phase[w][1] = wide_entry(e.y);
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
            V.wC = w * scaleC;
            V.wR = -w * lambdas[base + v] * scaleR;
            // extended precision: the root's rounding would enter every product twice
            const long double sq = sqrtl((long double)std::fabs(V.wC)) * (g->cubic ? (long double)q : 1.0L);
            V.neg = w < 0 ? 1 : 0;
            int ex = 0;
            if (sq > 0) frexpl(sq, &ex);
            const WideHalf h = wide_split(llrintl(ldexpl(sq, 62 - ex)));
            V.s.hi = h.hi;
            V.s.lo = h.lo;
            V.s.u = sq > 0 ? ex - 62 : kWideZero;
            V.s.pad = 0;
        }
        const int64_t nodes = (int64_t)P.X * P.Y * P.Z;
        const dim3 grid((unsigned)((2 * nodes + kGradThreads - 1) / kGradThreads), P.full ? 4 : 1);
        const double2* Xb = static_cast<const double2*>(X) + (int64_t)base * 3 * P.vstr;
        if (g->cubic) eig_grad_kernel<true><<<grid, kGradThreads, 0, s>>>(P, Xb, dC, drho, g->n);
        else eig_grad_kernel<false><<<grid, kGradThreads, 0, s>>>(P, Xb, dC, drho, g->n);
        note_launch();
        PC_CUDA_TRY(cudaGetLastError());
    }
    return PC_OK;
}
