// Tall-skinny complex128 products of the outer Krylov-Schur loop: the Gram blocks V^H M W of
// block classical Gram-Schmidt and Cholesky QR (M = the nodal mass, Eq. discrete_GEP_main),
// and the basis updates W <- beta W + alpha V h of the same steps, of the Ritz vectors and of
// the restarts.
//
// The shapes are a few to a few dozen columns of length 3 n_b (83k at N = 48, 3.1M at N = 160),
// so the work is a sum over a long index with a small dense result.  In FP64 arithmetic they are
// bound by GB300's FP64 pipe (2 lanes per clock and SM, 8 FMAs for every 16-byte operand), 4 to 6
// times above their memory time.  Gram products of more than four rows therefore run on the integer pipe in
// groups of eight (pc_wide.cuh): every value keeps its own exponent, a real product is four 32 x 32 + 64 bit
// multiply-adds and its place in the group's sum a rounding shift and an addition, and the FP64 pipe sees two
// instructions per group and result.  Operands are
// read once per register block with coalesced 16-byte loads, the mass weight is applied once per
// element of W (not per product), and Gram partial sums are reduced in a fixed order (per CTA, then
// across CTAs) so results are deterministic.
//
// Measured in an FP64 solve at N = 48 (sixteen spaces, vectors of 1.3 MB), FP64 / integer form: Gram products of
// more than four rows 0.56 / 0.34 ms.  Updates stay in FP64 (0.21 ms for 2 columns, 1.20 ms for 4): their rounding has
// to be free of any common offset, a long wave of the lattice that the shift-invert iteration would amplify, and with
// that the integer form took 0.18 and 1.11 ms.  (Eight values cut into limbs of one shared exponent took 0.19 ms for
// Gram products and 0.11 and 0.42 ms for updates, but lost small values next to large ones and made every squared norm
// 5e-17 too small.)
#include <algorithm>

#include "pc_solver.h"
#include "pc_wide.cuh"

namespace pc {

namespace {

constexpr int kGramThreads = 256;
constexpr int kGramCB = 2;  // columns of W per register block

template <int MATK>
__device__ __forceinline__ double node_weight(const void* __restrict__ mat, int64_t t, int64_t m, double rho0,
                                              double drho) {
    if (MATK == 0) return rho0 + drho * (double)static_cast<const uint8_t*>(mat)[t];
    if (MATK == 1) return rho0 + drho * (double)static_cast<const float*>(mat)[t];
    if (MATK == 2) return static_cast<const double*>(mat)[21 * m + t];
    return 1.0;
}

// Partial sums of out(i, j) = sum_e conj(A[i][e]) w(e) B[j][e] over the nodes [t0, t1) of chunk
// blockIdx.x (all three components), columns j0 and j0 + 1, into
// part[((base + i + j rows) 2 + re/im) nchunk + chunk].
// MATK: -1 = no weight, 0 = phase ids, 1 = inclusion fractions, 2 = nodewise material.
//
// FP64 form, rows i0 .. i0 + RB - 1: vectors too short for full groups of eight.
template <int RB, int MATK>
__device__ __forceinline__ void gram_chunk(const double2* __restrict__ A, int rows, const double2* __restrict__ B,
                                           int cols, int64_t m, const void* __restrict__ mat, double rho0, double drho,
                                           int i0, int j0, int nchunk, double* __restrict__ part, int64_t base) {
    constexpr int CB = kGramCB;
    const int64_t vs = 3 * m;
    const int64_t t0 = (int64_t)blockIdx.x * m / nchunk, t1 = (int64_t)(blockIdx.x + 1) * m / nchunk;
    double ar[RB][CB], ai[RB][CB];
#pragma unroll
    for (int i = 0; i < RB; ++i)
#pragma unroll
        for (int j = 0; j < CB; ++j) ar[i][j] = ai[i][j] = 0.0;
    for (int64_t t = t0 + threadIdx.x; t < t1; t += kGramThreads) {
        const double w = node_weight<MATK>(mat, t, m, rho0, drho);
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const int64_t e = c * m + t;
            double2 b[CB];
#pragma unroll
            for (int j = 0; j < CB; ++j) {
                b[j] = (j0 + j < cols) ? B[(int64_t)(j0 + j) * vs + e] : make_double2(0.0, 0.0);
                if (MATK >= 0) b[j] = make_double2(w * b[j].x, w * b[j].y);
            }
#pragma unroll
            for (int i = 0; i < RB; ++i) {
                if (i0 + i < rows) {
                    const double2 a = A[(int64_t)(i0 + i) * vs + e];
#pragma unroll
                    for (int j = 0; j < CB; ++j) {  // conj(a) b
                        ar[i][j] = fma(a.x, b[j].x, fma(a.y, b[j].y, ar[i][j]));
                        ai[i][j] = fma(a.x, b[j].y, fma(-a.y, b[j].x, ai[i][j]));
                    }
                }
            }
        }
    }
    // CTA reduction in a fixed order: warp shuffles, then the warps' sums in warp order
    constexpr int NV = RB * CB * 2;
    __shared__ double red[kGramThreads / 32][NV];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int i = 0; i < RB; ++i)
#pragma unroll
        for (int j = 0; j < CB; ++j) {
            double vr = ar[i][j], vi = ai[i][j];
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                vr += __shfl_down_sync(0xffffffffu, vr, o);
                vi += __shfl_down_sync(0xffffffffu, vi, o);
            }
            if (lane == 0) {
                red[warp][(i * CB + j) * 2 + 0] = vr;
                red[warp][(i * CB + j) * 2 + 1] = vi;
            }
        }
    __syncthreads();
    if (threadIdx.x < NV) {
        const int v = threadIdx.x, ij = v >> 1, ri = v & 1;
        const int gi = i0 + ij / CB, gj = j0 + ij % CB;
        if (gi < rows && gj < cols) {
            double s = 0.0;
            for (int q = 0; q < kGramThreads / 32; ++q) s += red[q][v];
            part[((base + gi + (int64_t)gj * rows) * 2 + ri) * nchunk + blockIdx.x] = s;
        }
    }
}

// Integer form, rows i0 .. i0 + 8 RW - 1 (warp w has rows i0 + w, i0 + w + 8, ...): a tile of 1024
// elements of the two columns is weighted and made factors once, and every warp runs its rows over the
// tile, eight elements of a lane to a group; a group whose largest value is out of range runs in FP64.
// Making a row's elements factors costs a third of their products, so two columns go together and the columns'
// own factors are shared by all rows through shared memory.
constexpr int kGramTile = 1024;

template <int RW, int MATK>
__device__ __forceinline__ void gram_tile(const double2* __restrict__ A, int rows, const double2* __restrict__ B,
                                          int cols, int64_t m, const void* __restrict__ mat, double rho0, double drho,
                                          int i0, int j0, int nchunk, double* __restrict__ part, int64_t base) {
    constexpr int CB = kGramCB, NB = 8;
    __shared__ WideC lb[CB][kGramTile];
    __shared__ short2 ub[CB][kGramTile];  // units of the two parts
    __shared__ bool okb[CB][kGramTile / NB];
    const int64_t vs = 3 * m;
    const int64_t t0 = (int64_t)blockIdx.x * m / nchunk, t1 = (int64_t)(blockIdx.x + 1) * m / nchunk;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int len = (int)(t1 - t0), total = 3 * len;  // elements of the chunk, component after component
    auto element = [&](int x) {                       // offset in a vector of element x of the chunk
        const int c = (x >= len) + (x >= 2 * len);
        return (int64_t)c * m + t0 + (x - c * len);
    };
    auto weighted = [&](int j, int x) {
        const int64_t e = element(x);
        double2 b = (j0 + j < cols) ? B[(int64_t)(j0 + j) * vs + e] : make_double2(0.0, 0.0);
        if (MATK >= 0) {
            const int c = (x >= len) + (x >= 2 * len);
            const double w = node_weight<MATK>(mat, e - (int64_t)c * m, m, rho0, drho);
            b = make_double2(w * b.x, w * b.y);
        }
        return b;
    };
    double ar[RW][CB], ai[RW][CB];
#pragma unroll
    for (int r = 0; r < RW; ++r)
#pragma unroll
        for (int j = 0; j < CB; ++j) ar[r][j] = ai[r][j] = 0.0;
    for (int x0 = 0; x0 < total; x0 += kGramTile) {
        {
            const int g = warp >> 1, j = warp & 1;
            double2 b[NB];
            int top = 0;
#pragma unroll
            for (int q = 0; q < NB; ++q) {
                const int x = x0 + g * 256 + q * 32 + lane;
                b[q] = x < total ? weighted(j, x) : make_double2(0.0, 0.0);
                top = wide_top(b[q], top);
            }
            const int E = top == 0 ? kWideLow : top >> 20;  // zeros, or values too small to count
#pragma unroll
            for (int q = 0; q < NB; ++q) {
                int ur, ui;
                lb[j][g * 256 + q * 32 + lane] = wide_factor(b[q], ur, ui);
                ub[j][g * 256 + q * 32 + lane] = make_short2((short)ur, (short)ui);
            }
            okb[j][g * 32 + lane] = E >= kWideLow && E <= kWideHigh;
        }
        __syncthreads();
#pragma unroll 1
        for (int g = 0; g < kGramTile / 256; ++g) {
            const int xg = x0 + g * 256 + lane;
            if (xg - lane >= total) break;
            const bool ok = okb[0][g * 32 + lane] && okb[1][g * 32 + lane];
#pragma unroll
            for (int r = 0; r < RW; ++r) {
                const int i = i0 + warp + 8 * r;
                if (i >= rows) break;
                const double2* __restrict__ Ai = A + (int64_t)i * vs;
                double2 a[NB];
                int top = 0;
#pragma unroll
                for (int q = 0; q < NB; ++q) {
                    const int x = xg + q * 32;
                    a[q] = x < total ? Ai[element(x)] : make_double2(0.0, 0.0);
                }
#pragma unroll
                for (int q = 0; q < NB; ++q) top = wide_top(a[q], top);
                const int E = top >> 20;
                if (ok && E >= kWideLow && E <= kWideHigh) {
                    WideSum re[CB], im[CB];
#pragma unroll
                    for (int j = 0; j < CB; ++j) re[j] = im[j] = wide_sum0();
#pragma unroll
                    for (int q = 0; q < NB; ++q) {
                        const int ur = wide_unit(a[q].x), ui = wide_unit(a[q].y);
#pragma unroll
                        for (int j = 0; j < CB; ++j) {
                            const short2 uv = ub[j][g * 256 + q * 32 + lane];
                            wide_reach(re[j], ur, uv.x, ui, uv.y);
                            wide_reach(im[j], ur, uv.y, ui, uv.x);
                        }
                    }
#pragma unroll
                    for (int q = 0; q < NB; ++q) {
                        int ur, ui;
                        const WideC la = wide_factor(a[q], ur, ui);
#pragma unroll
                        for (int j = 0; j < CB; ++j) {  // conj(a) b
                            const WideC lv = lb[j][g * 256 + q * 32 + lane];
                            const short2 uv = ub[j][g * 256 + q * 32 + lane];
                            wide_mac2<false>(re[j], la.re, ur, lv.re, uv.x, la.im, ui, lv.im, uv.y);
                            wide_mac2<true>(im[j], la.re, ur, lv.im, uv.y, la.im, ui, lv.re, uv.x);
                        }
                    }
#pragma unroll
                    for (int j = 0; j < CB; ++j) {
                        ar[r][j] += wide_to_double(re[j]);
                        ai[r][j] += wide_to_double(im[j]);
                    }
                } else if (top != 0 || !ok) {
#pragma unroll 1
                    for (int q = 0; q < NB; ++q) {
                        const int x = xg + q * 32;
                        if (x >= total) break;
                        const double2 av = Ai[element(x)];
#pragma unroll
                        for (int j = 0; j < CB; ++j) {
                            const double2 bv = weighted(j, x);
                            ar[r][j] = fma(av.x, bv.x, fma(av.y, bv.y, ar[r][j]));
                            ai[r][j] = fma(av.x, bv.y, fma(-av.y, bv.x, ai[r][j]));
                        }
                    }
                }
            }
        }
        __syncthreads();
    }
#pragma unroll
    for (int r = 0; r < RW; ++r) {
        const int i = i0 + warp + 8 * r;
        if (i >= rows) break;
#pragma unroll
        for (int j = 0; j < CB; ++j) {
            double vr = ar[r][j], vi = ai[r][j];
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                vr += __shfl_down_sync(0xffffffffu, vr, o);
                vi += __shfl_down_sync(0xffffffffu, vi, o);
            }
            if (lane == 0 && j0 + j < cols) {
                double* p = part + ((base + i + (int64_t)(j0 + j) * rows) * 2) * nchunk + blockIdx.x;
                p[0] = vr;
                p[nchunk] = vi;
            }
        }
    }
}

// One register block of a product: RB < 0 is the integer form with -RB rows per warp.
template <int RB, int MATK>
__device__ __forceinline__ void gram_block(const double2* __restrict__ A, int rows, const double2* __restrict__ B,
                                           int cols, int64_t m, const void* __restrict__ mat, double rho0, double drho,
                                           int rg, int cg, int nchunk, double* __restrict__ part, int64_t base) {
    if constexpr (RB < 0)
        gram_tile<-RB, MATK>(A, rows, B, cols, m, mat, rho0, drho, rg * -RB * 8, cg * kGramCB, nchunk, part, base);
    else
        gram_chunk<RB, MATK>(A, rows, B, cols, m, mat, rho0, drho, rg * RB, cg * kGramCB, nchunk, part, base);
}

// The form for `rows` rows of vectors of m nodes.  Integer form from vectors that fill two tiles of
// 1024 elements and 5 rows on (fewer rows leave its warps idle); rows per block in *rb.
int gram_form(int rows, int64_t m, int* rb) {
    const int f = (m >= 683 && rows > 4) ? (rows <= 8 ? -1 : rows <= 16 ? -2 : -3) : (rows <= 2 ? 2 : rows <= 4 ? 4 : 8);
    *rb = f < 0 ? -f * 8 : f;
    return f;
}

template <int RB, int MATK>
__global__ void __launch_bounds__(kGramThreads, RB < 0 ? 2 : 1)
    ts_gram_kernel(const double2* __restrict__ A, int rows, const double2* __restrict__ B, int cols, int64_t m,
                   const void* __restrict__ mat, double rho0, double drho, int ngc, int nchunk,
                   double* __restrict__ part) {
    gram_block<RB, MATK>(A, rows, B, cols, m, mat, rho0, drho, blockIdx.y / ngc, blockIdx.y % ngc, nchunk, part, 0);
}

// out[e] = sum over chunks of part[e][chunk]: one warp per entry, lane l sums the chunks
// l, l + 32, ... in order, then the lanes' sums are combined by a fixed shuffle tree
// (deterministic for a given chunk count).
__global__ void ts_gram_reduce(const double* __restrict__ part, int nentries, int nchunk, double2* __restrict__ out) {
    const int e = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    if (e >= nentries) return;
    double re = 0.0, im = 0.0;
    for (int c = lane; c < nchunk; c += 32) {
        re += part[((int64_t)e * 2 + 0) * nchunk + c];
        im += part[((int64_t)e * 2 + 1) * nchunk + c];
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        re += __shfl_down_sync(0xffffffffu, re, o);
        im += __shfl_down_sync(0xffffffffu, im, o);
    }
    if (lane == 0) out[e] = make_double2(re, im);
}

// C[:, j] = beta C[:, j] + alpha sum_k A[:, k] h(k, j) for the CB columns j0 .. j0 + CB - 1 of
// column group blockIdx.y, in FP64; h (k x cols, column-major) is staged in shared memory.  With
// beta == 0, C is not read (it may hold anything).
template <int CB>
__device__ __forceinline__ void update_columns(const double2* __restrict__ A, int k, const double2* __restrict__ h,
                                               int cols, double2* __restrict__ C, int64_t vs, double alpha,
                                               double beta, int j0) {
    extern __shared__ double2 hs[];  // [k][CB]
    for (int q = threadIdx.x; q < k * CB; q += blockDim.x) {
        const int kk = q / CB, j = q % CB;
        hs[q] = (j0 + j < cols) ? h[kk + (int64_t)(j0 + j) * k] : make_double2(0.0, 0.0);
    }
    __syncthreads();
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < vs; e += (int64_t)gridDim.x * blockDim.x) {
        double cr[CB], ci[CB];
#pragma unroll
        for (int j = 0; j < CB; ++j) cr[j] = ci[j] = 0.0;
        for (int kk = 0; kk < k; ++kk) {
            const double2 a = A[(int64_t)kk * vs + e];
#pragma unroll
            for (int j = 0; j < CB; ++j) {  // a h
                const double2 hv = hs[kk * CB + j];
                cr[j] = fma(a.x, hv.x, fma(-a.y, hv.y, cr[j]));
                ci[j] = fma(a.x, hv.y, fma(a.y, hv.x, ci[j]));
            }
        }
#pragma unroll
        for (int j = 0; j < CB; ++j) {
            if (j0 + j >= cols) continue;
            double2* cp = C + (int64_t)(j0 + j) * vs + e;
            double2 o = make_double2(alpha * cr[j], alpha * ci[j]);
            if (beta != 0.0) {
                const double2 cv = *cp;
                o.x = fma(beta, cv.x, o.x);
                o.y = fma(beta, cv.y, o.y);
            }
            *cp = o;
        }
    }
}

template <int CB>
__global__ void __launch_bounds__(256)
    ts_update_kernel(const double2* __restrict__ A, int k, const double2* __restrict__ h, int cols,
                     double2* __restrict__ C, int64_t vs, double alpha, double beta) {
    update_columns<CB>(A, k, h, cols, C, vs, alpha, beta, blockIdx.y * CB);
}

// Instantiations of a Gram kernel over the forms and weights: CALL(form, weight kind)
#define PC_GRAM_MK(CALL, RBV, mk)  \
    if (mk < 0) { CALL(RBV, -1); } \
    else if (mk == 0) { CALL(RBV, 0); } \
    else if (mk == 2) { CALL(RBV, 2); } \
    else { CALL(RBV, 1); }
#define PC_GRAM_FORM(CALL, form, mk)                    \
    switch (form) {                                     \
        case -1: PC_GRAM_MK(CALL, -1, mk) break;        \
        case -2: PC_GRAM_MK(CALL, -2, mk) break;        \
        case -3: PC_GRAM_MK(CALL, -3, mk) break;        \
        case 2: PC_GRAM_MK(CALL, 2, mk) break;          \
        case 4: PC_GRAM_MK(CALL, 4, mk) break;          \
        default: PC_GRAM_MK(CALL, 8, mk) break;         \
    }

// ---------------------------------------------------------------- batched forms (several spaces)
// The outer loop runs the same product for every active space of a solve (the four parity blocks
// times the Bloch vectors solved together); one launch serves them all, job j in blockIdx.z.
constexpr int kMaxJobs = 64;

struct GramBatch {
    GramJob j[kMaxJobs];
    int64_t off[kMaxJobs + 1];  // prefix sums of the jobs' result entries
    int n;
};

template <int RB, int MATK>
__global__ void __launch_bounds__(kGramThreads, RB < 0 ? 2 : 1)
    ts_gram_batch_kernel(const __grid_constant__ GramBatch B, int64_t m, double rho0, double drho, int ngc,
                         int nchunk, double* __restrict__ part) {
    const GramJob& J = B.j[blockIdx.z];
    const int rg = blockIdx.y / ngc, cg = blockIdx.y % ngc;
    constexpr int step = RB < 0 ? -RB * 8 : RB;
    if (rg * step >= J.rows || cg * kGramCB >= J.cols) return;  // this job has fewer blocks than the launch
    gram_block<RB, MATK>(J.A, J.rows, J.B, J.cols, m, J.mat, rho0, drho, rg, cg, nchunk, part, B.off[blockIdx.z]);
}

// Entry e of the concatenated results (job order) = fixed-order sum of its chunk partials.
__global__ void ts_gram_batch_reduce(const __grid_constant__ GramBatch B, const double* __restrict__ part,
                                     int nchunk) {
    const int64_t e = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    if (e >= B.off[B.n]) return;
    double re = 0.0, im = 0.0;
    for (int c = lane; c < nchunk; c += 32) {
        re += part[(e * 2 + 0) * nchunk + c];
        im += part[(e * 2 + 1) * nchunk + c];
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        re += __shfl_down_sync(0xffffffffu, re, o);
        im += __shfl_down_sync(0xffffffffu, im, o);
    }
    if (lane == 0) {
        int j = 0;
        while (e >= B.off[j + 1]) ++j;
        B.j[j].out[e - B.off[j]] = make_double2(re, im);
    }
}

struct UpdateBatch {
    UpdateJob j[kMaxJobs];
    int n;
};

template <int CB>
__global__ void __launch_bounds__(256)
    ts_update_batch_kernel(const __grid_constant__ UpdateBatch U, int64_t vs) {
    const UpdateJob& J = U.j[blockIdx.z];
    const int j0 = blockIdx.y * CB;
    if (j0 >= J.cols) return;
    update_columns<CB>(J.A, J.k, J.h, J.cols, J.C, vs, J.alpha, J.beta, j0);
}

}  // namespace

int ts_gram(const double2* A, int rows, const double2* B, int cols, int64_t m, const void* mat, int matkind,
            double rho0, double rho1, double2* d_out, double* d_part, size_t part_cap, cudaStream_t s) {
    if (rows <= 0 || cols <= 0) return PC_OK;
    if (!A || !B || !d_out || !d_part || m <= 0) return fail(PC_EINVAL, "ts_gram: bad argument");
    int rb;
    const int form = gram_form(rows, m, &rb);
    const int nrg = (rows + rb - 1) / rb, ngc = (cols + kGramCB - 1) / kGramCB;
    // chunks of the node range: about two CTAs per SM over all register blocks, at least 512
    // nodes (two per thread) per chunk so that the per-CTA reduction stays small next to the
    // products, and as many partials as the scratch holds
    const int64_t entries = (int64_t)rows * cols;
    int64_t nchunk = (2LL * device_sm_count() + nrg * ngc - 1) / (nrg * ngc);
    nchunk = std::min<int64_t>(nchunk, std::max<int64_t>(1, m / 512));
    nchunk = std::min<int64_t>(nchunk, (int64_t)(part_cap / (2 * entries)));
    if (nchunk < 1) return fail(PC_EINVAL, "ts_gram: partial-sum scratch too small");
    const double drho = rho1 - rho0;
    const int mk = mat ? matkind : -1;
    const dim3 grid((unsigned)nchunk, nrg * ngc);
#define PC_GRAM_1(RBV, MKV) \
    ts_gram_kernel<RBV, MKV><<<grid, kGramThreads, 0, s>>>(A, rows, B, cols, m, mat, rho0, drho, ngc, (int)nchunk, d_part)
    PC_GRAM_FORM(PC_GRAM_1, form, mk)
#undef PC_GRAM_1
    note_launch();
    ts_gram_reduce<<<(int)((entries + 7) / 8), 256, 0, s>>>(d_part, (int)entries, (int)nchunk, d_out);
    note_launch();
    PC_CUDA_TRY(cudaGetLastError());
    return PC_OK;
}

int ts_update(const double2* A, int k, const double2* d_h, int cols, double2* C, int64_t vs, double alpha,
              double beta, cudaStream_t s) {
    if (cols <= 0) return PC_OK;
    if (!C || vs <= 0) return fail(PC_EINVAL, "ts_update: bad argument");
    if (k <= 0) {  // empty product: C <- beta C
        if (beta == 1.0) return PC_OK;
        if (beta == 0.0) {
            for (int j = 0; j < cols; ++j)
                PC_CUDA_TRY(cudaMemsetAsync(C + (int64_t)j * vs, 0, sizeof(double2) * vs, s));
            return PC_OK;
        }
        return fail(PC_EINVAL, "ts_update: empty product with beta other than 0 or 1");
    }
    if (!A || !d_h) return fail(PC_EINVAL, "ts_update: bad argument");
    // column blocks of 2 when cols <= 2 (the Gram-Schmidt updates of a 2-wide Krylov block:
    // no FMAs on padding columns), else of 4
    const int CB = cols <= 2 ? 2 : 4;
    const size_t smem = sizeof(double2) * (size_t)k * CB;
    if (smem > 48 * 1024) return fail(PC_EINVAL, "ts_update: too many basis columns");
    const int ngc = (cols + CB - 1) / CB;
    int64_t gx = (vs + 255) / 256;
    gx = std::min<int64_t>(gx, std::max<int64_t>(1, 8LL * device_sm_count() / ngc));
    if (CB == 2)
        ts_update_kernel<2><<<dim3((unsigned)gx, ngc), 256, smem, s>>>(A, k, d_h, cols, C, vs, alpha, beta);
    else
        ts_update_kernel<4><<<dim3((unsigned)gx, ngc), 256, smem, s>>>(A, k, d_h, cols, C, vs, alpha, beta);
    note_launch();
    PC_CUDA_TRY(cudaGetLastError());
    return PC_OK;
}

int ts_gram_batch(const GramJob* jobs, int njobs, int64_t m, int matkind, double rho0, double rho1, double* d_part,
                  size_t part_cap, cudaStream_t s) {
    for (int base = 0; base < njobs; base += kMaxJobs) {
        GramBatch B;
        B.n = 0;
        B.off[0] = 0;
        int maxr = 0, maxc = 0;
        bool weighted = false;
        for (int i = base; i < njobs && B.n < kMaxJobs; ++i) {
            const GramJob& J = jobs[i];
            if (J.rows <= 0 || J.cols <= 0) continue;
            if (!J.A || !J.B || !J.out) return fail(PC_EINVAL, "ts_gram_batch: bad job");
            if (B.n > 0 && (J.mat != nullptr) != weighted) return fail(PC_EINVAL, "ts_gram_batch: mixed weights");
            weighted = J.mat != nullptr;
            B.j[B.n] = J;
            B.off[B.n + 1] = B.off[B.n] + (int64_t)J.rows * J.cols;
            ++B.n;
            maxr = std::max(maxr, J.rows);
            maxc = std::max(maxc, J.cols);
        }
        if (B.n == 0) continue;
        int rb;
        const int form = gram_form(maxr, m, &rb);
        const int nrg = (maxr + rb - 1) / rb, ngc = (maxc + kGramCB - 1) / kGramCB;
        const int64_t entries = B.off[B.n];
        int64_t nchunk = (2LL * device_sm_count() + (int64_t)nrg * ngc * B.n - 1) / ((int64_t)nrg * ngc * B.n);
        nchunk = std::min<int64_t>(nchunk, std::max<int64_t>(1, m / 512));
        nchunk = std::min<int64_t>(nchunk, (int64_t)(part_cap / (2 * entries)));
        if (nchunk < 1) return fail(PC_EINVAL, "ts_gram_batch: partial-sum scratch too small");
        const dim3 grid((unsigned)nchunk, nrg * ngc, B.n);
        const double drho = rho1 - rho0;
        const int mk = weighted ? matkind : -1;
#define PC_GRAM_B(RBV, MKV) \
    ts_gram_batch_kernel<RBV, MKV><<<grid, kGramThreads, 0, s>>>(B, m, rho0, drho, ngc, (int)nchunk, d_part)
        PC_GRAM_FORM(PC_GRAM_B, form, mk)
#undef PC_GRAM_B
        note_launch();
        ts_gram_batch_reduce<<<(unsigned)((entries + 7) / 8), 256, 0, s>>>(B, d_part, (int)nchunk);
        note_launch();
        PC_CUDA_TRY(cudaGetLastError());
    }
    return PC_OK;
}

int ts_update_batch(const UpdateJob* jobs, int njobs, int64_t vs, cudaStream_t s) {
    for (int base = 0; base < njobs; base += kMaxJobs) {
        UpdateBatch U;
        U.n = 0;
        int maxk = 0, maxc = 0;
        for (int i = base; i < njobs && U.n < kMaxJobs; ++i) {
            const UpdateJob& J = jobs[i];
            if (J.cols <= 0) continue;
            if (J.k <= 0 || !J.A || !J.h || !J.C) return fail(PC_EINVAL, "ts_update_batch: bad job");
            U.j[U.n++] = J;
            maxk = std::max(maxk, J.k);
            maxc = std::max(maxc, J.cols);
        }
        if (U.n == 0) continue;
        const int CB = maxc <= 2 ? 2 : 4;
        const size_t smem = sizeof(double2) * (size_t)maxk * CB;
        if (smem > 48 * 1024) return fail(PC_EINVAL, "ts_update_batch: too many basis columns");
        const int ngc = (maxc + CB - 1) / CB;
        int64_t gx = (vs + 255) / 256;
        gx = std::min<int64_t>(gx, std::max<int64_t>(1, 8LL * device_sm_count() / ((int64_t)ngc * U.n)));
        if (CB == 2)
            ts_update_batch_kernel<2><<<dim3((unsigned)gx, ngc, U.n), 256, smem, s>>>(U, vs);
        else
            ts_update_batch_kernel<4><<<dim3((unsigned)gx, ngc, U.n), 256, smem, s>>>(U, vs);
        note_launch();
        PC_CUDA_TRY(cudaGetLastError());
    }
    return PC_OK;
}

}  // namespace pc
