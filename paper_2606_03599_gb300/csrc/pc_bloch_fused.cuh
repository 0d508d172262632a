// Complex64 reference-medium preconditioner in three kernels with compile-time factors n = N1 N2 (the
// algorithm of pc_bloch_dft.cu; that file's runtime-factor and complex128 kernels serve all other
// sizes and precisions).
//
// A direct DFT stage works on groups of N1 or N2 values that one thread holds in registers, so the
// stages next to global memory read and write it themselves and shared memory is crossed only between
// stages:
//
//   plane_fwd : [load, pre-twiddle, rows stage A] [rows B] [columns A] [columns B, store]
//   pencil    : [load, stage A over k'] [stage B of all six pencils, butterfly, symbol solve, inverse
//               butterfly, inverse B] [inverse A, store]: a thread holds the 6 N2 values whose modes it
//               solves, so the middle of the transform needs no exchange at all
//   plane_inv : the plane stages backwards, with the post-twiddle and the partial Re<r, z>
//
// The work buffer keeps the digit-permuted mode order (mode k1 + N1 k2 at position k1 N2 + k2) in both
// plane axes, and the symbol table is stored in the same order, one array per entry, so every global
// access runs along consecutive addresses and no kernel permutes.  Plane rows are padded to an odd
// length: the rows' stage B reads a column of groups per warp.
#pragma once

#include "pc_complex.cuh"
#include "pc_fourier.h"
#include "pc_internal.h"
#include "pc_small_dft.cuh"

namespace pc {
namespace fused {

struct Args {
    const void* r;   // vectors in (V)
    void* z;         // vectors out (V)
    float2* W;
    const float2 *wn, *twa, *twb, *twk, *ea, *eb, *eg;
    const float* A;  // [9][2 n][n n], permuted planes
    const int *sys_block, *sys_k, *skip;
    int64_t tab_stride;
    float shift_rho, scale;
    double* part;
    int npart;
    int nsys;
};

__host__ __device__ constexpr int up32(int x) { return (x + 31) / 32 * 32; }
__host__ __device__ constexpr int cmax(int a, int b) { return a > b ? a : b; }
__host__ __device__ constexpr int cmin(int a, int b) { return a < b ? a : b; }

// threads of a plane CTA: one group each where that fits
template <int N1, int N2>
constexpr int plane_threads() { return cmin(512, up32(cmax(N1 * N2 * N2, N1 * N2 * N1))); }
// columns of a pencil CTA, and its threads: one (k1, column) each in the middle stage
template <int N1, int N2>
constexpr int pencil_cols() { return N1 <= 4 && N1 * N2 <= 32 ? 32 : 16; }
template <int N1, int N2>
constexpr int pencil_threads() { return cmax(64, up32(N1 * pencil_cols<N1, N2>())); }

template <int N1, int N2>
constexpr int plane_bytes() { return 8 * (N1 * N2 * ((N1 * N2) | 1) + N1 * N2); }
template <int N1, int N2>
constexpr int pencil_bytes() { return 8 * (6 * N1 * N2 * pencil_cols<N1, N2>() + N1 * N2); }

__device__ __forceinline__ float2 conj2(float2 a) { return make_float2(a.x, -a.y); }
__device__ __forceinline__ float2 to_c64(float2 v) { return v; }
__device__ __forceinline__ float2 to_c64(double2 v) { return make_float2((float)v.x, (float)v.y); }
__device__ __forceinline__ void from_c64(float2 v, float2& o) { o = v; }
__device__ __forceinline__ void from_c64(float2 v, double2& o) { o = make_double2(v.x, v.y); }

// w_n^{i k} twiddles of stage A (conjugate for the inverse)
template <int L, int N, bool INV>
__device__ __forceinline__ void twiddle(float2* v, const float2* wn, int i2) {
#pragma unroll
    for (int k = 1; k < L; ++k) {
        const float2 w = wn[i2 * k];  // i2 < N2, k < N1: below n
        v[k] = cmul(v[k], INV ? conj2(w) : w);
    }
}

// Plane id blockIdx.x = ((sys * 3 + comp) * 2 + par) * n + k'.
template <int N1, int N2, typename V>
__global__ void __launch_bounds__(plane_threads<N1, N2>()) plane_fwd(const __grid_constant__ Args P) {
    constexpr int n = N1 * N2, nn = n * n, LD = n | 1, T = plane_threads<N1, N2>();
    extern __shared__ __align__(16) float2 sm[];
    float2* buf = sm;
    float2* wn = sm + n * LD;
    const int pl = blockIdx.x, kp = pl % n, rest = pl / n;
    const int par = rest & 1, comp = (rest >> 1) % 3, sys = rest / 6;
    if (P.skip && P.skip[sys]) return;
    for (int j = threadIdx.x; j < n; j += T) wn[j] = P.wn[j];
    const int64_t nb = (int64_t)2 * n * nn, base = (int64_t)sys * 3 * nb + comp * nb;
    const int64_t to = P.sys_k ? (int64_t)P.sys_k[sys] * P.tab_stride : 0;
    const float2 tk = P.twk[to + kp];
    const V* __restrict__ src = static_cast<const V*>(P.r) + base + (int64_t)(2 * kp + par) * nn;
    __syncthreads();
    for (int g = threadIdx.x; g < n * N2; g += T) {
        const int b = g / N2, i2 = g - b * N2;
        const float2 tb = cmul(P.twb[to + b], tk);
        float2 v[16];
#pragma unroll
        for (int i = 0; i < N1; ++i) v[i] = cmul(to_c64(src[b * n + i * N2 + i2]), cmul(P.twa[to + i * N2 + i2], tb));
        small_dft_ct<N1, false>(v);
        twiddle<N1, n, false>(v, wn, i2);
#pragma unroll
        for (int i = 0; i < N1; ++i) buf[b * LD + i * N2 + i2] = v[i];
    }
    __syncthreads();
    for (int g = threadIdx.x; g < n * N1; g += T) {
        const int k1 = g / n, l = g - k1 * n;
        float2 v[16];
#pragma unroll
        for (int i = 0; i < N2; ++i) v[i] = buf[l * LD + k1 * N2 + i];
        small_dft_ct<N2, false>(v);
#pragma unroll
        for (int i = 0; i < N2; ++i) buf[l * LD + k1 * N2 + i] = v[i];
    }
    __syncthreads();
    for (int g = threadIdx.x; g < n * N2; g += T) {
        const int i2 = g / n, a = g - i2 * n;
        float2 v[16];
#pragma unroll
        for (int i = 0; i < N1; ++i) v[i] = buf[(i * N2 + i2) * LD + a];
        small_dft_ct<N1, false>(v);
        twiddle<N1, n, false>(v, wn, i2);
#pragma unroll
        for (int i = 0; i < N1; ++i) buf[(i * N2 + i2) * LD + a] = v[i];
    }
    __syncthreads();
    float2* __restrict__ dst = P.W + base + par * (nb / 2) + (int64_t)kp * nn;
    for (int g = threadIdx.x; g < n * N1; g += T) {
        const int k1 = g / n, a = g - k1 * n;
        float2 v[16];
#pragma unroll
        for (int i = 0; i < N2; ++i) v[i] = buf[(k1 * N2 + i) * LD + a];
        small_dft_ct<N2, false>(v);
#pragma unroll
        for (int i = 0; i < N2; ++i) dst[(k1 * N2 + i) * n + a] = v[i];
    }
}

template <int N1, int N2, typename V>
__global__ void __launch_bounds__(plane_threads<N1, N2>()) plane_inv(const __grid_constant__ Args P) {
    constexpr int n = N1 * N2, nn = n * n, LD = n | 1, T = plane_threads<N1, N2>();
    extern __shared__ __align__(16) float2 sm[];
    float2* buf = sm;
    float2* wn = sm + n * LD;
    const int pl = blockIdx.x, kp = pl % n, rest = pl / n;
    const int par = rest & 1, comp = (rest >> 1) % 3, sys = rest / 6;
    if (P.skip && P.skip[sys]) return;
    for (int j = threadIdx.x; j < n; j += T) wn[j] = P.wn[j];
    const int64_t nb = (int64_t)2 * n * nn, base = (int64_t)sys * 3 * nb + comp * nb;
    const float2* __restrict__ src = P.W + base + par * (nb / 2) + (int64_t)kp * nn;
    for (int g = threadIdx.x; g < n * N1; g += T) {
        const int k1 = g / n, a = g - k1 * n;
        float2 v[16];
#pragma unroll
        for (int i = 0; i < N2; ++i) v[i] = src[(k1 * N2 + i) * n + a];
        small_dft_ct<N2, true>(v);
#pragma unroll
        for (int i = 0; i < N2; ++i) buf[(k1 * N2 + i) * LD + a] = v[i];
    }
    __syncthreads();
    for (int g = threadIdx.x; g < n * N2; g += T) {
        const int i2 = g / n, a = g - i2 * n;
        float2 v[16];
#pragma unroll
        for (int i = 0; i < N1; ++i) v[i] = buf[(i * N2 + i2) * LD + a];
        twiddle<N1, n, true>(v, wn, i2);
        small_dft_ct<N1, true>(v);
#pragma unroll
        for (int i = 0; i < N1; ++i) buf[(i * N2 + i2) * LD + a] = v[i];
    }
    __syncthreads();
    for (int g = threadIdx.x; g < n * N1; g += T) {
        const int k1 = g / n, l = g - k1 * n;
        float2 v[16];
#pragma unroll
        for (int i = 0; i < N2; ++i) v[i] = buf[l * LD + k1 * N2 + i];
        small_dft_ct<N2, true>(v);
#pragma unroll
        for (int i = 0; i < N2; ++i) buf[l * LD + k1 * N2 + i] = v[i];
    }
    __syncthreads();
    const int64_t to = P.sys_k ? (int64_t)P.sys_k[sys] * P.tab_stride : 0;
    const float2 tk = P.twk[to + kp];
    const int64_t off = base + (int64_t)(2 * kp + par) * nn;
    V* dst = static_cast<V*>(P.z) + off;
    const V* r = static_cast<const V*>(P.r) + off;  // may be the output's own buffer: read before it is written
    decltype(V().x) acc = 0;  // per-thread sum in the vectors' precision, FP64 across threads
    for (int g = threadIdx.x; g < n * N2; g += T) {
        const int b = g / N2, i2 = g - b * N2;
        const float2 tb = cmul(P.twb[to + b], tk);
        float2 v[16];
#pragma unroll
        for (int i = 0; i < N1; ++i) v[i] = buf[b * LD + i * N2 + i2];
        twiddle<N1, n, true>(v, wn, i2);
        small_dft_ct<N1, true>(v);
#pragma unroll
        for (int i = 0; i < N1; ++i) {
            const int t = b * n + i * N2 + i2;
            V o;
            from_c64(cmul(v[i], conj2(cmul(P.twa[to + i * N2 + i2], tb))), o);
            if (P.part) acc = cdotre(r[t], o, acc);
            dst[t] = o;
        }
    }
    if (P.part) {
        __shared__ double red[T / 32];
        double v = (double)acc;
        for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
        if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
        __syncthreads();
        if (threadIdx.x == 0) {
            double t = 0.0;
            for (int i = 0; i < T / 32; ++i) t += red[i];
            P.part[(int64_t)sys * P.npart + (pl - sys * 6 * n)] = t;
        }
    }
}

// (A_ref(m) + shift)^-1 v in place by the adjugate; A: the mode's entries, `str` floats apart.
__device__ __forceinline__ void symbol_solve(const float* __restrict__ A, int64_t str, float shift, float scale,
                                             float2& v0, float2& v1, float2& v2) {
    const float d0 = A[0] + shift, d1 = A[str] + shift, d2 = A[2 * str] + shift;
    const float2 a01 = make_float2(A[3 * str], A[4 * str]), a02 = make_float2(A[5 * str], A[6 * str]),
                 a12 = make_float2(A[7 * str], A[8 * str]);
    const float c00 = d1 * d2 - (a12.x * a12.x + a12.y * a12.y);
    const float c11 = d0 * d2 - (a02.x * a02.x + a02.y * a02.y);
    const float c22 = d0 * d1 - (a01.x * a01.x + a01.y * a01.y);
    const float2 c01 = csub(cmul(a02, conj2(a12)), cscale(d2, a01));
    const float2 c02 = csub(cmul(a01, a12), cscale(d1, a02));
    const float2 c12 = csub(cmul(conj2(a01), a02), cscale(d0, a12));
    const float det = d0 * c00 + (a01.x * c01.x + a01.y * c01.y) + (a02.x * c02.x + a02.y * c02.y);
    const float inv = scale / det;
    const float2 z0 = cadd(cadd(cscale(c00, v0), cmul(c01, v1)), cmul(c02, v2));
    const float2 z1 = cadd(cadd(cmul(conj2(c01), v0), cscale(c11, v1)), cmul(c12, v2));
    const float2 z2 = cadd(cadd(cmul(conj2(c02), v0), cmul(conj2(c12), v1)), cscale(c22, v2));
    v0 = cscale(inv, z0);
    v1 = cscale(inv, z1);
    v2 = cscale(inv, z2);
}

// blockIdx.x = tile of PT columns (q position, p position) of the plane, blockIdx.y = system.
template <int N1, int N2>
__global__ void __launch_bounds__(pencil_threads<N1, N2>()) pencil(const __grid_constant__ Args P) {
    constexpr int n = N1 * N2, nn = n * n, PT = pencil_cols<N1, N2>(), T = pencil_threads<N1, N2>();
    extern __shared__ __align__(16) float2 sm[];
    float2* buf = sm;  // [pencil = comp * 2 + par][position over k'][column]
    float2* wn = sm + 6 * n * PT;
    const int sys = blockIdx.y;
    if (P.skip && P.skip[sys]) return;
    for (int j = threadIdx.x; j < n; j += T) wn[j] = P.wn[j];
    const int c0 = blockIdx.x * PT, pw = cmin(PT, nn - c0);
    const int64_t nb = (int64_t)2 * n * nn;
    float2* __restrict__ Ws = P.W + (int64_t)sys * 3 * nb + c0;
    __syncthreads();
#pragma unroll 3
    for (int g = threadIdx.x; g < 6 * N2 * PT; g += T) {
        const int pl = g % PT, i2 = (g / PT) % N2, pen = g / (PT * N2);
        const float2* __restrict__ src = Ws + (pen >> 1) * nb + (pen & 1) * (nb / 2) + pl;
        float2 v[16];
#pragma unroll
        for (int i = 0; i < N1; ++i) v[i] = pl < pw ? src[(int64_t)(i * N2 + i2) * nn] : make_float2(0.f, 0.f);
        small_dft_ct<N1, false>(v);
        twiddle<N1, n, false>(v, wn, i2);
#pragma unroll
        for (int i = 0; i < N1; ++i) buf[(pen * n + i * N2 + i2) * PT + pl] = v[i];
    }
    __syncthreads();
    const int b = P.sys_block[sys], p12 = b >> 1, p13 = b & 1;
    const int ks = P.sys_k ? P.sys_k[sys] : 0;
    const int64_t to = ks * P.tab_stride;
    const float* __restrict__ A = P.A + (int64_t)ks * 9 * nb;
    for (int g = threadIdx.x; g < N1 * PT; g += T) {
        const int pl = g % PT, k1 = g / PT;
        if (pl >= pw) continue;
        const int col = c0 + pl, qp = col / n, pp = col - qp * n;  // positions; modes:
        const int p = pp / N2 + N1 * (pp % N2), q = qp / N2 + N1 * (qp % N2);
        float2 B0 = make_float2(1.f, 0.f), B1 = B0;  // the butterfly's twiddles without e^{-i gamma_r}
        {
            const float2 va = P.ea[to + p], vb = P.eb[to + q];
            if (p13) B0 = va; else B1 = va;
            if ((p12 + p13) & 1) B0 = cmul(B0, vb); else B1 = cmul(B1, vb);
        }
        float2 v[6][N2];
#pragma unroll
        for (int pen = 0; pen < 6; ++pen) {
#pragma unroll
            for (int i = 0; i < N2; ++i) v[pen][i] = buf[(pen * n + k1 * N2 + i) * PT + pl];
            small_dft_ct<N2, false>(v[pen]);
        }
#pragma unroll
        for (int k2 = 0; k2 < N2; ++k2) {
            const int r = k1 + N1 * k2;
            const float2 T0 = B0, T1 = cmul(B1, P.eg[to + r]);
            float2 lo[3], hi[3];
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                const float2 w0 = cmul(T0, v[2 * c][k2]), w1 = cmul(T1, v[2 * c + 1][k2]);
                lo[c] = cadd(w0, w1);
                hi[c] = csub(w0, w1);
            }
            symbol_solve(A + (int64_t)r * nn + col, nb, P.shift_rho, P.scale, lo[0], lo[1], lo[2]);
            symbol_solve(A + (int64_t)(r + n) * nn + col, nb, P.shift_rho, P.scale, hi[0], hi[1], hi[2]);
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                v[2 * c][k2] = cmul(conj2(T0), cadd(lo[c], hi[c]));
                v[2 * c + 1][k2] = cmul(conj2(T1), csub(lo[c], hi[c]));
            }
        }
#pragma unroll
        for (int pen = 0; pen < 6; ++pen) {
            small_dft_ct<N2, true>(v[pen]);
#pragma unroll
            for (int i = 0; i < N2; ++i) buf[(pen * n + k1 * N2 + i) * PT + pl] = v[pen][i];
        }
    }
    __syncthreads();
#pragma unroll 2
    for (int g = threadIdx.x; g < 6 * N2 * PT; g += T) {
        const int pl = g % PT, i2 = (g / PT) % N2, pen = g / (PT * N2);
        float2 v[16];
#pragma unroll
        for (int i = 0; i < N1; ++i) v[i] = buf[(pen * n + i * N2 + i2) * PT + pl];
        twiddle<N1, n, true>(v, wn, i2);
        small_dft_ct<N1, true>(v);
        if (pl < pw) {
            float2* __restrict__ dst = Ws + (pen >> 1) * nb + (pen & 1) * (nb / 2) + pl;
#pragma unroll
            for (int i = 0; i < N1; ++i) dst[(int64_t)(i * N2 + i2) * nn] = v[i];
        }
    }
}

template <typename K>
int grant(K kern, int bytes) {
    if (bytes <= 48 * 1024) return PC_OK;
    PC_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes));
    return PC_OK;
}

template <int N1, int N2, typename V>
int launch(const Args& P, cudaStream_t s) {
    constexpr int n = N1 * N2, pb = plane_bytes<N1, N2>(), qb = pencil_bytes<N1, N2>(), PT = pencil_cols<N1, N2>();
    PC_TRY(grant(plane_fwd<N1, N2, V>, pb));
    PC_TRY(grant(pencil<N1, N2>, qb));
    PC_TRY(grant(plane_inv<N1, N2, V>, pb));
    const int planes = P.nsys * 6 * n;
    plane_fwd<N1, N2, V><<<planes, (plane_threads<N1, N2>()), pb, s>>>(P);
    note_launch();
    pencil<N1, N2><<<dim3((n * n + PT - 1) / PT, P.nsys), (pencil_threads<N1, N2>()), qb, s>>>(P);
    note_launch();
    plane_inv<N1, N2, V><<<planes, (plane_threads<N1, N2>()), pb, s>>>(P);
    note_launch();
    PC_CUDA_TRY(cudaGetLastError());
    return PC_OK;
}

// Sizes n = N1 N2 with a fused form: the solver's grids and the small lengths (bloch_dft_supported's factors).
#define PC_FUSED_A(X) X(2, 2) X(1, 5) X(2, 3) X(1, 7) X(2, 4) X(3, 3) X(2, 5) X(3, 4) X(2, 7) X(3, 5) X(4, 4) X(3, 6)
#define PC_FUSED_B(X) X(4, 5) X(3, 7) X(4, 6) X(5, 5) X(4, 7) X(5, 6) X(4, 8)
#define PC_FUSED_C(X) X(6, 6) X(5, 8) X(6, 7) X(6, 8) X(7, 7)
#define PC_FUSED_D(X) X(7, 8) X(6, 10) X(8, 8) X(8, 9) X(8, 10)

inline bool supported(int n) {
#define PC_FUSED_HAS(A, B) || n == A * B
    return false PC_FUSED_A(PC_FUSED_HAS) PC_FUSED_B(PC_FUSED_HAS) PC_FUSED_C(PC_FUSED_HAS) PC_FUSED_D(PC_FUSED_HAS);
#undef PC_FUSED_HAS
}

// wide: complex128 vectors.  *found = false when n is not among the part's sizes.
int launch_a(int n, bool wide, const Args& P, cudaStream_t s, bool* found);
int launch_b(int n, bool wide, const Args& P, cudaStream_t s, bool* found);
int launch_c(int n, bool wide, const Args& P, cudaStream_t s, bool* found);
int launch_d(int n, bool wide, const Args& P, cudaStream_t s, bool* found);

#define PC_FUSED_CASE(A, B) \
    case A * B: return wide ? launch<A, B, double2>(P, s) : launch<A, B, float2>(P, s);
#define PC_FUSED_TU(NAME, SIZES)                                                  \
    int NAME(int n, bool wide, const Args& P, cudaStream_t s, bool* found) {      \
        *found = true;                                                            \
        switch (n) {                                                              \
            SIZES(PC_FUSED_CASE)                                                  \
            default: *found = false; return PC_OK;                                \
        }                                                                         \
    }

}  // namespace fused
}  // namespace pc
