// Integer-pipe complex128 stencil apply (see pc_apply_int.cuh): kernel and launcher.
#include <algorithm>
#include <type_traits>

#include "pc_apply_int.cuh"

namespace pc {

namespace {

constexpr int kFixMaxItems = 64;

struct FixBatch {
    ApplyItem it[kFixMaxItems];
    double ph[kFixMaxItems][3][2];  // (cos, sin) of each item's Bloch phases
    int n;
};

// blockIdx.x = (tile, chunk of planes), blockIdx.y = item (full space: item * 4 + parity block).
// NP parts of a cell per thread: 2 / NP threads per cell.
template <bool CUBIC, int MATK, int NP>
__global__ void __launch_bounds__(2 / NP * kCells, NP)
    fix_apply(const __grid_constant__ FixParams F, const __grid_constant__ FixBatch B, const __grid_constant__ CellGeom G,
              double* __restrict__ dot_partials, int dot_stride) {
    using T = FixApply<CUBIC, MATK, NP>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int item = G.full ? (int)blockIdx.y >> 2 : (int)blockIdx.y;
    const ApplyItem& it = B.it[item];
    if (it.skip != nullptr && *it.skip) return;
    typename T::Shared sh;
    T::carve(sh, smem_raw);
    const int tid = threadIdx.x, cell = tid / (2 / NP), n = G.ncell;
    const bool live = cell < n;
    typename T::Ctx c;
    c.F = &F;
    c.G = &G;
    c.kph = B.ph[item];
    c.x = static_cast<const double2*>(it.x);
    c.y = static_cast<double2*>(it.y);
    c.mat = it.mat;
    c.shift = it.shift;
    c.dot = dot_partials != nullptr && it.dot_slot >= 0;
    const int tiles = G.ntx * G.nty;
    const int tile = (int)blockIdx.x % tiles, ch = (int)blockIdx.x / tiles;
    c.a0 = (tile % G.ntx) * G.TX;
    c.b0 = (tile / G.ntx) * G.TY;
    c.k0 = ch * G.tz;
    c.tz = min(G.tz, G.Z - c.k0);
    const int blk = G.full ? (int)(blockIdx.y & 3) : it.block;
    c.p12 = blk >> 1;
    c.p13 = blk & 1;
    typename T::Regs r;
    T::load_tables(c, sh, tid, blockDim.x);
    T::init(c, min(cell, n - 1), NP == 1 ? tid & 1 : 0, r);
    if (!live) r.flags = 0;
    const int klast = c.k0 + c.tz + 1;  // last plane of x
    // the first three planes go through the flux cells, which nothing uses yet; k0 is even, so planes
    // k0 - 2 .. k0 + 1 have parities 0, 1, 0, 1
    typename T::Shared pre[3] = {sh, sh, sh};
#pragma unroll
    for (int i = 0; i < 3; ++i) pre[i].raw = reinterpret_cast<double*>(sh.fs) + 3 * i * T::kRow;
    if (live) {
        T::template stage<0>(c, pre[0], r, cell, c.k0 - 2);
        T::template stage<1>(c, pre[1], r, cell, c.k0 - 1);
        T::template stage<0>(c, pre[2], r, cell, c.k0);
        T::template stage<1>(c, sh, r, cell, c.k0 + 1);
        r.mcur = T::template read_mat<1>(c, r, c.k0 - 1);
    }
    asm volatile("cp.async.commit_group;\ncp.async.wait_group 0;" ::: "memory");
    __syncthreads();  // phase table
    if (live) {
        T::template convert<0>(c, pre[0], r, cell, c.k0 - 2, 0);
        T::template convert<1>(c, pre[1], r, cell, c.k0 - 1, 1);
        T::template convert<0>(c, pre[2], r, cell, c.k0, 2);
    }
    __syncthreads();
    int sm = 0, sc = 1, sp = 2;
    auto step = [&](auto parity, int kf) {
        constexpr int Q = decltype(parity)::value;
        if (live) {
            if (kf < c.k0 + c.tz) r.mnext = T::template read_mat<1 - Q>(c, r, kf + 1);
            T::template flux<Q>(c, sh, r, kf, sm, sc, sp);
            T::template load_own<Q>(c, r, kf);
        }
        __syncthreads();
        T::template gather<Q>(c, sh, r, kf);
        if (kf + 2 <= klast && live) {
            asm volatile("cp.async.wait_group 0;" ::: "memory");
            T::template convert<Q>(c, sh, r, cell, kf + 2, sm);
            if (kf + 3 <= klast) T::template stage<1 - Q>(c, sh, r, cell, kf + 3);
            asm volatile("cp.async.commit_group;" ::: "memory");
        }
        T::next_mat(r);
        __syncthreads();
        const int t = sm;
        sm = sc;
        sc = sp;
        sp = t;
    };
    for (int kf = c.k0 - 1; kf <= c.k0 + c.tz; kf += 2) {
        step(std::integral_constant<int, 1>(), kf);
        step(std::integral_constant<int, 0>(), kf + 1);
    }
    if (r.ks < c.k0 + c.tz && r.part() == 0) r.dot += T::slow_column(c, r.ks, r.off[0], r.off[1]);  // both parts
    if (c.dot) {
        double v = r.dot;
        double* red = reinterpret_cast<double*>(sh.fs);
        for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
        if ((tid & 31) == 0) red[tid >> 5] = v;
        __syncthreads();
        if (tid == 0) {
            double s = 0.0;
            for (int w = 0; w < (int)(blockDim.x >> 5); ++w) s += red[w];
            const int sub = G.full ? (int)(blockIdx.y & 3) * (int)gridDim.x : 0;
            dot_partials[(int64_t)it.dot_slot * dot_stride + sub + blockIdx.x] = s;
        }
    }
}

template <bool CUBIC, int MATK, int NP>
int launch_fix_np(const FixParams& F, const FixBatch& B, const CellGeom& G, double* dp, int ds, cudaStream_t s) {
    using T = FixApply<CUBIC, MATK, NP>;
    auto kern = fix_apply<CUBIC, MATK, NP>;
    // set on every launch: an attribute of the kernel on the current device
    PC_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)T::shared_bytes()));
    const dim3 grid(G.ntx * G.nty * G.nch, B.n * (G.full ? 4 : 1));
    kern<<<grid, (2 / NP * G.ncell + 31) / 32 * 32, T::shared_bytes(), s>>>(F, B, G, dp, ds);
    note_launch();
    note_apply_launch();
    PC_CUDA_TRY(cudaGetLastError());
    return PC_OK;
}

template <bool CUBIC, int MATK>
int launch_fix_t(const FixParams& F, const FixBatch& B, const CellGeom& G, double* dp, int ds, cudaStream_t s) {
    // Two threads per cell (see FixApply) in launches of one CTA per SM at most, and where a tile has so few cells
    // that its CTA has half the threads and two still share an SM (N = 16, 64 items: 28.9 us, 44.9 us with one
    // thread per cell; N = 10 26.8 / 39.1, N = 18 43.9 / 67.3 us).
    const long ctas = (long)G.ntx * G.nty * G.nch * B.n * (G.full ? 4 : 1);
    return ctas <= device_sm_count() || G.ncell <= kCells / 2 ? launch_fix_np<CUBIC, MATK, 1>(F, B, G, dp, ds, s)
                                     : launch_fix_np<CUBIC, MATK, 2>(F, B, G, dp, ds, s);
}

}  // namespace

int fix_apply_ctas(int N, bool full, int nitems, int tz_in, int* tz) {
    CellGeom G;
    make_cell_geom(G, N, full, false);
    if (tz_in > 0) {
        cell_planes(G, tz_in);
    } else {
        const double rate[2] = {1.0, 1.8};
        cell_chunks(G, std::min(nitems, kFixMaxItems), device_sm_count(), rate, 2);
    }
    if (tz) *tz = G.tz;
    return G.ntx * G.nty * G.nch * (full ? 4 : 1);
}

bool fix_apply_ok(const StencilParams<double>& P, bool cubic, int matkind) {
    FixParams F;
    return make_fix_params(F, P, cubic, matkind);
}

int launch_apply_fix(bool full, bool cubic, int matkind, const StencilParams<double>& P, const ApplyItem* items,
                     const double* item_ph, int nitems, int tz, double* dp, int ds, cudaStream_t s) {
    CellGeom G;
    make_cell_geom(G, P.N, full, false);
    cell_planes(G, tz);
    if (dp != nullptr && G.ntx * G.nty * G.nch * (full ? 4 : 1) > ds)
        return fail(PC_EINVAL, "apply: launch has more CTAs than partial-sum slots");
    FixParams F;
    if (!make_fix_params(F, P, cubic, matkind)) return fail(PC_EINVAL, "apply: a stiffness entry is not finite");
    for (int base = 0; base < nitems; base += kFixMaxItems) {
        FixBatch B;
        B.n = std::min(nitems - base, kFixMaxItems);
        for (int i = 0; i < B.n; ++i) {
            B.it[i] = items[base + i];
            for (int e = 0; e < 6; ++e) B.ph[i][e / 2][e % 2] = item_ph[(size_t)6 * (base + i) + e];
        }
        int rc;
        if (cubic) rc = matkind == 2 ? launch_fix_t<true, 2>(F, B, G, dp, ds, s)
                        : matkind    ? launch_fix_t<true, 1>(F, B, G, dp, ds, s)
                                     : launch_fix_t<true, 0>(F, B, G, dp, ds, s);
        else rc = matkind == 2 ? launch_fix_t<false, 2>(F, B, G, dp, ds, s)
                  : matkind    ? launch_fix_t<false, 1>(F, B, G, dp, ds, s)
                               : launch_fix_t<false, 0>(F, B, G, dp, ds, s);
        PC_TRY(rc);
    }
    return PC_OK;
}

}  // namespace pc
