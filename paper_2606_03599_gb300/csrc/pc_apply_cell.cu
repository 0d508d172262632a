// Complex64 cell apply (see pc_apply_cell.cuh): kernel and launcher.
#include <algorithm>
#include <type_traits>

#include "pc_apply_cell.cuh"
#include "pc_apply_tma.cuh"  // mbarrier helpers

namespace pc {

namespace {

constexpr int kCellMaxItems = 64;

struct CellBatch {
    ApplyItem it[kCellMaxItems];
    float ph[kCellMaxItems][3][2];  // (cos, sin) of each item's Bloch phases
    int n;
    uint32_t wait_limit;
    int* err;
};

// Arrive on bar once this thread's copies so far have landed.
__device__ __forceinline__ void copies_arrive(uint64_t* bar) {
    asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ bool bounded_wait(uint64_t* bar, uint32_t parity, uint32_t limit) {
    for (uint32_t n = 0; n < limit; ++n)
        if (mbar_try_wait(bar, parity)) return true;
    return false;
}

// blockIdx.x = (tile, chunk of planes), blockIdx.y = item (full space: item * 4 + parity block).
template <bool CUBIC, int MATK>
__global__ void __launch_bounds__(kCells, 3)
    cell_apply(const __grid_constant__ StencilParams<float> P, const __grid_constant__ CellBatch B,
               const __grid_constant__ CellGeom G, double* __restrict__ dot_partials, int dot_stride) {
    using T = CellApply<CUBIC, MATK>;
    constexpr int NS = T::NS;
    extern __shared__ float4 smem_cell[];
    __shared__ uint64_t full[NS];
    __shared__ double red[kCells / 32];
    const int item = G.full ? (int)blockIdx.y >> 2 : (int)blockIdx.y;
    const ApplyItem& it = B.it[item];
    if (it.skip != nullptr && *it.skip) return;
    typename T::Shared sh;
    T::carve(sh, smem_cell);
    const int tid = threadIdx.x, n = G.ncell;
    const bool live = tid < n;
    typename T::Ctx c;
    c.P = &P;
    c.G = &G;
    c.kph = B.ph[item];
    c.x = static_cast<const float2*>(it.x);
    c.y = static_cast<float2*>(it.y);
    c.mat = it.mat;
    c.shift = (float)it.shift;
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
    T::init(c, min(tid, n - 1), r);
    if (!live) r.flags = 0;
    if (tid < NS) mbar_init(&full[tid], n);
    fence_mbar_init();
    __syncthreads();
    const int kfirst = c.k0 - 2, klast = c.k0 + c.tz + 1;  // planes of x
    if (live) {  // k0 is even: planes k0 - 2 .. k0 + 1 have parities 0, 1, 0, 1
        T::template stage<0>(c, sh, r, kfirst, 0);
        copies_arrive(&full[0]);
        T::template stage<1>(c, sh, r, kfirst + 1, 1);
        copies_arrive(&full[1]);
        T::template stage<0>(c, sh, r, kfirst + 2, 2);
        copies_arrive(&full[2]);
        T::template stage<1>(c, sh, r, kfirst + 3, 3);
        copies_arrive(&full[3]);
        r.mcur = T::template read_mat<1>(c, r, c.k0 - 1);
    }
    bool ok = bounded_wait(&full[0], 0, B.wait_limit) && bounded_wait(&full[1], 0, B.wait_limit) &&
              bounded_wait(&full[2], 0, B.wait_limit);
    if (ok && live) {
        T::template settle<0>(c, sh, r, kfirst, 0);
        T::template settle<1>(c, sh, r, kfirst + 1, 1);
        T::template settle<0>(c, sh, r, kfirst + 2, 2);
    }
    ok = __syncthreads_and(ok);
    auto step = [&](auto parity, int kf, int j) {
        constexpr int Q = decltype(parity)::value;
        const int sm = j & 3, sn = (j + 3) & 3;
        if (live) {
            if (kf < c.k0 + c.tz) r.mnext = T::template read_mat<1 - Q>(c, r, kf + 1);
            T::template flux<Q>(c, sh, r, sm, (j + 1) & 3, (j + 2) & 3);
        }
        __syncthreads();
        T::template gather<Q>(c, sh, r, kf, sm);
        if (kf + 3 <= klast && live) {  // plane kf - 1 has had its last reader
            T::template stage<1 - Q>(c, sh, r, kf + 3, sm);
            copies_arrive(&full[sm]);
        }
        if (kf + 2 <= klast) {
            ok = bounded_wait(&full[sn], ((j + 3) >> 2) & 1, B.wait_limit);
            if (ok && live) T::template settle<Q>(c, sh, r, kf + 2, sn);
        }
        r.mcur = r.mnext;
        ok = __syncthreads_and(ok);
    };
    for (int kf = c.k0 - 1, j = 0; ok && kf <= c.k0 + c.tz; kf += 2, j += 2) {
        step(std::integral_constant<int, 1>(), kf, j);
        if (!ok) break;
        step(std::integral_constant<int, 0>(), kf + 1, j + 1);
    }
    asm volatile("cp.async.wait_all;" ::: "memory");  // nothing lands after the CTA has gone
    if (!ok && tid == 0) atomicExch(B.err, 1);
    if (c.dot) {
        double v = (double)r.dot;
        for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
        if ((tid & 31) == 0) red[tid >> 5] = v;
        __syncthreads();
        if (tid == 0) {
            double s = 0.0;
            for (int w = 0; w < (int)(blockDim.x >> 5); ++w) s += red[w];
            const int sub = G.full ? (int)(blockIdx.y & 3) * (int)gridDim.x : 0;
            dot_partials[(int64_t)it.dot_slot * dot_stride + sub + blockIdx.x] =
                ok ? s : __longlong_as_double(0x7ff8000000000000LL);
        }
    }
}

template <bool CUBIC, int MATK>
int launch_cell_t(const StencilParams<float>& P, const CellBatch& B, const CellGeom& G, double* dp, int ds, cudaStream_t s) {
    using T = CellApply<CUBIC, MATK>;
    auto kern = cell_apply<CUBIC, MATK>;
    PC_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, 56 << 10));
    const dim3 grid(G.ntx * G.nty * G.nch, B.n * (G.full ? 4 : 1));
    kern<<<grid, (G.ncell + 31) / 32 * 32, T::shared_bytes(), s>>>(P, B, G, dp, ds);
    note_launch();
    note_apply_launch();
    PC_CUDA_TRY(cudaGetLastError());
    return PC_OK;
}

}  // namespace

int cell_apply_ctas(int N, bool full, int nitems, int tz_in, int* tz) {
    CellGeom G;
    make_cell_geom(G, N, full, true);
    if (tz_in > 0) {
        cell_planes(G, tz_in);
    } else {
        const double rate[3] = {1.0, 1.9, 2.6};
        cell_chunks(G, std::min(nitems, kCellMaxItems), device_sm_count(), rate, 3);
    }
    if (tz) *tz = G.tz;
    return G.ntx * G.nty * G.nch * (full ? 4 : 1);
}

int launch_apply_cell(bool full, bool cubic, int matkind, const StencilParams<float>& P, const ApplyItem* items,
                      const double* item_ph, int nitems, int tz, double* dp, int ds, int* err, cudaStream_t s) {
    CellGeom G;
    make_cell_geom(G, P.N, full, true);
    cell_planes(G, tz);
    if (dp != nullptr && G.ntx * G.nty * G.nch * (full ? 4 : 1) > ds)
        return fail(PC_EINVAL, "apply: launch has more CTAs than partial-sum slots");
    for (int base = 0; base < nitems; base += kCellMaxItems) {
        CellBatch B;
        B.n = std::min(nitems - base, kCellMaxItems);
        B.wait_limit = wait_limit();
        B.err = err;
        for (int i = 0; i < B.n; ++i) {
            B.it[i] = items[base + i];
            for (int e = 0; e < 6; ++e) B.ph[i][e / 2][e % 2] = (float)item_ph[(size_t)6 * (base + i) + e];
        }
        int rc;
        if (cubic) rc = matkind ? launch_cell_t<true, 1>(P, B, G, dp, ds, s) : launch_cell_t<true, 0>(P, B, G, dp, ds, s);
        else rc = matkind ? launch_cell_t<false, 1>(P, B, G, dp, ds, s) : launch_cell_t<false, 0>(P, B, G, dp, ds, s);
        PC_TRY(rc);
    }
    return PC_OK;
}

}  // namespace pc
