// Tiles of one cell per thread, shared by the integer-pipe complex128 apply (pc_apply_int.cuh) and the
// complex64 cell apply (pc_apply_cell.cuh).
//
// A CTA owns TX x TY columns of the quarter grid and marches through tz planes; a full-space vector is
// treated as its four parity blocks with strided addresses (the blocks do not couple), so one geometry
// serves both layouts.  Which columns beyond its own a tile touches follows from the operator (see
// pc_apply_tile.cuh): the flux of a node reads x at column offset i0 - 1 and row offsets j0 - 1, j0 of
// the planes next to it, and an output reads fluxes at column offset i0 and row offsets j0, j0 - 1, with
// i0 = (k + p13) mod 2, j0 = (k + p12 + p13) mod 2 of the plane.  So every plane needs one more column,
// a0 + TX or a0 - 1 by its parity, and the rows b0 - 1 and b0 + TY.
//
// Threads: the TX x TY output columns first, then that column, then the row b0 + TY, then the row b0 - 1,
// so that whatever wraps around the unit cell sits in the last warps.  In shared memory the cells of a
// plane lie row by row with TX + 1 columns in their order in space (which of the two extra columns a row
// holds depends on the plane's parity), so the accesses of a warp run along consecutive cells.
#pragma once

#include <stdint.h>

#include "pc_complex.cuh"

namespace pc {

constexpr int kCells = 256;  // most cells (threads) of a CTA, and the stride of its shared arrays: a
                             // constant, so that an access is a register and an immediate offset

struct CellGeom {
    int X, Y, Z;   // quarter-grid extents (N/2, N/2, N)
    int N, full;   // full-space layout: addresses of the full grid
    int TX, TY, ntx, nty, ncell;
    int tz, nch;
    int plane, vstr;  // nodes per plane and per component of the vector layout (N <= 1024: below 2^31)
};

// Tile extents: least warps over the whole plane with at most kCells cells per CTA (ties: the larger
// tile).  rows16 (complex64): widths that are no multiple of 16 count 15 % more, because half-warps of
// 8-byte accesses then straddle two rows and the gap between them costs a bank conflict (N = 160, 4 items:
// 106 us with 16-wide tiles, 143 us with 20-wide ones; N = 128, 8 items: 119 to 105 us), and narrow tiles,
// which read short rows of x, 30 %.
inline void make_cell_geom(CellGeom& G, int N, bool full, bool rows16) {
    G.N = N;
    G.full = full ? 1 : 0;
    G.X = N / 2;
    G.Y = N / 2;
    G.Z = N;
    G.plane = full ? N * N : G.X * G.Y;
    G.vstr = G.plane * N;
    double best = -1;
    for (int nx = 1; nx <= G.X; ++nx) {
        int tx = (G.X + nx - 1) / nx;
        if (rows16 && tx > 16 && tx % 16 >= 12) tx = (tx + 15) / 16 * 16;  // a little ragged, but whole half-warps
        const int most = kCells / (tx + 1) - 2;
        if (most < 1) continue;
        const int ny0 = (G.Y + most - 1) / most;
        for (int ny = ny0; ny <= G.Y && ny < ny0 + 3; ++ny) {
            const int ty = (G.Y + ny - 1) / ny;
            const int cells = (tx + 1) * (ty + 2);
            const double cost = (double)nx * ny * ((cells + 31) / 32) *
                                (!rows16 || tx % 16 == 0 ? 1.0 : tx < 12 && tx < G.X ? 1.3 : 1.15);
            if (best < 0 || cost < best) {
                best = cost;
                G.TX = tx;
                G.TY = ty;
                G.ntx = (G.X + tx - 1) / tx;
                G.nty = (G.Y + ty - 1) / ty;
                G.ncell = cells;
            }
        }
    }
    G.tz = G.Z;
    G.nch = 1;
}

// Chunks of planes per tile for a launch of nitems vectors on sm SMs.  A chunk repeats two flux planes
// and loads three more of x (counted as four planes), so few chunks are best once every SM has work;
// below that more CTAs shorten the march.  rate[r - 1]: planes per unit of time that r resident CTAs of an
// SM finish together (r = 1 .. rmax); the fullest SM's CTAs run in waves of rmax.
inline void cell_chunks(CellGeom& G, int nitems, int sm, const double* rate, int rmax) {
    const long base = (long)G.ntx * G.nty * (G.full ? 4 : 1) * (nitems > 1 ? nitems : 1);
    double best = -1;
    for (int tz = 2; tz <= G.Z; tz += 2) {
        const int nch = (G.Z + tz - 1) / tz;
        const long per = (base * nch + sm - 1) / sm, rem = per % rmax;
        const double cost = (tz + 4) * (per / rmax * (rmax / rate[rmax - 1]) + (rem ? rem / rate[rem - 1] : 0.0));
        if (best < 0 || cost < best) {
            best = cost;
            G.tz = tz;
            G.nch = nch;
        }
    }
}

// Planes per CTA: even, so that every chunk starts on an even plane and the march's plane parities are
// known at compile time (step kf = k0 - 1 is odd).
inline void cell_planes(CellGeom& G, int tz) {
    G.tz = tz < 1 ? 2 : (tz >= G.Z ? G.Z : (tz + 1) / 2 * 2);
    G.nch = (G.Z + G.tz - 1) / G.tz;
}

// A thread's cell: where its node lies and which cells it exchanges with, by plane parity.
struct CellMap {
    int off[2];  // in-plane offset of the cell's node
    int wab[2];  // (wa + 1) + 3 (wb + 1) of that node
    int own[2];  // its place among the plane's cells
    int nb[2];   // backward neighbour cells (next planes), s2 = +1 low half, -1 high half (flux)
    int gn[2];   // forward flux cells (next planes), s2 = +1 low half, -1 high half (gather)
    int flags;   // bit 0, 1: flux on even, odd planes; bit 2: output
};

PC_HD int cell_wrap(int v, int n, int& w) {
    w = v < 0 ? -1 : (v >= n ? 1 : 0);
    return v - w * n;
}

// place of tile column cx in [-i0, TX - i0], row r in [-1, TY] on a plane of offset i0
PC_HD int cell_of(const CellGeom& G, int i0, int cx, int r) { return (r + 1) * (G.TX + 1) + cx + i0; }

PC_HD void cell_init(const CellGeom& G, int a0, int b0, int p12, int p13, int tid, CellMap& r) {
    const int main = G.TX * G.TY;
    int cx, row;
    if (tid < main) {
        row = tid / G.TX;
        cx = tid - row * G.TX;
    } else if (tid < main + G.TY) {
        cx = G.TX;
        row = tid - main;
    } else {
        const int e = tid - main - G.TY;
        row = e > G.TX ? -1 : G.TY;
        cx = e > G.TX ? e - (G.TX + 1) : e;
    }
    r.flags = 0;
    if (tid < main && a0 + cx < G.X && b0 + row < G.Y) r.flags |= 4;
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        const int i0 = (q + p13) & 1, j0 = (q + p12 + p13) & 1;
        int wa, wb;
        if (cx == G.TX && i0) r.own[q] = cell_of(G, i0, -1, row);
        else r.own[q] = cell_of(G, i0, cx, row);
        const int a = cell_wrap(a0 + ((cx == G.TX && i0) ? -1 : cx), G.X, wa);
        const int b = cell_wrap(b0 + row, G.Y, wb);
        r.off[q] = G.full ? (2 * a + i0) + G.N * (2 * b + j0) : a + G.X * b;
        r.wab[q] = (wa + 1) + 3 * (wb + 1);
        // fluxes: columns a0 .. a0 + TX - i0, rows b0 - j0 .. b0 + TY - j0
        const bool f = (cx < G.TX || !i0) && row >= -j0 && row <= G.TY - j0;
        if (f) r.flags |= 1 << q;
        r.nb[q] = r.gn[q] = 0;
        if (f) r.nb[q] = cell_of(G, 1 - i0, cx + i0 - 1, row + j0 - 1) | (cell_of(G, 1 - i0, cx + i0 - 1, row + j0) << 16);
        if (tid < main) r.gn[q] = cell_of(G, 1 - i0, cx + i0, row + j0) | (cell_of(G, 1 - i0, cx + i0, row + j0 - 1) << 16);
    }
}

}  // namespace pc
