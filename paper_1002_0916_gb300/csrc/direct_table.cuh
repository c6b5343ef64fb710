// direct_table.cuh -- the per-axis tables of the direct kernel for a block of
// points, shared by the single-hologram tables kernel (direct.cu) and the
// batch's (batch.cu).  Internal to libcgh.
#pragma once

#include "common.cuh"
#include "direct_tile.cuh"
#include "sep32.cuh"

namespace cgh {

// Points per block: their records are staged in shared memory once, and each
// thread writes one coordinate of DT_SPAN for every point, or, in a rotation
// table, four coordinates of a group for one point at a time.
constexpr int DT_POINTS = 16;
constexpr int DT_SPAN = 256;  // coordinates (and threads) per block

// One coordinate w (column or row, axis 0 = x, 1 = y) of a tile's angle
// table for the npts points of srec: dst[q * stride] = its angle for point q.
__device__ __forceinline__ void angle_column(const PointRec *srec, int npts, int w, int axis,
                                             float *dst, int stride) {
    for (int q = 0; q < npts; ++q) {
        const PointRec &r = srec[q];
        const uint64_t b = axis ? r.by : r.bx, a = axis ? r.ay : r.ax;
        dst[(size_t)q * stride] = (float)phase_hi(axis_phase(r.c, b, a, w)) * RAD_PER_U32;
    }
}

// Four coordinates g0 + k0 .. g0 + k0 + 3 (k0 = 4 h) of one rotation group
// of gs coordinates along an axis (0 = x, 1 = y), for one point: slots k0 ..
// k0 + 3 (cosines of the offsets; slot 0 is the angle at g0) and gs + k0 ..
// gs + k0 + 3 (sines; slot gs is 0), one 16-byte store each into the
// point's row of the table (ng groups per tile).  The offsets are exact in
// fixed point: Phi(g0 + k) - Phi(g0) = k (c (2 g0 + k) - b) for the first,
// then each next one adds the first difference c (2 u + 1) - b, which grows
// by 2 c per coordinate (Eq. 2 on the axis).  sincos_fixed instead of
// sincospif of the rounded offset: 226 -> 199 us at 3840x2160x16384, of which
// writing the 786 MB takes 116.
__device__ __forceinline__ void rotation_quarter(const PointRec &r, int axis, int g0, int g,
                                                 int h, int gs, int ng, float *row) {
    const uint64_t c = r.c, b = axis ? r.by : r.bx, a = axis ? r.ay : r.ax;
    const int k0 = 4 * h;
    uint64_t d = (uint64_t)k0 * (c * (uint64_t)(2 * g0 + k0) - b);
    uint64_t step = c * (uint64_t)(2 * (g0 + k0) + 1) - b;
    float co[4], si[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        sincos_fixed(d, si[i], co[i]);
        d += step;
        step += 2 * c;
    }
    if (k0 == 0) {
        co[0] = (float)phase_hi(axis_phase(c, b, a, g0)) * RAD_PER_U32;
        si[0] = 0.0f;
    }
    *reinterpret_cast<float4 *>(row + rotation_pos(g, k0, ng)) =
        make_float4(co[0], co[1], co[2], co[3]);
    *reinterpret_cast<float4 *>(row + rotation_pos(g, gs + k0, ng)) =
        make_float4(si[0], si[1], si[2], si[3]);
}

// The tables of one hologram: [x tile][point][x in tile], [y tile][point]
// [y in tile] (rotation groups of xg, yg coordinates; 0: plain angles).
struct DirectTables {
    int Npad, TX, TY, xg, yg, nxt, nyt;
    float *phx, *phy, *amp;
    // blocks of DT_SPAN coordinates: the x coordinates, then the y ones
    __host__ __device__ int spans_x() const { return (nxt * TX + DT_SPAN - 1) / DT_SPAN; }
    __host__ __device__ int spans() const {
        return spans_x() + (nyt * TY + DT_SPAN - 1) / DT_SPAN;
    }
};

// Span `span` of the tables for the npts points j0 .. of srec, by DT_SPAN threads.
__device__ __forceinline__ void direct_table_block(const DirectTables &dt, const PointRec *srec,
                                                   int j0, int npts, int span) {
    const int nbx = dt.spans_x();
    const int axis = span >= nbx ? 1 : 0;
    const int w0 = (span - axis * nbx) * DT_SPAN;  // the block's first coordinate
    const int T = axis ? dt.TY : dt.TX, gs = axis ? dt.yg : dt.xg;
    const int n = T * (axis ? dt.nyt : dt.nxt);
    float *tab = axis ? dt.phy : dt.phx;
    if (gs) {
        // a rotation table: one thread per four coordinates and point
        for (int it = threadIdx.x; it < DT_SPAN / 4 * npts; it += DT_SPAN) {
            const int w = w0 + 4 * (it % (DT_SPAN / 4)), q = it / (DT_SPAN / 4);
            if (w >= n) continue;
            const int t = w / T, i = w - t * T, g = i / gs, h = (i - g * gs) >> 2;
            rotation_quarter(srec[q], axis, w - 4 * h, g, h, gs, T / gs,
                             tab + ((size_t)t * dt.Npad + j0 + q) * T * 2);
        }
    } else {
        const int u = w0 + threadIdx.x;
        if (u < n) {
            const int t = u / T, i = u - t * T;
            angle_column(srec, npts, u, axis, tab + ((size_t)t * dt.Npad + j0) * T + i, T);
        }
    }
    if (span == 0 && threadIdx.x < npts) dt.amp[j0 + threadIdx.x] = srec[threadIdx.x].A;
}

}  // namespace cgh
