// direct.cu -- the direct FP32 evaluation of Eq. 1 (steps A2-A5).
//
// Design (sm_103a):
//  * Phase.  The phase of Eq. 1 in turns splits exactly into an x part and a
//    y part, Q_j (x - x_j)^2 + Q_j (y - y_j)^2.  Each part is evaluated once
//    per (point, pixel column) and (point, pixel row) -- not per pixel -- in
//    64-bit fixed-point turns (exact modulo one turn; this is the exact
//    integer form of the paper's Eq. 2 recurrence, Section 2.1, which also
//    avoids recomputing the full phase per pixel), then rounded to an FP32
//    angle in [-pi, pi).  Per pixel only theta_x + theta_y remains: one add.
//  * Tables.  These per-axis angles are written once per call into tables
//    laid out tile by tile, so that the slice a CTA needs for one stage of
//    points is one contiguous block: [x tile][point][x in tile].
//  * Staging.  Point tiles are staged in shared memory by 1-D bulk copies
//    (cp.async.bulk, mbarrier completion), NST stages deep -- the paper's
//    shared-memory staging of 256 points per barrier (Section 2.1).
//  * Work per thread.  Each thread owns a VX x VY block of pixels (the
//    paper's float8 "eight pixels per item", Section 2.1).  The rotation
//    tiles (the heuristic's choice) take one hardware sincos per thread and
//    point and reach the block's other pixels by angle addition with the
//    tables' cosines and sines; the others a cosine per pixel (the paper's
//    native cos).
//  * Bound.  The rotation tiles: the FMA pipe (2 multiply-adds per update) and
//    the shared-memory reads beside it.  With packed 16x4 blocks the pipe is
//    73% and the shared-memory data path 76% busy (3840x2160x2048): 41.5
//    updates per clock and SM of 58.5.  1920x1024x1024 204 -> 167 us,
//    3840x2160x16384 11.13 -> 10.28 ms against scalar 16x4 blocks with the
//    groups' sums stored in place.  Cosine-per-pixel tiles: the MUFU.
//
// Accuracy: angle rounding about 2^-22 rad per axis, __cosf absolute error
// about 2^-21 on |x| <= pi, FP32 accumulation: far inside
// max |I - I_ref| <= 1e-4 sum |A_j|.
#include <math.h>

#include "common.cuh"
#include "direct_table.cuh"
#include "direct_tile.cuh"
#include "point_rec.cuh"

namespace cgh {

// ------------------------------------------------------------ tables
// One block per DT_POINTS points (grid x) and DT_SPAN pixel columns or rows
// (grid y: the x range, then the y range); see direct_table.cuh.
// FUSE: the block builds its DT_POINTS records itself from the caller's
// points (step A1, as in prologue.cu) instead of reading them from `rec`;
// each record is then built once per block row of grid y, a few FP64
// operations each, which costs less than a separate kernel in the chain.
template <bool FUSE>
__global__ void __launch_bounds__(DT_SPAN)
direct_tables_kernel(const PointRec *__restrict__ rec, PointSource src, DirectTables dt,
                     unsigned *__restrict__ zero, int nzero) {
    __shared__ PointRec srec[DT_POINTS];
    // No early trigger for the direct kernel: placed while this kernel still
    // runs, its CTAs would double up on the SMs that are free first
    // (640x480x300: 26 us against 18; nothing gained elsewhere).
    pdl_wait();  // the records (or the caller's points) come from the kernel before
    // the split schedule's per-tile arrival counters start at zero (every
    // earlier kernel on the stream has finished: pdl_wait above)
    if (blockIdx.x == 0)
        for (int k = blockIdx.y * blockDim.x + threadIdx.x; k < nzero;
             k += gridDim.y * blockDim.x)
            zero[k] = 0u;
    const int j0 = blockIdx.x * DT_POINTS;
    if (threadIdx.x < DT_POINTS && j0 + (int)threadIdx.x < dt.Npad) {
        if constexpr (FUSE)
            srec[threadIdx.x] =
                make_point_rec(src.points, src.A, src.z, src.N, j0 + threadIdx.x,
                               src.K, src.status, src.y0);
        else
            srec[threadIdx.x] = rec[j0 + threadIdx.x];
    }
    __syncthreads();
    const int npts = dt.Npad - j0 < DT_POINTS ? dt.Npad - j0 : DT_POINTS;
    direct_table_block(dt, srec, j0, npts, blockIdx.y);
}

// ------------------------------------------------------- direct kernel
// One CTA per pixel tile (1-D grid, tiles in row-major order), except for
// the last tiles when their count does not spread evenly over the SMs: the
// tiles from `tail` on are each cut into `m` chunks of point stages, one CTA
// per chunk, placed after the whole tiles in the grid so that they fill the
// SMs that finish first.  Each chunk CTA writes its partial tile to `part`
// (slot = chunk index) and counts itself in count[tile - tail]; the last to
// arrive adds the m partials in chunk order -- the same order whoever is
// last, so the result is deterministic -- and writes the tile.  No CTA waits
// for another.
template <int TX, int TY, int VX, int VY, int PT, int NST, int NP, int G, int PK>
__global__ void __launch_bounds__(DirectTileLoop<TX, TY, VX, VY, PT, NST, NP, G, PK>::S::THREADS,
                                    DirectTileLoop<TX, TY, VX, VY, PT, NST, NP, G, PK>::MIN_CTAS)
direct_fwd_kernel(const float *__restrict__ phx, const float *__restrict__ phy,
                  const float *__restrict__ amp, int Npad, int Nx, int Ny,
                  int nxt, int tail, int m, float *__restrict__ out,
                  int vec_store, float *__restrict__ part,
                  unsigned *__restrict__ count, unsigned *status) {
    using L = DirectTileLoop<TX, TY, VX, VY, PT, NST, NP, G, PK>;
    using S = typename L::S;
    extern __shared__ __align__(128) float smem[];
    __shared__ __align__(8) uint64_t full[NST];
    __shared__ volatile int abort_flag;
    __shared__ int s_last;

    if (threadIdx.x == 0) {
        abort_flag = 0;
        for (int s = 0; s < NST; ++s) mbar_init(&full[s], 1);
        mbar_fence_init();
    }
    pdl_wait();  // the tables (and zeroed counters) come from the kernel before
    __syncthreads();

    const int nst = Npad / PT;  // point stages per tile
    int tile = (int)blockIdx.x, s0 = 0, s1 = nst, q = -1;
    if (tile >= tail) {  // a chunk of a split tile
        q = tile - tail;
        tile = tail + q / m;
        const int k = q % m;
        s0 = (int)((long long)nst * k / m);
        s1 = (int)((long long)nst * (k + 1) / m);
    }
    const int xt = tile % nxt, yt = tile / nxt;
    typename L::Acc acc;
    acc.zero();
    if (!L::accumulate(smem, full, &abort_flag,
                       phx + (size_t)xt * Npad * TX * L::XF + (size_t)s0 * S::SX,
                       phy + (size_t)yt * Npad * TY * L::YF + (size_t)s0 * S::SY,
                       amp + (size_t)s0 * PT, s1 - s0, acc, status))
        return;
    // only the stores are left: the next kernel of the stream may launch
    pdl_trigger();
    if (q < 0) {
        L::store(acc, smem, xt, yt, Nx, Ny, out, vec_store);
        return;
    }
    // publish this chunk's partial tile, then count in
    if constexpr (L::QUADS) {
        float4 v[L::NQ];
        L::reduce_quads(acc, smem, v);
        float4 *dst = reinterpret_cast<float4 *>(part + (size_t)q * TX * TY);
#pragma unroll
        for (int i = 0; i < L::NQ; ++i) dst[threadIdx.x + i * S::THREADS] = v[i];
        __threadfence();
        __syncthreads();
        if (threadIdx.x == 0)
            s_last = atomicAdd(&count[tile - tail], 1u) == (unsigned)(m - 1);
        __syncthreads();
        if (!s_last) return;
        __threadfence();
        const float4 *src =
            reinterpret_cast<const float4 *>(part + (size_t)(tile - tail) * m * TX * TY);
#pragma unroll
        for (int i = 0; i < L::NQ; ++i) v[i] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        for (int k = 0; k < m; ++k, src += TX * TY / 4)
#pragma unroll
            for (int i = 0; i < L::NQ; ++i) {
                const float4 p = __ldcg(src + threadIdx.x + i * S::THREADS);
                v[i].x += p.x;
                v[i].y += p.y;
                v[i].z += p.z;
                v[i].w += p.w;
            }
        L::write_quads(v, xt, yt, Nx, Ny, out, vec_store);
        return;
    }
    L::reduce_groups(acc, smem);
    const int lt = threadIdx.x % S::GT, grp = threadIdx.x / S::GT;
    const int tx = lt % S::NTX, ty = lt / S::NTX;
    const int off = (ty * VY) * TX + tx * VX;
    if (grp == 0) {
        float *dst = part + (size_t)q * TX * TY + off;
#pragma unroll
        for (int r = 0; r < VY; ++r)
#pragma unroll
            for (int k = 0; k < VX; ++k) dst[r * TX + k] = acc.get(r, k);
        __threadfence();
    }
    __syncthreads();
    if (threadIdx.x == 0)
        s_last = atomicAdd(&count[tile - tail], 1u) == (unsigned)(m - 1);
    __syncthreads();
    if (s_last && grp == 0) {
        __threadfence();
        acc.zero();
        const float *src = part + (size_t)(tile - tail) * m * TX * TY + off;
        for (int k = 0; k < m; ++k, src += TX * TY)
#pragma unroll
            for (int r = 0; r < VY; ++r)
#pragma unroll
                for (int c = 0; c < VX; ++c) acc.add(r, c, __ldcg(src + r * TX + c));
        L::write_out(acc, xt, yt, Nx, Ny, out, vec_store);
    }
}

// ------------------------------------------------------- naive kernel
// One thread per pixel, plain loop over points (the paper's unoptimised
// kernel, Fig. 2b, restated): exact 64-bit fixed-point phase, cospif.
__global__ void naive_fwd_kernel(const PointRec *__restrict__ rec, int N,
                                 int Nx, int Ny, float *__restrict__ out) {
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    const int y = blockIdx.y;
    if (x >= Nx || y >= Ny) return;
    float acc = 0.0f;
    for (int j = 0; j < N; ++j) {
        const PointRec r = rec[j];
        uint64_t ph = axis_phase(r.c, r.bx, r.ax, x) + axis_phase(r.c, r.by, r.ay, y);
        float turns = (float)phase_hi(ph) * TURN_PER_U32;
        acc = fmaf(r.A, cospif(2.0f * turns), acc);
    }
    out[(size_t)y * Nx + x] = acc;
}

// ------------------------------------------------------------ registry

static const DirectTile kTiles[] = {
#define X(tx, ty, vx, vy, pt, ns, np, g, pk) {tx, ty, vx, vy, pt, np, g, pk},
    CGH_DIRECT_TILES(X)
#undef X
};
static constexpr int kNumTiles = sizeof(kTiles) / sizeof(kTiles[0]);

int direct_tile_count() { return kNumTiles; }
DirectTile direct_tile_get(int i) { return kTiles[i]; }
int direct_tile_index(const DirectTile &t) {
    for (int i = 0; i < kNumTiles; ++i)
        if (kTiles[i].tx == t.tx && kTiles[i].ty == t.ty && kTiles[i].vx == t.vx &&
            kTiles[i].vy == t.vy && kTiles[i].pt == t.pt && kTiles[i].np == t.np &&
            kTiles[i].g == t.g && kTiles[i].pk == t.pk)
            return i;
    return -1;
}

size_t direct_phase_table_floats(const DirectTile &t, int Npad, int Nx,
                                 int Ny) {
    const int nxt = (Nx + t.tx - 1) / t.tx, nyt = (Ny + t.ty - 1) / t.ty;
    return direct_x_floats(t, nxt, Npad) + direct_y_floats(t, nyt, Npad);
}

static cudaError_t launch_tables(const PointRec *rec, const PointSource *src,
                                 int Npad, int Nx, int Ny, const DirectTile &t,
                                 float *phx, float *phy, float *amp,
                                 unsigned *zero, int nzero, cudaStream_t s) {
    const DirectTables dt{Npad, t.tx, t.ty, direct_xg(t), direct_yg(t), (Nx + t.tx - 1) / t.tx,
                          (Ny + t.ty - 1) / t.ty, phx, phy, amp};
    dim3 grid((Npad + DT_POINTS - 1) / DT_POINTS, dt.spans());
    if (src)  // (builds the records itself: the call's first kernel)
        return launch_kernel(false, direct_tables_kernel<true>, grid, dim3(DT_SPAN), 0, s,
                             (const PointRec *)nullptr, *src, dt, zero, nzero);
    return launch_dependent(direct_tables_kernel<false>, grid, dim3(DT_SPAN), 0, s, rec,
                            PointSource{}, dt, zero, nzero);
}

cudaError_t launch_direct_tables(const PointRec *rec, int Npad, int Nx, int Ny,
                                 const DirectTile &t, float *phx, float *phy,
                                 float *amp, unsigned *zero, int nzero,
                                 cudaStream_t s) {
    return launch_tables(rec, nullptr, Npad, Nx, Ny, t, phx, phy, amp, zero, nzero, s);
}

cudaError_t launch_direct_tables_fused(const PointSource &src, int Npad, int Nx,
                                       int Ny, const DirectTile &t, float *phx,
                                       float *phy, float *amp, unsigned *zero,
                                       int nzero, cudaStream_t s) {
    return launch_tables(nullptr, &src, Npad, Nx, Ny, t, phx, phy, amp, zero, nzero, s);
}

static const int kTileCtas[] = {
#define X(tx, ty, vx, vy, pt, ns, np, g, pk) \
    DirectTileLoop<tx, ty, vx, vy, pt, ns, np, g, pk>::SM_CTAS,
    CGH_DIRECT_TILES(X)
#undef X
};

int direct_tile_ctas(int i) { return kTileCtas[i]; }

// Which tiles to cut, and into how many chunks.  An SM gets through its CTAs
// at about the same rate however many it holds (one alone 7% slower), so the
// whole tiles are as many as share out evenly, and the others are cut so that
// the busiest SM has the fewest points left, a chunk counted 20 points more
// than its share, the cutting itself 60, and the sum of a tile's chunks the
// time of 34000 updates (0.4 us) each.  All tiles
// are cut where the whole ones would fill some of an SM's places only: 800x600
// x2000 (247 tiles) 96 us against 110 with one whole tile per SM.  Kernel
// times by the count of chunks follow this: 1023x767x1999, 80 tiles to cut,
// 138 us in 11 chunks, 143 in 4 (always two chunks per SM, the former rule),
// 156 in 2 or whole; 300x200x5000, 35 tiles, 41 us in 8, 51 in 9; 1920x1080
// x4096, 108 tiles, 660 us in 4, 684 in 3; 1500x900x200 39 whole, 42 cut.
// full: up to 8 chunks per SM, else 2 (less scratch).
DirectSplit direct_split_plan(int tile_index, int sm_count, int Npad, int Nx,
                              int Ny, bool split, bool full) {
    const DirectTile &t = kTiles[tile_index];
    DirectSplit d;
    d.tiles = ((Nx + t.tx - 1) / t.tx) * ((Ny + t.ty - 1) / t.ty);
    d.tail = d.tiles;
    d.m = 1;
    const int nst = Npad / t.pt;
    d.points = sm_count > 0 ? (double)((d.tiles + sm_count - 1) / sm_count) * Npad : 0.0;
    if (!split || sm_count < 1 || nst < 2 || d.tiles % sm_count == 0) return d;
    const int slots = sm_count * kTileCtas[tile_index];
    const int most = (full ? 8 : 2) * sm_count;
    const int even = d.tiles - d.tiles % sm_count;
    for (int tail = even; tail >= 0; tail -= even > 0 ? even : 1) {
        const int rest = d.tiles - tail;
        for (int m = 2; m <= nst && rest * m <= most; ++m) {
            const int ctas = tail + rest * m;
            if (tail > 0 && tail < slots && ctas > slots) break;
            const int rounds = (rest * m + sm_count - 1) / sm_count;
            double points = (double)tail / sm_count * Npad +
                            rounds * (double)((nst + m - 1) / m * t.pt + 20) + 60.0 +
                            m * 34000.0 / (t.tx * t.ty);
            if (ctas <= sm_count) points *= 1.07;
            if (points < d.points) {
                d.points = points;
                d.tail = tail;
                d.m = m;
            }
        }
        if (even >= slots) break;
    }
    return d;
}

template <int TX, int TY, int VX, int VY, int PT, int NST, int NP, int G, int PK>
static cudaError_t launch_one(const float *phx, const float *phy,
                              const float *amp, int Npad, int Nx, int Ny,
                              float *out, const DirectSplit &d, float *part,
                              unsigned *count, unsigned *status, cudaStream_t s) {
    using S = typename DirectTileLoop<TX, TY, VX, VY, PT, NST, NP, G, PK>::S;
    auto kern = direct_fwd_kernel<TX, TY, VX, VY, PT, NST, NP, G, PK>;
    static bool attr_set[64] = {};
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev < 0 || dev >= 64 || !attr_set[dev]) {
        cudaError_t e = cudaFuncSetAttribute(
            kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)S::SMEM);
        if (e != cudaSuccess) return e;
        if (dev >= 0 && dev < 64) attr_set[dev] = true;
    }
    const int nxt = (Nx + TX - 1) / TX;
    const unsigned grid = (unsigned)d.tail + (unsigned)(d.tiles - d.tail) * d.m;
    int vec_store = (Nx % 4 == 0) && (((uintptr_t)out & 15) == 0);
    return launch_dependent(kern, dim3(grid), dim3(S::THREADS), S::SMEM, s, phx, phy,
                            amp, Npad, Nx, Ny, nxt, d.tail, d.m, out, vec_store, part,
                            count, status);
}

cudaError_t launch_direct_forward(int tile_index, const float *phx,
                                  const float *phy, const float *amp, int Npad,
                                  int Nx, int Ny, float *out,
                                  const DirectSplit &d, float *part,
                                  unsigned *count, unsigned *status,
                                  cudaStream_t s) {
    if (d.tail < d.tiles && (!part || !count)) return cudaErrorInvalidValue;
    int i = 0;
#define X(tx, ty, vx, vy, pt, ns, np, g, pk)                                   \
    if (tile_index == i)                                                       \
        return launch_one<tx, ty, vx, vy, pt, ns, np, g, pk>(                   \
            phx, phy, amp, Npad, Nx, Ny, out, d, part, count, status, s);      \
    ++i;
    CGH_DIRECT_TILES(X)
#undef X
    return cudaErrorInvalidValue;
}

cudaError_t launch_naive_forward(const PointRec *rec, int N, int Nx, int Ny,
                                 float *out, cudaStream_t s) {
    dim3 grid((Nx + 127) / 128, Ny);
    naive_fwd_kernel<<<grid, 128, 0, s>>>(rec, N, Nx, Ny, out);
    return cudaGetLastError();
}

}  // namespace cgh
