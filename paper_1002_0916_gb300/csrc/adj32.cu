// adj32.cu -- the separable adjoint of Eq. 1 at FP32 accuracy on the tensor
// cores.
//
// For a loss with G = dL/dI (Ny x Nx), phi = P_j r^2, dx = x - x_j, dy = y -
// y_j (Section 1, Eq. 1):
//     dL/dA_j = sum G cos(phi)
//     dL/dx_j = 2 P_j A_j sum G sin(phi) dx      (and the same for y)
//     dL/dz_j = (P_j A_j / z_j) sum G sin(phi) (dx^2 + dy^2)
// With U = e^{i th_x}, V = e^{i th_y}, sum_{x,y} G e^{i phi} w(x) = sum_x w(x)
// U[x] (sum_y G[y][x] V[y]): two products,
//     D1[2j+c][x] = sum_y V'[2j+c][y] G[y][x],  D2[2j+c][y] = sum_x U'[2j+c][x] G[y][x],
// U', V' the cosine and sine rows, whose epilogues (sep32.cu) weight D1 with
// U and 1, dx, dx^2, and D2 with V and dy, dy^2.
//
// Both run on the product kernel of sep32.cu: every FP32 factor as two FP16
// numbers, partial sums added in FP32 every 64 values of k.  U', V' are
// scaled by 2^14 and G by the power of two that brings max |G| into [2^13,
// 2^14); the sums come out in units of 2^floor(log2 max |G|), an FP32 number
// for every G.  Four launches:
//   1. the largest |G| of a run of pixels per block, and, in the blocks
//      behind those, the tables U', V' with their point records;
//   2. G to FP16 hi and lo in both orientations;
//   3. both products, one grid;
//   4. the partial sums added in a fixed order, per-point factors
//      (backward.cu).
// Points are taken in chunks whose tables stay within TABLE_BYTES.
// Bound: the MMAs of 3 (76% of the tensor pipe's cycles, 128 us of 166 at
// 1920x1080x4096).  The whole adjoint there took 1577 us as FP32 sums on the
// FMA pipe, and 232 us as split-FP16 products with one accumulation over all of
// K; the gradients are closer to FP64 than either's.
#include <cuda_fp16.h>
#include <math.h>

#include "api_internal.h"
#include "common.cuh"
#include "point_rec.cuh"
#include "sep32.cuh"

namespace cgh {

constexpr int A32_THREADS = 256;
constexpr int A32_MAX_BLOCKS = 304;            // blocks of the |G| maximum
constexpr int A32_POINTS = 32;                 // points per table block
constexpr int A32_RUN = 8;                     // coordinates per thread and point
constexpr int A32_SPAN = 32 * A32_RUN;         // coordinates per table block
constexpr size_t TABLE_BYTES = (size_t)1 << 30;

// max |G| over this block's share, NaN kept.
__device__ __forceinline__ float nan_max(float a, float b) { return b > a || b != b ? b : a; }

__device__ __forceinline__ float block_max(float m, float *sm) {
    for (int o = 16; o > 0; o >>= 1) m = nan_max(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((threadIdx.x & 31) == 0) sm[threadIdx.x >> 5] = m;
    __syncthreads();
    m = sm[0];
    for (int w = 1; w < A32_THREADS / 32; ++w) m = nan_max(m, sm[w]);
    return m;
}

struct Adj32Tables {
    PointSource src;  // the chunk's points
    int Nx, Ny, ldx, ldy, nbx;
    __half *Uhi, *Ulo, *Vhi, *Vlo;  // [2n][ldx], [2n][ldy]
    PointRec *rec;                  // n, for the products' epilogue
};

// One point's run of A32_RUN coordinates from u0: rows 2j (cos) and 2j + 1
// (sin), hi and lo, one 16-byte store each; the phase is stepped by Eq. 2 in
// exact fixed point.
__device__ __forceinline__ void adj32_run(const PointRec &r, int axis, int u0, __half *hi,
                                          __half *lo, int ld) {
    const uint64_t b = axis ? r.by : r.bx, a = axis ? r.ay : r.ax;
    uint64_t ph = axis_phase(r.c, b, a, u0);
    uint64_t d = r.c * (uint64_t)(2 * (int64_t)u0 + 1) - b;
    const uint64_t dd = 2 * r.c;
    __half2 ch[A32_RUN / 2], cl[A32_RUN / 2], sh[A32_RUN / 2], sl[A32_RUN / 2];
#pragma unroll
    for (int i = 0; i < A32_RUN / 2; ++i) {
        float s[2], c[2];
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            sincos_fixed(ph, s[e], c[e]);
            s[e] *= S32_R_SCALE;
            c[e] *= S32_R_SCALE;
            ph += d;
            d += dd;
        }
        ch[i] = __floats2half2_rn(c[0], c[1]);
        sh[i] = __floats2half2_rn(s[0], s[1]);
        const float2 fc = __half22float2(ch[i]), fs = __half22float2(sh[i]);
        cl[i] = __floats2half2_rn(c[0] - fc.x, c[1] - fc.y);
        sl[i] = __floats2half2_rn(s[0] - fs.x, s[1] - fs.y);
    }
    *reinterpret_cast<uint4 *>(hi) = *reinterpret_cast<const uint4 *>(ch);
    *reinterpret_cast<uint4 *>(lo) = *reinterpret_cast<const uint4 *>(cl);
    *reinterpret_cast<uint4 *>(hi + ld) = *reinterpret_cast<const uint4 *>(sh);
    *reinterpret_cast<uint4 *>(lo + ld) = *reinterpret_cast<const uint4 *>(sl);
}

// Blocks 0 .. nmax - 1: gmax[block].  The others: tables of A32_POINTS
// points over A32_SPAN coordinates (nbx spans of x, then those of y).
__global__ void __launch_bounds__(A32_THREADS)
adj32_prep_kernel(const float *__restrict__ G, long long ng, float *__restrict__ gmax, int nmax,
                  Adj32Tables tb, int spans) {
    __shared__ PointRec srec[A32_POINTS];
    __shared__ float sm[A32_THREADS / 32];
    if ((int)blockIdx.x < nmax) {
        // 16-byte loads from the first aligned element on
        const long long head0 = (long long)((16 - ((uintptr_t)G & 15)) & 15) / 4;
        const long long head = head0 < ng ? head0 : ng, nv = (ng - head) / 4;
        const float4 *V = reinterpret_cast<const float4 *>(G + head);
        const long long step = (long long)nmax * A32_THREADS;
        long long i = (long long)blockIdx.x * A32_THREADS + threadIdx.x;
        float m = 0.0f;
        if (i < head) m = nan_max(m, fabsf(G[i]));
        if (i < ng - head - 4 * nv) m = nan_max(m, fabsf(G[head + 4 * nv + i]));
        for (; i < nv; i += 4 * step) {
            float4 v[4];
#pragma unroll
            for (int k = 0; k < 4; ++k)
                v[k] = i + k * step < nv ? __ldg(V + i + k * step)
                                         : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
#pragma unroll
            for (int k = 0; k < 4; ++k)
                m = nan_max(nan_max(nan_max(m, fabsf(v[k].x)), nan_max(0.0f, fabsf(v[k].y))),
                            nan_max(fabsf(v[k].z), fabsf(v[k].w)));
        }
        m = block_max(m, sm);
        if (threadIdx.x == 0) gmax[blockIdx.x] = m;
        pdl_trigger();
        return;
    }
    const int b = (int)blockIdx.x - nmax;
    const int span = b % spans, j0 = (b / spans) * A32_POINTS;
    const int axis = span >= tb.nbx;
    const int n = axis ? tb.Ny : tb.Nx, ld = axis ? tb.ldy : tb.ldx;
    if (threadIdx.x < A32_POINTS) {
        const int j = j0 + threadIdx.x;
        srec[threadIdx.x] = make_point_rec(tb.src.points, tb.src.A, tb.src.z, tb.src.N, j,
                                           tb.src.K, tb.src.status);
        if (span == 0 && j < tb.src.N) tb.rec[j] = srec[threadIdx.x];
    }
    __syncthreads();
    const int u0 = (span - axis * tb.nbx) * A32_SPAN + (threadIdx.x & 31) * A32_RUN;
    __half *hi = axis ? tb.Vhi : tb.Uhi, *lo = axis ? tb.Vlo : tb.Ulo;
    if (u0 < n)
        for (int q = threadIdx.x >> 5; q < A32_POINTS && j0 + q < tb.src.N; q += A32_THREADS / 32) {
            const size_t off = (size_t)(2 * (j0 + q)) * ld + u0;
            adj32_run(srec[q], axis, u0, hi + off, lo + off, ld);
        }
    pdl_trigger();
}

// G -> scaled FP16 hi and lo, [y][x] (row stride ldx) and [x][y] (ldy), 64 x
// 64 pixels per block through shared memory, two pixels per store.  The pad
// of a row (up to its stride) is written as zero.
constexpr int GC_T = 64;

__global__ void __launch_bounds__(A32_THREADS)
adj32_convert_kernel(const float *__restrict__ G, int Nx, int Ny, const float *__restrict__ gmax,
                     int nmax, float *__restrict__ gunit, __half *__restrict__ Gr_hi,
                     __half *__restrict__ Gr_lo, int ldx, __half *__restrict__ Gt_hi,
                     __half *__restrict__ Gt_lo, int ldy) {
    __shared__ float tile[GC_T][GC_T + 1];
    __shared__ float sm[A32_THREADS / 32];
    pdl_wait();  // the maxima come from the kernel before
    float m = 0.0f;
    for (int i = threadIdx.x; i < nmax; i += A32_THREADS) m = nan_max(m, gmax[i]);
    m = block_max(m, sm);
    // (no scaling if max |G| is 0 or not finite)
    const int e = m > 0.0f && isfinite(m) ? ilogbf(m) : S32_EXP - 1;
    if (blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0) *gunit = scalbnf(1.0f, e);
    // in two steps: 2^(S32_EXP - 1 - e) itself is no FP32 number for a small G
    const int k = S32_EXP - 1 - e;
    const float s0 = scalbnf(1.0f, k / 2), s1 = scalbnf(1.0f, k - k / 2);
    const int bx = blockIdx.x * GC_T, by = blockIdx.y * GC_T;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int r = warp; r < GC_T; r += A32_THREADS / 32)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int y = by + r, x = bx + lane + 32 * h;
            tile[r][lane + 32 * h] =
                y < Ny && x < Nx ? __ldg(G + (size_t)y * Nx + x) * s0 * s1 : 0.0f;
        }
    __syncthreads();
#pragma unroll
    for (int r = warp; r < GC_T; r += A32_THREADS / 32) {
        const int y = by + r, x = bx + 2 * lane;
        if (y < Ny && x < ldx) {
            const float v0 = tile[r][2 * lane], v1 = tile[r][2 * lane + 1];
            const __half2 h = __floats2half2_rn(v0, v1);
            const float2 f = __half22float2(h);
            *reinterpret_cast<__half2 *>(Gr_hi + (size_t)y * ldx + x) = h;
            *reinterpret_cast<__half2 *>(Gr_lo + (size_t)y * ldx + x) =
                __floats2half2_rn(v0 - f.x, v1 - f.y);
        }
        const int xr = bx + r, yc = by + 2 * lane;
        if (xr < Nx && yc < ldy) {
            const float v0 = tile[2 * lane][r], v1 = tile[2 * lane + 1][r];
            const __half2 h = __floats2half2_rn(v0, v1);
            const float2 f = __half22float2(h);
            *reinterpret_cast<__half2 *>(Gt_hi + (size_t)xr * ldy + yc) = h;
            *reinterpret_cast<__half2 *>(Gt_lo + (size_t)xr * ldy + yc) =
                __floats2half2_rn(v0 - f.x, v1 - f.y);
        }
    }
    pdl_trigger();
}

}  // namespace cgh

using namespace cgh;

cgh_status cgh_ctx::backward_sep32(const float *points, const float *A, const float *z, int N,
                                   double lambda, double p, int Nx, int Ny, const float *G,
                                   float *gpts, float *gA, float *gz, int timer,
                                   cudaStream_t s) {
    const int ldx = pad_to(Nx, 8), ldy = pad_to(Ny, 8);
    const size_t per_point = 8 * ((size_t)ldx + ldy);  // table bytes
    long long most = (long long)(TABLE_BYTES / per_point) / 128 * 128;
    if (most < 128) most = 128;
    const int chunk = N < most ? N : (int)most;
    const Adj32Plan plan = adj32_plan(chunk, Nx, Ny, sm_count);
    // product 0 has the longer K: the x columns' sum runs over y
    const int first = Ny > Nx ? 0 : 1;  // axis of product 0's columns
    const int axis[2] = {first, 1 - first};
    const int cols[2] = {first ? Ny : Nx, first ? Nx : Ny};
    const int K[2] = {first ? Nx : Ny, first ? Ny : Nx};
    const int npad = pad_to(chunk, 32);
    int tiles[2], T[2];
    size_t part_b[2];
    for (int i = 0; i < 2; ++i) {
        tiles[i] = (cols[i] + plan.bn - 1) / plan.bn;
        T[i] = tiles[i] * plan.S[i] * 2;
        part_b[i] = align256((size_t)T[i] * npad * 3 * sizeof(float));
    }
    const size_t u_b = align256((size_t)2 * chunk * ldx * 2);
    const size_t v_b = align256((size_t)2 * chunk * ldy * 2);
    const size_t gr_b = align256((size_t)Ny * ldx * 2), gt_b = align256((size_t)Nx * ldy * 2);
    const size_t max_b = align256((A32_MAX_BLOCKS + 1) * sizeof(float));
    const size_t rec_b = align256((size_t)chunk * sizeof(PointRec));
    cgh_status st = ensure(ws2, max_b + rec_b + part_b[0] + part_b[1] + 2 * (u_b + v_b + gr_b + gt_b), s,
                           "adjoint workspace");
    if (st) return st;
    char *b = (char *)ws2.ptr;
    auto take = [&b](size_t bytes) {
        char *q = b;
        b += bytes;
        return q;
    };
    float *gmax = (float *)take(max_b), *gunit = gmax + A32_MAX_BLOCKS;
    PointRec *rec = (PointRec *)take(rec_b);
    float *part[2] = {(float *)take(part_b[0]), (float *)take(part_b[1])};
    __half *Uhi = (__half *)take(u_b), *Ulo = (__half *)take(u_b);
    __half *Vhi = (__half *)take(v_b), *Vlo = (__half *)take(v_b);
    __half *Grh = (__half *)take(gr_b), *Grl = (__half *)take(gr_b);
    __half *Gth = (__half *)take(gt_b), *Gtl = (__half *)take(gt_b);

    const double Kz = fresnel_scale(lambda, p);
    const long long ng = (long long)Nx * Ny;
    const int spans_x = (Nx + A32_SPAN - 1) / A32_SPAN, spans_y = (Ny + A32_SPAN - 1) / A32_SPAN;
    for (int j0 = 0; j0 < N; j0 += chunk) {
        const int n = N - j0 < chunk ? N - j0 : chunk;
        const PointSource src{points + 2 * (size_t)j0, A + j0, z + j0, n, Kz, d_status};
        long long nmax = (ng + 4 * 4 * A32_THREADS - 1) / (4 * 4 * A32_THREADS);
        if (nmax > A32_MAX_BLOCKS) nmax = A32_MAX_BLOCKS;
        {
            TimedLaunch tl(this, CGH_K_SEP_TABLES, s);
            const int nm = j0 == 0 ? (int)nmax : 0;
            const long long blocks =
                nm + (long long)(spans_x + spans_y) * ((n + A32_POINTS - 1) / A32_POINTS);
            cudaError_t e = launch_kernel(
                false, adj32_prep_kernel, dim3((unsigned)blocks), dim3(A32_THREADS), 0, s, G, ng,
                gmax, nm, Adj32Tables{src, Nx, Ny, ldx, ldy, spans_x, Uhi, Ulo, Vhi, Vlo,
                                                rec},
                spans_x + spans_y);
            if (e != cudaSuccess) return cuda_fail(e, "adjoint tables launch");
            tl.done();
        }
        if (j0 == 0) {
            TimedLaunch tl(this, CGH_K_AUX, s);
            dim3 grid((ldx + GC_T - 1) / GC_T, (ldy + GC_T - 1) / GC_T);
            cudaError_t e =
                launch_dependent(adj32_convert_kernel, grid, dim3(A32_THREADS), 0, s, G, Nx, Ny,
                                 (const float *)gmax, (int)nmax, gunit, Grh, Grl, ldx, Gth, Gtl,
                                 ldy);
            if (e != cudaSuccess) return cuda_fail(e, "G convert launch");
            tl.done();
        }
        {
            TimedLaunch tl(this, timer, s);
            Adj32Args ga{};
            Sep32Operands op[2];
            for (int i = 0; i < 2; ++i) {
                const bool x = axis[i] == 0;
                ga.p[i] = Adj32Prod{((2 * n + 255) / 256) * tiles[i] * plan.S[i],
                                    tiles[i],
                                    plan.S[i],
                                    (K[i] + 63) / 64,
                                    axis[i],
                                    part[i]};
                op[i] = x ? Sep32Operands{Vhi, Vlo, Gth, Gtl, ldy, ldy}
                          : Sep32Operands{Uhi, Ulo, Grh, Grl, ldx, ldx};
            }
            ga.n = n;
            ga.npad = npad;
            ga.tiles_m = (2 * n + 255) / 256;
            ga.rec = rec;
            ga.points = src.points;
            cudaError_t e = launch_adj32(plan.bn, op, cols, K, ga, d_status, s);
            if (e != cudaSuccess) return cuda_fail(e, "adjoint product launch");
            tl.done();
        }
        {
            TimedLaunch tl(this, CGH_K_BWD_REDUCE, s);
            const int ix = axis[0] == 0 ? 0 : 1, iy = 1 - ix;
            const AdjointParts pp{part[ix], part[iy] + npad, T[ix],       T[iy],
                                  3 * (size_t)npad, (size_t)npad};
            cudaError_t e = launch_adjoint_sum(src, pp, gunit,
                                               gpts ? gpts + 2 * (size_t)j0 : nullptr,
                                               gA ? gA + j0 : nullptr, gz ? gz + j0 : nullptr, s);
            if (e != cudaSuccess) return cuda_fail(e, "adjoint reduce launch");
            tl.done();
        }
    }
    return CGH_OK;
}
