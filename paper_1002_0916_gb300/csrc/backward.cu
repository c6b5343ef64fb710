// backward.cu -- the hand-written adjoint of Eq. 1 (step A8).
//
// For a loss L with G = dL/dI (Ny x Nx) and phi = P_j r^2 (Section 1,
// Eq. 1; P_j = 2 pi Q_j, dx = x - x_j, dy = y - y_j, dP_j/dz_j = -P_j/z_j):
//     dL/dA_j = sum G cos(phi)
//     dL/dx_j = 2 P_j A_j sum G sin(phi) dx
//     dL/dy_j = 2 P_j A_j sum G sin(phi) dy
//     dL/dz_j = (P_j A_j / z_j) sum G sin(phi) (dx^2 + dy^2)
// The direct method (FP32, here) produces per-strip partial sums
//     part_x[t][j] = (sum G cos phi, sum G sin phi dx, sum G sin phi dx^2)
//     part_y[t][j] = (-, sum G sin phi dy, sum G sin phi dy^2)
// and one reduction kernel adds the strips in a fixed order (deterministic)
// and applies the per-point factors: each thread owns one point and walks a
// 16-pixel-wide column strip of G top to bottom; the x angles of the strip
// stay in registers and the y angle follows the exact fixed-point form of the
// paper's Eq. 2 recurrence.  A quarter of the columns take sin and cos from
// FMA-pipe polynomials, the rest from the hardware sincos (two MUFU
// operations per point-pixel update).
//
// The separable methods run on the tensor cores (adj32.cu).
#include <math.h>

#include "api_internal.h"
#include "common.cuh"
#include "cos_poly.h"
#include "umma.cuh"

namespace cgh {

constexpr float PI_F = 3.14159265358979323846f;

// ------------------------------------------------------ direct adjoint
// Each thread owns one point and a BWD_STRIP-column strip; the arithmetic
// runs on column pairs in packed FP32x2.  NPOLY columns (pairs spread evenly
// over the strip) take sin and cos from FMA-pipe polynomials (u = |theta| - pi: cos theta = -C(u^2),
// sin theta = -sign(theta) u S(u^2); cos_poly.h), the others from the
// hardware sincos (two MUFU operations).  The offset dx = x - x_j is
// constant down a column, so the x sums of G sin(phi) dx and G sin(phi) dx^2
// are taken as dx and dx^2 times each column's sum of G sin(phi), formed once
// at the end: per update 5 FP32 operations and 2 MUFU on the hardware path
// (angle add, argument scale, and the cos, column and row sums), 17 on the
// polynomial path.  The polynomial columns accumulate negated sums, whose
// sign is restored at the end.
constexpr int BWD_STRIP = 16;    // pixels per column strip
// points per CTA: 256 with G staged through shared memory (each staged row
// serves more points), 128 reading G rows from global memory (measured on
// the direct adjoint at 1920x1080x4096, before the per-column sums: 3.34
// against 3.44 ms staged, 3.59 against 4.10 ms unstaged); points are padded
// to the larger
constexpr int BWD_THREADS_STAGED = 256;
constexpr int BWD_THREADS_GLOBAL = 128;
constexpr int BWD_PAD = 256;
constexpr int BWD_NP2 = BWD_STRIP / 2;
// G staged through shared memory (bwd_staged_walk): BWD_RB rows of the
// CTA's strip per stage, BWD_NST stages in flight
constexpr int BWD_RB = 32;
constexpr int BWD_NST = 4;

// One thread's sums over its strip: G cos(phi) of the hardware columns (+)
// and of the polynomial columns (negated), G sin(phi) per column pair (the
// polynomial pairs negated), and the y sums.
struct BwdAcc {
    float2 sC, nC;
    float2 S[BWD_NP2];
    float sY, sYY;
};

// The x angles of the thread's strip, and the start of its exact
// fixed-point y recurrence.
struct BwdPoint {
    float2 tx[BWD_NP2];
    uint64_t th, dth, d2;
    float xj, yj;
    bool valid;
};

// Polynomial column pairs, spread evenly among the hardware ones.
template <int NPOLY>
__device__ __forceinline__ constexpr bool bwd_poly_pair(int k) {
    return NPOLY > 0 && k % (BWD_STRIP / (NPOLY > 0 ? NPOLY : 1)) == 0 &&
           k / (BWD_STRIP / (NPOLY > 0 ? NPOLY : 1)) < NPOLY / 2;
}

__device__ __forceinline__ void bwd_point(const PointRec *__restrict__ rec,
                                          const float *__restrict__ points, int N,
                                          int j, int x0, BwdPoint &P, BwdAcc &acc) {
    P.valid = j < N;
    PointRec pr{};
    P.xj = 0.0f;
    P.yj = 0.0f;
    if (P.valid) {
        pr = rec[j];
        P.xj = points[2 * j];
        P.yj = points[2 * j + 1];
    }
#pragma unroll
    for (int k = 0; k < BWD_NP2; ++k)
        P.tx[k] = make_float2(
            (float)phase_hi(axis_phase(pr.c, pr.bx, pr.ax, x0 + 2 * k)) * RAD_PER_U32,
            (float)phase_hi(axis_phase(pr.c, pr.bx, pr.ax, x0 + 2 * k + 1)) * RAD_PER_U32);
    // y angle by the fixed-point recurrence: th(y+1) = th(y) + d(y),
    // d(y+1) = d(y) + 2c (exact modulo one turn)
    P.th = pr.ay;
    P.dth = pr.c - pr.by;
    P.d2 = 2 * pr.c;
    const float2 z2 = make_float2(0.0f, 0.0f);
    acc.sC = acc.nC = z2;
#pragma unroll
    for (int k = 0; k < BWD_NP2; ++k) acc.S[k] = z2;
    acc.sY = acc.sYY = 0.0f;
}

// One row y of the strip with G values g.
template <int NPOLY>
__device__ __forceinline__ void bwd_row(BwdPoint &P, int y, const float2 (&g)[BWD_NP2],
                                        BwdAcc &acc) {
    const float ty = (float)phase_hi(P.th) * RAD_PER_U32;
    P.th += P.dth;
    P.dth += P.d2;
    const float dy = (float)y - P.yj;
    const float2 ty2 = make_float2(ty, ty);
    const float2 z2 = make_float2(0.0f, 0.0f);
    float2 rs = z2, nrs = z2;
#pragma unroll
    for (int k = 0; k < BWD_NP2; ++k) {
        const float2 a = __fadd2_rn(P.tx[k], ty2);
        if (bwd_poly_pair<NPOLY>(k)) {
            const float2 u = make_float2(fabsf(a.x) - PI_F, fabsf(a.y) - PI_F);
            const float2 w = __fmul2_rn(u, u);
            float2 c = make_float2(COS5_C5, COS5_C5);
            c = __ffma2_rn(c, w, make_float2(COS5_C4, COS5_C4));
            c = __ffma2_rn(c, w, make_float2(COS5_C3, COS5_C3));
            c = __ffma2_rn(c, w, make_float2(COS5_C2, COS5_C2));
            c = __ffma2_rn(c, w, make_float2(COS5_C1, COS5_C1));
            c = __ffma2_rn(c, w, make_float2(COS5_C0, COS5_C0));  // -cos a
            float2 sn = make_float2(SIN5_C5, SIN5_C5);
            sn = __ffma2_rn(sn, w, make_float2(SIN5_C4, SIN5_C4));
            sn = __ffma2_rn(sn, w, make_float2(SIN5_C3, SIN5_C3));
            sn = __ffma2_rn(sn, w, make_float2(SIN5_C2, SIN5_C2));
            sn = __ffma2_rn(sn, w, make_float2(SIN5_C1, SIN5_C1));
            sn = __ffma2_rn(sn, w, make_float2(SIN5_C0, SIN5_C0));
            float2 v = __fmul2_rn(sn, u);  // sin u
            // -sin a = sign(a) sin u: flip the sign bit where a < 0
            v = make_float2(
                __int_as_float(__float_as_int(v.x) ^ (__float_as_int(a.x) & 0x80000000)),
                __int_as_float(__float_as_int(v.y) ^ (__float_as_int(a.y) & 0x80000000)));
            acc.nC = __ffma2_rn(g[k], c, acc.nC);
            acc.S[k] = __ffma2_rn(g[k], v, acc.S[k]);
            nrs = __ffma2_rn(g[k], v, nrs);
        } else {
            float2 sv, cv;
            __sincosf(a.x, &sv.x, &cv.x);
            __sincosf(a.y, &sv.y, &cv.y);
            acc.sC = __ffma2_rn(g[k], cv, acc.sC);
            acc.S[k] = __ffma2_rn(g[k], sv, acc.S[k]);
            rs = __ffma2_rn(g[k], sv, rs);
        }
    }
    const float r = (rs.x + rs.y) - (nrs.x + nrs.y);
    acc.sY = fmaf(r, dy, acc.sY);
    acc.sYY = fmaf(r * dy, dy, acc.sYY);
}

template <int NPOLY>
__device__ __forceinline__ void bwd_store(const BwdPoint &P, const BwdAcc &acc, int strip,
                                          int j, int Npad, float *__restrict__ part_x,
                                          float *__restrict__ part_y) {
    if (!P.valid) return;
    float *px = part_x + ((size_t)strip * Npad + j) * 3;
    float *py = part_y + ((size_t)strip * Npad + j) * 3;
    const int x0 = strip * BWD_STRIP;
    // the x sums: dx and dx^2 times each column's sum of G sin(phi)
    float sX = 0.0f, sXX = 0.0f;
#pragma unroll
    for (int k = 0; k < BWD_NP2; ++k) {
        const float sgn = bwd_poly_pair<NPOLY>(k) ? -1.0f : 1.0f;
        const float dx0 = (float)(x0 + 2 * k) - P.xj, dx1 = (float)(x0 + 2 * k + 1) - P.xj;
        const float t0 = sgn * acc.S[k].x * dx0, t1 = sgn * acc.S[k].y * dx1;
        sX += t0 + t1;
        sXX = fmaf(t0, dx0, fmaf(t1, dx1, sXX));
    }
    px[0] = (acc.sC.x + acc.sC.y) - (acc.nC.x + acc.nC.y);
    px[1] = sX;
    px[2] = sXX;
    py[0] = 0.0f;
    py[1] = acc.sY;
    py[2] = acc.sYY;
}

// ------------------------------------------------ walks down a strip
// G read from global memory row by row (any alignment, any Nx): calls
// row(y, g) for y = 0 .. Ny-1 with the strip's 16 values as 8 column pairs
// (zero beyond the frame).
template <class ROW>
__device__ __forceinline__ void bwd_global_walk(const float *__restrict__ G, int Nx,
                                                int Ny, int x0, ROW &&row) {
    const int ncols = Nx - x0 < BWD_STRIP ? Nx - x0 : BWD_STRIP;
    // whole 16-byte vectors: a full strip of a 16-byte aligned G whose rows
    // start 16-byte aligned (Nx a multiple of 4)
    const bool vec = (ncols == BWD_STRIP) && ((Nx & 3) == 0) && (((uintptr_t)G & 15) == 0);
#pragma unroll 1
    for (int y = 0; y < Ny; ++y) {
        const float *grow = G + (size_t)y * Nx + x0;
        float2 g[BWD_NP2];
        if (vec) {
#pragma unroll
            for (int k = 0; k < BWD_NP2; k += 2) {
                const float4 v = __ldg(reinterpret_cast<const float4 *>(grow + 2 * k));
                g[k] = make_float2(v.x, v.y);
                g[k + 1] = make_float2(v.z, v.w);
            }
        } else {
#pragma unroll
            for (int k = 0; k < BWD_NP2; ++k)
                g[k] = make_float2(2 * k < ncols ? __ldg(grow + 2 * k) : 0.0f,
                                   2 * k + 1 < ncols ? __ldg(grow + 2 * k + 1) : 0.0f);
        }
        row(y, g);
    }
}

// G staged through shared memory: the CTA's 16-column strip arrives BWD_RB
// rows at a time by 2-D TMA loads (zero fill beyond the frame), BWD_NST
// stages in flight, so the row loads do not wait on L2 in the loop.  The
// rows are read from shared memory by every thread at the same address
// (broadcast).  Calls row(y, g) for y = 0 .. Ny-1.  Waits are bounded; after
// a timeout (DEV_TIMEOUT recorded) the CTA's own copies are let land and the
// walk returns false.  Needs G 16-byte aligned and Nx a multiple of 4; every
// thread of the CTA must call it.
template <class ROW>
__device__ __forceinline__ bool bwd_staged_walk(const CUtensorMap &tG, int Ny, int x0,
                                                unsigned *status, ROW &&row) {
    constexpr uint32_t STAGE_BYTES = BWD_RB * BWD_STRIP * sizeof(float);
    __shared__ __align__(128) float sgrow[BWD_NST][BWD_RB][BWD_STRIP];
    __shared__ __align__(8) uint64_t full[BWD_NST];
    __shared__ volatile int abort_flag;
    const int nstage = (Ny + BWD_RB - 1) / BWD_RB;
    if (threadIdx.x == 0) {
        abort_flag = 0;
        for (int s = 0; s < BWD_NST; ++s) mbar_init(&full[s], 1);
        mbar_fence_init();
        umma::prefetch_tmap(&tG);
    }
    __syncthreads();
    int issued = 0;  // thread 0 only
    if (threadIdx.x == 0)
        for (int s = 0; s < BWD_NST && s < nstage; ++s) {
            mbar_arrive_expect_tx(&full[s], STAGE_BYTES);
            umma::tma_load_2d(&sgrow[s][0][0], &tG, x0, s * BWD_RB, &full[s]);
            ++issued;
        }
    int t = 0;
    for (; t < nstage; ++t) {
        const int s = t % BWD_NST;
        if (!mbar_wait_bounded(&full[s], (uint32_t)((t / BWD_NST) & 1))) {
            abort_flag = 1;
            set_status(status, DEV_TIMEOUT);
        } else {
            const int y0 = t * BWD_RB;
            const int rows = Ny - y0 < BWD_RB ? Ny - y0 : BWD_RB;
#pragma unroll 1
            for (int r = 0; r < rows; ++r) {
                const float4 *src = reinterpret_cast<const float4 *>(&sgrow[s][r][0]);
                float2 g[BWD_NP2];
#pragma unroll
                for (int k = 0; k < BWD_NP2; k += 2) {
                    const float4 v = src[k >> 1];
                    g[k] = make_float2(v.x, v.y);
                    g[k + 1] = make_float2(v.z, v.w);
                }
                row(y0 + r, g);
            }
        }
        __syncthreads();  // every thread is done with slot s
        if (abort_flag) break;
        if (threadIdx.x == 0 && t + BWD_NST < nstage) {
            fence_proxy_async_smem();
            mbar_arrive_expect_tx(&full[s], STAGE_BYTES);
            umma::tma_load_2d(&sgrow[s][0][0], &tG, x0, (t + BWD_NST) * BWD_RB, &full[s]);
            ++issued;
        }
    }
    if (abort_flag) {
        if (threadIdx.x == 0)
            for (int u = t; u < issued; ++u)
                mbar_wait_bounded(&full[u % BWD_NST], (uint32_t)((u / BWD_NST) & 1));
        return false;
    }
    return true;
}

// --------------------------------------------------- direct adjoint
template <int NPOLY>
__global__ void __launch_bounds__(BWD_THREADS_GLOBAL)
direct_bwd_kernel(const PointRec *__restrict__ rec, const float *__restrict__ points,
                  int N, int Npad, int Nx, int Ny, const float *__restrict__ G,
                  float *__restrict__ part_x, float *__restrict__ part_y) {
    static_assert(NPOLY % 2 == 0 && NPOLY <= BWD_STRIP, "polynomial column pairs");
    const int strip = blockIdx.x;
    const int j = blockIdx.y * BWD_THREADS_GLOBAL + threadIdx.x;
    const int x0 = strip * BWD_STRIP;
    BwdPoint P;
    BwdAcc acc;
    bwd_point(rec, points, N, j, x0, P, acc);
    bwd_global_walk(G, Nx, Ny, x0, [&](int y, const float2 (&g)[BWD_NP2]) {
        bwd_row<NPOLY>(P, y, g, acc);
    });
    bwd_store<NPOLY>(P, acc, strip, j, Npad, part_x, part_y);
}

template <int NPOLY>
__global__ void __launch_bounds__(BWD_THREADS_STAGED)
direct_bwd_staged_kernel(const __grid_constant__ CUtensorMap tG,
                         const PointRec *__restrict__ rec,
                         const float *__restrict__ points, int N, int Npad, int Ny,
                         float *__restrict__ part_x, float *__restrict__ part_y,
                         unsigned *status) {
    static_assert(NPOLY % 2 == 0 && NPOLY <= BWD_STRIP, "polynomial column pairs");
    const int strip = blockIdx.x;
    const int j = blockIdx.y * BWD_THREADS_STAGED + threadIdx.x;
    const int x0 = strip * BWD_STRIP;
    BwdPoint P;
    BwdAcc acc;
    bwd_point(rec, points, N, j, x0, P, acc);
    if (bwd_staged_walk(tG, Ny, x0, status, [&](int y, const float2 (&g)[BWD_NP2]) {
            bwd_row<NPOLY>(P, y, g, acc);
        }))
        bwd_store<NPOLY>(P, acc, strip, j, Npad, part_x, part_y);
}

// ------------------------------------------------------------ reduce
// One block per RD_PTS points; its RD_SL slices of threads take every
// RD_SL-th partial-sum tile of their point (FP64), then slice 0 adds the
// slices' sums in slice order: deterministic, and enough threads in flight
// to cover the loads' latency (one thread per point walking ~100 tiles
// left the SMs nearly empty).
constexpr int RD_PTS = 32, RD_SL = 8;

__global__ void __launch_bounds__(RD_PTS * RD_SL)
adjoint_reduce_kernel(const PointRec *__restrict__ rec, const float *__restrict__ z,
                      int N, int Npad, const float *__restrict__ part_x, int Tx,
                      const float *__restrict__ part_y, int Ty, float *gpts, float *gA, float *gz) {
    __shared__ double part[RD_SL][5][RD_PTS];
    const int lj = threadIdx.x % RD_PTS, sl = threadIdx.x / RD_PTS;
    const int j = blockIdx.x * RD_PTS + lj;
    double sC = 0, sX = 0, sXX = 0, sY = 0, sYY = 0;
    if (j < N) {
        for (int t = sl; t < Tx; t += RD_SL) {
            const float *p = part_x + ((size_t)t * Npad + j) * 3;
            sC += p[0];
            sX += p[1];
            sXX += p[2];
        }
        for (int t = sl; t < Ty; t += RD_SL) {
            const float *p = part_y + ((size_t)t * Npad + j) * 3;
            sY += p[1];
            sYY += p[2];
        }
    }
    part[sl][0][lj] = sC;
    part[sl][1][lj] = sX;
    part[sl][2][lj] = sXX;
    part[sl][3][lj] = sY;
    part[sl][4][lj] = sYY;
    __syncthreads();
    if (sl != 0 || j >= N) return;
    sC = sX = sXX = sY = sYY = 0;
#pragma unroll
    for (int q = 0; q < RD_SL; ++q) {
        sC += part[q][0][lj];
        sX += part[q][1][lj];
        sXX += part[q][2][lj];
        sY += part[q][3][lj];
        sYY += part[q][4][lj];
    }
    const PointRec r = rec[j];
    const bool ok = r.Q32 > 0.0f;
    const double P = 6.283185307179586 * (double)r.Q32;
    const double a = (double)r.A;
    if (gA) gA[j] = ok ? (float)(sC) : 0.0f;
    if (gpts) {
        gpts[2 * j] = ok ? (float)(2.0 * P * a * sX) : 0.0f;
        gpts[2 * j + 1] = ok ? (float)(2.0 * P * a * sY) : 0.0f;
    }
    if (gz) gz[j] = ok ? (float)(P * a / (double)z[j] * (sXX + sYY)) : 0.0f;
}

}  // namespace cgh

using namespace cgh;

static cgh_status run_direct_backward(cgh_ctx *h, const float *points, const float *A,
                                      const float *z, int N, double lambda, double p, int Nx,
                                      int Ny, const float *G, float *gpts, float *gA, float *gz,
                                      cudaStream_t s) {
    const int Npad = pad_to(N, BWD_PAD);
    const int Tx = (Nx + BWD_STRIP - 1) / BWD_STRIP;  // partial-sum tiles: one per strip
    const size_t rec_b = align256((size_t)Npad * sizeof(PointRec));
    const size_t part_b = align256((size_t)Tx * Npad * 3 * sizeof(float));
    cgh_status st = h->ensure(h->ws2, rec_b + 2 * part_b, s, "adjoint workspace");
    if (st) return st;
    char *b = (char *)h->ws2.ptr;
    PointRec *rec = (PointRec *)b;
    float *part_x = (float *)(b + rec_b);
    float *part_y = (float *)(b + rec_b + part_b);
    {
        TimedLaunch tl(h, CGH_K_PROLOGUE, s);
        cudaError_t e = launch_prologue(points, A, z, N, Npad, lambda, p, rec,
                                        h->d_status, s);
        if (e != cudaSuccess) return h->cuda_fail(e, "prologue launch");
        tl.done();
    }
    {
        TimedLaunch tl(h, CGH_K_BWD_DIRECT, s);
        const dim3 grid_st(Tx, Npad / BWD_THREADS_STAGED);
        const dim3 grid_gl(Tx, Npad / BWD_THREADS_GLOBAL);
        // G through shared memory by TMA when its layout allows (16-byte
        // aligned rows), else row loads from global memory
        CUtensorMap tG;
        const bool staged = h->bwd_staged && (((uintptr_t)G & 15) == 0) && (Nx % 4 == 0) &&
                            make_f32_map(&tG, G, Nx, Ny, Nx, BWD_STRIP, BWD_RB);
        if (staged) {
            if (h->bwd_poly == 0)
                direct_bwd_staged_kernel<0><<<grid_st, BWD_THREADS_STAGED, 0, s>>>(
                    tG, rec, points, N, Npad, Ny, part_x, part_y, h->d_status);
            else if (h->bwd_poly == 6)
                direct_bwd_staged_kernel<6><<<grid_st, BWD_THREADS_STAGED, 0, s>>>(
                    tG, rec, points, N, Npad, Ny, part_x, part_y, h->d_status);
            else
                direct_bwd_staged_kernel<4><<<grid_st, BWD_THREADS_STAGED, 0, s>>>(
                    tG, rec, points, N, Npad, Ny, part_x, part_y, h->d_status);
        } else if (h->bwd_poly == 0) {
            direct_bwd_kernel<0><<<grid_gl, BWD_THREADS_GLOBAL, 0, s>>>(rec, points, N, Npad, Nx,
                                                               Ny, G, part_x, part_y);
        } else if (h->bwd_poly == 6) {
            direct_bwd_kernel<6><<<grid_gl, BWD_THREADS_GLOBAL, 0, s>>>(rec, points, N, Npad, Nx,
                                                               Ny, G, part_x, part_y);
        } else {
            direct_bwd_kernel<4><<<grid_gl, BWD_THREADS_GLOBAL, 0, s>>>(rec, points, N, Npad, Nx,
                                                               Ny, G, part_x, part_y);
        }
        cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return h->cuda_fail(e, "direct adjoint launch");
        tl.done();
    }
    {
        TimedLaunch tl(h, CGH_K_BWD_REDUCE, s);
        adjoint_reduce_kernel<<<(N + RD_PTS - 1) / RD_PTS, RD_PTS * RD_SL, 0, s>>>(
            rec, z, N, Npad, part_x, Tx, part_y, Tx, gpts, gA, gz);
        cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return h->cuda_fail(e, "adjoint reduce launch");
        tl.done();
    }
    return CGH_OK;
}

extern "C" cgh_status cgh_backward(cgh_handle h, const float *points,
                                   const float *A, const float *z, int N,
                                   double lambda, double p, int Nx, int Ny,
                                   const float *grad_out, float *grad_points,
                                   float *grad_A, float *grad_z, int method,
                                   void *stream) {
    NvtxRange range("cgh_backward");
    if (!h) return CGH_ERR_INVALID_ARG;
    int prev = 0;
    cudaGetDevice(&prev);
    if (prev != h->device) cudaSetDevice(h->device);
    h->err[0] = 0;
    cgh_status st = h->check_problem(points, A, z, N, lambda, p, Nx, Ny, grad_out);
    if (st == CGH_OK && method != CGH_DIRECT_FP32 && method != CGH_SEP_FP16X3 &&
        method != CGH_SEP_FP32)
        st = h->fail(CGH_ERR_INVALID_ARG,
                     "adjoint method must be CGH_DIRECT_FP32, CGH_SEP_FP32 or CGH_SEP_FP16X3");
    if (st == CGH_OK &&
        ((((uintptr_t)grad_points) | ((uintptr_t)grad_A) | ((uintptr_t)grad_z)) & 3))
        st = h->fail(CGH_ERR_INVALID_ARG, "gradient arrays must be 4-byte aligned");
    if (st == CGH_OK && N > 0 && (grad_points || grad_A || grad_z)) {
        if (method == CGH_DIRECT_FP32)
            st = run_direct_backward(h, points, A, z, N, lambda, p, Nx, Ny, grad_out,
                                     grad_points, grad_A, grad_z, (cudaStream_t)stream);
        else
            st = h->backward_sep32(points, A, z, N, lambda, p, Nx, Ny, grad_out, grad_points,
                                   grad_A, grad_z,
                                   method == CGH_SEP_FP32 ? CGH_K_BWD_SIMT : CGH_K_BWD_GEMM,
                                   (cudaStream_t)stream);
    }
    if (prev != h->device) cudaSetDevice(prev);
    return st;
}
