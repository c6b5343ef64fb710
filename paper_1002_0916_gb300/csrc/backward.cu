// backward.cu -- the hand-written adjoint of Eq. 1 (step A8).
//
// For a loss L with G = dL/dI (Ny x Nx) and phi = P_j r^2 (Section 1,
// Eq. 1; P_j = 2 pi Q_j, dx = x - x_j, dy = y - y_j, dP_j/dz_j = -P_j/z_j):
//     dL/dA_j = sum G cos(phi)
//     dL/dx_j = 2 P_j A_j sum G sin(phi) dx
//     dL/dy_j = 2 P_j A_j sum G sin(phi) dy
//     dL/dz_j = (P_j A_j / z_j) sum G sin(phi) (dx^2 + dy^2)
// The direct method is here: FP32 point-owned sums.  Each thread owns one
// point and walks a 16- or 32-pixel-wide column strip of G over a run of rows; the
// cosines and sines of the strip's columns stay in registers, the row angle
// follows the exact fixed-point form of the paper's Eq. 2 recurrence, and the
// cosine and sine of each summed phase are expanded by angle addition.  One
// reduction kernel adds the strips' and runs' partial sums in a fixed order
// (deterministic) and applies the per-point factors.
//
// The separable methods run on the tensor cores (adj32.cu), small and low
// frames (sep_by_strips) on the same sums.
#include <math.h>

#include "api_internal.h"
#include "common.cuh"
#include "point_rec.cuh"
#include "sep32.cuh"

namespace cgh {

// ------------------------------------------------------ direct adjoint
// With (cx, sx) of each column's angle and (cy, sy) of each row's,
//     sum_y G cos(phi) = cx U - sx V,   sum_y G sin(phi) = sx U + cx V,
//     U = sum_y G cy,   V = sum_y G sy           (per column, down the strip)
//     sum_x G sin(phi) = cy P + sy Q,
//     P = sum_x G sx,   Q = sum_x G cx           (per row, across the strip)
// Per update: 4 FP32 multiply-adds (U, V, P, Q), packed in column pairs; the
// row's hardware sincos is shared by the strip's updates, the columns' (to FP32
// rounding) by a whole run of rows.  The offset dx is constant down a column,
// so the x sums are taken from the columns' sums once at the end.
//
// Bound: the FMA pipe, 128 / 4 = 32 updates per clock and SM.  A sincos per
// update, a quarter of them as polynomials, was bound by the MUFU instead:
// 2954 us at 1920x1080x4096 against 1273 here (0.66 of the bound; a packed
// multiply-add holds the pipe two cycles, and a row costs 28 instructions
// beside its 64).  24 columns with 96 threads: 1775; two rows unrolled at 32
// columns: 1310; stages of 8, 12, 24 or 32 rows there: 1290 to 1330; split P
// and Q chains or the columns' phases stepped instead of evaluated: 1330.
// 16 columns, four CTAs per SM and two rows unrolled: 1446 us there, but less
// set-up per CTA: 8.2 us against 9.8 at 256x256x64, 29 both at 1023x767x100.
template <int STRIP>
struct BwdShape {
    static constexpr int NP2 = STRIP / 2;
    static constexpr int CTAS = STRIP == 32 ? 3 : 4;  // per SM (168 or 128 registers)
    // rows of the strip per shared-memory stage (two stages): the CTA's
    // threads load the next stage into registers, any alignment and width,
    // before they compute on this one
    static constexpr int RB = STRIP == 32 ? 16 : 32;
    static constexpr int UNROLL = STRIP == 32 ? 1 : 2;  // rows
};
constexpr int BWD_THREADS = 128;  // points per CTA
// Strips of 32 columns from 2^25 updates on.
static int bwd_strip(int Nx, int Ny, int N) {
    return (double)Nx * Ny * N < (double)(1 << 25) ? 16 : 32;
}

// Grid: x = column strips, y = groups of BWD_THREADS points, z = runs of
// `rows` rows.  part: [strip * runs + run][5][Npad], the sums of G cos, G sin
// dx, G sin dx^2, G sin dy, G sin dy^2.
// ROW32: the rows' sines and cosines to FP32 rounding too (sep_by_strips).
template <int STRIP, bool ROW32>
__global__ void __launch_bounds__(BWD_THREADS, BwdShape<STRIP>::CTAS)
direct_bwd_kernel(PointSource src, int Npad, int Nx, int Ny, int rows,
                  const float *__restrict__ G, float *__restrict__ part) {
    constexpr int NP2 = BwdShape<STRIP>::NP2, RB = BwdShape<STRIP>::RB;
    constexpr int LOADS = RB * STRIP / BWD_THREADS, UNROLL = BwdShape<STRIP>::UNROLL;
    __shared__ __align__(16) float sg[2][RB][STRIP];
    const int strip = blockIdx.x, x0 = strip * STRIP;
    const int j = blockIdx.y * BWD_THREADS + threadIdx.x;
    const int ya = blockIdx.z * rows, yb = ya + rows < Ny ? ya + rows : Ny;
    const int lc = threadIdx.x % STRIP, lr = threadIdx.x / STRIP;
    const float *gcol = G + x0 + lc;
    const bool in_x = x0 + lc < Nx;
    float next[LOADS];
    auto load = [&](int y0) {
#pragma unroll
        for (int k = 0; k < LOADS; ++k) {
            const int y = y0 + lr + k * (BWD_THREADS / STRIP);
            next[k] = in_x && y < yb ? __ldg(gcol + (size_t)y * Nx) : 0.0f;
        }
    };
    auto store = [&](int b) {
#pragma unroll
        for (int k = 0; k < LOADS; ++k)
            sg[b][lr + k * (BWD_THREADS / STRIP)][lc] = next[k];
    };
    load(ya);

    // the point's record (a rejected point reports once per CTA column)
    const PointRec pr = make_point_rec(src.points, src.A, src.z, src.N, j, src.K, src.status);
    const float2 z2 = make_float2(0.0f, 0.0f);
    float2 cx[NP2], sx[NP2], U[NP2], V[NP2];
#pragma unroll
    for (int k = 0; k < NP2; ++k) {
        sincos_fixed(axis_phase(pr.c, pr.bx, pr.ax, x0 + 2 * k), sx[k].x, cx[k].x);
        sincos_fixed(axis_phase(pr.c, pr.bx, pr.ax, x0 + 2 * k + 1), sx[k].y, cx[k].y);
        U[k] = V[k] = z2;
    }
    const float yj = j < src.N ? src.points[2 * j + 1] : 0.0f;
    uint64_t th = axis_phase(pr.c, pr.by, pr.ay, ya);
    uint64_t dth = pr.c * (uint64_t)(2 * (int64_t)ya + 1) - pr.by;
    const uint64_t d2 = 2 * pr.c;
    float dy = (float)ya - yj;
    float sY = 0.0f, sYY = 0.0f;

    store(0);
    __syncthreads();
    int b = 0;
    for (int y0 = ya; y0 < yb; y0 += RB, b ^= 1) {
        const bool more = y0 + RB < yb;
        if (more) load(y0 + RB);
        const int n = yb - y0 < RB ? yb - y0 : RB;
#pragma unroll UNROLL
        for (int r = 0; r < n; ++r) {
            float sy, cy;
            if constexpr (ROW32) sincos_fixed(th, sy, cy);
            else __sincosf((float)phase_hi(th) * RAD_PER_U32, &sy, &cy);
            th += dth;
            dth += d2;
            const float2 cy2 = make_float2(cy, cy), sy2 = make_float2(sy, sy);
            const float4 *row = reinterpret_cast<const float4 *>(&sg[b][r][0]);
            float2 p = z2, q = z2;
#pragma unroll
            for (int k = 0; k < NP2; k += 2) {
                const float4 v = row[k >> 1];
                const float2 g[2] = {make_float2(v.x, v.y), make_float2(v.z, v.w)};
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    U[k + e] = __ffma2_rn(g[e], cy2, U[k + e]);
                    V[k + e] = __ffma2_rn(g[e], sy2, V[k + e]);
                    p = __ffma2_rn(g[e], sx[k + e], p);
                    q = __ffma2_rn(g[e], cx[k + e], q);
                }
            }
            const float t = fmaf(cy, p.x + p.y, sy * (q.x + q.y)) * dy;
            sY += t;
            sYY = fmaf(t, dy, sYY);
            dy += 1.0f;
        }
        if (more) store(b ^ 1);
        __syncthreads();
    }
    if (j >= src.N) return;
    const float xj = src.points[2 * j];
    float C = 0.0f, sX = 0.0f, sXX = 0.0f;
#pragma unroll
    for (int k = 0; k < NP2; ++k) {
        C += fmaf(cx[k].x, U[k].x, -sx[k].x * V[k].x) + fmaf(cx[k].y, U[k].y, -sx[k].y * V[k].y);
        const float dx0 = (float)(x0 + 2 * k) - xj, dx1 = (float)(x0 + 2 * k + 1) - xj;
        const float t0 = fmaf(sx[k].x, U[k].x, cx[k].x * V[k].x) * dx0;
        const float t1 = fmaf(sx[k].y, U[k].y, cx[k].y * V[k].y) * dx1;
        sX += t0 + t1;
        sXX = fmaf(t0, dx0, fmaf(t1, dx1, sXX));
    }
    float *dst = part + ((size_t)(strip * gridDim.z + blockIdx.z) * 5) * Npad + j;
    dst[0] = C;
    dst[(size_t)Npad] = sX;
    dst[(size_t)2 * Npad] = sXX;
    dst[(size_t)3 * Npad] = sY;
    dst[(size_t)4 * Npad] = sYY;
}

// --------------------------------------------------------------- sums
// The partial sums of the points, both methods: one block per RD_PTS points,
// up to RD_SL slices of threads; a slice takes every so-many-th tile of its
// point and adds its fields as FP32 pairs (two-sum: value and accumulated
// rounding error, about 48 bits), then one warp per field adds the slices'
// pairs in slice order: deterministic.  Adding everything in FP64 was bound by
// this GPU's FP64 rate, 2 per clock and SM (35 us at 1920x1080x4096 with 360
// tiles; 15 here).
// Few tiles take 8 slices: with 32 the slices' own sums dominate (1920x1080x
// 16384, 28 tiles: 39 us against 13).
constexpr int RD_PTS = 32, RD_SL = 32;

__device__ __forceinline__ void two_sum(float &s, float &e, float v) {
    const float t = __fadd_rn(s, v), b = __fsub_rn(t, s);
    e = __fadd_rn(e, __fadd_rn(__fsub_rn(s, __fsub_rn(t, b)), __fsub_rn(v, b)));
    s = t;
}

__global__ void __launch_bounds__(RD_PTS * RD_SL)
adjoint_sum_kernel(PointSource src, AdjointParts pp, const float *__restrict__ unit, float *gpts,
                   float *gA, float *gz) {
    __shared__ float2 part[RD_SL][5][RD_PTS];
    __shared__ double sums[5][RD_PTS];
    const int lj = threadIdx.x % RD_PTS, sl = threadIdx.x / RD_PTS;
    const int nsl = blockDim.x / RD_PTS;  // slices
    const int j = blockIdx.x * RD_PTS + lj;
    pdl_wait();  // the partial sums come from the kernel before
    float s[5] = {0, 0, 0, 0, 0}, e[5] = {0, 0, 0, 0, 0};
    if (j < src.N) {
        const float *x = pp.x + j, *y = pp.y + j;
#pragma unroll 4
        for (int t = sl; t < pp.Tx; t += nsl)
#pragma unroll
            for (int k = 0; k < 3; ++k)
                two_sum(s[k], e[k], __ldcg(x + t * pp.stride + k * pp.npad));
#pragma unroll 4
        for (int t = sl; t < pp.Ty; t += nsl)
#pragma unroll
            for (int k = 0; k < 2; ++k)
                two_sum(s[3 + k], e[3 + k], __ldcg(y + t * pp.stride + k * pp.npad));
    }
#pragma unroll
    for (int k = 0; k < 5; ++k) part[sl][k][lj] = make_float2(s[k], e[k]);
    __syncthreads();
    for (int k = sl; k < 5; k += nsl) {
        float v = 0.0f, w = 0.0f;
        for (int q = 0; q < nsl; ++q) {
            two_sum(v, w, part[q][k][lj].x);
            w += part[q][k][lj].y;
        }
        double sum = (double)v + (double)w;
        if (!isfinite(sum) && j < src.N) {
            // an infinite partial sum, whose rounding error is NaN, or a
            // total past FP32's range: once more in FP64
            const bool is_x = k < 3;
            const float *p = (is_x ? pp.x + k * pp.npad : pp.y + (k - 3) * pp.npad) + j;
            const int T = is_x ? pp.Tx : pp.Ty;
            sum = 0.0;
            for (int t = 0; t < T; ++t) sum += (double)__ldcg(p + t * pp.stride);
        }
        sums[k][lj] = sum;
    }
    __syncthreads();
    if (sl != 0 || j >= src.N) return;
    const PointRec r =
        make_point_rec(src.points, src.A, src.z, src.N, j, src.K, (unsigned *)nullptr);
    const bool ok = r.Q32 > 0.0f;
    const double g = unit ? (double)*unit : 1.0;  // the unit of the sums
    const double P = 6.283185307179586 * (double)r.Q32;
    const double a = (double)r.A;
    if (gA) gA[j] = ok ? (float)(sums[0][lj] * g) : 0.0f;
    if (gpts) {
        gpts[2 * j] = ok ? (float)(2.0 * P * a * sums[1][lj] * g) : 0.0f;
        gpts[2 * j + 1] = ok ? (float)(2.0 * P * a * sums[3][lj] * g) : 0.0f;
    }
    if (gz)
        gz[j] = ok ? (float)(P * a / (double)src.z[j] * (sums[2][lj] + sums[4][lj]) * g) : 0.0f;
}

cudaError_t launch_adjoint_sum(const PointSource &src, const AdjointParts &pp, const float *unit,
                               float *gpts, float *gA, float *gz, cudaStream_t s) {
    const int tiles = pp.Tx > pp.Ty ? pp.Tx : pp.Ty;
    const int slices = tiles > 64 ? RD_SL : 8;  // (few tiles: the slices' own sum dominates)
    return launch_dependent(adjoint_sum_kernel, dim3((src.N + RD_PTS - 1) / RD_PTS),
                            dim3(RD_PTS * slices), 0, s, src, pp, unit, gpts, gA, gz);
}

// Frames whose adjoint the separable methods take by the strips: the products
// of adj32.cu (four launches; K in 64s, columns in 192s at least) are mostly
// padding on small and on low frames.  Strips against products, us: 16x16x16384
// 8.5 and 39, 64x64x4000 11.8 and 20, 512x32x1000 14.7 and 19, 181x181x300 13.7
// and 19, 2048x16x4000 50 and 61, 32768x3x500 76 and 375; on the other side of
// the lines 91x91x100000 184 and 180, 256x128x760 20 and 18.5, 48x200x16384 54
// and 44, 2048x24x1000 27 and 26, 32768x16x16 69 and 53.  With the rows' sines to
// FP32 rounding (3% of the time) the strips are no less accurate: 64x64x4000 x
// 1.4e-7, A 1.6e-7, z 1.3e-7 from FP64, the products 2.3e-7, 1.9e-7, 2.5e-7.
// Their partial sums, 20 bytes per point and 32 columns, take 1 GiB at most, like
// the products' tables.
static bool sep_by_strips(int N, int Nx, int Ny) {
    const long long pixels = (long long)Nx * Ny;
    const bool small = Nx <= 8192 && Ny <= 1024 &&
                       (pixels <= 8192 ||
                        (pixels <= 32768 && pixels * N <= (Ny <= 64 ? 25000000 : 12000000)));
    return (small || (Ny <= 20 && N >= 256)) && (long long)Nx * N <= 1700000000;
}

// Rows per run: the fewest runs (each repeats the columns' sincos, worth
// about 16 rows) whose CTAs fill the SMs' slots in nearly whole waves.
static int bwd_rows(int strip, int Nx, int Ny, int N, int sms) {
    const int rb = strip == 32 ? BwdShape<32>::RB : BwdShape<16>::RB;
    const int per_sm = strip == 32 ? BwdShape<32>::CTAS : BwdShape<16>::CTAS;
    const long long ctas = (long long)((Nx + strip - 1) / strip) *
                           ((N + BWD_THREADS - 1) / BWD_THREADS);
    const long long slots = (long long)per_sm * (sms > 0 ? sms : 1);
    int best = Ny;
    double best_cost = 1e300;
    for (int runs = 1; runs <= 16; ++runs) {
        const int rows = pad_to((Ny + runs - 1) / runs, rb);
        const long long n = (Ny + rows - 1) / rows;
        const double cost = (double)((ctas * n + slots - 1) / slots) * (rows + 16);
        if (cost < best_cost * 0.99) {
            best_cost = cost;
            best = rows;
        }
    }
    return best;
}

}  // namespace cgh

using namespace cgh;

// timer: the cgh_kernel_id of the strips' launch
static cgh_status run_direct_backward(cgh_ctx *h, const float *points, const float *A,
                                      const float *z, int N, double lambda, double p, int Nx,
                                      int Ny, const float *G, float *gpts, float *gA, float *gz,
                                      bool row32, int timer, cudaStream_t s) {
    const int Npad = pad_to(N, 32);
    const int strip = bwd_strip(Nx, Ny, N), strips = (Nx + strip - 1) / strip;
    const int rows = bwd_rows(strip, Nx, Ny, N, h->sm_count), runs = (Ny + rows - 1) / rows;
    const size_t part_b = (size_t)strips * runs * 5 * Npad * sizeof(float);
    cgh_status st = h->ensure(h->ws2, part_b, s, "adjoint workspace");
    if (st) return st;
    float *part = (float *)h->ws2.ptr;
    const PointSource src{points, A, z, N, fresnel_scale(lambda, p), h->d_status};
    {
        auto kern = strip == 32 ? (row32 ? direct_bwd_kernel<32, true> : direct_bwd_kernel<32, false>)
                                : (row32 ? direct_bwd_kernel<16, true> : direct_bwd_kernel<16, false>);
        // as many groups of points as grid y takes (one grid dimension for
        // strips and groups together made the kernel 4% slower)
        const int most = 65535 * BWD_THREADS;
        for (int j0 = 0; j0 < N; j0 += most) {
            TimedLaunch tl(h, timer, s);
            const int n = N - j0 < most ? N - j0 : most;
            const PointSource some{points + 2 * (size_t)j0, A + j0, z + j0, n, src.K, src.status};
            const dim3 grid(strips, (n + BWD_THREADS - 1) / BWD_THREADS, runs);
            cudaError_t e = launch_kernel(false, kern, grid, dim3(BWD_THREADS), 0, s, some, Npad,
                                          Nx, Ny, rows, G, part + j0);
            if (e != cudaSuccess) return h->cuda_fail(e, "direct adjoint launch");
            tl.done();
        }
    }
    {
        TimedLaunch tl(h, CGH_K_BWD_REDUCE, s);
        const AdjointParts pp{part, part + 3 * (size_t)Npad, strips * runs, strips * runs,
                              5 * (size_t)Npad, (size_t)Npad};
        cudaError_t e = launch_adjoint_sum(src, pp, nullptr, gpts, gA, gz, s);
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
            st = run_direct_backward(h, points, A, z, N, lambda, p, Nx, Ny, grad_out, grad_points,
                                     grad_A, grad_z, false, CGH_K_BWD_DIRECT,
                                     (cudaStream_t)stream);
        else {
            const int timer = method == CGH_SEP_FP32 ? CGH_K_BWD_SIMT : CGH_K_BWD_GEMM;
            if (sep_by_strips(N, Nx, Ny))
                st = run_direct_backward(h, points, A, z, N, lambda, p, Nx, Ny, grad_out,
                                         grad_points, grad_A, grad_z, true, timer,
                                         (cudaStream_t)stream);
            else
                st = h->backward_sep32(points, A, z, N, lambda, p, Nx, Ny, grad_out, grad_points,
                                       grad_A, grad_z, timer, (cudaStream_t)stream);
        }
    }
    if (prev != h->device) cudaSetDevice(prev);
    return st;
}
