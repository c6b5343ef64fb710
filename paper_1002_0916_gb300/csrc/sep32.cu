// sep32.cu -- the separable form of Eq. 1 at FP32 accuracy on the tensor
// cores.
//
// The phase of Eq. 1 is a sum of an x part and a y part, so with
//     L[x][2j] = A_j cos theta_x,  L[x][2j+1] = -A_j sin theta_x,
//     R[y][2j] =     cos theta_y,  R[y][2j+1] =      sin theta_y,
// I[y][x] = sum_k R[y][k] L[x][k], a matrix product of depth K = 2N.
//
// Precision.  Each FP32 table entry v is held as two FP16 numbers, hi =
// fp16(v) and lo = fp16(v - hi): 22 significant bits and a sign, an error of
// at most 2^-23 |v|.  The product is hi*hi + hi*lo + lo*hi (lo*lo, 2^-24 of
// a term, is dropped).  Two things keep this at FP32 accuracy:
//   * Range.  R is scaled by 2^14 and the L entries of every 32 points (one
//     K block of 64 values) by the power of two that brings their largest
//     |A_j| into [2^13, 2^14), so that hi and lo are normal FP16 numbers
//     for amplitudes of any size.  Powers of two change no bits; the block's
//     factor is taken out again in FP32.
//   * Accumulation.  The tensor cores add into FP32 but drop the low bits of
//     every sum, a bias toward zero that grows with the number of adds.  Here
//     tensor memory accumulates one K block at a time -- the cross products
//     first, while the sum is small, then four hi*hi steps -- and the
//     epilogue warps add each block's partial product, times its factor, to
//     FP32 registers with round to nearest while the next block runs.
//
// Kernel: CTA pairs (tcgen05 cta_group::2, 256 x BNP tiles), the loads and
// synchronisation of umma2.cu; two tensor-memory buffers of 256 columns
// alternate between the MMAs and the epilogue.  Eight epilogue warps hold
// the CTA's 128 x BNP sums, each thread one row and half of the columns (at
// most 128 registers).  What bounds it is the MMA rate (12 steps per K
// block): at 256 columns a K block takes 0.81 us, the same with the promotion
// as without it; at 112 to 160 columns it takes 0.64 to 0.69 us against 0.60,
// or 0.52 with no loads.  The epilogue's barrier waits are at CTA scope and
// its arrivals relaxed (tensor memory is ordered by the tcgen05 fences, and no
// generic memory is handed over): with cluster-scope acquire and release a
// block took 1.1 to 1.4 us.
// Measured, whole call, against an FP32 product on the FMA pipe (0.70 of its
// bound): 1920x1024x3584 543 -> 84 us, 3840x2160x16384 9.85 -> 1.12 ms;
// relative RMS error against FP64 6.8e-7 -> 1.9e-7 and 1.6e-6 -> 2.3e-7.
//
// Long products on few tiles are cut along K into S slices: each slice's
// CTA writes its partial tile, and the last slice of a tile to finish adds
// the S partials in slice order (deterministic).
#include <cudaTypedefs.h>
#include <math.h>

#include "api_internal.h"
#include "common.cuh"
#include "cos_poly.h"
#include "point_rec.cuh"
#include "sep_table.cuh"
#include "umma.cuh"
#include "umma_pair.cuh"

namespace cgh {

bool make_gemm_map(CUtensorMap *m, const void *base, long long inner, long long rows,
                   long long ld, int box_rows, bool bf16);

// ---------------------------------------------------------------- tables
// R entries are scaled by 2^S32_EXP, a block's L entries to below it.
constexpr int S32_EXP = 14;
constexpr float S32_R_SCALE = 16384.0f;

// sin and cos of a 0.64 fixed-point phase: the nearest quarter turn is taken
// off in fixed point, so that the remainder x (quarter turns, |x| <= 1/2)
// rounds to FP32 with a relative error (2^-25) however large the phase, then
// polynomials (cos_poly.h), a swap and two sign bits.  The hardware sincos of
// the rounded angle would be cheaper but has an absolute error of 2^-21, more
// than the rest of this path together; sincospif of the rounded turn took 9.1
// us against 7.6 (tables at 1023x767x1999) and left more error in the hologram
// (1.76e-7 against 1.62e-7 at 1920x1024x1024).
__device__ __forceinline__ void sincos_fixed(uint64_t ph, float &s, float &c) {
    const float x = (float)(int)(uint32_t)(ph >> 30) * TURN_PER_U32;
    const uint32_t t = (uint32_t)(ph >> 32) + 0x20000000u;  // top 2 bits: the quadrant
    const float z = x * x;
    float ps = fmaf(QSIN_C3, z, QSIN_C2), pc = fmaf(QCOS_C4, z, QCOS_C3);
    ps = fmaf(ps, z, QSIN_C1);
    pc = fmaf(pc, z, QCOS_C2);
    ps = fmaf(ps, z, QSIN_C0);
    pc = fmaf(pc, z, QCOS_C1);
    ps *= x;
    pc = fmaf(pc, z, QCOS_C0);
    const bool odd = (t & 0x40000000u) != 0;
    const float a = odd ? ps : pc, b = odd ? pc : ps;
    c = __uint_as_float(__float_as_uint(a) ^ ((t + 0x40000000u) & 0x80000000u));
    s = __uint_as_float(__float_as_uint(b) ^ (t & 0x80000000u));
}

// One point's walk along an axis: the exact fixed-point phase and its first
// and second differences (Eq. 2, modulo one turn), and the factors of its
// cosine and sine entries (0 for a padding point).
struct Sep32Walk {
    uint64_t ph, d, dd;
    float re, im;
    __device__ __forceinline__ Sep32Walk(const PointRec &p, bool valid, bool is_x, int u) {
        const uint64_t b = is_x ? p.bx : p.by;
        ph = axis_phase(p.c, b, is_x ? p.ax : p.ay, u);
        d = p.c * (uint64_t)(2 * (int64_t)u + 1) - b;
        dd = 2 * p.c;
        re = valid ? (is_x ? p.A : S32_R_SCALE) : 0.0f;
        im = is_x ? -re : re;
    }
    // the entry pair as FP16 hi and lo, and one step on
    __device__ __forceinline__ void entry(__half2 &hi, __half2 &lo) {
        float s, c;
        sincos_fixed(ph, s, c);
        ph += d;
        d += dd;
        const float vr = re * c, vi = im * s;
        hi = __floats2half2_rn(vr, vi);
        const float2 h = __half22float2(hi);
        lo = __floats2half2_rn(vr - h.x, vi - h.y);
    }
};

// As sep_tables_kernel (separable.cu): one block per 64 points and 8 runs
// of ST_ROWS table rows; block (*, 0) also writes the blocks' factors, and
// the first block column zeroes the split schedule's arrival counters.
constexpr int S32_POINTS = 64;
constexpr int S32_BLOCK_ROWS = 8 * ST_ROWS;

__global__ void __launch_bounds__(256)
sep32_tables_kernel(PointSource src, int Npad, int Nx, int Ny, int Kp,
                    __half *__restrict__ Lhi, __half *__restrict__ Llo,
                    __half *__restrict__ Rhi, __half *__restrict__ Rlo,
                    float *__restrict__ scale, unsigned *__restrict__ zero, int nzero) {
    __shared__ PointRec srec[S32_POINTS];
    if (blockIdx.x == 0)
        for (int k = blockIdx.y * blockDim.x + threadIdx.x; k < nzero;
             k += gridDim.y * blockDim.x)
            zero[k] = 0u;
    const int j0 = blockIdx.x * S32_POINTS;
    if (threadIdx.x < S32_POINTS) {  // whole warps: one K block of 32 points each
        PointRec r{};
        if (j0 + (int)threadIdx.x < Npad)
            r = make_point_rec(src.points, src.A, src.z, src.N, j0 + threadIdx.x, src.K,
                               src.status, src.y0);
        const unsigned top =
            __reduce_max_sync(0xffffffffu, __float_as_uint(r.A) & 0x7fffffffu);
        // exponent of the block's largest |A_j|, kept where both factors are
        // FP32 numbers
        int e = top ? ilogbf(__uint_as_float(top)) : 0;
        e = e < -110 ? -110 : e;
        r.A = scalbnf(r.A, S32_EXP - 1 - e);
        srec[threadIdx.x] = r;
        if (blockIdx.y == 0 && (threadIdx.x & 31) == 0 && j0 + (int)threadIdx.x < Npad)
            scale[(j0 + threadIdx.x) / 32] = scalbnf(1.0f, e + 1 - 2 * S32_EXP);
    }
    __syncthreads();
    const int pair = threadIdx.x & 31, run = threadIdx.x >> 5;
    const int jj = j0 + 2 * pair;  // even; Npad is even, so jj + 1 < Npad too
    if (jj >= Npad) return;
    const int r0 = blockIdx.y * S32_BLOCK_ROWS + run * ST_ROWS;
    const int rows = Nx + Ny;
    if (r0 >= rows) return;
    const int r1 = r0 + ST_ROWS < rows ? r0 + ST_ROWS : rows;
#pragma unroll
    for (int seg = 0; seg < 2; ++seg) {  // the x rows, then the y rows
        const bool is_x = seg == 0;
        const int ra = is_x ? r0 : (r0 > Nx ? r0 : Nx);
        const int rb = is_x ? (r1 < Nx ? r1 : Nx) : r1;
        if (ra >= rb) continue;
        const int u = is_x ? ra : ra - Nx;
        Sep32Walk w0(srec[2 * pair], jj < src.N, is_x, u);
        Sep32Walk w1(srec[2 * pair + 1], jj + 1 < src.N, is_x, u);
        const size_t off = (size_t)u * Kp + 2 * (size_t)jj;
        __half *hi = (is_x ? Lhi : Rhi) + off, *lo = (is_x ? Llo : Rlo) + off;
#pragma unroll 2
        for (int r = ra; r < rb; ++r, hi += Kp, lo += Kp) {
            __half2 h[2], l[2];
            w0.entry(h[0], l[0]);
            w1.entry(h[1], l[1]);
            *reinterpret_cast<uint2 *>(hi) = *reinterpret_cast<const uint2 *>(h);
            *reinterpret_cast<uint2 *>(lo) = *reinterpret_cast<const uint2 *>(l);
        }
    }
    pdl_trigger();
}

// ------------------------------------------------------------------ GEMM
constexpr int S32_EPI_WARPS = 8;
constexpr int S32_THREADS = 64 + 32 * S32_EPI_WARPS;

struct Sep32Args {
    int M, N, K;
    float *D;
    long long ldd;
    const float *scale;  // one factor per K block
    float *part;         // [unit][cta rank][column / 4][row][4] partial tiles (S > 1)
    unsigned *count;     // [tile][cta rank] arrival counters, zero at launch (S > 1)
    int S;               // K slices
    int vec;             // stores of 4 consecutive columns are 16-byte aligned
    unsigned *status;
};

// Columns are handled in units of 16: the warps of half 0 take the first
// ceil(units / 2) units of a tile, those of half 1 the rest.
template <int BNP>
struct Sep32Cols {
    static constexpr int UNITS = BNP / 16;
    static constexpr int U0 = (UNITS + 1) / 2;  // units of half 0 (the larger)
    static constexpr int U1 = UNITS - U0;
    // tensor-memory buffers (512 columns in all) and their stride
    static constexpr int NBUF = BNP <= 128 ? 4 : 2;
    static constexpr uint32_t STRIDE = 512 / NBUF;
};

// acc += factor * tensor-memory buffer, nu units of 16 columns.
template <int U0>
__device__ __forceinline__ void sep32_promote(uint32_t taddr, int nu, float f,
                                              float (&acc)[U0 * 16]) {
    // two loads of 16 columns in flight ahead of the one being added
    uint32_t r[2][16];
    umma::tmem_ld16(taddr, r[0]);
#pragma unroll
    for (int u = 0; u < U0; ++u) {
        if (u >= nu) break;
        umma::tmem_ld_wait();
        uint32_t v[16];
#pragma unroll
        for (int i = 0; i < 16; ++i) v[i] = r[u & 1][i];
        if (u + 1 < nu) umma::tmem_ld16(taddr + (u + 1) * 16, r[(u + 1) & 1]);
#pragma unroll
        for (int i = 0; i < 16; ++i)
            acc[u * 16 + i] = fmaf(__uint_as_float(v[i]), f, acc[u * 16 + i]);
    }
}

// Grid: x = 2 x column tiles, y = row tiles of 256, z = K slices; clusters of
// two CTAs along x.
template <int BNP, int STAGES>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(S32_THREADS, 1)
sep32_pair_kernel(const __grid_constant__ CUtensorMap tA,
                  const __grid_constant__ CUtensorMap tB,
                  const __grid_constant__ CUtensorMap tA2,
                  const __grid_constant__ CUtensorMap tB2, Sep32Args g, uint32_t idesc) {
    using S = PairShape<BNP, true, STAGES>;
    using C = Sep32Cols<BNP>;
    extern __shared__ uint8_t smem_raw[];
    __shared__ __align__(8) uint64_t full[STAGES];   // (even CTA) both halves landed
    __shared__ __align__(8) uint64_t empty[STAGES];
    __shared__ __align__(8) uint64_t acc_full[C::NBUF];
    __shared__ __align__(8) uint64_t acc_empty[C::NBUF];  // (even CTA) both epilogues done
    __shared__ uint32_t tmem_base;
    __shared__ volatile int abort_flag;
    __shared__ int s_last;

    uint8_t *smem = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    const uint32_t rank = umma2::cluster_rank();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int m0 = blockIdx.y * 2 * S::BM + (int)rank * S::BM;  // this CTA's rows
    const int np0 = (blockIdx.x >> 1) * BNP;                     // the pair's columns
    const int nb = np0 + (int)rank * S::BNH;                     // this CTA's B rows
    const int KB = (g.K + S::BK - 1) / S::BK;
    const int kb0 = (int)((long long)KB * blockIdx.z / g.S);
    const int nkb = (int)((long long)KB * (blockIdx.z + 1) / g.S) - kb0;

    if (threadIdx.x == 0) {
        abort_flag = 0;
        for (int s = 0; s < STAGES; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        for (int b = 0; b < C::NBUF; ++b) {
            mbar_init(&acc_full[b], 1);
            mbar_init(&acc_empty[b], 2 * S32_EPI_WARPS);
        }
        mbar_fence_init();
        umma::prefetch_tmap(&tA);
        umma::prefetch_tmap(&tB);
        umma::prefetch_tmap(&tA2);
        umma::prefetch_tmap(&tB2);
    }
    if (warp == 1) {
        umma2::tmem_alloc2(&tmem_base, 512);
        umma2::tmem_relinquish2();
    }
    umma::fence_before_sync();
    umma2::cluster_sync();
    umma::fence_after_sync();
    const uint32_t tmem = tmem_base;
    pdl_wait();  // the tables and factors come from the kernel before

    if (warp == 0 && lane == 0) {
        // ------------------------------------------ producer (both CTAs)
        int issued = 0;
        for (int i = 0; i < nkb; ++i) {
            const int s = i % STAGES;
            if (i >= STAGES &&
                !mbar_wait_bounded(&empty[s], (uint32_t)(((i / STAGES) - 1) & 1))) {
                abort_flag = 1;
                set_status(g.status, DEV_TIMEOUT);
            }
            if (abort_flag) break;
            uint8_t *st = smem + (size_t)s * S::STAGE_BYTES;
            // the even CTA's barrier counts the bytes of both CTAs' loads
            if (rank == 0) mbar_arrive_expect_tx(&full[s], 2 * S::STAGE_BYTES);
            const uint32_t bar = umma2::map_to_rank(&full[s], 0);
            const int k = (kb0 + i) * S::BK;
            umma2::tma_load_2d_pair(st, &tA, k, m0, bar);
            umma2::tma_load_2d_pair(st + S::A_BYTES, &tB, k, nb, bar);
            umma2::tma_load_2d_pair(st + S::A_BYTES + S::B_BYTES, &tA2, k, m0, bar);
            umma2::tma_load_2d_pair(st + 2 * S::A_BYTES + S::B_BYTES, &tB2, k, nb, bar);
            ++issued;
        }
        if (abort_flag && rank == 0) {
            // let the stages' copies land before shared memory goes (the odd
            // CTA leaves only after the closing cluster barrier)
            for (int i = issued - STAGES < 0 ? 0 : issued - STAGES; i < issued; ++i)
                mbar_wait_bounded(&full[i % STAGES], (uint32_t)((i / STAGES) & 1));
        } else if (!abort_flag) {
            // wait (bounded) for the commits of the last stages, so that no
            // arrive is in flight when the CTA's shared memory passes on
            for (int i = nkb - STAGES < 0 ? 0 : nkb - STAGES; i < nkb; ++i)
                mbar_wait_bounded(&empty[i % STAGES], (uint32_t)((i / STAGES) & 1));
        }
    } else if (warp == 1 && lane == 0) {
        if (rank == 0) {
            // ---------------------------------------- MMA issuer (even CTA)
            for (int i = 0; i < nkb; ++i) {
                const int s = i % STAGES, b = i % C::NBUF;
                if (!mbar_wait_bounded(&acc_empty[b],
                                                 (uint32_t)(((i / C::NBUF) & 1) ^ 1)) ||
                    !mbar_wait_bounded(&full[s], (uint32_t)((i / STAGES) & 1))) {
                    abort_flag = 1;
                    set_status(g.status, DEV_TIMEOUT);
                }
                if (abort_flag) break;
                umma::fence_after_sync();
                const uint32_t a = smem_u32(smem + (size_t)s * S::STAGE_BYTES);
                const uint32_t bb = a + S::A_BYTES;
                const uint32_t a2 = bb + S::B_BYTES, b2 = a2 + S::A_BYTES;
                const uint64_t ad = umma::sw128_kmajor_desc(a);
                const uint64_t bd = umma::sw128_kmajor_desc(bb);
                const uint64_t ad2 = umma::sw128_kmajor_desc(a2);
                const uint64_t bd2 = umma::sw128_kmajor_desc(b2);
                const uint32_t d = tmem + (uint32_t)b * C::STRIDE;
                // the small cross products first: the sum's low bits are
                // dropped only by the four hi*hi steps
#pragma unroll
                for (int kk = 0; kk < 4; ++kk)
                    umma2::mma2_f16(d, ad + 2 * kk, bd2 + 2 * kk, idesc, kk != 0);
#pragma unroll
                for (int kk = 0; kk < 4; ++kk)
                    umma2::mma2_f16(d, ad2 + 2 * kk, bd + 2 * kk, idesc, 1);
#pragma unroll
                for (int kk = 0; kk < 4; ++kk)
                    umma2::mma2_f16(d, ad + 2 * kk, bd + 2 * kk, idesc, 1);
                umma2::commit2(&empty[s], 0x3);
                umma2::commit2(&acc_full[b], 0x3);
            }
        }
    } else if (warp >= 2) {
        // --------------------------------------- epilogue (both CTAs)
        const int q = warp & 3;               // the 32-lane quarter of TMEM
        const int half = (warp - 2) >> 2;     // the columns' half
        const int nu = half ? C::U1 : C::U0;  // its units of 16 columns
        const int c0 = half * C::U0 * 16;
        const int lrow = q * 32 + lane;
        const uint32_t t0 = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)c0;
        const uint32_t lead_empty = umma2::map_to_rank(&acc_empty[0], 0);
        float acc[C::U0 * 16];
#pragma unroll
        for (int i = 0; i < C::U0 * 16; ++i) acc[i] = 0.0f;
        bool ok = true;
        float f_next = __ldg(g.scale + kb0);
        for (int i = 0; i < nkb; ++i) {
            const int b = i % C::NBUF;
            const float f = f_next;
            f_next = __ldg(g.scale + kb0 + (i + 1 < nkb ? i + 1 : i));
            ok = __all_sync(0xffffffffu, mbar_wait_bounded(
                                             &acc_full[b], (uint32_t)((i / C::NBUF) & 1)));
            umma::fence_after_sync();
            if (!ok || abort_flag) {
                if (!ok) set_status(g.status, DEV_TIMEOUT);
                ok = false;
                break;
            }
            sep32_promote<C::U0>(t0 + (uint32_t)b * C::STRIDE, nu, f, acc);
            umma::fence_before_sync();
            __syncwarp();
            if (lane == 0) umma2::arrive_pair(lead_empty + (uint32_t)b * 8u);
        }
        bool store = ok;
        if (g.S > 1) {
            // publish the partial tile ([column / 4][row][4 columns]: 16-byte
            // stores of neighbouring rows are consecutive), then count in
            const size_t tile = (size_t)blockIdx.y * (gridDim.x >> 1) + (blockIdx.x >> 1);
            const size_t plane = (size_t)S::BM * BNP;
            float *dst = g.part + ((tile * g.S + blockIdx.z) * 2 + rank) * plane;
            if (ok) {
#pragma unroll
                for (int c = 0; c < C::U0 * 16; c += 4)
                    if (c < nu * 16)
                        *reinterpret_cast<float4 *>(
                            dst + ((size_t)((c0 + c) >> 2) * S::BM + lrow) * 4) =
                            make_float4(acc[c], acc[c + 1], acc[c + 2], acc[c + 3]);
            }
            __threadfence();
            asm volatile("bar.sync 1, %0;" ::"n"(32 * S32_EPI_WARPS) : "memory");
            if (threadIdx.x == 64)
                s_last = atomicAdd(&g.count[tile * 2 + rank], 1u) == (unsigned)(g.S - 1);
            asm volatile("bar.sync 1, %0;" ::"n"(32 * S32_EPI_WARPS) : "memory");
            store = ok && s_last;
            if (store) {
                __threadfence();
#pragma unroll
                for (int c = 0; c < C::U0 * 16; ++c) acc[c] = 0.0f;
                for (int z = 0; z < g.S; ++z) {
                    const float *src = g.part + ((tile * g.S + z) * 2 + rank) * plane;
#pragma unroll
                    for (int c = 0; c < C::U0 * 16; c += 4)
                        if (c < nu * 16) {
                            const float4 v = __ldcg(reinterpret_cast<const float4 *>(
                                src + ((size_t)((c0 + c) >> 2) * S::BM + lrow) * 4));
                            acc[c] += v.x;
                            acc[c + 1] += v.y;
                            acc[c + 2] += v.z;
                            acc[c + 3] += v.w;
                        }
                }
            }
        }
        const int row = m0 + lrow;
        if (store && row < g.M) {
            float *drow = g.D + (long long)row * g.ldd;
#pragma unroll
            for (int c = 0; c < C::U0 * 16; c += 4) {
                const int col = np0 + c0 + c;
                if (c >= nu * 16 || col >= g.N) break;
                if (g.vec && col + 4 <= g.N) {
                    *reinterpret_cast<float4 *>(drow + col) =
                        make_float4(acc[c], acc[c + 1], acc[c + 2], acc[c + 3]);
                } else {
#pragma unroll
                    for (int e = 0; e < 4; ++e)
                        if (col + e < g.N) drow[col + e] = acc[c + e];
                }
            }
        }
    }
    umma::fence_before_sync();
    umma2::cluster_sync();  // no MMA, commit or remote arrive still aims at either CTA
    if (warp == 1) {
        umma::fence_after_sync();
        umma2::tmem_dealloc2(tmem, 512);
    }
}

// ------------------------------------------------------------- host side
struct Sep32Plan {
    int bn, S;
};

static const int kSep32BN[] = {112, 128, 160, 192, 256};
constexpr int S32_MAX_SPLIT = 64;

// The tile width and the number of K slices with the least modelled time:
// waves of the SM pairs times (K blocks of a slice + fill and epilogue), plus
// the partial tiles of a split.  The constants are fits in microseconds to a
// sweep of every width and 1 to 64 slices over 13 frames (128 x 128 to
// 3840 x 2160, 64 to 16,384 points): a K block takes 0.69 us at 112 columns
// and 0.87 at 256 -- below 160 columns the MMA steps stop getting shorter
// (90 SM cycles each, for operand reads) -- so the narrow tiles only serve to
// fill the SMs, and a small frame is better cut along K: 128x128x16384 36 us
// in 32 slices against 327 in one, 640x480x2000 22.7 us in 6 against 49.
static Sep32Plan sep32_plan(int M, int N, int KB, int sms) {
    Sep32Plan best{256, 1};
    double best_cost = 1e300;
    const int pairs = sms / 2 > 0 ? sms / 2 : 1;
    for (int bn : kSep32BN) {
        const long long tiles = (long long)((M + 255) / 256) * ((N + bn - 1) / bn);
        for (int S = 1; S <= S32_MAX_SPLIT && S <= KB; ++S) {
            const long long waves = (tiles * S + pairs - 1) / pairs;
            const double cost =
                (double)waves * (((KB + S - 1) / S) * (0.55 + 0.00125 * bn) + 2.0 + 0.012 * bn) +
                (S > 1 ? 4.0 + 0.0065 * bn * S : 0.0);
            if (cost < best_cost) {
                best_cost = cost;
                best = Sep32Plan{bn, S};
            }
        }
    }
    return best;
}

struct Sep32Operands {
    const __half *A_hi, *A_lo, *B_hi, *B_lo;
    long long lda, ldb;
};

template <int BNP, int STAGES>
static cudaError_t launch_sep32_t(const Sep32Operands &op, const Sep32Args &g, cudaStream_t s) {
    using S = PairShape<BNP, true, STAGES>;
    CUtensorMap tA, tB, tA2, tB2;
    if (!make_gemm_map(&tA, op.A_hi, g.K, g.M, op.lda, S::BM, false) ||
        !make_gemm_map(&tB, op.B_hi, g.K, g.N, op.ldb, S::BNH, false) ||
        !make_gemm_map(&tA2, op.A_lo, g.K, g.M, op.lda, S::BM, false) ||
        !make_gemm_map(&tB2, op.B_lo, g.K, g.N, op.ldb, S::BNH, false))
        return cudaErrorInvalidValue;
    auto kern = sep32_pair_kernel<BNP, STAGES>;
    static bool attr_set[64] = {};
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev < 0 || dev >= 64 || !attr_set[dev]) {
        cudaError_t e = cudaFuncSetAttribute(
            kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)S::SMEM);
        if (e != cudaSuccess) return e;
        if (dev >= 0 && dev < 64) attr_set[dev] = true;
    }
    dim3 grid(2 * ((g.N + BNP - 1) / BNP), (g.M + 255) / 256, g.S);
    return launch_dependent(kern, grid, dim3(S32_THREADS), S::SMEM, s, tA, tB, tA2, tB2, g,
                            umma::idesc_f16(2 * S::BM, BNP, false));
}

static cudaError_t launch_sep32(int bn, const Sep32Operands &op, const Sep32Args &g,
                                cudaStream_t s) {
    switch (bn) {
    case 112: return launch_sep32_t<112, 4>(op, g, s);
    case 128: return launch_sep32_t<128, 4>(op, g, s);
    case 160: return launch_sep32_t<160, 4>(op, g, s);
    case 192: return launch_sep32_t<192, 4>(op, g, s);
    case 256: return launch_sep32_t<256, 3>(op, g, s);
    }
    return cudaErrorInvalidValue;
}

}  // namespace cgh

using namespace cgh;

cgh_status cgh_ctx::forward_sep32(const float *points, const float *A, const float *z, int N,
                                  double lambda, double p, int Nx, int Ny, float *out,
                                  cudaStream_t s) {
    const int Kp = pad_to(2 * N, 64);
    const int Npad = Kp / 2;
    const Sep32Plan plan = sep32_plan(Ny, Nx, Kp / 64, sm_count);
    const size_t tiles = (size_t)((Ny + 255) / 256) * ((Nx + plan.bn - 1) / plan.bn);
    const size_t l_b = align256((size_t)Nx * Kp * 2);
    const size_t r_b = align256((size_t)Ny * Kp * 2);
    const size_t sc_b = align256((size_t)(Kp / 64) * sizeof(float));
    const size_t part_b =
        plan.S > 1 ? align256(tiles * plan.S * 256 * plan.bn * sizeof(float)) : 0;
    const size_t cnt_b = plan.S > 1 ? align256(tiles * 2 * sizeof(unsigned)) : 0;
    cgh_status st = ensure(ws, 2 * (l_b + r_b) + sc_b + part_b + cnt_b, s,
                           "FP32 separable workspace");
    if (st) return st;
    char *base = (char *)ws.ptr;
    __half *Lhi = (__half *)base, *Rhi = (__half *)(base + l_b);
    __half *Llo = (__half *)(base + l_b + r_b), *Rlo = (__half *)(base + 2 * l_b + r_b);
    char *rest = base + 2 * (l_b + r_b);
    float *scale = (float *)rest;
    float *part = plan.S > 1 ? (float *)(rest + sc_b) : nullptr;
    unsigned *count = plan.S > 1 ? (unsigned *)(rest + sc_b + part_b) : nullptr;
    {
        TimedLaunch tl(this, CGH_K_SEP_TABLES, s);
        const int rows = Nx + Ny;
        dim3 grid((Npad + S32_POINTS - 1) / S32_POINTS,
                  (rows + S32_BLOCK_ROWS - 1) / S32_BLOCK_ROWS);
        cudaError_t e = launch_kernel(
            false, sep32_tables_kernel, grid, dim3(256), 0, s,
            PointSource{points, A, z, N, fresnel_scale(lambda, p), d_status, row_origin}, Npad,
            Nx, Ny, Kp, Lhi, Llo, Rhi, Rlo, scale, count, plan.S > 1 ? (int)(2 * tiles) : 0);
        if (e != cudaSuccess) return cuda_fail(e, "FP32 separable tables launch");
        tl.done();
    }
    {
        TimedLaunch tl(this, CGH_K_SIMT, s);
        Sep32Args g{};
        g.M = Ny;
        g.N = Nx;
        g.K = Kp;
        g.D = out;
        g.ldd = Nx;
        g.scale = scale;
        g.part = part;
        g.count = count;
        g.S = plan.S;
        g.vec = (Nx % 4 == 0) && (((uintptr_t)out & 15) == 0);
        g.status = d_status;
        cudaError_t e = launch_sep32(plan.bn, Sep32Operands{Rhi, Rlo, Lhi, Llo, Kp, Kp}, g, s);
        if (e != cudaSuccess) return cuda_fail(e, "FP32 separable product launch");
        tl.done();
    }
    return CGH_OK;
}
