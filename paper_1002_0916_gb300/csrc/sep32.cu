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
// block): a K block takes 0.81 us at 256 columns and 0.37 at 112 (one pair
// alone), 139 and 63 SM cycles a step.  Two things cost more than the MMAs
// before: issued from one lane's branch instead of an elected lane of a
// converged warp, a step took 105 to 120 cycles at any width below 192 (see
// elect_one); and with cluster-scope acquire and release on the epilogue's
// barriers a block took 1.1 to 1.4 us (the waits are at CTA scope and the
// arrivals relaxed: tensor memory is ordered by the tcgen05 fences, and no
// generic memory is handed over).
// Measured, whole call, against an FP32 product on the FMA pipe (0.70 of its
// bound): 1920x1024x3584 543 -> 73 us, 3840x2160x16384 9.85 -> 1.02 ms;
// relative RMS error against FP64 6.8e-7 -> 2.3e-7 and 1.6e-6 -> 4.3e-7.
//
// A tile's columns are equal shares at the plan's number of waves, as in
// umma2.cu (3840x2160x16384 1060 -> 1040 us, 640x480x300 13.3 -> 12.2).
// Long products on few tiles are cut along K into S slices: each slice's
// CTA writes its partial tile, and the last slice of a tile to finish adds
// the S partials in slice order (deterministic).
#include <cudaTypedefs.h>
#include <math.h>

#include "api_internal.h"
#include "common.cuh"
#include "point_rec.cuh"
#include "sep32.cuh"
#include "sep_table.cuh"
#include "umma.cuh"
#include "umma_epi.cuh"
#include "umma_pair.cuh"

namespace cgh {

int sm_count_of_current_device();
bool make_gemm_map(CUtensorMap *m, const void *base, long long inner, long long rows,
                   long long ld, int box_rows, bool bf16);

// ---------------------------------------------------------------- tables
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
// One warpgroup with the producer and the MMA issuer, two of epilogue warps.
// 384 threads get 168 registers each at launch; the first group gives up all
// but 56, the others take 224 (56 + 2 x 224 = 3 x 168), which holds a
// thread's 128 sums and two tensor-memory loads without spills (at 168: 5 to
// 10% slower).
constexpr int S32_THREADS = 128 + 32 * S32_EPI_WARPS;
constexpr int S32_ROLE_REGS = 56, S32_EPI_REGS = 224;

struct Sep32Args {
    int units, tiles_m, tiles_n, KB;  // forward: tiles, K blocks; units of either
    int bw;                           // columns per tile, at most BNP
    int M, N;
    float *D;
    long long ldd;
    const float *scale;  // one factor per K block
    float *part;         // [unit][cta rank][column / 4][row][4] partial tiles (S > 1)
    unsigned *count;     // [tile][cta rank] arrival counters, zero at launch (S > 1)
    int S;               // K slices
    int vec;             // store_width(D, ldd)
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

// Forward epilogue: with K slices, publish the partial tile ([column / 4]
// [row][4 columns]: 16-byte stores of neighbouring rows are consecutive),
// count in, and let the last slice add all of them; then store the row,
// clipped to the frame.  Called by every epilogue warp.
template <int BNP>
__device__ __forceinline__ void sep32_store(const Sep32Args &g, bool ok, int mt, int nt, int slice,
                                            int rank, int half, int lrow, int m0, int np0,
                                            int *s_last, float *stage,
                                            float (&acc)[Sep32Cols<BNP>::U0 * 16]) {
    using C = Sep32Cols<BNP>;
    constexpr int BM = 128;
    const int nu = half ? C::U1 : C::U0, c0 = half * C::U0 * 16;
    const int end = np0 + g.bw < g.N ? np0 + g.bw : g.N;  // of the tile's columns
    bool store = ok;
    if (g.S > 1) {
        const size_t tile = (size_t)mt * g.tiles_n + nt;
        const size_t plane = (size_t)BM * BNP;
        float *dst = g.part + ((tile * g.S + slice) * 2 + rank) * plane;
        if (ok) {
#pragma unroll
            for (int c = 0; c < C::U0 * 16; c += 4)
                if (c < nu * 16)
                    *reinterpret_cast<float4 *>(dst + ((size_t)((c0 + c) >> 2) * BM + lrow) * 4) =
                        make_float4(acc[c], acc[c + 1], acc[c + 2], acc[c + 3]);
        }
        __threadfence();
        asm volatile("bar.sync 1, %0;" ::"n"(32 * S32_EPI_WARPS) : "memory");
        if (threadIdx.x == 128)
            *s_last = atomicAdd(&g.count[tile * 2 + rank], 1u) == (unsigned)(g.S - 1);
        asm volatile("bar.sync 1, %0;" ::"n"(32 * S32_EPI_WARPS) : "memory");
        store = ok && *(volatile int *)s_last;
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
                            src + ((size_t)((c0 + c) >> 2) * BM + lrow) * 4));
                        acc[c] += v.x;
                        acc[c + 1] += v.y;
                        acc[c + 2] += v.z;
                        acc[c + 3] += v.w;
                    }
            }
        }
    }
    const int row = m0 + lrow;
    if (!store) return;  // (the same in every lane)
    if (!g.vec) {
        const int lane = lrow & 31, row0 = row - lane;
#pragma unroll
        for (int u = 0; u < C::U0; ++u)
            if (u < nu)
                epilogue_store_odd(stage, acc + u * 16, g.D + (long long)row0 * g.ldd, g.ldd,
                                   g.M - row0, np0 + c0 + u * 16, end, false, lane);
        return;
    }
    if (row >= g.M) return;
    float *drow = g.D + (long long)row * g.ldd;
#pragma unroll
    for (int c = 0; c < C::U0 * 16; c += 8) {
        const int col = np0 + c0 + c;
        if (c >= nu * 16 || col >= end) break;
        if (g.vec == 2 && col + 8 <= end) {
            store8(drow + col, acc + c);
        } else if (col + 8 <= end) {
            *reinterpret_cast<float4 *>(drow + col) =
                make_float4(acc[c], acc[c + 1], acc[c + 2], acc[c + 3]);
            *reinterpret_cast<float4 *>(drow + col + 4) =
                make_float4(acc[c + 4], acc[c + 5], acc[c + 6], acc[c + 7]);
        } else {
#pragma unroll
            for (int e = 0; e < 8; ++e)
                if (col + e < end) drow[col + e] = acc[c + e];
        }
    }
}

// Adjoint epilogue.  GEMM row k = 2j + c (c = 0: cosine row, 1: sine row of
// point j); with (W_c, W_s) = rows 2j, 2j + 1 of D at column u, (cu, su) =
// cos, sin of theta_axis(u, j) and d = u - u_j, sum over the columns
//     C = cu W_c - su W_s,   S = su W_c + cu W_s
// with weights 1 for C and d, d^2 for S.  The two lanes of a point hold the
// two rows: the even lane takes the first half of the warp's columns, the odd
// lane the second, and each sends the other the value it lacks.  With the odd
// lane's phase a quarter turn ahead, (c', s') its cosine and sine, and r the
// received value (negated when it comes from the odd lane), both lanes compute
// C = own c' + r s' and -S = r c' - own s'.  d = i + delta with i the column's
// index in the lane's run: the sums are taken with i and shifted at the end.
// Columns beyond the frame have zero operands, hence W = 0.
// (Reading the weights from the split tables instead of stepping the phase by
// Eq. 2 and taking sincos_fixed cost 7.8 us a tile, waiting on L2.)
template <int U0>
__device__ __forceinline__ void adj32_reduce(const Adj32Prod &pr, const Adj32Args &ga, int t,
                                             int row, int n0, const float (&acc)[U0 * 16]) {
    constexpr int RUN = U0 * 8;  // columns per lane
    const int j = row >> 1;
    const bool odd = (row & 1) != 0, valid = j < ga.n;
    const int u0 = n0 + (odd ? RUN : 0);
    uint64_t ph = 0, d = 0, dd = 0;
    if (valid) {
        const PointRec &r = ga.rec[j];
        const uint64_t b = pr.axis ? r.by : r.bx;
        ph = axis_phase(r.c, b, pr.axis ? r.ay : r.ax, u0) + (odd ? 1ull << 62 : 0ull);
        d = r.c * (uint64_t)(2 * (int64_t)u0 + 1) - b;
        dd = 2 * r.c;
    }
    // (C by eights of columns: one chain of two roundings a column left the
    // amplitudes' gradient at 2.2e-7 from FP64, against 1.7e-7; what is left is
    // the tensor cores' truncation, a shrink of 7e-8 in each product on random
    // phases)
    float C = 0.0f, C8 = 0.0f, S0 = 0.0f, S1 = 0.0f, S2 = 0.0f;
#pragma unroll
    for (int i = 0; i < RUN; ++i) {
        const float own = odd ? acc[RUN + i] : acc[i];
        const float r = __shfl_xor_sync(0xffffffffu, odd ? -acc[i] : acc[RUN + i], 1);
        float s, c;
        sincos_fixed(ph, s, c);
        ph += d;
        d += dd;
        C8 = fmaf(own, c, fmaf(r, s, C8));
        if (i % 8 == 7) {
            C += C8;
            C8 = 0.0f;
        }
        const float v = fmaf(own, s, -r * c);
        S0 += v;
        S1 = fmaf(v, (float)i, S1);
        S2 = fmaf(v, (float)(i * i), S2);
    }
    const float delta = valid ? (float)u0 - ga.points[2 * j + pr.axis] : 0.0f;
    S2 = fmaf(delta, fmaf(delta, S0, 2.0f * S1), S2);
    S1 = fmaf(delta, S0, S1);
    C += __shfl_xor_sync(0xffffffffu, C, 1);
    S1 += __shfl_xor_sync(0xffffffffu, S1, 1);
    S2 += __shfl_xor_sync(0xffffffffu, S2, 1);
    if (valid && !odd) {
        float *p = pr.part + (size_t)t * 3 * ga.npad + j;
        p[0] = C;
        p[ga.npad] = S1;
        p[2 * ga.npad] = S2;
    }
}

struct Sep32Maps {
    CUtensorMap A, B, A2, B2;  // hi and lo planes: M x K and N x K, K-major
};

// One unit of work: a tile of one product over one K slice.
struct Sep32Unit {
    int which, mt, nt, slice, kb0, nkb;
};

template <bool ADJ>
__device__ __forceinline__ Sep32Unit sep32_unit(int u, const Sep32Args &g, const Adj32Args &ga) {
    Sep32Unit w;
    int tn = g.tiles_n, tm = g.tiles_m, S = g.S, KB = g.KB;
    w.which = 0;
    if constexpr (ADJ) {
        tm = ga.tiles_m;
        w.which = u >= ga.p[0].units;
        if (w.which) u -= ga.p[0].units;
        tn = w.which ? ga.p[1].tiles_n : ga.p[0].tiles_n;
        S = w.which ? ga.p[1].S : ga.p[0].S;
        KB = w.which ? ga.p[1].KB : ga.p[0].KB;
    }
    w.nt = u % tn;
    u /= tn;
    w.mt = u % tm;
    w.slice = u / tm;
    w.kb0 = (int)((long long)KB * w.slice / S);
    w.nkb = (int)((long long)KB * (w.slice + 1) / S) - w.kb0;
    return w;
}

// Persistent: clusters of two CTAs (one per SM) take the units in
// group_item_index order; loads and MMAs run ahead into the next unit while
// the epilogue of the last one finishes.  ADJ: both products of the adjoint
// in one list, the longer K first.
template <int BNP, int STAGES, bool ADJ>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(S32_THREADS, 1)
sep32_pair_kernel(const __grid_constant__ Sep32Maps maps0,
                  const __grid_constant__ Sep32Maps maps1, const __grid_constant__ Sep32Args g,
                  const __grid_constant__ Adj32Args ga, uint32_t idesc) {
    using S = PairShape<BNP, true, STAGES>;
    using C = Sep32Cols<BNP>;
    extern __shared__ uint8_t smem_raw[];
    __shared__ __align__(8) uint64_t full[STAGES];   // (even CTA) both halves landed
    __shared__ __align__(8) uint64_t empty[STAGES];
    __shared__ __align__(8) uint64_t acc_full[C::NBUF];
    __shared__ __align__(8) uint64_t acc_empty[C::NBUF];  // (even CTA) both epilogues done
    __shared__ __align__(8) uint64_t drain;  // (even CTA) after a timeout: MMAs done
    __shared__ uint32_t tmem_base;
    __shared__ volatile int abort_flag;
    __shared__ int s_last;

    uint8_t *smem = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    const uint32_t rank = umma2::cluster_rank();
    const int warp = umma::warp_index(), lane = threadIdx.x & 31;
    const int cl = blockIdx.x >> 1, ncl = gridDim.x >> 1;

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
        mbar_init(&drain, 1);
        mbar_fence_init();
        umma::prefetch_tmap(&maps0.A);
        umma::prefetch_tmap(&maps0.B);
        umma::prefetch_tmap(&maps0.A2);
        umma::prefetch_tmap(&maps0.B2);
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

    if (warp < 4) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(S32_ROLE_REGS));
        if (warp == 0) {
            // -------------------------------------- producer (both CTAs)
            unsigned n = 0;  // K blocks issued
            bool ok = true;
            const int bw = ADJ ? BNP : g.bw;
            const uint32_t bytes = 4 * (S::A_BYTES + (uint32_t)bw * S::BK);
            for (int r = 0; r * ncl < g.units && ok; ++r) {
                const int u = group_item_index(r, cl, ncl);
                if (u >= g.units) break;
                const Sep32Unit w = sep32_unit<ADJ>(u, g, ga);
                const Sep32Maps *maps = w.which ? &maps1 : &maps0;
                const int m0 = w.mt * 2 * S::BM + (int)rank * S::BM;  // this CTA's rows
                const int nb = w.nt * bw + (int)rank * (bw / 2);      // its B rows
                for (int i = 0; i < w.nkb; ++i, ++n) {
                    const int s = (int)(n % STAGES);
                    if (n >= STAGES && !mbar_wait_bounded(&empty[s], ((n / STAGES) - 1) & 1)) {
                        abort_flag = 1;
                        set_status(g.status, DEV_TIMEOUT);
                    }
                    ok = __all_sync(0xffffffffu, !abort_flag);
                    if (!ok) break;
                    uint8_t *st = smem + (size_t)s * S::STAGE_BYTES;
                    const uint32_t bar = umma2::map_to_rank(&full[s], 0);
                    const int k = (w.kb0 + i) * S::BK;
                    if (umma::elect_one()) {
                        // the even CTA's barrier counts the bytes of both CTAs' loads
                        if (rank == 0) mbar_arrive_expect_tx(&full[s], bytes);
                        umma2::tma_load_2d_pair(st, &maps->A, k, m0, bar);
                        umma2::tma_load_2d_pair(st + S::A_BYTES, &maps->B, k, nb, bar);
                        umma2::tma_load_2d_pair(st + S::A_BYTES + S::B_BYTES, &maps->A2, k, m0,
                                                bar);
                        umma2::tma_load_2d_pair(st + 2 * S::A_BYTES + S::B_BYTES, &maps->B2, k,
                                                nb, bar);
                    }
                }
            }
            const unsigned lo = n > STAGES ? n - STAGES : 0;
            if (!ok && rank == 0) {
                // let the stages' copies land before shared memory goes (the odd
                // CTA leaves only after the closing cluster barrier)
                for (unsigned i = lo; i < n; ++i)
                    mbar_wait_bounded(&full[i % STAGES], (i / STAGES) & 1);
            } else if (ok) {
                // wait (bounded) for the commits of the last stages, so that no
                // arrive is in flight when the CTA's shared memory passes on
                for (unsigned i = lo; i < n; ++i)
                    mbar_wait_bounded(&empty[i % STAGES], (i / STAGES) & 1);
            }
        } else if (warp == 1 && rank == 0) {
            // ---------------------------------------- MMA issuer (even CTA)
            unsigned n = 0;
            bool ok = true;
            for (int r = 0; r * ncl < g.units && ok; ++r) {
                const int u = group_item_index(r, cl, ncl);
                if (u >= g.units) break;
                const int nkb = sep32_unit<ADJ>(u, g, ga).nkb;
                for (int i = 0; i < nkb; ++i, ++n) {
                    const int s = (int)(n % STAGES), b = (int)(n % C::NBUF);
                    if (!mbar_wait_bounded(&acc_empty[b], ((n / C::NBUF) & 1) ^ 1) ||
                        !mbar_wait_bounded(&full[s], (n / STAGES) & 1)) {
                        abort_flag = 1;
                        set_status(g.status, DEV_TIMEOUT);
                    }
                    ok = __all_sync(0xffffffffu, !abort_flag);
                    if (!ok) break;
                    umma::fence_after_sync();
                    const uint32_t a = smem_u32(smem + (size_t)s * S::STAGE_BYTES);
                    const uint32_t bb = a + S::A_BYTES;
                    const uint32_t a2 = bb + S::B_BYTES, b2 = a2 + S::A_BYTES;
                    const uint64_t ad = umma::sw128_kmajor_desc(a);
                    const uint64_t bd = umma::sw128_kmajor_desc(bb);
                    const uint64_t ad2 = umma::sw128_kmajor_desc(a2);
                    const uint64_t bd2 = umma::sw128_kmajor_desc(b2);
                    const uint32_t d = tmem + (uint32_t)b * C::STRIDE;
                    if (umma::elect_one()) {
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
                    __syncwarp();
                }
            }
            if (!ok) {
                // the blocks issued so far use the stages and tensor memory of
                // both CTAs, which are released after the closing barrier
                if (umma::elect_one()) umma2::commit2(&drain, 0x1);
                mbar_wait_bounded(&drain, 0);
            }
        }
    } else {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(S32_EPI_REGS));
        // --------------------------------------- epilogue (both CTAs)
        const int q = warp & 3;               // the 32-lane quarter of TMEM
        const int half = (warp - 4) >> 2;     // the columns' half
        const int nu = half ? C::U1 : C::U0;  // its units of 16 columns
        const int c0 = half * C::U0 * 16;
        const int lrow = q * 32 + lane;
        const uint32_t t0 = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)c0;
        const uint32_t lead_empty = umma2::map_to_rank(&acc_empty[0], 0);
        float *stage = reinterpret_cast<float *>(smem + (size_t)STAGES * S::STAGE_BYTES) +
                       (warp - 4) * EPI_WARP_FLOATS;  // (forward only)
        bool ok = true;
        unsigned n = 0;
        for (int r = 0; r * ncl < g.units; ++r) {
            const int u = group_item_index(r, cl, ncl);
            if (u >= g.units) break;
            const Sep32Unit w = sep32_unit<ADJ>(u, g, ga);
            float acc[C::U0 * 16];
#pragma unroll
            for (int i = 0; i < C::U0 * 16; ++i) acc[i] = 0.0f;
            float f_next = ADJ ? S32_ADJ_FACTOR : __ldg(g.scale + w.kb0);
            for (int i = 0; i < w.nkb && ok; ++i, ++n) {
                const int b = (int)(n % C::NBUF);
                const float f = f_next;
                if (!ADJ) f_next = __ldg(g.scale + w.kb0 + (i + 1 < w.nkb ? i + 1 : i));
                const bool landed = mbar_wait_bounded(&acc_full[b], (n / C::NBUF) & 1);
                if (!landed) set_status(g.status, DEV_TIMEOUT);
                ok = __all_sync(0xffffffffu, landed && !abort_flag);
                if (!ok) break;
                umma::fence_after_sync();
                sep32_promote<C::U0>(t0 + (uint32_t)b * C::STRIDE, nu, f, acc);
                umma::fence_before_sync();
                __syncwarp();
                if (lane == 0) umma2::arrive_pair(lead_empty + (uint32_t)b * 8u);
            }
            const int m0 = w.mt * 2 * S::BM + (int)rank * S::BM;
            if constexpr (ADJ) {
                static_assert(C::U0 == C::U1, "equal column halves");
                if (ok)
                    adj32_reduce<C::U0>(ga.p[w.which], ga, (w.slice * (w.which ? ga.p[1].tiles_n : ga.p[0].tiles_n) + w.nt) * 2 + half,
                                        m0 + lrow, w.nt * BNP + c0, acc);
            } else {
                // (every warp, also after a timeout: it meets at barriers)
                sep32_store<BNP>(g, ok, w.mt, w.nt, w.slice, (int)rank, half, lrow, m0,
                                 w.nt * g.bw, &s_last, stage, acc);
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

static const int kSep32BN[] = {112, 128, 144, 160, 192, 224, 256};
constexpr int S32_MAX_SPLIT = 64;

// The tile width and the number of K slices with the least modelled time:
// waves of the SM pairs times (K blocks of a slice + fill and epilogue), plus
// the partial tiles of a split.  The constants are fits in microseconds to a
// sweep of every width and 1 to 64 slices over 13 frames (128 x 128 to
// 3840 x 2160, 64 to 16,384 points), taken with slower MMA issue: a K block of
// 0.44 us at 112 columns and 0.87 at 256 (0.37 and 0.81 since).  A small frame is
// better cut along K: 128x128x16384 31 us
// in 24 slices against 187 in one, 640x480x2000 21 us in 5 against 39.
static Sep32Plan sep32_plan(int M, int N, int KB, int sms) {
    Sep32Plan best{256, 1};
    double best_cost = 1e300;
    const int pairs = sms / 2 > 0 ? sms / 2 : 1;
    for (int bn : kSep32BN) {
        const long long tiles = (long long)((M + 255) / 256) * ((N + bn - 1) / bn);
        for (int S = 1; S <= S32_MAX_SPLIT && S <= KB && (S == 1 || tiles * S <= 2 * pairs); ++S) {
            const long long waves = (tiles * S + pairs - 1) / pairs;
            const double cost =
                (double)waves * (((KB + S - 1) / S) * (0.10 + 0.0030 * bn) + 2.0 + 0.012 * bn) +
                (S > 1 ? 4.0 + 0.0065 * bn * S : 0.0);
            if (cost < best_cost) {
                best_cost = cost;
                best = Sep32Plan{bn, S};
            }
        }
    }
    return best;
}

static bool make_sep32_maps(Sep32Maps *m, const Sep32Operands &op, int M, int N, int K, int bw) {
    return make_gemm_map(&m->A, op.A_hi, K, M, op.lda, 128, false) &&
           make_gemm_map(&m->B, op.B_hi, K, N, op.ldb, bw / 2, false) &&
           make_gemm_map(&m->A2, op.A_lo, K, M, op.lda, 128, false) &&
           make_gemm_map(&m->B2, op.B_lo, K, N, op.ldb, bw / 2, false);
}

template <int BNP, int STAGES, bool ADJ>
static cudaError_t launch_sep32_kernel(const Sep32Maps &m0, const Sep32Maps &m1,
                                       const Sep32Args &g, const Adj32Args &ga, int bw,
                                       cudaStream_t s) {
    using S = PairShape<BNP, true, STAGES>;
    constexpr size_t SMEM = ADJ ? S::RING : S::SMEM;
    static_assert(SMEM <= 232448 - 1024, "shared memory");
    auto kern = sep32_pair_kernel<BNP, STAGES, ADJ>;
    static bool attr_set[64] = {};
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev < 0 || dev >= 64 || !attr_set[dev]) {
        cudaError_t e = cudaFuncSetAttribute(
            kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SMEM);
        if (e != cudaSuccess) return e;
        if (dev >= 0 && dev < 64) attr_set[dev] = true;
    }
    const int pairs = sm_count_of_current_device() / 2;
    const int clusters = g.units < pairs ? g.units : pairs > 0 ? pairs : 1;
    return launch_dependent(kern, dim3(2 * clusters), dim3(S32_THREADS), SMEM, s, m0, m1, g, ga,
                            umma::idesc_f16(2 * S::BM, bw, false));
}

template <int BNP, int STAGES>
static cudaError_t launch_sep32_t(const Sep32Operands &op, const Sep32Args &g, cudaStream_t s) {
    Sep32Maps m;
    if (!make_sep32_maps(&m, op, g.M, g.N, 64 * g.KB, g.bw)) return cudaErrorInvalidValue;
    return launch_sep32_kernel<BNP, STAGES, false>(m, m, g, Adj32Args{}, g.bw, s);
}

static cudaError_t launch_sep32(int bn, const Sep32Operands &op, const Sep32Args &g,
                                cudaStream_t s) {
    switch (bn) {
    case 112: return launch_sep32_t<112, 4>(op, g, s);
    case 128: return launch_sep32_t<128, 4>(op, g, s);
    case 144: return launch_sep32_t<144, 4>(op, g, s);
    case 160: return launch_sep32_t<160, 4>(op, g, s);
    case 192: return launch_sep32_t<192, 3>(op, g, s);
    case 224: return launch_sep32_t<224, 3>(op, g, s);
    case 256: return launch_sep32_t<256, 3>(op, g, s);
    }
    return cudaErrorInvalidValue;
}

// ------------------------------------------------------ adjoint products
static const int kAdj32BN[] = {192, 224, 256};

// The width and slices with the least modelled time (the constants of
// sep32_plan): units of both products on the SM pairs, longest first, so the
// total spread over the pairs plus part of a unit, or the longest unit alone.
// A unit's epilogue adds about 2.9 us that the next unit's MMAs do not cover
// (1920x1080x4096: 128 us at 224 columns, 134 at 192, 141 at 256); a K slice
// costs nothing else, since the epilogue is linear in D and every slice writes
// its own partial sums.
Adj32Plan adj32_plan(int n, int Nx, int Ny, int sms) {
    Adj32Plan best{256, {1, 1}};
    double best_cost = 1e300;
    const double pairs = sms / 2 > 0 ? sms / 2 : 1;
    const long long mt = (2LL * n + 255) / 256;
    const int N[2] = {Nx <= Ny ? Nx : Ny, Nx <= Ny ? Ny : Nx};  // columns; K = the other
    const int KB[2] = {(N[1] + 63) / 64, (N[0] + 63) / 64};
    for (int bn : kAdj32BN) {
        const double tkb = 1.1 * (0.10 + 0.0030 * bn), epi = 2.9;
        // (slices only where the tiles alone leave pairs idle)
        const long long t0 = mt * ((N[0] + bn - 1) / bn), t1 = mt * ((N[1] + bn - 1) / bn);
        const int most = t0 + t1 >= 4 * pairs ? 1 : 16;
        for (int S0 = 1; S0 <= most && S0 <= KB[0]; ++S0)
            for (int S1 = 1; S1 <= most && S1 <= KB[1]; ++S1) {
                if (S0 + S1 > 2 && t0 * S0 + t1 * S1 > 2 * pairs) break;
                const double n0 = (double)(t0 * S0), n1 = (double)(t1 * S1);
                const double u0 = ((KB[0] + S0 - 1) / S0) * tkb + epi;
                const double u1 = ((KB[1] + S1 - 1) / S1) * tkb + epi;
                const double longest = u0 > u1 ? u0 : u1;
                const double total = (n0 * u0 + n1 * u1) / pairs;
                const double cost = n0 + n1 <= pairs ? longest : total + 0.3 * longest;
                if (cost < best_cost * 0.99) {
                    best_cost = cost;
                    best = Adj32Plan{bn, {S0, S1}};
                }
            }
    }
    // Whole units of the longer K that outlast a pair's share of all the work (a
    // low wide frame's few tiles over x beside its many over y) are cut until
    // they do not: 32768x32x500 376 -> 113 us, 3564x195x1456 76 -> 52.
    if (best.S[0] == 1 && best.S[1] == 1) {
        const double tkb = 1.1 * (0.10 + 0.0030 * best.bn), epi = 2.9;
        const double n0 = (double)(mt * ((N[0] + best.bn - 1) / best.bn));
        const double n1 = (double)(mt * ((N[1] + best.bn - 1) / best.bn));
        for (int S0 = 1; S0 <= 16 && S0 <= KB[0]; ++S0) {
            const double u0 = ((KB[0] + S0 - 1) / S0) * tkb + epi, u1 = KB[1] * tkb + epi;
            best.S[0] = S0;
            if (u0 <= (n0 * S0 * u0 + n1 * u1) / pairs) break;
        }
    }
    return best;
}

template <int BNP, int STAGES>
static cudaError_t launch_adj32_t(const Sep32Operands (&op)[2], const int (&N)[2],
                                  const int (&K)[2], const Adj32Args &ga, unsigned *status,
                                  cudaStream_t s) {
    Sep32Maps m[2];
    for (int i = 0; i < 2; ++i)
        if (!make_sep32_maps(&m[i], op[i], 2 * ga.n, N[i], K[i], BNP)) return cudaErrorInvalidValue;
    Sep32Args g{};
    g.status = status;
    g.units = ga.p[0].units + ga.p[1].units;
    return launch_sep32_kernel<BNP, STAGES, true>(m[0], m[1], g, ga, BNP, s);
}

cudaError_t launch_adj32(int bn, const Sep32Operands (&op)[2], const int (&N)[2],
                         const int (&K)[2], const Adj32Args &ga, unsigned *status,
                         cudaStream_t s) {
    switch (bn) {
    case 192: return launch_adj32_t<192, 4>(op, N, K, ga, status, s);
    case 224: return launch_adj32_t<224, 3>(op, N, K, ga, status, s);
    case 256: return launch_adj32_t<256, 3>(op, N, K, ga, status, s);
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
    const int bw = pair_columns(Ny, Nx, plan.bn, sm_count, plan.S);
    const size_t tiles = (size_t)((Ny + 255) / 256) * ((Nx + bw - 1) / bw);
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
        g.tiles_m = (Ny + 255) / 256;
        g.tiles_n = (Nx + bw - 1) / bw;
        g.bw = bw;
        g.units = g.tiles_m * g.tiles_n * plan.S;
        g.KB = Kp / 64;
        g.D = out;
        g.ldd = Nx;
        g.scale = scale;
        g.part = part;
        g.count = count;
        g.S = plan.S;
        g.vec = store_width(out, Nx);
        g.status = d_status;
        cudaError_t e = launch_sep32(plan.bn, Sep32Operands{Rhi, Rlo, Lhi, Llo, Kp, Kp}, g, s);
        if (e != cudaSuccess) return cuda_fail(e, "FP32 separable product launch");
        tl.done();
    }
    return CGH_OK;
}
