// umma_epi.cuh -- arguments and row store shared by the one-CTA (umma.cu) and
// CTA-pair (umma2.cu) tensor-core GEMMs.  Internal to libcgh.
#pragma once

#include "common.cuh"
#include "umma.cuh"

namespace cgh {

struct GemmArgs {
    int M, N, K;
    float *D;
    long long ldd;
    float lo_scale;
    unsigned *status;
    int accumulate;  // 0: D = product; 1: D += product (a later K chunk)
};

// Widest aligned store of D's rows: 2 = 32 bytes, 1 = 16, 0 = single floats.
__host__ __device__ inline int store_width(const void *D, long long ldd) {
    return (ldd & 7) == 0 && ((uintptr_t)D & 31) == 0   ? 2
           : (ldd & 3) == 0 && ((uintptr_t)D & 15) == 0 ? 1
                                                        : 0;
}

// Eight consecutive floats to a 32-byte aligned address: a thread's row is its
// own in the epilogues, so a whole 32-byte sector goes out at once (with eight
// epilogue warps, 1920x1024x1024 split FP16 23.2 -> 21.5 us, 3840x2160x16384
// BF16 329 -> 317 against 16-byte stores and four).
__device__ __forceinline__ void store8(float *p, const float *v) {
    asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p), "f"(v[0]),
                 "f"(v[1]), "f"(v[2]), "f"(v[3]), "f"(v[4]), "f"(v[5]), "f"(v[6]), "f"(v[7])
                 : "memory");
}

// Rows that no vector store can take (ldd not a multiple of 4, or D not
// 16-byte aligned): a warp's 32 rows x 16 columns go through its own piece of
// shared memory, and each store covers 16 consecutive columns of two rows.
// (One float per lane and row touched 32 sectors a store: the split FP16 GEMM of
// 1366x768x777 took 27 us, 21 this way.)
constexpr int EPI_COLS = 16, EPI_LD = EPI_COLS + 1;
constexpr int EPI_WARP_FLOATS = 32 * EPI_LD;  // shared memory per epilogue warp

// v: the lane's row (row0 + lane) at columns col .. col + 15; D(row0, 0) at
// d0.  The whole warp calls it.
__device__ __forceinline__ void epilogue_store_odd(float *stage, const float *v, float *d0,
                                                   long long ldd, int rows, int col, int ncols,
                                                   bool accumulate, int lane) {
#pragma unroll
    for (int i = 0; i < EPI_COLS; ++i) stage[lane * EPI_LD + i] = v[i];
    __syncwarp();
    const int c = lane & 15, r0 = lane & 16;
    if (col + c < ncols) {
        float *d = d0 + col + c;
#pragma unroll
        for (int r = 0; r < 16; ++r)
            if (r0 + r < rows) {
                float *p = d + (long long)(r0 + r) * ldd;
                const float x = stage[(r0 + r) * EPI_LD + c];
                *p = accumulate ? *p + x : x;
            }
    }
    __syncwarp();
}

// Store CH consecutive FP32 values of one output row (row < M checked by the
// caller; col a multiple of 8), clipped to N columns; with g.accumulate the
// row's current values are added first (FP32, round to nearest).
template <int CH>
__device__ __forceinline__ void epilogue_store_row(float *drow, int col, float (&v)[CH],
                                                   const GemmArgs &g, int vec) {
    if (vec == 2 && !g.accumulate && col + CH <= g.N) {
#pragma unroll
        for (int i = 0; i < CH; i += 8) store8(drow + col + i, v + i);
        return;
    }
    if (vec && col + CH <= g.N) {
        if (g.accumulate) {
            // all of the chunk's loads before any of its stores: one memory
            // latency per chunk instead of one per vector
            float4 d[CH / 4];
#pragma unroll
            for (int i = 0; i < CH; i += 4)
                d[i / 4] = *reinterpret_cast<const float4 *>(drow + col + i);
#pragma unroll
            for (int i = 0; i < CH; i += 4) {
                d[i / 4].x += v[i];
                d[i / 4].y += v[i + 1];
                d[i / 4].z += v[i + 2];
                d[i / 4].w += v[i + 3];
            }
#pragma unroll
            for (int i = 0; i < CH; i += 4)
                *reinterpret_cast<float4 *>(drow + col + i) = d[i / 4];
            return;
        }
#pragma unroll
        for (int i = 0; i < CH; i += 4)
            *reinterpret_cast<float4 *>(drow + col + i) =
                make_float4(v[i], v[i + 1], v[i + 2], v[i + 3]);
    } else {
#pragma unroll
        for (int i = 0; i < CH; ++i)
            if (col + i < g.N) drow[col + i] = g.accumulate ? drow[col + i] + v[i] : v[i];
    }
}

}  // namespace cgh
