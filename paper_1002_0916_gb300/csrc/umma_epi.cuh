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

// Store CH consecutive FP32 values of one output row (row < M checked by the
// caller), clipped to N columns; with g.accumulate the row's current values
// are added first (FP32, round to nearest).
template <int CH>
__device__ __forceinline__ void epilogue_store_row(float *drow, int col, float (&v)[CH],
                                                   const GemmArgs &g, bool vec) {
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
