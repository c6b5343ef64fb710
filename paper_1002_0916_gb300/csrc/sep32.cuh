// sep32.cuh -- pieces shared by the FP32-accurate tensor-core products:
// sep32.cu (the product kernel and the forward) and adj32.cu (the adjoint).
// Internal to libcgh.
#pragma once

#include <cuda_fp16.h>

#include "common.cuh"
#include "cos_poly.h"

namespace cgh {

// R entries are scaled by 2^S32_EXP, a block's L entries to below it.
constexpr int S32_EXP = 14;
constexpr float S32_R_SCALE = 16384.0f;
// The adjoint's products are taken out of both factors' scales, 2^S32_EXP and
// 2^(S32_EXP - 1), as they are added up: sums in units of max |G| rounded down
// to a power of two, whatever its size.
constexpr float S32_ADJ_FACTOR = 1.0f / 134217728.0f;  // 2^-27

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

struct Sep32Operands {
    const __half *A_hi, *A_lo, *B_hi, *B_lo;
    long long lda, ldb;
};

// One product of the adjoint (adj32.cu): D = T' G over one image axis, its
// columns the coordinates u of the other axis.
struct Adj32Prod {
    int units;    // row tiles x column tiles x slices
    int tiles_n;  // column tiles
    int S;        // K slices
    int KB;       // K blocks of 64
    int axis;     // the columns' axis: 0 x, 1 y
    float *part;  // [(slice, column tile, half)][3][npad]
};

struct Adj32Args {
    Adj32Prod p[2];
    int n;                // points
    int npad;             // partial-sum stride (points)
    int tiles_m;          // row tiles of 256 (128 points)
    const PointRec *rec;  // n
    const float *points;  // n x 2
};

// How the adjoint's two products are tiled for n points: tile width and the
// K slices of each.
struct Adj32Plan {
    int bn, S[2];
};
Adj32Plan adj32_plan(int n, int Nx, int Ny, int sms);
// Both products in one launch: op[0], K[0] and ga.p[0] the longer K first;
// N[i] columns.
cudaError_t launch_adj32(int bn, const Sep32Operands (&op)[2], const int (&N)[2],
                         const int (&K)[2], const Adj32Args &ga, unsigned *status,
                         cudaStream_t s);

}  // namespace cgh
