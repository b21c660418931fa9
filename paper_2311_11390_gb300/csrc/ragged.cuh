// Rows whose windows start at any 4-byte boundary (T not a multiple of 16, or an unaligned base).
//
// Both warp-per-row kernels are bound by issue slots, so what counts is instructions.  Where rows stay
// 16-byte aligned (T a multiple of 4) a window is one 1-D bulk copy, read and written by 16 bytes.
// Elsewhere the lanes' E single reads stay: a copy of the granules covering the window, shifted in
// registers, took more instructions and measured the same or slower (forward 296 -> 312 us, backward
// without dL/dI 414 -> 467 us at 32768 rows of 4001 steps).  Single writes do not: E stores of 32
// sectors each against two of 16 bytes, shifted to the boundary with the next lane's first floats.
// 32768 rows: forward with both traces 908 -> 348 us at 4004 steps and 914 -> 455 us at 4001, backward
// 502 -> 415 us at 4004 and 505 -> 491 us at 4001.
#pragma once

#include "common.cuh"

namespace alif {
namespace ragged {

// This lane's E floats (steps t0 ..) of the window at src, steps past cnt left 0.
template <int E>
__device__ __forceinline__ void read_direct(const float *src, int t0, int cnt, float (&x)[E]) {
#pragma unroll
    for (int k = 0; k < E; ++k) x[k] = t0 + k < cnt ? __ldg(src + t0 + k) : 0.0f;
}

// Stores steps 0 .. cnt - 1 of a window at dst, this lane holding y = steps t0 .. t0 + E - 1.  Called by
// the whole warp; cnt <= 32 E.
template <int E>
__device__ __forceinline__ void store(float *dst, int t0, int cnt, const float (&y)[E]) {
    const int h = (4 - ((int)((uintptr_t)dst >> 2) & 3)) & 3;  // steps before the first 16-byte boundary
    float z[E];                                                // steps t0 + h .. t0 + h + E - 1
    if (h == 0) {
#pragma unroll
        for (int k = 0; k < E; ++k) z[k] = y[k];
    } else {
        float n[E + 3], u[E + 2];
#pragma unroll
        for (int k = 0; k < E; ++k) n[k] = y[k];
#pragma unroll
        for (int k = 0; k < 3; ++k) n[E + k] = __shfl_down_sync(FULL, y[k], 1);
#pragma unroll
        for (int k = 0; k < E + 2; ++k) u[k] = (h & 1) ? n[k + 1] : n[k];
#pragma unroll
        for (int k = 0; k < E; ++k) z[k] = (h & 2) ? u[k + 2] : u[k];
        if (t0 == 0) {
#pragma unroll
            for (int k = 0; k < 3; ++k)
                if (k < h && k < cnt) dst[k] = y[k];
        }
    }
#pragma unroll
    for (int q = 0; q < E / 4; ++q) {
        const int t = t0 + h + 4 * q;
        if (t + 4 <= cnt) {
            *reinterpret_cast<float4 *>(dst + t) = make_float4(z[4 * q], z[4 * q + 1], z[4 * q + 2], z[4 * q + 3]);
        } else {
#pragma unroll
            for (int k = 0; k < 4; ++k)
                if (t + k < cnt) dst[t + k] = z[4 * q + k];
        }
    }
}

}  // namespace ragged
}  // namespace alif
