// Exact sums of one pair by one thread.
#pragma once

#include "yy_internal.cuh"

namespace yy {

// S1 and S2 of one pair over all coordinates in increasing order, loads a stage ahead.
__device__ __forceinline__ void pair_sums_thread(const float* __restrict__ ut, const float* __restrict__ ft,
                                                 const float* __restrict__ us, int r_pad, float& s1, float& s2) {
    constexpr int Q = 4;   // float4 per stage and operand
    float4 a[Q], f[Q], c[Q];
    auto get = [&](int d) {
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            a[q] = *reinterpret_cast<const float4*>(ut + d + 4 * q);
            f[q] = *reinterpret_cast<const float4*>(ft + d + 4 * q);
            c[q] = *reinterpret_cast<const float4*>(us + d + 4 * q);
        }
    };
    s1 = s2 = 0.f;
    get(0);
    for (int d = 0; d < r_pad; d += 4 * Q) {   // padded coordinates are zero in all three
        float4 x[Q], y[Q], z[Q];
#pragma unroll
        for (int q = 0; q < Q; ++q) { x[q] = a[q]; y[q] = f[q]; z[q] = c[q]; }
        if (d + 4 * Q < r_pad) get(d + 4 * Q);
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            const float xs[4] = {x[q].x, x[q].y, x[q].z, x[q].w}, ys[4] = {y[q].x, y[q].y, y[q].z, y[q].w};
            const float zs[4] = {z[q].x, z[q].y, z[q].z, z[q].w};
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const float dl = xs[e] - zs[e];
                s1 = fmaf(dl, dl, s1);
                s2 = fmaf(dl, ys[e], s2);
            }
        }
    }
}

// The same over the r coordinates in stages of 16 whose loads are not ahead of the stage before: for a
// kernel short of registers (48 words at a time).
__device__ __forceinline__ void pair_sums_staged(const float* __restrict__ ut, const float* __restrict__ ft,
                                                 const float* __restrict__ us, int r, float& s1, float& s2) {
    constexpr int Q = 4;
    s1 = s2 = 0.f;
#pragma unroll 1
    for (int d = 0; d < r; d += 4 * Q) {   // padded coordinates are zero in all three
        float4 x[Q], y[Q], z[Q];
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            x[q] = *reinterpret_cast<const float4*>(ut + d + 4 * q);
            y[q] = *reinterpret_cast<const float4*>(ft + d + 4 * q);
            z[q] = *reinterpret_cast<const float4*>(us + d + 4 * q);
        }
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            const float xs[4] = {x[q].x, x[q].y, x[q].z, x[q].w}, ys[4] = {y[q].x, y[q].y, y[q].z, y[q].w};
            const float zs[4] = {z[q].x, z[q].y, z[q].z, z[q].w};
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const float dl = xs[e] - zs[e];
                s1 = fmaf(dl, dl, s1);
                s2 = fmaf(dl, ys[e], s2);
            }
        }
    }
}

}  // namespace yy
