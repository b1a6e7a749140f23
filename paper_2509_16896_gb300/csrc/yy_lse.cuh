// Log-sum-exp reductions shared by the preparation and update passes.
#pragma once

#include "yy_internal.cuh"

namespace yy {

// (max, sum) of up to 8 warps' log-sum-exp states, by one warp: the rescale factors side by side
// in 8 lanes (a float64 exponential takes about 1100 clocks here, one after the other eight
// times that); lane 0 has the result.
__device__ __forceinline__ void lse_merge8(double m, double s, double& M, double& S) {
    const int lane = threadIdx.x & 31;
    if (lane >= 8) m = -INFINITY;
    float mf = (m == -INFINITY) ? -INFINITY : __double2float_ru(m);   // any bound near the largest serves ...
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) mf = fmaxf(mf, __shfl_xor_sync(0xffffffffu, mf, o));
    mf = __shfl_sync(0xffffffffu, mf, 0);
    M = (double)mf;   // ... as the maximum the sum is taken relative to
    S = (m == -INFINITY) ? 0.0 : s * exp(m - M);
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) S += __shfl_xor_sync(0xffffffffu, S, o);
}

}  // namespace yy
