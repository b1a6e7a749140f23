// Float64 prediction of filters with short rows (r <= 64): float32 picks the pairs, float64
// evaluates them.
//
// What bounds the form is the float64 pipe: two lane operations per clock and SM (0.62 T/s
// measured), and an exponential is about twenty of them.  Most kernel terms of a node are zero
// next to its largest, so each pair is first scored in float32 (the coordinates are float32
// numbers; 64 times the rate) and only pairs that can carry more than e^-(ln n + 40) of their
// row's largest term are evaluated in float64: everything dropped from a row adds up to less
// than e^-40, a thirtieth of a unit in the last place.  Both sides of the comparison carry the
// bound of their float32 rounding (kErr): a pair's score its upper, the row's largest its lower.
//
// One warp per target row.  A block's eight warps share tiles of sources staged in shared
// memory; a warp scores the tile in float32 twice, for the largest score (the reference of the
// selection, and of the log-sum-exp: close below the maximum is all it has to be) and for the
// survivors, which it queues and then evaluates 32 at a time, one per lane, with one exponential
// per scale and no comparison in float64.  Where a survivor's magnitudes are so large that its
// float32 score is off by more than kMaxErr nats (weights spread over 1e8 nats, a step far
// shorter than the box is wide), e^(score - reference) could overflow, and the tile's
// reference is the largest of the survivors' float64 scores, evaluated once more.  The lanes' sums are added at the end, and the eight
// rows' combinations are taken side by side by eight lanes.  Measured at r = 2, n = 1024, N = 2
// (box 8 wide): every pair in float64, coordinates padded to 16: 370 us; selection against
// the row's own term: 62 us (a row far from the posterior's peak keeps a third of the
// sources); against the largest score: 33 us.
#include <algorithm>

#include "yy_combine.cuh"

namespace yy {

namespace {

constexpr int kRows = 8;          // target rows (warps) per block
constexpr int kTileFloats = 4096; // coordinates of one source tile in shared memory, at most
constexpr int kTileMax = 1024;    // sources of one tile, at most
// A float32 score of at most 64 coordinates is off by less than kErr times the magnitudes that
// enter it (two chains of 64 FMAs, 3.9e-6, and the roundings of the operands).
constexpr float kErr = 1e-5f;
constexpr float kMaxErr = 100.0f;  // up to here a float32 bound serves as the sums' reference

__device__ __forceinline__ int tile_sources(int r) { return min(kTileMax, kTileFloats / (r + 1) / 32 * 32); }

template <int N>
__global__ void __launch_bounds__(32 * kRows, 1)
    k_ksum_f64(const __grid_constant__ Consts<double> k, const __grid_constant__ Bufs<double> b) {
    __shared__ float us[kTileFloats];               // [source][r + 1]
    __shared__ float lsf[kTileMax];                 // log-weights (float), -inf: not live
    __shared__ unsigned short queue[kRows][kTileMax];
    __shared__ float uf[kRows][64], ff[kRows][64];
    __shared__ double smx[kRows][N], ssm[kRows][N];
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const int r = k.r, rs = r + 1;
    const int TS = tile_sources(r);
    const long long i = k.row0 + (long long)blockIdx.x * kRows + w;
    const bool target = i < k.row1 && i < k.n && !b.mask[i];
    const double* fi = b.f + (size_t)i * k.r_pad;
    double rowc[N], sm[N], ref[N];   // sums of e^(score - ref)
    float top[N];                    // lower bounds of the row's largest score
    const double nf = target ? b.nf[i] : 0.0;
    if (target)
        for (int d = lane; d < r; d += 32) {
            uf[w][d] = b.u[(size_t)i * k.r_pad + d];
            ff[w][d] = (float)fi[d];
        }
    __syncwarp();
    const float gap = logf((float)k.n) + 41.0f;
    float rowf[N], i2t[N];
#pragma unroll
    for (int j = 0; j < N; ++j) {
        rowc[j] = -0.5 * k.tau[j] * nf;
        rowf[j] = (float)rowc[j];
        i2t[j] = (float)k.inv2tau[j];
        sm[j] = 0.0;
        ref[j] = -INFINITY;
        top[j] = -INFINITY;
    }
    for (long long s0 = 0; s0 < k.n; s0 += TS) {
        __syncthreads();
        const int ts = (int)min((long long)TS, k.n - s0);
        for (int e = tid; e < ts * r; e += 32 * kRows) {
            const int s = e / r, d = e - s * r;
            us[s * rs + d] = b.u[(size_t)(s0 + s) * k.r_pad + d];
        }
        for (int s = tid; s < ts; s += 32 * kRows) {
            // -inf in float only where the double is (a finite weight below float's range has no
            // neighbour it could count next to, and is kept as float's lowest)
            const double v = b.mask[s0 + s] ? -INFINITY : b.logw[s0 + s];
            lsf[s] = (v == -INFINITY) ? -INFINITY : fmaxf((float)v, -3.0e38f);
            if (v != v) lsf[s] = NAN;
        }
        __syncthreads();
        if (!target) continue;
        // float32 scores of source s of the tile; *err: a bound of their rounding
        auto scores = [&](int s, float ls, float (&sc)[N], float* err) {
            const float* p = us + s * rs;
            float s1 = 0.f, s2 = 0.f, a2 = 0.f;
            for (int d = 0; d < r; ++d) {
                const float dl = uf[w][d] - p[d], f = ff[w][d];
                s1 = fmaf(dl, dl, s1);
                s2 = fmaf(dl, f, s2);
                a2 = fmaf(fabsf(dl), fabsf(f), a2);
            }
            float m = a2 + fabsf(ls);
#pragma unroll
            for (int j = 0; j < N; ++j) {
                sc[j] = fmaf(-s1, i2t[j], s2) + (rowf[j] + ls);
                m = fmaxf(m, fmaf(s1, i2t[j], a2 + fabsf(ls) + fabsf(rowf[j])));
            }
            *err = kErr * m;
        };
        // 1. a lower bound of the tile's largest score per scale (an undefined one bounds nothing)
        float fm[N];
#pragma unroll
        for (int j = 0; j < N; ++j) fm[j] = -INFINITY;
        for (int s = lane; s < ts; s += 32) {
            const float ls = lsf[s];
            if (ls == -INFINITY) continue;
            float sc[N], err;
            scores(s, ls, sc, &err);
#pragma unroll
            for (int j = 0; j < N; ++j) fm[j] = fmaxf(fm[j], sc[j] - err);
        }
#pragma unroll
        for (int j = 0; j < N; ++j) {
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) fm[j] = fmaxf(fm[j], __shfl_xor_sync(0xffffffffu, fm[j], o));
            top[j] = fmaxf(top[j], fm[j]);
        }
        // 2. the sources that can count next to it (an undefined score is kept)
        int nq = 0;
        bool exact_ref = false;
        for (int c = 0; c < ts; c += 32) {
            const int s = c + lane;
            bool keep = false;
            const float ls = s < ts ? lsf[s] : -INFINITY;
            if (ls != -INFINITY) {
                float sc[N], err;
                scores(s, ls, sc, &err);
#pragma unroll
                for (int j = 0; j < N; ++j) keep |= !(sc[j] + err < top[j] - gap);
                exact_ref |= keep && !(err < kMaxErr);
            }
            const uint32_t bal = __ballot_sync(0xffffffffu, keep);
            if (keep) queue[w][nq + __popc(bal & ((1u << lane) - 1u))] = (unsigned short)s;
            nq += __popc(bal);
        }
        __syncwarp();
        // 3. their terms, in float64
        auto scores64 = [&](int q, double (&sc)[N]) {
            const int s = q < nq ? queue[w][q] : 0;
            const float* p = us + s * rs;
            double s1 = 0.0, s2 = 0.0;
            for (int d = 0; d < r; ++d) {
                const double dl = (double)uf[w][d] - (double)p[d];
                s1 = fma(dl, dl, s1);
                s2 = fma(dl, fi[d], s2);
            }
            const double ls = q < nq ? b.logw[s0 + s] : -INFINITY;
#pragma unroll
            for (int j = 0; j < N; ++j) sc[j] = fma(-s1, k.inv2tau[j], s2) + (rowc[j] + ls);
        };
        double tref[N];   // the tile's reference
#pragma unroll
        for (int j = 0; j < N; ++j) tref[j] = (double)fm[j];
        if (__any_sync(0xffffffffu, exact_ref)) {
#pragma unroll
            for (int j = 0; j < N; ++j) tref[j] = -INFINITY;
            for (int q0 = 0; q0 < nq; q0 += 32) {
                double sc[N];
                scores64(q0 + lane, sc);
#pragma unroll
                for (int j = 0; j < N; ++j) tref[j] = fmax(tref[j], sc[j]);
            }
#pragma unroll
            for (int j = 0; j < N; ++j)
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) tref[j] = fmax(tref[j], __shfl_xor_sync(0xffffffffu, tref[j], o));
        }
#pragma unroll
        for (int j = 0; j < N; ++j)
            if (tref[j] > ref[j]) {
                if (ref[j] != -INFINITY) sm[j] *= exp(ref[j] - tref[j]);
                ref[j] = tref[j];
            }
        for (int q0 = 0; q0 < nq; q0 += 32) {
            const bool on = q0 + lane < nq;
            double e[N];
            scores64(q0 + lane, e);
#pragma unroll
            for (int j = 0; j < N; ++j) e[j] = exp(e[j] - ref[j]);
#pragma unroll
            for (int j = 0; j < N; ++j) sm[j] += on && ref[j] != -INFINITY ? e[j] : 0.0;
        }
        __syncwarp();
    }
    if (target) {
#pragma unroll
        for (int j = 0; j < N; ++j) {
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) sm[j] += __shfl_xor_sync(0xffffffffu, sm[j], o);
            if (lane == 0) { smx[w][j] = ref[j]; ssm[w][j] = sm[j]; }
        }
    }
    __syncthreads();
    if (tid < kRows) {
        const long long ii = k.row0 + (long long)blockIdx.x * kRows + tid;
        if (ii < k.row1 && ii < k.n) {
            if (b.mask[ii]) {
                b.logw_pred[ii] = -INFINITY;
            } else {
                double mx[N];
#pragma unroll
                for (int j = 0; j < N; ++j) { mx[j] = smx[tid][j]; sm[j] = ssm[tid][j]; }
                b.logw_pred[ii] = combine_scales<double, N>(k, mx, sm, b.divf[ii], b.logw[ii], b.stats->c_ref,
                                                            &b.stats->clamps);
            }
        }
    }
}

}  // namespace

bool ksum_f64_fits(const Consts<double>& k) { return k.r <= 64 && k.noise != YY_NOISE_DIAG; }

cudaError_t launch_ksum_f64(const Consts<double>& k, const Bufs<double>& b, cudaStream_t s, int* launches) {
    const long long rows = k.row1 - k.row0;
    if (rows <= 0) return cudaSuccess;
    const unsigned grid = (unsigned)((rows + kRows - 1) / kRows);
    switch (k.N) {
        case 1: k_ksum_f64<1><<<grid, 32 * kRows, 0, s>>>(k, b); break;
        case 2: k_ksum_f64<2><<<grid, 32 * kRows, 0, s>>>(k, b); break;
        case 3: k_ksum_f64<3><<<grid, 32 * kRows, 0, s>>>(k, b); break;
        case 4: k_ksum_f64<4><<<grid, 32 * kRows, 0, s>>>(k, b); break;
        default: return cudaErrorInvalidValue;
    }
    if (launches) *launches += 1;
    return cudaGetLastError();
}

}  // namespace yy
