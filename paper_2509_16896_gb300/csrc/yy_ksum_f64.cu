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
// rows' combinations are taken side by side by eight lanes.  Where most pairs count, the form
// is bound by the float64 pipe as the general one is: three operations per coordinate and the
// exponentials.  Measured, N = 2, us (general form -> this one): r = 2, n = 2048, box 8 wide 1151
// -> 85; every pair in reach (box 0.04 wide): r = 2 1103 -> 493, r = 16 1100 -> 851, r = 31 1518
// -> 1271, r = 47 1934 -> 1722, r = 64 2352 -> 2195; a restart's weights: r = 16 1102 -> 203, r = 64
// 2375 -> 585.
#include "yy_combine.cuh"

namespace yy {

namespace {

constexpr int kRows = 8;          // target rows (warps) per block
constexpr int kMaxDim = 64;
constexpr int kTileMax = 1024;    // sources of one tile, at most
constexpr size_t kTileBytes = 100 * 1024;   // of one tile, at most: two blocks per SM

// A tile holds each source's coordinates as doubles and as floats (converting them for every
// pair costs the float64 pipe two thirds of the pair's own operations; r = 64, every pair kept, n =
// 2048: 3.4 ms so), in rows of an odd length (lanes take consecutive sources: no bank conflicts; rows
// of r + 1 words made odd r up to 32-way, 4.9 ms at r = 63), its log-weight and its
// place in each row's queue.
__host__ __device__ __forceinline__ int tile_row(int r) { return r | 1; }
__host__ __device__ __forceinline__ size_t source_bytes(int r) {
    return (size_t)tile_row(r) * (sizeof(double) + sizeof(float)) + sizeof(float) + kRows * sizeof(unsigned short);
}
__host__ __device__ __forceinline__ int tile_sources(int r, long long n) {
    const long long fit = (long long)(kTileBytes / source_bytes(r)) / 32 * 32, all = (n + 31) / 32 * 32;
    return (int)(fit < all ? (fit < kTileMax ? fit : kTileMax) : (all < kTileMax ? all : kTileMax));
}

// A float32 score of at most 64 coordinates is off by less than kErr times the magnitudes that
// enter it (two chains of 64 FMAs, 3.9e-6, and the roundings of the operands).
constexpr float kErr = 1e-5f;
constexpr float kMaxErr = 100.0f;  // up to here a float32 bound serves as the sums' reference

template <int N>
__global__ void __launch_bounds__(32 * kRows, 2)
    k_ksum_f64(const __grid_constant__ Consts<double> k, const __grid_constant__ Bufs<double> b) {
    extern __shared__ __align__(16) char f64_smem[];
    __shared__ double ud[kRows][kMaxDim], fd[kRows][kMaxDim];   // the rows' coordinates and drifts
    __shared__ float uf[kRows][kMaxDim], ff[kRows][kMaxDim];
    __shared__ double smx[kRows][N], ssm[kRows][N];
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const int r = k.r, rs = tile_row(r);
    const int TS = tile_sources(r, k.n);
    double* const tud = reinterpret_cast<double*>(f64_smem);                 // [TS][rs]
    float* const tuf = reinterpret_cast<float*>(tud + (size_t)TS * rs);      // [TS][rs]
    float* const lsf = tuf + (size_t)TS * rs;                                // [TS] (float), -inf: not live
    unsigned short* const queue = reinterpret_cast<unsigned short*>(lsf + TS) + w * TS;
    const long long i = k.row0 + (long long)blockIdx.x * kRows + w;
    const bool target = i < k.row1 && i < k.n && !b.mask[i];
    double rowc[N], sm[N], ref[N];   // sums of e^(score - ref)
    float top[N];                    // lower bounds of the row's largest score
    const double nf = target ? b.nf[i] : 0.0;
    if (target)
        for (int d = lane; d < r; d += 32) {
            uf[w][d] = b.u[(size_t)i * k.r_pad + d];
            ud[w][d] = (double)uf[w][d];
            fd[w][d] = b.f[(size_t)i * k.r_pad + d];
            ff[w][d] = (float)fd[w][d];
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
    const int ls0 = tid / r, ld0 = tid % r, ls1 = 32 * kRows / r, ld1 = 32 * kRows % r;
    for (long long s0 = 0; s0 < k.n; s0 += TS) {
        __syncthreads();
        const int ts = (int)min((long long)TS, k.n - s0);
        for (int s = ls0, d = ld0; s < ts;) {   // element tid, tid + 256, ... of the tile
            const float v = b.u[(size_t)(s0 + s) * k.r_pad + d];
            tuf[s * rs + d] = v;
            tud[s * rs + d] = (double)v;
            s += ls1;
            d += ld1;
            if (d >= r) { d -= r; ++s; }
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
            const float* p = tuf + s * rs;
            float s1 = 0.f, s2 = 0.f, a2 = 0.f;
#pragma unroll 4
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
            if (keep) queue[nq + __popc(bal & ((1u << lane) - 1u))] = (unsigned short)s;
            nq += __popc(bal);
        }
        __syncwarp();
        // 3. their terms, in float64
        auto scores64 = [&](int q, double (&sc)[N]) {
            const int s = q < nq ? queue[q] : 0;
            const double* p = tud + s * rs;
            double s1 = 0.0, s2 = 0.0;
#pragma unroll 4
            for (int d = 0; d < r; ++d) {
                const double dl = ud[w][d] - p[d];
                s1 = fma(dl, dl, s1);
                s2 = fma(dl, fd[w][d], s2);
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

// Up to kMaxDim coordinates this form is the faster one whatever the weights (figures above);
// above, the rows' copies in shared memory would have to grow and nothing has been measured.
bool ksum_f64_fits(const Consts<double>& k) { return k.r <= kMaxDim && k.noise != YY_NOISE_DIAG; }

// Opts the kernel into its shared memory on the current device (at creation, so that no
// attribute call happens during stream capture).
cudaError_t prepare_ksum_f64() {
    const auto a = cudaFuncAttributeMaxDynamicSharedMemorySize;
    cudaError_t e = cudaFuncSetAttribute(k_ksum_f64<1>, a, (int)kTileBytes);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_ksum_f64<2>, a, (int)kTileBytes);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_ksum_f64<3>, a, (int)kTileBytes);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_ksum_f64<4>, a, (int)kTileBytes);
    return e;
}

cudaError_t launch_ksum_f64(const Consts<double>& k, const Bufs<double>& b, cudaStream_t s, int* launches) {
    const long long rows = k.row1 - k.row0;
    if (rows <= 0) return cudaSuccess;
    const unsigned grid = (unsigned)((rows + kRows - 1) / kRows);
    const size_t sm = (size_t)tile_sources(k.r, k.n) * source_bytes(k.r);
    switch (k.N) {
        case 1: k_ksum_f64<1><<<grid, 32 * kRows, sm, s>>>(k, b); break;
        case 2: k_ksum_f64<2><<<grid, 32 * kRows, sm, s>>>(k, b); break;
        case 3: k_ksum_f64<3><<<grid, 32 * kRows, sm, s>>>(k, b); break;
        case 4: k_ksum_f64<4><<<grid, 32 * kRows, sm, s>>>(k, b); break;
        default: return cudaErrorInvalidValue;
    }
    if (launches) *launches += 1;
    return cudaGetLastError();
}

}  // namespace yy
