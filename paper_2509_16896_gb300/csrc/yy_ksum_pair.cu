// Plain float32 prediction (and the materialised operator's build) on the pair loop of
// yy_pair.cuh: single filters, with and without noise coefficients.
//
// For every target i and scale j (tau_j = dt / 2^(j-1)), in units relative to c_ref:
//   L_j(i) - c_ref = (C_j - c_ref) - tau_j div f(x_i)
//                    + LSE_s [ -|u_i - tau_j f_i - u_s|^2 / (2 tau_j) + ell_s ],
//   C_j = -(r/2) log(2 pi tau_j) + log w_q,
// which is log sum_s K_{tau_j}(x_i, x_s) w_q e^{ell_s} for the first-order kernel of
// eq. kernel ("First-Order Kernel Construction") after completing the square:
//   -|x-y|^2/(2 tau) - (y-x).f(x) - tau(div f + |f|^2/2) = -|x - tau f(x) - y|^2/(2 tau) - tau div f,
//   |u_i - tau f_i - u_s|^2 = S1 - 2 tau S2 + tau^2 |f_i|^2,  S1 = |D|^2, S2 = D.f_i, D = u_i - u_s,
// so one pass over the coordinates serves all N scales.  The N terms are combined with the
// identity term of eq. general_kernel by a signed log-sum-exp; a non-positive total gives
// -inf (counted).  Noise coefficients (diagonal): S1 and S2 take the target's metric a(x_i)^+,
// |f_i|^2 likewise, and -1/2 log det_+ a(x_i) is added in the combination.
#include <algorithm>

#include "yy_pair.cuh"

namespace yy {

namespace {

using namespace pair;

template <int N, bool NOISE>
__global__ void __launch_bounds__(THREADS, BLOCKS_PER_SM)
    k_pair(const __grid_constant__ Consts<float> k, const __grid_constant__ Bufs<float> b, int nsplit) {
    extern __shared__ __align__(16) float pair_smem[];
    block<N, NOISE, false>(k, b, k.row0 + (long long)(blockIdx.x / nsplit) * BM, (int)(blockIdx.x % nsplit), nsplit,
                           pair_smem);
}

// The same with terms that cannot count left out (see block); flags: per target block of 32, a
// bit per tile of 128 sources (fwords words per block), or nullptr.
template <int N>
__global__ void __launch_bounds__(THREADS, BLOCKS_PER_SM)
    k_pair_skip(const __grid_constant__ Consts<float> k, const __grid_constant__ Bufs<float> b, int nsplit,
                const __grid_constant__ SkipTest skip, const uint32_t* __restrict__ flags, int fwords) {
    extern __shared__ __align__(16) float pair_smem[];
    const long long i0 = k.row0 + (long long)(blockIdx.x / nsplit) * BM;
    block<N, false, false, true>(k, b, i0, (int)(blockIdx.x % nsplit), nsplit, pair_smem, &skip,
                                 flags ? flags + (size_t)(i0 / BM) * fwords : nullptr);
}

// Lower bounds of every target row's largest score, per scale: the larger of the row's own
// term (u_i - u_i = 0) and its exact score against the live source of the largest log-weight.
// The second is taken down by what its rounding and the pair loop's, which adds up in
// another order, can differ by (see yy_pair.cuh).  Each block finds that source for itself (n words from L2); then one warp per row.
template <int N>
__global__ void __launch_bounds__(256) k_pair_ref(const __grid_constant__ Consts<float> k,
                                                  const __grid_constant__ Bufs<float> b) {
    __shared__ float sm[8];
    __shared__ long long si[8];
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    float m = -INFINITY;
    long long top = -1;
    for (long long s = threadIdx.x; s < k.n; s += blockDim.x) {
        const float v = b.mask[s] ? -INFINITY : b.logw[s];
        if (v > m) { m = v; top = s; }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const float m2 = __shfl_xor_sync(0xffffffffu, m, o);
        const long long t2 = __shfl_xor_sync(0xffffffffu, top, o);
        if (m2 > m || (m2 == m && t2 > top)) { m = m2; top = t2; }
    }
    if (lane == 0) { sm[wib] = m; si[wib] = top; }
    __syncthreads();
    for (int w = 0; w < 8; ++w)
        if (sm[w] > m || (sm[w] == m && si[w] > top)) { m = sm[w]; top = si[w]; }
    const float* us = b.u + (size_t)max(top, 0ll) * k.r_pad;
    for (long long i = k.row0 + (long long)blockIdx.x * 8 + wib; i < k.row1; i += (long long)gridDim.x * 8) {
        const float* ui = b.u + (size_t)i * k.r_pad;
        const float* fi = b.f + (size_t)i * k.r_pad;
        float s1 = 0.f, s2 = 0.f;
        for (int d = lane; d < k.r; d += 32) {
            const float dl = ui[d] - us[d];
            s1 = fmaf(dl, dl, s1);
            s2 = fmaf(dl, fi[d], s2);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            s1 += __shfl_xor_sync(0xffffffffu, s1, o);
            s2 += __shfl_xor_sync(0xffffffffu, s2, o);
        }
        if (lane == 0) {
            const float nf = b.nf[i], li = b.logw[i], gam = skip_gamma(k.r);
#pragma unroll
            for (int j = 0; j < N; ++j) {
                const float rc = __fmul_rn(-0.5f * k.tau[j], nf);   // rounded as in the pair loop
                const float err = gam * (5.0f * s1 * k.inv2tau[j] - 4.0f * rc) + 1e-6f * fabsf(m);
                b.pair_ref[(size_t)i * kMaxScales + j] = fmaxf(rc + li, fmaf(-s1, k.inv2tau[j], s2) + (rc + m) - err);
            }
        }
    }
}

template <int N, bool NOISE>
__global__ void __launch_bounds__(256) k_pair_merge(const __grid_constant__ Consts<float> k,
                                                    const __grid_constant__ Bufs<float> b, int nsplit) {
    const long long i = k.row0 + (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= k.row1 || i >= k.n) return;
    merge_row<N, NOISE>(k, b, i, nsplit);
}

// Materialised operator: built only when the node set moved since the last build (the flag
// is set by restarts and state changes, cleared by the apply), unless forced.
template <int N>
__global__ void __launch_bounds__(THREADS, BLOCKS_PER_SM)
    k_op_build(const __grid_constant__ Consts<float> k, const __grid_constant__ Bufs<float> b, int nsplit, int force) {
    if (!force && b.stats->op_stale == 0) return;
    extern __shared__ __align__(16) float pair_smem[];
    block<N, false, true>(k, b, k.row0 + (long long)(blockIdx.x / nsplit) * BM, (int)(blockIdx.x % nsplit), nsplit,
                          pair_smem);
}

// batched: block x processes item x = (member, target block)
template <int N>
__global__ void __launch_bounds__(THREADS, BLOCKS_PER_SM) kb_pair(const Traj<float>* __restrict__ tr,
                                                                  const int2* __restrict__ items) {
    extern __shared__ __align__(16) float pair_smem[];
    const int2 it = items[blockIdx.x];
    const Traj<float>& t = tr[it.x];
    block<N, false, false>(t.k, t.b, (long long)it.y * BM, 0, 1, pair_smem);
}

// The skipping form: from this many coordinates (its reference pass and masks cost about 10 us,
// and a tile is not given up before 64 coordinates: at r = 100 nothing is), up to this much
// mask.  Measured, large-scale model at r = 1000, n = 2000, N = 2, full form 545 us per prediction:
// weights of a restart 165 us (tiles given up after 192 to 256 coordinates; 300 us while the
// rows' own pairs kept their tiles), weights of an update 95 us (one heavy node; 350 us before
// thin tiles).
// With at most 512 sources a prediction waits out one stage after the other, and the reference
// pass and the tests add a quarter to it: measured at n <= 512, us, full form -> skipping, weights of a
// restart / nothing to skip: r = 128 29 -> 42 / 42, r = 200 35 -> 41 / 50, r = 300 43 -> 43 / 63, r =
// 500 59 -> 50 / 89, r = 1000 98 -> 51 / 150; so rows of 512 and more skip there.
constexpr int kSkipMinDim = 128, kSkipMinDimSmall = 512;
constexpr long long kSkipSmall = 512;
// Masks of a source range: one million sources in the plain form, which has another way (behind the
// screen kMaxMaskBytesScreen, 5 million, as all pairs of so many rows would take minutes).
constexpr size_t kMaxMaskBytes = 32768;
constexpr float kSkipGap = 110.0f;

// Source ranges per target row (at most kSimtMaxSplit, none beyond the source groups): two
// blocks of 64 targets per SM where the filter has few targets and the workspace holds the
// partial states.
int pair_splits(const Consts<float>& k, const Bufs<float>& b, long long rows) {
    if (!b.simt_part) return 1;
    const long long blocks = (rows + 63) / 64;
    long long sp = (2 * kSms + blocks - 1) / blocks;
    sp = std::min<long long>(sp, kSimtMaxSplit);
    sp = std::min<long long>(sp, k.n_pad / 64);
    return (int)std::max<long long>(sp, 1);
}

template <int N>
cudaError_t set_attr_n() {
    const auto a = cudaFuncAttributeMaxDynamicSharedMemorySize;
    cudaError_t e = cudaFuncSetAttribute(k_pair<N, false>, a, (int)smem_bytes<N, false, false>());
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_pair<N, true>, a, (int)smem_bytes<N, true, false>());
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_pair_skip<N>, a, (int)(smem_bytes<N, false, false, true>() + kMaxMaskBytesScreen));
    if (e == cudaSuccess) e = cudaFuncSetAttribute(kb_pair<N>, a, (int)smem_bytes<N, false, false>());
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_op_build<N>, a, (int)smem_bytes<N, false, true>());
    return e;
}

template <int N>
cudaError_t launch_ref_n(const Consts<float>& k, const Bufs<float>& b, cudaStream_t s) {
    const long long rows = k.row1 - k.row0;
    k_pair_ref<N><<<(unsigned)std::min<long long>((rows + 7) / 8, 2 * kSms), 256, 0, s>>>(k, b);
    return cudaGetLastError();
}

template <int N, bool NOISE>
cudaError_t merge_n(const Consts<float>& k, const Bufs<float>& b, int S, cudaStream_t s) {
    if (S > 1) k_pair_merge<N, NOISE><<<(unsigned)((k.row1 - k.row0 + 127) / 128), 128, 0, s>>>(k, b, S);
    return cudaGetLastError();
}
template <int N>
cudaError_t launch_skip_n(const Consts<float>& k, const Bufs<float>& b, int S, float gap, const uint32_t* flags,
                          int fwords, cudaStream_t s) {
    const unsigned grid = (unsigned)((k.row1 - k.row0 + BM - 1) / BM * S);
    SkipTest t{gap, skip_gamma(k.r), {}};
    for (int j = 0; j < k.N; ++j) t.i2t[j] = k.inv2tau[j] * std::max(1.0f - 5.0f * t.gam, 0.0f);
    k_pair_skip<N><<<grid, THREADS, smem_bytes<N, false, false, true>() + pair_mask_bytes(k.n, S), s>>>(k, b, S, t, flags,
                                                                                                  fwords);
    const cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? merge_n<N, false>(k, b, S, s) : e;
}
template <int N, bool NOISE>
cudaError_t launch_n(const Consts<float>& k, const Bufs<float>& b, int S, cudaStream_t s, int* l) {
    if (!NOISE && k.r >= (k.n > kSkipSmall ? kSkipMinDim : kSkipMinDimSmall) && pair_skip_fits(k, b)) {
        if (l) *l += 1;
        const cudaError_t e = launch_ref_n<N>(k, b, s);
        return e == cudaSuccess ? launch_skip_n<N>(k, b, S, kSkipGap, nullptr, 0, s) : e;
    }
    const unsigned grid = (unsigned)((k.row1 - k.row0 + BM - 1) / BM * S);
    k_pair<N, NOISE><<<grid, THREADS, smem_bytes<N, NOISE, false>(), s>>>(k, b, S);
    const cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? merge_n<N, NOISE>(k, b, S, s) : e;
}

}  // namespace

// Opts the kernels into their shared-memory sizes on the current device (at creation, so
// that no attribute call happens during stream capture).
cudaError_t prepare_pair() {
    cudaError_t e = set_attr_n<1>();
    if (e == cudaSuccess) e = set_attr_n<2>();
    if (e == cudaSuccess) e = set_attr_n<3>();
    if (e == cudaSuccess) e = set_attr_n<4>();
    return e;
}

cudaError_t launch_pair(const Consts<float>& k, const Bufs<float>& b, cudaStream_t s, int* launches) {
    const long long rows = k.row1 - k.row0;
    if (rows <= 0) return cudaSuccess;
    const int S = pair_splits(k, b, rows);
    const bool noise = k.noise == YY_NOISE_DIAG;
    if (launches) *launches += S > 1 ? 2 : 1;
    switch (k.N) {
        case 1: return noise ? launch_n<1, true>(k, b, S, s, launches) : launch_n<1, false>(k, b, S, s, launches);
        case 2: return noise ? launch_n<2, true>(k, b, S, s, launches) : launch_n<2, false>(k, b, S, s, launches);
        case 3: return noise ? launch_n<3, true>(k, b, S, s, launches) : launch_n<3, false>(k, b, S, s, launches);
        case 4: return noise ? launch_n<4, true>(k, b, S, s, launches) : launch_n<4, false>(k, b, S, s, launches);
    }
    return cudaErrorInvalidValue;
}

// The masks of a source range fit the skipping form's shared memory.
bool pair_skip_fits(const Consts<float>& k, const Bufs<float>& b) {
    return b.pair_ref && pair_mask_bytes(k.n, pair_splits(k, b, k.row1 - k.row0)) <= kMaxMaskBytes;
}

cudaError_t launch_pair_ref(const Consts<float>& k, const Bufs<float>& b, cudaStream_t s) {
    if (k.row1 <= k.row0) return cudaSuccess;
    switch (k.N) {
        case 1: return launch_ref_n<1>(k, b, s);
        case 2: return launch_ref_n<2>(k, b, s);
        case 3: return launch_ref_n<3>(k, b, s);
        case 4: return launch_ref_n<4>(k, b, s);
    }
    return cudaErrorInvalidValue;
}

cudaError_t launch_pair_flagged(const Consts<float>& k, const Bufs<float>& b, float gap, const uint32_t* flags,
                                int fwords, cudaStream_t s, int* launches) {
    const long long rows = k.row1 - k.row0;
    if (rows <= 0) return cudaSuccess;
    const int S = pair_splits(k, b, rows);
    if (launches) *launches += S > 1 ? 2 : 1;
    switch (k.N) {
        case 1: return launch_skip_n<1>(k, b, S, gap, flags, fwords, s);
        case 2: return launch_skip_n<2>(k, b, S, gap, flags, fwords, s);
        case 3: return launch_skip_n<3>(k, b, S, gap, flags, fwords, s);
        case 4: return launch_skip_n<4>(k, b, S, gap, flags, fwords, s);
    }
    return cudaErrorInvalidValue;
}

cudaError_t launch_op_build(const Consts<float>& k, const Bufs<float>& b, bool force, cudaStream_t s) {
    if (!b.op) return cudaErrorInvalidValue;
    const long long rows = k.row1 - k.row0;
    if (rows <= 0) return cudaSuccess;
    // entries are independent, so the source ranges only balance the SMs
    const int S = (int)std::max<long long>(1, std::min<long long>(8, k.n_pad / 512));
    const unsigned grid = (unsigned)((rows + BM - 1) / BM * S);
    const int f = force ? 1 : 0;
    switch (k.N) {
        case 1: k_op_build<1><<<grid, THREADS, smem_bytes<1, false, true>(), s>>>(k, b, S, f); break;
        case 2: k_op_build<2><<<grid, THREADS, smem_bytes<2, false, true>(), s>>>(k, b, S, f); break;
        case 3: k_op_build<3><<<grid, THREADS, smem_bytes<3, false, true>(), s>>>(k, b, S, f); break;
        case 4: k_op_build<4><<<grid, THREADS, smem_bytes<4, false, true>(), s>>>(k, b, S, f); break;
        default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

long long pair_batch_blocks(long long n) { return (n + BM - 1) / BM; }

cudaError_t launch_pair_batch(const Traj<float>* d_traj, int N, const int2* d_items, int n_items, cudaStream_t s,
                              int* launches) {
    if (n_items == 0) return cudaSuccess;
    switch (N) {
        case 1: kb_pair<1><<<n_items, THREADS, smem_bytes<1, false, false>(), s>>>(d_traj, d_items); break;
        case 2: kb_pair<2><<<n_items, THREADS, smem_bytes<2, false, false>(), s>>>(d_traj, d_items); break;
        case 3: kb_pair<3><<<n_items, THREADS, smem_bytes<3, false, false>(), s>>>(d_traj, d_items); break;
        case 4: kb_pair<4><<<n_items, THREADS, smem_bytes<4, false, false>(), s>>>(d_traj, d_items); break;
        default: return cudaErrorInvalidValue;
    }
    if (launches) *launches += 1;
    return cudaGetLastError();
}

}  // namespace yy
