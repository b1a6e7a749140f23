// Float32 screen on the FMA pipes (YY_PREC_FP32_SCREEN): a Gram pass marks the tiles whose
// pairs can count, and the skipping form of the pair loop (yy_pair.cuh) evaluates those exactly.
//
// Bound.  With T = ln n + 20 and ref_j(i) a lower bound of row i's largest score (k_pair_ref: its
// own term, or its term against the heaviest source),
//     rho_i = max_j [tau_j |f_i| + sqrt(2 tau_j max(0, lmax - ref_j(i) + T))],
// lmax the largest live log-weight of the tile's sources.  By the triangle inequality
// |u_i - tau_j f_i - u_s| >= |u_i - u_s| - tau_j |f_i|, a pair beyond rho_i scores below ref_j(i) by
// more than T at every scale; all such terms together are below e^-20 of the row's sum.  The
// squared distance over the first k coordinates is a lower bound of the full one, and in its
// Gram form q_i + q_s - 2 G (one FMA per coordinate; q the norms over those coordinates from the
// preparation pass) it is bounded from below by taking off (3 gamma_k + 10^-5)(q_i + q_s), gamma_k
// = k 2^-24 / (1 - k 2^-24) for the FMA chain (2 |u_i||u_s| <= q_i + q_s), 10^-5 for the norms.
//
// The pass is bound by the FP32 pipe (one FMA per pair and coordinate, packed in pairs) and by
// shared-memory loads next to it: 8 x 8 pairs per thread (64 x 128 per block) load 8 words per
// 32 packed FMAs.  G is symmetric, so only the tiles on and above the diagonal are formed and
// tested in both directions; a tile is dropped at the first multiple of 64 coordinates at which
// no pair is left.  At r = 1000, n = 16384, N = 3 that is after 192 to 256 coordinates.
#include <algorithm>

#include "yy_pair.cuh"

namespace yy {

namespace {

using namespace pair;

constexpr int GM = 64, GN = 128;                  // targets, sources per block
constexpr int GAS = GM + 4, GBS = GN + 4;
constexpr int GSW = BK * (GAS + GBS);

template <int N>
__global__ void __launch_bounds__(THREADS, 4)
    k_scr_gram(const __grid_constant__ Consts<float> k, const __grid_constant__ Bufs<float> b, int k1, float T,
               uint32_t* __restrict__ flags, int fwords) {
    __shared__ __align__(16) float st[2 * GSW];
    __shared__ float rho_r[GM], rho_c[GN], q_r[GM], q_c[GN], red[8];
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4, lane = tid & 31, wib = tid >> 5;
    const int ta = blockIdx.x, tc = blockIdx.y;   // block of 64 rows, tile of 128 columns (up to 65535)
    if (tc < ta / 2) return;                      // its pairs belong to the block with the roles swapped
    const long long i0 = (long long)ta * GM, c0 = (long long)tc * GN;
    const bool rows_in = i0 < k.row1 && i0 + GM > k.row0, cols_in = c0 < k.row1 && c0 + GN > k.row0;
    if (!rows_in && !cols_in) return;             // targets of other shards
    if (tc == ta / 2) {                           // the rows' own pairs: always evaluated
        if (tid < 2) atomicOr(&flags[(size_t)(ta * 2 + tid) * fwords + (tc >> 5)], 1u << (tc & 31));
        return;
    }
    const int rp = k.r_pad, nq = rp / 64;
    const int lc = tid & 15, lr = tid >> 4;
    auto load = [&](int c, int buf) {
        float* A = st + buf * GSW;
        float* B = A + BK * GAS;
        const size_t step = (size_t)8 * rp;
        const float* pa = b.u + (size_t)(i0 + lr) * rp + c * BK + lc;
        const float* pb = b.u + (size_t)(c0 + lr) * rp + c * BK + lc;
#pragma unroll
        for (int q = 0; q < GM / 8; ++q, pa += step) cp4(A + lc * GAS + lr + 8 * q, pa);
#pragma unroll
        for (int q = 0; q < GN / 8; ++q, pb += step) cp4(B + lc * GBS + lr + 8 * q, pb);
        cp_commit();
    };
    load(0, 0);
    // largest live log-weight of the rows and of the columns (as sources)
    {
        auto live = [&](long long s) -> float { return (s < k.n && !b.mask[s]) ? b.logw[s] : -INFINITY; };
        float lr_ = tid < GM ? live(i0 + tid) : -INFINITY, lc_ = live(c0 + tid);
        // an undefined weight keeps its tile
        if (lr_ != lr_) lr_ = INFINITY;
        if (lc_ != lc_) lc_ = INFINITY;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            lr_ = fmaxf(lr_, __shfl_xor_sync(0xffffffffu, lr_, o));
            lc_ = fmaxf(lc_, __shfl_xor_sync(0xffffffffu, lc_, o));
        }
        if (lane == 0) { red[wib] = lr_; red[4 + wib] = lc_; }
        __syncthreads();
        const float lmr = fmaxf(fmaxf(red[0], red[1]), fmaxf(red[2], red[3]));
        const float lmc = fmaxf(fmaxf(red[4], red[5]), fmaxf(red[6], red[7]));
        // squared screening radius of target i against sources of weight at most lmax (-1: no
        // candidates)
        auto radius = [&](long long i, float lmax) -> float {
            if (i >= k.n || b.mask[i] || lmax == -INFINITY) return -1.f;
            const float Fi = sqrtf(b.nf[i]);
            float rho = 0.f;
#pragma unroll
            for (int j = 0; j < N; ++j) {
                const float ref = b.pair_ref[(size_t)i * kMaxScales + j];
                if (!(ref > -INFINITY)) return INFINITY;   // no reference: every pair
                rho = fmaxf(rho, k.tau[j] * Fi + sqrtf(2.f * k.tau[j] * fmaxf(lmax - ref + T, 0.f)));
            }
            return rho * rho * 1.0001f + 1e-30f;
        };
        if (tid < GM) rho_r[tid] = rows_in ? radius(i0 + tid, lmc) : -1.f;
        rho_c[tid] = cols_in ? radius(c0 + tid, lmr) : -1.f;
    }
    uint64_t G[4][8];
#pragma unroll
    for (int p = 0; p < 4; ++p)
#pragma unroll
        for (int c = 0; c < 8; ++c) G[p][c] = 0ull;
    float qr = 0.f, qc = 0.f;   // norms of row tid (< 64) and column tid over the coordinates so far
    const int nch = min(k1, rp) / BK;
    int buf = 0;
    for (int c = 0; c < nch; ++c, buf ^= 1) {
        cp_wait_all();
        __syncthreads();
        if (c + 1 < nch) load(c + 1, buf ^ 1);
        const float* A = st + buf * GSW + ty * 4;
        const float* B = st + buf * GSW + BK * GAS + tx * 4;
#pragma unroll 4
        for (int kk = 0; kk < BK; ++kk) {
            uint64_t a[4];
#pragma unroll
            for (int g = 0; g < 2; ++g) {
                const ulonglong2 av = *reinterpret_cast<const ulonglong2*>(A + kk * GAS + 32 * g);
                a[2 * g] = av.x;
                a[2 * g + 1] = av.y;
            }
#pragma unroll
            for (int g = 0; g < 2; ++g) {
                const float4 bv = *reinterpret_cast<const float4*>(B + kk * GBS + 64 * g);
                const float bs[4] = {bv.x, bv.y, bv.z, bv.w};
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const uint64_t bb = dup2(bs[e]);
#pragma unroll
                    for (int p = 0; p < 4; ++p) G[p][4 * g + e] = fma2(a[p], bb, G[p][4 * g + e]);
                }
            }
        }
        if ((c & 3) != 3) continue;
        const int cq = c >> 2;
        if (tid < GM) q_r[tid] = qr += b.nu_chunk[(size_t)(i0 + tid) * nq + cq];
        q_c[tid] = qc += b.nu_chunk[(size_t)(c0 + tid) * nq + cq];
        __syncthreads();
        const float keep = 1.f - (3.03f * (float)((c + 1) * BK) * 5.9604645e-8f + 1e-5f);
        const bool last = c + 1 == nch;
        bool any = false;
        bool row_any[2] = {false, false}, col_any[2] = {false, false};
        float qcv[8], rcv[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            const int col = (e >> 2) * 64 + tx * 4 + (e & 3);
            qcv[e] = q_c[col];
            rcv[e] = rho_c[col];
        }
#pragma unroll
        for (int p = 0; p < 4; ++p)
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int row = (p >> 1) * 32 + ty * 4 + 2 * (p & 1) + h;
                const float qi = q_r[row], ri = rho_r[row];
#pragma unroll
                for (int e = 0; e < 8; ++e) {
                    const float lower = fmaf(-2.f, lane2(G[p][e], h), (qi + qcv[e]) * keep);
                    if (!last) {
                        any |= !(lower > fmaxf(ri, rcv[e]));
                    } else {
                        row_any[p >> 1] |= !(lower > ri);
                        col_any[e >> 2] |= !(lower > rcv[e]);
                    }
                }
            }
        if (!last) {
            if (!__syncthreads_or(any)) {
                cp_wait_all();   // the stage under way
                return;
            }
            continue;
        }
        // what is left is evaluated exactly: flags per block of 32 targets and tile of 128 sources
#pragma unroll
        for (int g = 0; g < 2; ++g) {
            if (__any_sync(0xffffffffu, row_any[g]) && lane == 0)
                atomicOr(&flags[(size_t)(ta * 2 + g) * fwords + (tc >> 5)], 1u << (tc & 31));
            const uint32_t bal = __ballot_sync(0xffffffffu, col_any[g]);
            if (lane < 2 && (bal & (lane ? 0xff00ff00u : 0x00ff00ffu)))
                atomicOr(&flags[(size_t)(tc * 4 + 2 * g + lane) * fwords + (ta >> 6)], 1u << ((ta >> 1) & 31));
        }
    }
}

}  // namespace

// Where the screen runs.  Below 64 coordinates the plain form is as fast as a screen that drops
// everything but needs 64 coordinates to see it was before the packed loops (r = 64, n = 16384, N = 2:
// 2.35 ms against 2.2 ms plain), and with few targets its passes cost more than they
// save.  Measured at N = 2, us, plain form -> screen where no pair is left / every tile is left:
// r = 64 n = 2048 60 -> 58 / 68, n = 4096 193 -> 82 / 107; r = 100 n = 2048 79 -> 67 / 118, n = 4096 277 -> 93 /
// 304, n = 16384 3280 -> 511 / 4088; r = 127 n = 4096 331 -> 81 / 329, n = 16384 3989 -> 496 / 3826.
// Longer rows are screened at any size: their tiles are also given up on the way.
static bool screen_pays(int r, long long n) { return r >= 128 || (r >= 64 && n >= 4096); }

// Flags of a filter that is screened: one bit per block of 32 targets and tile of 128 sources.  None (0)
// where the plain form is what runs: see above, or beyond what the masks of one source range hold.
size_t scr_flag_words(int r, long long n, long long n_pad) {
    if (!screen_pays(r, n) || pair_mask_bytes(n, 1) > kMaxMaskBytesScreen) return 0;
    return (size_t)(n_pad / 32) * (size_t)((n_pad / 128 + 31) / 32);
}

// First pass over at most k1 coordinates (a multiple of 64: the norms come in chunks of 64),
// then exact evaluation of every flagged tile.
cudaError_t launch_ksum_scr32(const Consts<float>& k, const Bufs<float>& b, int k1, cudaStream_t s, int* launches) {
    const size_t words = scr_flag_words(k.r, k.n, k.n_pad);
    if (words == 0) return launch_pair(k, b, s, launches);
    if (!b.nu_chunk || !b.scr_flags || !b.pair_ref) return cudaErrorInvalidValue;
    k1 = std::max(64, std::min((k1 + 63) / 64 * 64, k.r_pad));
    const float T = logf((float)k.n) + 20.0f;
    const int fwords = (int)((k.n_pad / 128 + 31) / 32);
    cudaError_t e = cudaMemsetAsync(b.scr_flags, 0, words * sizeof(uint32_t), s);
    if (e != cudaSuccess) return e;
    if ((e = launch_pair_ref(k, b, s)) != cudaSuccess) return e;
    const dim3 grid((unsigned)(k.n_pad / GM), (unsigned)(k.n_pad / GN));
    switch (k.N) {
        case 1: k_scr_gram<1><<<grid, THREADS, 0, s>>>(k, b, k1, T, b.scr_flags, fwords); break;
        case 2: k_scr_gram<2><<<grid, THREADS, 0, s>>>(k, b, k1, T, b.scr_flags, fwords); break;
        case 3: k_scr_gram<3><<<grid, THREADS, 0, s>>>(k, b, k1, T, b.scr_flags, fwords); break;
        case 4: k_scr_gram<4><<<grid, THREADS, 0, s>>>(k, b, k1, T, b.scr_flags, fwords); break;
        default: return cudaErrorInvalidValue;
    }
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    if (launches) *launches += 2;
    return launch_pair_flagged(k, b, T + 1.0f, b.scr_flags, fwords, s, launches);
}

}  // namespace yy
