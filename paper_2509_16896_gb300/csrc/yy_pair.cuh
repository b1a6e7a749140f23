// Pair loop of the float32 forms that evaluate exact differences: for a block of targets and
// a range of sources it accumulates, per pair and over the coordinates in increasing order,
//     S1 = |u_i - u_s|^2,   S2 = (u_i - u_s) . f_i      (difference first, then one FMA each)
// and hands them to an online log-sum-exp per target and scale (plain form) or to the
// materialised operator.
//
// What bounds it: the FP32 pipe.  A pair and coordinate cost one subtraction and two FMAs
// (noise coefficients: one product more); the pipe does 128 lane operations per clock and
// SM, scalar or packed (measured 122 scalar, 116-126 packed), but a packed instruction
// (two lanes of operands) takes half the issue slots, which leaves room for the
// shared-memory loads.  So the arithmetic is packed over pairs of target rows, whose
// coordinates lie side by side in shared memory, with the source coordinate duplicated.
//
// Tile: 32 targets x 128 sources, 128 threads of 4 x 8 pairs (rows 4 ty + 0..3, columns 4 tx + 64 g
// + 0..3, so every shared-memory load is 16 bytes, conflict-free over the columns and a
// broadcast over the rows), four blocks per SM at 128 registers.  Measured at r = 100, n =
// 16384, N = 2 (6.8 ms unpacked, one word per load, 4 x 4 pairs): 8 x 8 pairs and two blocks per SM
// 3.9 ms, 4 x 8 at three blocks 3.4 ms (FMA pipe 68 % busy, waiting on fixed latencies), at
// four 3.3 ms = 24.4 T pair-coordinate operations a second, 0.61 of the pipe; r = 17, n = 9001,
// N = 1: 0.62 -> 0.29 ms; r = 1000, n = 2000: 0.95 -> 0.55 ms (8 source ranges: blocks of unequal
// number per SM).  16 coordinates per stage, double-buffered and filled by 4-byte
// asynchronous copies that transpose on the way (coordinate-major rows padded by 4 words:
// two-way conflicts at most); the copies of the next stage, across source tiles, run under
// the arithmetic of this one.
//
// Order of the sums: a target row has 16 chains (tx) per source range; a chain takes columns
// 4 tx .. 4 tx + 3 of one group of 64 sources after the other, four scores at a time, and the
// chains are merged in a butterfly, whatever the tile: results depend only on the
// number of source ranges.
#pragma once

#include "yy_combine.cuh"
#include "yy_pair_sums.cuh"
#include "yy_tcgen05.cuh"

namespace yy {
namespace pair {

constexpr int BK = 16;        // coordinates per stage
constexpr int THREADS = 128;
constexpr int BLOCKS_PER_SM = 4;
constexpr int TM = 4, TN = 8;                    // pairs per thread
constexpr int BM = 8 * TM, BN = 16 * TN;         // targets, sources per tile
constexpr int AS = BM + 4, BS = BN + 4;          // padded row lengths (words)

// Words of one stage: targets' u and f (and metric), sources' u.
template <bool NOISE>
__host__ __device__ constexpr int stage_words() {
    return BK * ((NOISE ? 3 : 2) * AS + BS);
}
// Skipping form: words of a chain's mask, one bit per group of 64 sources of a range.
__host__ __device__ __forceinline__ int mask_words(long long n, int nsplit) {
    const long long groups = (n + 63) / 64;
    return (int)(((groups + nsplit - 1) / nsplit + 31) / 32);
}
constexpr size_t kMaxMaskBytesScreen = 160 * 1024;   // as much as a block can have
inline size_t pair_mask_bytes(long long n, int nsplit) { return 16 * sizeof(uint32_t) * (size_t)mask_words(n, nsplit); }
// Two stages | log-sum-exp states per thread [TM][N][2][THREADS] | source terms of two tiles |
// |f|^2 of the targets | skipping form: thresholds [BM][N], group tables of two tiles [2][2][16],
// four words, chain masks [16][mask_words].
template <int N, bool NOISE, bool OP, bool SKIP = false>
__host__ __device__ constexpr size_t smem_bytes() {
    return sizeof(float) * (2 * (size_t)stage_words<NOISE>() + (OP ? 0 : TM * N * 2 * THREADS) + 2 * BN + BM +
                            (SKIP ? BM * N + 2 * 2 * 16 + 4 : 0));
}

__device__ __forceinline__ void cp4(float* dst, const float* src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(ptx::smem_u32(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void cp_wait_all() { asm volatile("cp.async.wait_group 0;" ::: "memory"); }

// Two float lanes in one 64-bit register pair; every operation rounds each lane as its
// scalar form does.
__device__ __forceinline__ uint64_t dup2(float v) {
    uint64_t d;
    asm("mov.b64 %0, {%1, %1};" : "=l"(d) : "f"(v));
    return d;
}
__device__ __forceinline__ uint64_t sub2(uint64_t a, uint64_t b) {
    uint64_t d;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ uint64_t mul2(uint64_t a, uint64_t b) {
    uint64_t d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
    uint64_t d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ float lane2(uint64_t v, int h) {
    return __uint_as_float(h ? (uint32_t)(v >> 32) : (uint32_t)v);
}

constexpr float kLog2e = 1.4426950408889634f;
// e^x by the hardware base-2 exponential (results below 2^-126 flush to zero)
__device__ __forceinline__ float exp_hw(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x * kLog2e));
    return y;
}
// maximum that keeps a NaN
__device__ __forceinline__ float max_nan(float a, float b) {
    float d;
    asm("max.NaN.f32 %0, %1, %2;" : "=f"(d) : "f"(a), "f"(b));
    return d;
}
// A term this far below the running maximum is zero in float32 (e^-105 is below the smallest
// denormal's half).
constexpr float kZeroGap = 105.0f;

constexpr int kThinGroups = 2;
// Bound of a chain of r products' rounding, relative to the sum of their magnitudes (and of the
// few operations around it).
__host__ __device__ __forceinline__ float skip_gamma(int r) { return (float)(r + 16) * 6.03e-8f; }
// What the skipping form tests with (a kernel parameter: a register per value would spill).
struct SkipTest {
    float gap, gam;           // nats below the reference; skip_gamma
    float i2t[kMaxScales];    // 1 / (2 tau_j), shrunk by 5 gamma
};
// One block: targets i0 .. i0 + BM - 1 against the groups of 64 sources in the range [split /
// nsplit, (split + 1) / nsplit), TN / 4 groups per source tile.  nsplit > 1: the rows' (max,
// sum) go to b.simt_part and a merge kernel applies the combination.  OP: every pair's score
// without the source weight, A_j(i, s) = -S1 / (2 tau_j) + S2 - tau_j |f_i|^2 / 2, is written to
// b.op instead.
//
// SKIP: terms that provably cannot count are not evaluated.  b.pair_ref[i][j] is a lower bound
// of row i's largest score at scale j (k_pair_ref); a pair whose score is below it by more than
// gap at every scale is dropped.  A score is ell_s minus a sum of squares over the coordinates,
// S1 / (2 tau) - S2 + Q of them with Q = tau |f_i|^2 / 2, so a part of the sum bounds it from above up
// to rounding.  That is at most skip_gamma = (r + 16) u times the magnitudes, u = 2^-24, and |D||f| <= D^2 / (2
// tau) + tau f^2 / 2: a computed score exceeds the bound computed on the way, the thresholds' own
// rounding included, by less than 5 gamma S1 / (2 tau) + 8 gamma Q + 16 u |ref|.  The first is taken off by
// shrinking 1 / (2 tau) in the test, the others from the threshold.  Two bounds are tested:
//   - a chain's group of 4 sources is left out when its largest ell_s is below the block's lowest
//     threshold (weights spread over many nats: the large-scale model after an update); the
//     remaining groups of a chain keep their order;
//   - a tile is given up when, every 64 coordinates, -S1 / (2 tau_j) + S2 + ell_s of every pair is
//     below its row's threshold (a row's own pair, D = 0, aside: its score is known).
// A tile of one or two groups (one heavy node) is taken by one thread per target and source:
// with the full tile's loop its few blocks would wait out one stage after the other.
// With gap = 110 every dropped term is zero in float32 next to the row's largest: the row's sum
// is bit for bit that of the full evaluation.  flags != nullptr: only groups of tiles
// flagged for this target block ([tile of 128 sources] bits) are taken.
template <int N, bool NOISE, bool OP, bool SKIP = false>
__device__ __forceinline__ void block(const Consts<float>& k, const Bufs<float>& b, long long i0, int split,
                                      int nsplit, float* smem, const SkipTest* skip = nullptr, const uint32_t* flags = nullptr) {
    static_assert(!SKIP || (!NOISE && !OP), "the skipping form is the plain one");
    constexpr int SW = stage_words<NOISE>();
    constexpr int RP = TM / 2;   // row pairs per thread
    float* st0 = smem;
    float* lse = smem + 2 * SW;                                // [TM][N][2][THREADS]
    float* lsrc = lse + (OP ? 0 : TM * N * 2 * THREADS);       // [2][BN]
    float* nfs = lsrc + 2 * BN;                                // [BM]
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    const int rp = k.r_pad;
    const int nch = (k.r + BK - 1) / BK;
    const long long groups = (k.n + 63) / 64;
    const long long s_begin = (groups * split / nsplit) * 64;
    const long long s_end = min(k.n, (groups * (split + 1) / nsplit) * 64);
    int nt = s_end > s_begin ? (int)((s_end - s_begin + BN - 1) / BN) : 0;   // source tiles
    float* thr = nfs + BM;                                               // [BM][N]
    int* grp = reinterpret_cast<int*>(thr + (SKIP ? BM * N : 0));        // [2][2][16]
    int* gcnt = grp + 64;                                                // [2]: groups of two tiles
    float* red = reinterpret_cast<float*>(gcnt + 2);                     // [2]
    uint32_t* cmask = reinterpret_cast<uint32_t*>(red + 2);              // [16][mw]
    const int mw = SKIP ? mask_words(k.n, nsplit) : 0;
    uint32_t mword = 0u;   // thread tid < 16: the rest of chain tid's current mask word
    int mpos = -1;

    for (int r = tid; r < BM; r += THREADS) nfs[r] = (i0 + r < k.n) ? b.nf[i0 + r] : 0.f;
    if constexpr (!OP) {
#pragma unroll
        for (int e = 0; e < TM * N; ++e) {
            lse[(2 * e) * THREADS + tid] = -INFINITY;
            lse[(2 * e + 1) * THREADS + tid] = 0.f;
        }
    }
    // thread's share of a stage: coordinate tid & 15 of rows (tid >> 4) + 8 q
    const int lc = tid & 15, lr = tid >> 4;
    auto load = [&](int t, int c, int buf) {
        float* A = st0 + buf * SW;
        float* F = A + BK * AS;
        float* M = F + BK * AS;
        float* B = A + (NOISE ? 3 : 2) * BK * AS;
        const size_t step = (size_t)8 * rp;
        const size_t ti = (size_t)(i0 + lr) * rp + c * BK + lc;
        const float* pu = b.u + ti;
        const float* pf = b.f + ti;
        const float* pm = NOISE ? b.minv + ti : nullptr;
#pragma unroll
        for (int q = 0; q < BM / 8; ++q, pu += step, pf += step) {
            cp4(A + lc * AS + lr + 8 * q, pu);
            cp4(F + lc * AS + lr + 8 * q, pf);
            if constexpr (NOISE) { cp4(M + lc * AS + lr + 8 * q, pm); pm += step; }
        }
        // rows past the range belong to others and carry no weight; none past n_pad is read
        if constexpr (SKIP) {
            const int* gt = grp + (t & 1) * 32;
            const float* ps = b.u + (size_t)s_begin * rp + c * BK + lc;
#pragma unroll
            for (int q = 0; q < BN / 8; ++q) {
                const int j = lr + 8 * q;
                const int g = max(gt[(j >> 6) * 16 + ((j & 63) >> 2)], 0);
                cp4(B + lc * BS + j, ps + (size_t)(g * 64 + (j & 63)) * rp);
            }
            cp_commit();
            return;
        }
        const long long s0 = s_begin + (long long)t * BN;
        const float* ps = b.u + (size_t)(s0 + lr) * rp + c * BK + lc;
        const int rows = (int)min((long long)BN, k.n_pad - s0);   // BN or 64 (uniform)
#pragma unroll
        for (int q = 0; q < BN / 8; ++q, ps += step)
            if (8 * q < rows) cp4(B + lc * BS + lr + 8 * q, ps);
        cp_commit();
    };
    auto source_term = [&](int t) -> float {   // of this thread's source (tid < BN) of tile t
        long long s = s_begin + (long long)t * BN + tid;
        if constexpr (SKIP) {
            const int g = grp[(t & 1) * 32 + (tid >> 6) * 16 + ((tid & 63) >> 2)];
            s = g < 0 ? s_end : s_begin + (long long)g * 64 + (tid & 63);
        }
        return (tid < BN && s < s_end && !b.mask[s]) ? b.logw[s] : -INFINITY;
    };
    // SKIP: the next two groups of every chain, for tile t (threads 0..15)
    auto next_groups = [&](int t) {
        if (tid >= 16) return;
        int cnt = 0;
#pragma unroll
        for (int g = 0; g < 2; ++g) {
            while (mword == 0u && mpos + 1 < mw) mword = cmask[tid * mw + ++mpos];
            int v = -1;
            if (mword != 0u) {
                v = mpos * 32 + __ffs(mword) - 1;
                mword &= mword - 1u;
            }
            grp[(t & 1) * 32 + g * 16 + tid] = v;
            cnt += __popc(__ballot_sync(0xffffu, v >= 0));
        }
        if (tid == 0) gcnt[t & 1] = cnt;
    };
    // a tile of so few groups that one thread per target and source takes it
    auto thin = [&](int t) -> bool { return SKIP && gcnt[t & 1] <= kThinGroups; };
    if constexpr (SKIP) {
        // thresholds of the rows and the lowest of them
        float lo = INFINITY;
        if (tid < BM) {
            const long long i = i0 + tid;
            const bool target = i < k.n && !b.mask[i];
#pragma unroll
            for (int j = 0; j < N; ++j) {
                float v = INFINITY;
                if (target) {
                    const float ref = b.pair_ref[(size_t)i * kMaxScales + j];
                    v = ref - (skip->gap + 8.0f * skip->gam * (0.5f * k.tau[j] * b.nf[i]) + 1e-6f * fabsf(ref));
                }
                thr[tid * N + j] = v;
                lo = (v != v) ? -INFINITY : fminf(lo, v);   // an undefined bound drops nothing
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) lo = fminf(lo, __shfl_xor_sync(0xffffffffu, lo, o));
            if (tid == 0) red[0] = lo;
        }
        for (int w = tid; w < 16 * mw; w += THREADS) cmask[w] = 0u;
        __syncthreads();
        lo = red[0];
        // the chains' groups that can count, one group of 64 sources per warp at a time
        const int lane = tid & 31, ng = (int)((s_end - s_begin + 63) / 64);
        for (int g = tid >> 5; g < ng; g += THREADS / 32) {
            const long long s0 = s_begin + (long long)g * 64;
            if (flags && !((flags[(s0 >> 7) >> 5] >> ((s0 >> 7) & 31)) & 1u)) continue;
            bool act = false;
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const long long s = s0 + 2 * lane + e;
                const float v = (s < s_end && !b.mask[s]) ? b.logw[s] : -INFINITY;
                act |= v != -INFINITY && !(v < lo);
            }
            const uint32_t bal = __ballot_sync(0xffffffffu, act);
            if (lane < 16 && ((bal >> (2 * lane)) & 3u)) atomicOr(&cmask[lane * mw + (g >> 5)], 1u << (g & 31));
        }
        __syncthreads();
        if (tid < 32) {   // tiles: two groups of each chain per tile
            int c = 0;
            if (tid < 16)
                for (int w = 0; w < mw; ++w) c += __popc(cmask[tid * mw + w]);
            c = __reduce_max_sync(0xffffffffu, c);
            if (tid == 0) red[1] = __int_as_float((c + 1) / 2);
        }
        next_groups(0);
        __syncthreads();
        nt = __float_as_int(red[1]);
    }

    // which of the thread's two groups of tile t holds its own target rows (-1: neither; rows and
    // groups are aligned to 4)
    auto own_group = [&](int t) -> int {
        const long long row = i0 + ty * 4 - s_begin;
#pragma unroll
        for (int g = 0; g < 2; ++g) {
            const int v = grp[(t & 1) * 32 + g * 16 + tx];
            if (v >= 0 && (long long)v * 64 + tx * 4 == row) return g;
        }
        return -1;
    };
    // four scores into state sp of a chain (maximum, sum)
    auto add4 = [&](float* sp, const float (&sc)[4]) {
        float tmax = max_nan(max_nan(sc[0], sc[1]), max_nan(sc[2], sc[3]));
        float mx = sp[0];
        // every term zero in float32 (a NaN compares false and is taken in)
        if (tmax < mx - kZeroGap) return;
        if (tmax != tmax) tmax = fmaxf(fmaxf(sc[0], sc[1]), fmaxf(sc[2], sc[3]));
        if (!(tmax > -INFINITY)) return;   // no live source
        float sm = sp[THREADS];
        if (tmax > mx) {
            sm = (mx == -INFINITY) ? 0.f : sm * exp_hw(mx - tmax);
            mx = tmax;
        }
#pragma unroll
        for (int c = 0; c < 4; ++c) sm += exp_hw(sc[c] - mx);
        sp[0] = mx;
        sp[THREADS] = sm;
    };
    if (nt > 0) {
        if (!thin(0)) load(0, 0, 0);
        if (tid < BN) lsrc[tid] = source_term(0);
    }
    int buf = 0;
    for (int t = 0; t < nt; ++t) {
        if (SKIP && thin(t)) {
            __syncthreads();   // the chains' states are written by other threads here
            const int row = tid >> 2, e = tid & 3;
            const float nf = nfs[row];
#pragma unroll 1
            for (int x = 0; x < 32; ++x) {   // the tile's groups, chain by chain in order
                const int v = grp[(t & 1) * 32 + x];
                if (v < 0) continue;
                const long long s = s_begin + (long long)v * 64 + (x & 15) * 4 + e;
                const float ls = (s < s_end && !b.mask[s]) ? b.logw[s] : -INFINITY;
                float s1, s2;
                pair_sums_thread(b.u + (size_t)(i0 + row) * rp, b.f + (size_t)(i0 + row) * rp, b.u + (size_t)s * rp, rp, s1, s2);
#pragma unroll
                for (int j = 0; j < N; ++j) {
                    const float v0 = fmaf(-s1, k.inv2tau[j], s2) + (__fmul_rn(-0.5f * k.tau[j], nf) + ls);
                    float sc[4];
#pragma unroll
                    for (int c = 0; c < 4; ++c) sc[c] = __shfl_sync(0xffffffffu, v0, (tid & 28) + c);
                    if (e == 0) add4(lse + (size_t)((row & 3) * N + j) * 2 * THREADS + (row >> 2) * 16 + (x & 15), sc);
                }
            }
            if (t + 1 < nt) next_groups(t + 1);
            __syncthreads();
            if (t + 1 < nt) {
                if (!thin(t + 1)) load(t + 1, 0, buf);
                if (tid < BN) lsrc[((t + 1) & 1) * BN + tid] = source_term(t + 1);
            }
            continue;
        }
        uint64_t S1[RP][TN], S2[RP][TN];
#pragma unroll
        for (int p = 0; p < RP; ++p)
#pragma unroll
            for (int c = 0; c < TN; ++c) { S1[p][c] = 0ull; S2[p][c] = 0ull; }
        bool dead = false;
        for (int c = 0; c < nch; ++c, buf ^= 1) {
            cp_wait_all();
            __syncthreads();   // the stage landed; the other buffer and the last tile are done with
            const bool last = c + 1 == nch;
            if (!last) load(t, c + 1, buf ^ 1);
            else if (t + 1 < nt && !thin(t + 1)) load(t + 1, 0, buf ^ 1);
            // the next tile's source terms (SKIP: its groups first, one stage earlier)
            if (SKIP && c == 0 && t + 1 < nt) next_groups(t + 1);
            const bool take = c == (SKIP ? 1 : 0) && t + 1 < nt;
            const float nls = take ? source_term(t + 1) : 0.f;
            const float* A = st0 + buf * SW + ty * 4;
            const float* F = A + BK * AS;
            const float* M = F + BK * AS;
            const float* B = st0 + buf * SW + (NOISE ? 3 : 2) * BK * AS + tx * 4;
            // the last stage stops at the filter's last coordinate
            const int kc = last ? k.r - c * BK : BK;
            auto coord = [&](int kk) {
                uint64_t a[RP], f[RP], m[NOISE ? RP : 1];
                const ulonglong2 av = *reinterpret_cast<const ulonglong2*>(A + kk * AS);
                const ulonglong2 fv = *reinterpret_cast<const ulonglong2*>(F + kk * AS);
                a[0] = av.x; a[1] = av.y;
                f[0] = fv.x; f[1] = fv.y;
                if constexpr (NOISE) {
                    const ulonglong2 mv = *reinterpret_cast<const ulonglong2*>(M + kk * AS);
                    m[0] = mv.x; m[1] = mv.y;
                    f[0] = mul2(f[0], mv.x);
                    f[1] = mul2(f[1], mv.y);
                }
#pragma unroll
                for (int g = 0; g < TN / 4; ++g) {
                    const float4 bv = *reinterpret_cast<const float4*>(B + kk * BS + 64 * g);
                    const float bs[4] = {bv.x, bv.y, bv.z, bv.w};
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        const uint64_t bb = dup2(bs[e]);
#pragma unroll
                        for (int p = 0; p < RP; ++p) {
                            const uint64_t d = sub2(a[p], bb);
                            S1[p][4 * g + e] = fma2(NOISE ? mul2(m[p], d) : d, d, S1[p][4 * g + e]);
                            S2[p][4 * g + e] = fma2(d, f[p], S2[p][4 * g + e]);
                        }
                    }
                }
            };
            if (kc == BK) {
#pragma unroll 4
                for (int kk = 0; kk < BK; ++kk) coord(kk);
            } else {
#pragma unroll 1
                for (int kk = 0; kk < kc; ++kk) coord(kk);
            }
            if (take && tid < BN) lsrc[((t + 1) & 1) * BN + tid] = nls;
            if (SKIP && (c & 3) == 3 && nch - 1 - c >= 4) {
                // every pair of the tile already below its row's threshold at every scale?
                float ls[TN];
#pragma unroll
                for (int g = 0; g < TN / 4; ++g) {
                    const float4 lv = *reinterpret_cast<const float4*>(lsrc + (t & 1) * BN + 64 * g + tx * 4);
                    ls[4 * g] = lv.x; ls[4 * g + 1] = lv.y; ls[4 * g + 2] = lv.z; ls[4 * g + 3] = lv.w;
                }
                // (a row's own term, D = 0, is known: it does not keep the tile)
                const int own = own_group(t);
                bool alive = false;
#pragma unroll
                for (int a = 0; a < TM; ++a)
#pragma unroll
                    for (int j = 0; j < N; ++j) {
                        float m = -INFINITY;
#pragma unroll
                        for (int e = 0; e < TN; ++e)
                            if (!((e & 3) == a && (e >> 2) == own)) m = max_nan(m, fmaf(-lane2(S1[a >> 1][e], a & 1), skip->i2t[j], lane2(S2[a >> 1][e], a & 1)) + ls[e]);
                        alive |= !(m < thr[(ty * 4 + a) * N + j]);
                    }
                if (!__syncthreads_or(alive)) {
                    if (own >= 0) {
#pragma unroll
                        for (int a = 0; a < TM; ++a)
#pragma unroll
                            for (int j = 0; j < N; ++j) {
                                float sc[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
                                sc[a] = 0.f + (__fmul_rn(-0.5f * k.tau[j], nfs[ty * 4 + a]) + (own ? ls[4 + a] : ls[a]));
                                add4(lse + (size_t)(a * N + j) * 2 * THREADS + tid, sc);
                            }
                    }
                    cp_wait_all();   // the stage under way is of no use
                    __syncthreads();
                    if (t + 1 < nt && !thin(t + 1)) load(t + 1, 0, buf ^ 1);
                    dead = true;
                    buf ^= 1;
                    break;
                }
            }
        }
        if (SKIP && dead) continue;
        if constexpr (OP) {
            const size_t plane = (size_t)k.n_pad * (size_t)k.n_pad;
#pragma unroll
            for (int a = 0; a < TM; ++a) {
                const int row = ty * 4 + a;
                const float nf = nfs[row];
#pragma unroll
                for (int j = 0; j < N; ++j) {
                    const float rc = __fmul_rn(-0.5f * k.tau[j], nf);   // rounded before the sum
#pragma unroll
                    for (int g = 0; g < TN / 4; ++g) {
                        float v[4];
#pragma unroll
                        for (int e = 0; e < 4; ++e)
                            v[e] = fmaf(-lane2(S1[a >> 1][4 * g + e], a & 1), k.inv2tau[j],
                                        lane2(S2[a >> 1][4 * g + e], a & 1)) + rc;
                        const long long s = s_begin + (long long)t * BN + 64 * g;
                        if (s < s_end)   // whole groups of 64 (n_pad is a multiple of 256)
                            *reinterpret_cast<float4*>(b.op + j * plane + (size_t)(i0 + row) * k.n_pad + s + tx * 4) =
                                make_float4(v[0], v[1], v[2], v[3]);
                    }
                }
            }
        } else {
            // scores and online log-sum-exp, one group of 64 sources after the other (the
            // tile's source terms were written before the barrier of its first stage)
#pragma unroll
            for (int g = 0; g < TN / 4; ++g) {
                const float4 lv = *reinterpret_cast<const float4*>(lsrc + (t & 1) * BN + 64 * g + tx * 4);
                const float ls[4] = {lv.x, lv.y, lv.z, lv.w};
#pragma unroll
                for (int a = 0; a < TM; ++a) {
                    const float nf = nfs[ty * 4 + a];
#pragma unroll
                    for (int j = 0; j < N; ++j) {
                        const float rc = __fmul_rn(-0.5f * k.tau[j], nf);   // rounded before the sum
                        float sc[4];
#pragma unroll
                        for (int c = 0; c < 4; ++c)
                            sc[c] = fmaf(-lane2(S1[a >> 1][4 * g + c], a & 1), k.inv2tau[j],
                                         lane2(S2[a >> 1][4 * g + c], a & 1)) + (rc + ls[c]);
                        add4(lse + (size_t)(a * N + j) * 2 * THREADS + tid, sc);
                    }
                }
            }
        }
    }
    if constexpr (!OP) {
        // merge the 16 threads that share a target row (lanes differing in the low 4 bits)
#pragma unroll 1
        for (int a = 0; a < TM; ++a) {
            float mx[N], sm[N];
#pragma unroll
            for (int j = 0; j < N; ++j) {
                const float* sp = lse + (size_t)(a * N + j) * 2 * THREADS + tid;
                float m = sp[0], s = sp[THREADS];
#pragma unroll
                for (int o = 1; o < 16; o <<= 1) {
                    const float m2 = __shfl_xor_sync(0xffffffffu, m, o);
                    const float s2 = __shfl_xor_sync(0xffffffffu, s, o);
                    if (m2 != -INFINITY) {
                        if (m == -INFINITY) { m = m2; s = s2; }
                        else if (m2 > m) { s = s * exp_hw(m - m2) + s2; m = m2; }
                        else { s += s2 * exp_hw(m2 - m); }
                    }
                }
                mx[j] = m;
                sm[j] = s;
            }
            if (tx != 0) continue;
            const long long i = i0 + ty * 4 + a;
            if (i >= k.n) continue;
            if (nsplit > 1) {   // this range's states; the merge applies the combination
#pragma unroll
                for (int j = 0; j < N; ++j)
                    *reinterpret_cast<float2*>(b.simt_part + (((size_t)i * kSimtMaxSplit + split) * kMaxScales + j) * 2) =
                        make_float2(mx[j], sm[j]);
            } else if (b.mask[i]) {
                b.logw_pred[i] = -INFINITY;
            } else {
                const float hld = NOISE ? b.hld[i] : 0.f;
                b.logw_pred[i] = combine_scales<float, N>(k, mx, sm, b.divf[i], b.logw[i], b.stats->c_ref,
                                                          &b.stats->clamps, hld);
            }
        }
    }
}

// Merges the source ranges' (max, sum) states of target row i in range order and applies the
// multi-scale combination (four ranges' states are loaded before any is used).
template <int N, bool NOISE>
__device__ __forceinline__ void merge_row(const Consts<float>& k, const Bufs<float>& b, long long i,
                                          int nsplit) {
    if (b.mask[i]) { b.logw_pred[i] = -INFINITY; return; }
    float mx[N], sm[N];
#pragma unroll
    for (int j = 0; j < N; ++j) { mx[j] = -INFINITY; sm[j] = 0.f; }
    for (int q0 = 0; q0 < nsplit; q0 += 4) {
        float2 v[4][N];
#pragma unroll
        for (int q = 0; q < 4; ++q)
#pragma unroll
            for (int j = 0; j < N; ++j)
                v[q][j] = (q0 + q < nsplit)
                              ? *reinterpret_cast<const float2*>(b.simt_part + (((size_t)i * kSimtMaxSplit + q0 + q) * kMaxScales + j) * 2)
                              : make_float2(-INFINITY, 0.f);
#pragma unroll
        for (int j = 0; j < N; ++j)
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const float m2 = v[q][j].x, s2 = v[q][j].y;
                if (m2 == -INFINITY) continue;
                if (mx[j] == -INFINITY) { mx[j] = m2; sm[j] = s2; }
                else if (m2 > mx[j]) { sm[j] = sm[j] * exp_hw(mx[j] - m2) + s2; mx[j] = m2; }
                else { sm[j] += s2 * exp_hw(m2 - mx[j]); }
            }
    }
    const float hld = NOISE ? b.hld[i] : 0.f;
    b.logw_pred[i] = combine_scales<float, N>(k, mx, sm, b.divf[i], b.logw[i], b.stats->c_ref, &b.stats->clamps, hld);
}

}  // namespace pair
}  // namespace yy
