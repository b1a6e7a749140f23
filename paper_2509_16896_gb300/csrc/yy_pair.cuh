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
// N = 1: 0.62 -> 0.29 ms; r = 1000, n = 2000: 0.93 -> 0.62 ms (8 source ranges: blocks of unequal
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
// Two stages | log-sum-exp states per thread [TM][N][2][THREADS] | source terms of two tiles |
// |f|^2 of the targets.
template <int N, bool NOISE, bool OP>
__host__ __device__ constexpr size_t smem_bytes() {
    return sizeof(float) * (2 * (size_t)stage_words<NOISE>() + (OP ? 0 : TM * N * 2 * THREADS) + 2 * BN + BM);
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

// One block: targets i0 .. i0 + BM - 1 against the groups of 64 sources in the range [split /
// nsplit, (split + 1) / nsplit), TN / 4 groups per source tile.  nsplit > 1: the rows' (max,
// sum) go to b.simt_part and a merge kernel applies the combination.  OP: every pair's score
// without the source weight, A_j(i, s) = -S1 / (2 tau_j) + S2 - tau_j |f_i|^2 / 2, is written to b.op instead.
template <int N, bool NOISE, bool OP>
__device__ __forceinline__ void block(const Consts<float>& k, const Bufs<float>& b, long long i0, int split,
                                      int nsplit, float* smem) {
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
    const int nt = s_end > s_begin ? (int)((s_end - s_begin + BN - 1) / BN) : 0;   // source tiles

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
        const long long s0 = s_begin + (long long)t * BN;
        const float* ps = b.u + (size_t)(s0 + lr) * rp + c * BK + lc;
        const int rows = (int)min((long long)BN, k.n_pad - s0);   // BN or 64 (uniform)
#pragma unroll
        for (int q = 0; q < BN / 8; ++q, ps += step)
            if (8 * q < rows) cp4(B + lc * BS + lr + 8 * q, ps);
        cp_commit();
    };
    auto source_term = [&](int t) -> float {   // of this thread's source (tid < BN) of tile t
        const long long s = s_begin + (long long)t * BN + tid;
        return (tid < BN && s < s_end && !b.mask[s]) ? b.logw[s] : -INFINITY;
    };

    if (nt > 0) {
        load(0, 0, 0);
        if (tid < BN) lsrc[tid] = source_term(0);
    }
    int buf = 0;
    for (int t = 0; t < nt; ++t) {
        uint64_t S1[RP][TN], S2[RP][TN];
#pragma unroll
        for (int p = 0; p < RP; ++p)
#pragma unroll
            for (int c = 0; c < TN; ++c) { S1[p][c] = 0ull; S2[p][c] = 0ull; }
        for (int c = 0; c < nch; ++c, buf ^= 1) {
            cp_wait_all();
            __syncthreads();   // the stage landed; the other buffer and the last tile are done with
            const bool last = c + 1 == nch;
            if (!last) load(t, c + 1, buf ^ 1);
            else if (t + 1 < nt) load(t + 1, 0, buf ^ 1);
            const float nls = (c == 0 && t + 1 < nt) ? source_term(t + 1) : 0.f;
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
            if (c == 0 && t + 1 < nt && tid < BN) lsrc[((t + 1) & 1) * BN + tid] = nls;
        }
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
                        float tmax = max_nan(max_nan(sc[0], sc[1]), max_nan(sc[2], sc[3]));
                        float* sp = lse + (size_t)(a * N + j) * 2 * THREADS + tid;
                        float mx = sp[0];
                        // every term zero in float32 (a NaN compares false and is taken in)
                        if (tmax < mx - kZeroGap) continue;
                        if (tmax != tmax) tmax = fmaxf(fmaxf(sc[0], sc[1]), fmaxf(sc[2], sc[3]));
                        if (!(tmax > -INFINITY)) continue;   // no live source
                        float sm = sp[THREADS];
                        if (tmax > mx) {
                            sm = (mx == -INFINITY) ? 0.f : sm * exp_hw(mx - tmax);
                            mx = tmax;
                        }
#pragma unroll
                        for (int c = 0; c < 4; ++c) sm += exp_hw(sc[c] - mx);
                        sp[0] = mx;
                        sp[THREADS] = sm;
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
