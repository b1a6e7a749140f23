// Correction, normalisation, estimate and restart test: the online stage and step 4 of
// "Procedure for the Improved Yau-Yau Algorithm", the observation update and normalisation
// of "Log-Domain Computation", and "Local Resampling-Restart Mechanism".
//
// The Ito-corrected log-likelihood h(x).dy - dt/2 |h(x)|^2 is split as
//     lambda(c) + sum_d dh_d (g_d - dt/2 dh_d),   dh_d = h(c_d + u_d) - h(c_d),
//     g_d = dy_d - dt h(c_d),
// which is an exact rewrite: lambda(c) (float64, once per step) absorbs the large common
// part, and the per-node sum has no cancellation (cubic: dh = u (3c^2 + 3cu + u^2); the
// large-scale model's (x - 100)^3 is the same expansion about c - 100).
// The log-weights kept in T are therefore relative to c_ref + lambda(c); the absolute
// normaliser Lambda_k = c_ref + lambda(c) + LSE(relative) is accumulated in float64.
//
// Passes (all coalesced, one warp per node row or one thread per coordinate):
//   obs_prep        g, centre in T, lambda(c)                             (1 block)
//   loglik          ell' = ell_pred + sum_d ..., per-block (max, sum)     (HBM pass over u)
//   lse_merge       Lambda_rel                                            (1 block, float64)
//   moments         ell_hat = ell' - Lambda_rel, w = e^ell_hat; per block the weight sum,
//                   sum of squares, weighted mean and centred second moment of u over
//                   32-row chunks merged with Chan's update                (HBM pass over u)
//   finalize        merge of the block moments (float64): x_hat = c + mean, v_hat, ESS =
//                   W^2 / sum w^2, Z += Lambda, restart test, history row
//
// Every pass is a __device__ body taking the block index and block count explicitly;
// a single-filter __global__ wrapper runs it over blockIdx.x, and a batched wrapper
// (prefix kb_) runs it for trajectory blockIdx.y of a Traj array, so that one launch
// covers a whole batch of ragged filters.
#include "yy_internal.cuh"
#include "yy_lse.cuh"
#include "yy_prep_dims.cuh"

namespace yy {

template <typename T>
__device__ __forceinline__ T warp_sum_u(T v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

template <typename T> __device__ __forceinline__ T sin_u(T x);
template <> __device__ __forceinline__ float sin_u<float>(float x) { return sinf(x); }
template <> __device__ __forceinline__ double sin_u<double>(double x) { return sin(x); }

template <typename T>
__device__ __forceinline__ T exp_t(T x);
template <>
__device__ __forceinline__ float exp_t<float>(float x) { return expf(x); }
template <>
__device__ __forceinline__ double exp_t<double>(double x) { return exp(x); }

// Moment partials: 4 + 2 r_pad doubles per block (the log-sum-exp partials reuse the
// first 2 x (blocks of their pass, at most 4 kNumPartBlocks) doubles earlier in the step).
size_t part_bytes(int r_pad) {
    return (size_t)kNumPartBlocks * (size_t)(4 + 2 * r_pad) * sizeof(double);
}

// ---------------------------------------------------------------------------------------
// bodies
// ---------------------------------------------------------------------------------------

template <typename T>
__device__ __forceinline__ void obs_prep_body(const Consts<T>& k, const Bufs<T>& b, const double* __restrict__ dy) {
    __shared__ double red[32];
    double acc = 0.0;
    for (int d = threadIdx.x; d < k.r_pad; d += blockDim.x) {
        if (d < k.r) {
            const double c = b.centre[d];
            // h(c) and the centre of the cubic expansion: x^3 about c, (x - 100)^3 about c - 100
            const double cc = (k.model == YY_MODEL_PAPER_E1) ? c - 100.0 : c;
            const double hc = (k.model == YY_MODEL_LINEAR) ? c : cc * cc * cc;
            const double y = dy[d];
            b.dy_last[d] = y;
            b.obs_g[d] = (T)(y - (double)k.dt * hc);
            b.obs_c[d] = (T)cc;
            const double lcd = hc * y - 0.5 * (double)k.dt * hc * hc;
            if (k.noise == YY_NOISE_DIAG) {
                // weighted by 1 / b_d(c); the nodes' own 1 / b_d(x) enters in the likelihood pass
                const double sc = sin(c);
                const double V = (double)k.nz_v * (1.0 + (double)k.nz_vk * sc * sc);
                const double ibc = 1.0 / (V * V);
                b.obs_l[d] = (T)lcd;
                b.obs_ibc[d] = (T)ibc;
                acc += lcd * ibc;
            } else {
                acc += lcd;
            }
        } else {
            b.obs_g[d] = T(0);
            b.obs_c[d] = T(0);
            b.obs_l[d] = T(0);
            b.obs_ibc[d] = T(0);
        }
    }
    acc = warp_sum_u(acc);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x < 32) {
        double v = threadIdx.x < (blockDim.x >> 5) ? red[threadIdx.x] : 0.0;
        v = warp_sum_u(v);
        if (threadIdx.x == 0) b.stats->lam_c = v;
    }
}

// ell'(i) = ell_pred(i) + sum_d dh_d (g_d - dt/2 dh_d); per-block (max, sum) partials.
// One warp per row; lane l holds float2 l + 32 q of the row (the whole row is loaded
// before any arithmetic, so that up to r_pad / 64 loads per lane are in flight); the
// per-step vectors g and c sit in shared memory.  Coordinates r..r_pad-1 are zero in u and
// in g, so they add nothing.
constexpr int kRowQ = YY_MAX_DIM / 64, kShortQ = 2;

// dh = (c + u)^3 - c^3 = u (3c^2 + 3cu + u^2), and two coordinates' terms dh (g - dt/2 dh), of short
// rows: the roundings are spelt out, so that they do not depend on how an instance is compiled.
__device__ __forceinline__ float cubic_dh(float u, float c) {
    const float t = __fmul_rn(3.0f, c);
    return __fmul_rn(u, fmaf(u, u, fmaf(t, u, __fmul_rn(t, c))));
}
__device__ __forceinline__ double cubic_dh(double u, double c) { return u * (3.0 * c * c + 3.0 * c * u + u * u); }
__device__ __forceinline__ float two_terms(float h0, float g0, float h1, float g1, float half_dt) {
    return fmaf(h0, fmaf(-half_dt, h0, g0), __fmul_rn(h1, fmaf(-half_dt, h1, g1)));
}
__device__ __forceinline__ double two_terms(double h0, double g0, double h1, double g1, double half_dt) {
    return h0 * (g0 - half_dt * h0) + h1 * (g1 - half_dt * h1);
}

// NOISE (diagonal noise coefficients): per coordinate the update is
//     (h_d dy_d - dt/2 h_d^2) / b_d(x) = (l_d + dh_d (g_d - dt/2 dh_d)) / b_d(x),
// l_d = h(c_d) dy_d - dt/2 h(c_d)^2, stored relative to l_d / b_d(c) (whose sum is lambda(c)).
// NQ: float2 per lane of the longest row the instance takes (r_pad <= 64 NQ).  Short rows (NQ = 2, r <= 128)
// are bound by latency, one row of a warp after the other, so the next row is loaded under the
// arithmetic of this one; the short loop also stays in the instruction cache.
template <typename T, bool NOISE, int NQ>
__device__ __forceinline__ void loglik_body(const Consts<T>& k, const Bufs<T>& b, int bid, int nblk) {
    __shared__ double sm[8], ss[8];
    __shared__ T s_g[YY_MAX_DIM], s_c[YY_MAX_DIM];
    __shared__ T s_l[NOISE ? YY_MAX_DIM : 1], s_ibc[NOISE ? YY_MAX_DIM : 1];
    for (int d = threadIdx.x; d < k.r_pad; d += blockDim.x) {
        s_g[d] = b.obs_g[d];
        s_c[d] = b.obs_c[d];
        if constexpr (NOISE) { s_l[d] = b.obs_l[d]; s_ibc[d] = b.obs_ibc[d]; }
    }
    __syncthreads();
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    const long long warp = (bid * (long long)blockDim.x + threadIdx.x) >> 5;
    const long long nwarps = ((long long)nblk * blockDim.x) >> 5;
    const T half_dt = T(0.5) * k.dt;
    const bool cubic = k.model != YY_MODEL_LINEAR;   // cubic in u about obs_c
    const int nq = k.r_pad >> 6;
    T m = T(-INFINITY), s = T(0);   // working precision (see below)
    float2 un[NQ];
    T pn = T(0);
    auto load_row = [&](long long i) {
        if (i >= k.row1) return;
        const float2* ui = reinterpret_cast<const float2*>(b.u + (size_t)i * k.r_pad);
        pn = b.logw_pred[i];
#pragma unroll
        for (int q = 0; q < NQ; ++q) un[q] = (q < nq) ? ui[lane + 32 * q] : make_float2(0.f, 0.f);
    };
    constexpr bool ahead = NQ <= kShortQ;
    if (ahead) load_row(k.row0 + warp);
    for (long long i = k.row0 + warp; i < k.row1; i += nwarps) {
        if (!ahead) load_row(i);
        const T p = pn;
        float2 uu[NQ];
#pragma unroll
        for (int q = 0; q < NQ; ++q) uu[q] = un[q];
        if (ahead) load_row(i + nwarps);
        T acc[2] = {T(0), T(0)};
#pragma unroll
        for (int q = 0; q < NQ; ++q) {
            if (q >= nq) break;   // uniform over the warp
            const int d = 64 * q + 2 * lane;
            const T u0 = (T)uu[q].x, u1 = (T)uu[q].y;
            const T c0 = s_c[d], c1 = s_c[d + 1];
            T h0 = u0, h1 = u1;
            if constexpr (NQ <= kShortQ) {
                h0 = cubic ? cubic_dh(u0, c0) : u0;
                h1 = cubic ? cubic_dh(u1, c1) : u1;
            } else {
                h0 = cubic ? u0 * (T(3) * c0 * c0 + T(3) * c0 * u0 + u0 * u0) : u0;
                h1 = cubic ? u1 * (T(3) * c1 * c1 + T(3) * c1 * u1 + u1 * u1) : u1;
            }
            if constexpr (NOISE) {
                // 1 / b_d at the node x = c + u (padded coordinates: u = l = 0, no term)
                const T sx0 = sin_u<T>(c0 + u0), sx1 = sin_u<T>(c1 + u1);
                const T v0 = k.nz_v * (T(1) + k.nz_vk * sx0 * sx0), v1 = k.nz_v * (T(1) + k.nz_vk * sx1 * sx1);
                const T ib0 = T(1) / (v0 * v0), ib1 = T(1) / (v1 * v1);
                acc[q & 1] += (s_l[d] + h0 * (s_g[d] - half_dt * h0)) * ib0 - s_l[d] * s_ibc[d] +
                              (s_l[d + 1] + h1 * (s_g[d + 1] - half_dt * h1)) * ib1 - s_l[d + 1] * s_ibc[d + 1];
            } else {
                if constexpr (NQ <= kShortQ) acc[q & 1] += two_terms(h0, s_g[d], h1, s_g[d + 1], half_dt);
                else acc[q & 1] += h0 * (s_g[d] - half_dt * h0) + h1 * (s_g[d + 1] - half_dt * h1);
            }
        }
        T tot = acc[0] + acc[1];
        tot = warp_sum_u(tot);
        const T lw = (p == T(-INFINITY)) ? T(-INFINITY) : p + tot;
        if (lane == 0) {
            b.logw[i] = lw;
            // running (max, sum) of this warp's rows in the working precision (float64 issue
            // time per row is large on this part); blocks merge in float64
            if (lw != T(-INFINITY)) {
                if (lw > m) {
                    s = (m == T(-INFINITY)) ? T(1) : s * exp_t<T>(m - lw) + T(1);
                    m = lw;
                } else {
                    s += exp_t<T>(lw - m);
                }
            }
        }
    }
    if (lane == 0) { sm[wib] = (double)m; ss[wib] = (double)s; }
    __syncthreads();
    if (threadIdx.x < 32) {
        double M, S;
        lse_merge8(sm[lane & 7], ss[lane & 7], M, S);
        if (lane == 0) { b.part[2 * bid] = M; b.part[2 * bid + 1] = S; }
    }
}

// LSE partials of b.logw (used after init / restart weights).
template <typename T>
__device__ __forceinline__ void lse_partials_body(const Consts<T>& k, const Bufs<T>& b, int conditional, int bid,
                                                  int nblk) {
    if (conditional && b.stats->restart_flag == 0) return;
    __shared__ float smf[8];
    __shared__ double ss[8];
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    const long long i0 = bid * (long long)blockDim.x + threadIdx.x, step = (long long)nblk * blockDim.x;
    // an upper bound of the block's maximum within a float rounding, then one exponential per
    // weight relative to it
    float m = -INFINITY;
    for (long long i = i0; i < k.n; i += step) m = fmaxf(m, __double2float_ru((double)b.logw[i]));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    if (lane == 0) smf[wib] = m;
    __syncthreads();
    for (int w = 0; w < 8; ++w) m = fmaxf(m, smf[w]);
    double s = 0.0;
    if (m != -INFINITY)
        for (long long i = i0; i < k.n; i += step) {
            const double l = (double)b.logw[i];
            if (l != -INFINITY) s += exp(l - (double)m);
        }
    s = warp_sum_u(s);
    if (lane == 0) ss[wib] = s;
    __syncthreads();
    if (threadIdx.x < 32) {
        s = lane < 8 ? ss[lane] : 0.0;
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (lane == 0) { b.part[2 * bid] = (double)m; b.part[2 * bid + 1] = s; }
    }
}

// The partials' sums are float64; the rescale factors e^(m_b - M) in [0, 1] are taken in the
// filter's working precision T (a float64 exponential per partial is costly on this part, and
// float filters carry their log-weights in float).  The maxima of float filters are float
// numbers and are compared as such.  Called by every thread of the block.
template <typename T>
__device__ __forceinline__ void lse_merge_body(const double* __restrict__ part, int nb, DevStats* st, int report = 1) {
    __shared__ double red[32];
    __shared__ T redm[32];
    const int nw = (int)(blockDim.x >> 5);
    // phase 1: the largest block maximum
    T mt = T(-INFINITY);
    for (int i = threadIdx.x; i < nb; i += blockDim.x) mt = fmax(mt, (T)part[2 * i]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) mt = fmax(mt, __shfl_xor_sync(0xffffffffu, mt, o));
    if ((threadIdx.x & 31) == 0) redm[threadIdx.x >> 5] = mt;
    __syncthreads();
    for (int w = 0; w < nw; ++w) mt = fmax(mt, redm[w]);
    const double M = (double)mt;
    // phase 2: sum of the block sums rescaled to M
    double s = 0.0;
    if (mt != T(-INFINITY))
        for (int i = threadIdx.x; i < nb; i += blockDim.x) {
            const double mb = part[2 * i];
            if (mb != -INFINITY)
                s += part[2 * i + 1] * (sizeof(T) == 4 ? (double)expf((float)mb - (float)mt) : exp(mb - M));
        }
    s = warp_sum_u(s);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        double S = 0.0;
        for (int w = 0; w < nw; ++w) S += red[w];
        if (mt == T(-INFINITY)) {
            if (report) st->status |= kStatusDegenerate;   // a shard's own rows may all be empty
            st->lam_rel = 0.0;
        } else {
            st->lam_rel = M + log(S);
            if (!isfinite(st->lam_rel)) { st->status |= kStatusNonFinite; st->lam_rel = 0.0; }
        }
    }
}

template <typename T>
__device__ __forceinline__ void subtract_body(const Consts<T>& k, const Bufs<T>& b, int conditional, int bid,
                                              int nblk) {
    if (conditional && b.stats->norm_flag == 0) return;
    const T lam = (T)b.stats->lam_rel;
    for (long long i = bid * (long long)blockDim.x + threadIdx.x; i < k.n; i += (long long)nblk * blockDim.x)
        b.logw[i] = b.logw[i] - lam;
}

constexpr int kMomDims = YY_MAX_DIM / 256;   // coordinates per thread in the moments pass

// One round of the moments pass over the cnt listed rows, for a warp whose threads have up to SL
// coordinates (tid + 256 q): the round's weighted mean, then its centred second moment, merged
// into the block's running values.  Every slot's loads of several rows are in flight together;
// per slot the sums run over the rows in order.  Warps without coordinates do not come here: with
// all eight at four slots each a filter of few coordinates spent 10,000 instructions a block
// (r = 100, n = 16384: 19 us, 10 so; r = 2, n = 1024 in double: 35 us, 8).
template <typename T, int SL>
__device__ __forceinline__ void moments_rows(const Consts<T>& k, const Bufs<T>& b, long long c0, int cnt,
                                             const int* s_rows, const T* s_w, double W, double Wc,
                                             double (&mu)[kMomDims], double (&M2)[kMomDims]) {
    const int tid = threadIdx.x;
    const bool in = tid + 256 * (SL - 1) < k.r;   // the last slot's coordinate exists
    T S[SL], muc[SL], m2[SL];
#pragma unroll
    for (int q = 0; q < SL; ++q) { S[q] = T(0); m2[q] = T(0); }
#pragma unroll 4
    for (int l = 0; l < cnt; ++l) {
        const float* ur = b.u + (size_t)(c0 + s_rows[l]) * k.r_pad + tid;
        const T wl = s_w[l];
#pragma unroll
        for (int q = 0; q < SL; ++q) {
            const T v = (q < SL - 1 || in) ? (T)ur[256 * q] : T(0);
            S[q] += wl * v;
        }
    }
#pragma unroll
    for (int q = 0; q < SL; ++q) muc[q] = S[q] / (T)Wc;
#pragma unroll 4
    for (int l = 0; l < cnt; ++l) {
        const float* ur = b.u + (size_t)(c0 + s_rows[l]) * k.r_pad + tid;
        const T wl = s_w[l];
#pragma unroll
        for (int q = 0; q < SL; ++q) {
            const T v = (q < SL - 1 || in) ? (T)ur[256 * q] : T(0);
            const T dv = v - muc[q];
            m2[q] += wl * dv * dv;
        }
    }
    if (W == 0.0) {   // the first round with weight is taken as it is
#pragma unroll
        for (int q = 0; q < SL; ++q) { mu[q] = (double)muc[q]; M2[q] = (double)m2[q]; }
    } else {
        const double Wn = W + Wc, a = Wc / Wn, c = W * Wc / Wn;
#pragma unroll
        for (int q = 0; q < SL; ++q) {
            const double delta = (double)muc[q] - mu[q];
            mu[q] += delta * a;
            M2[q] += (double)m2[q] + delta * delta * c;
        }
    }
}

// Normalises ell' and accumulates per-block weighted moments of u.  The block's rows are
// taken 256 at a time (one per thread): ell_hat = ell' - Lambda_rel and w = e^ell_hat, the
// round's weight sum and sum of squares (float64), and the rows with w > 0 compacted in
// row order (ballot prefix sums, so the result does not depend on scheduling).  Only those
// rows are read: per coordinate the round's weighted mean, then its centred second moment,
// merged into the block's running values with Chan's rule (float64).  With posteriors
// concentrated on few nodes most rounds read no coordinates at all.
template <typename T>
__device__ __forceinline__ void moments_body(const Consts<T>& k, const Bufs<T>& b, int bid, int nblk) {
    __shared__ int s_rows[256];
    __shared__ T s_w[256];
    __shared__ int s_wcnt[8];
    __shared__ double s_red[2][8];
    const int tid = threadIdx.x, lane = tid & 31, wib = tid >> 5;
    const long long rows_per = (k.row1 - k.row0 + nblk - 1) / nblk;
    const long long i0 = k.row0 + bid * rows_per;
    const long long i1 = min(k.row1, i0 + rows_per);
    const T lam = (T)b.stats->lam_rel;
    double W = 0.0, Q = 0.0;
    double mu[kMomDims], M2[kMomDims];
#pragma unroll
    for (int q = 0; q < kMomDims; ++q) { mu[q] = 0.0; M2[q] = 0.0; }
    // coordinate slots of this warp (0: none of its threads has one; it only normalises rows)
    const int slots = k.r > 32 * wib ? (k.r - 32 * wib + 255) / 256 : 0;
    for (long long c0 = i0; c0 < i1; c0 += 256) {
        const long long i = c0 + tid;
        T w = T(0);
        if (i < i1) {
            const T lh = b.logw[i] - lam;
            b.logw[i] = lh;
            w = exp_t<T>(lh);
        }
        // round sums and the compacted list of rows with weight (float64 arithmetic only in and
        // over warps that have some: an addition takes 64 clocks, more with every warp at it)
        const uint32_t bal = __ballot_sync(0xffffffffu, !(w <= T(0)));
        if (bal) {
            const double wsum = warp_sum_u((double)w), wsq = warp_sum_u((double)w * (double)w);
            if (lane == 0) { s_red[0][wib] = wsum; s_red[1][wib] = wsq; }
        }
        if (lane == 0) s_wcnt[wib] = __popc(bal);
        __syncthreads();
        int off = 0, cnt = 0;
        double Wc = 0.0, Qc = 0.0;
        for (int g = 0; g < 8; ++g) {
            if (g < wib) off += s_wcnt[g];
            cnt += s_wcnt[g];
            if (s_wcnt[g]) {
                Wc += s_red[0][g];
                Qc += s_red[1][g];
            }
        }
        if (!(w <= T(0))) {
            const int slot = off + __popc(bal & ((1u << lane) - 1u));
            s_rows[slot] = (int)(i - c0);
            s_w[slot] = w;
        }
        __syncthreads();
        if (cnt > 0 && Wc > 0.0) {
            switch (slots) {   // uniform over a warp
                case 1: moments_rows<T, 1>(k, b, c0, cnt, s_rows, s_w, W, Wc, mu, M2); break;
                case 2: moments_rows<T, 2>(k, b, c0, cnt, s_rows, s_w, W, Wc, mu, M2); break;
                case 3: moments_rows<T, 3>(k, b, c0, cnt, s_rows, s_w, W, Wc, mu, M2); break;
                case 4: moments_rows<T, 4>(k, b, c0, cnt, s_rows, s_w, W, Wc, mu, M2); break;
            }
            W += Wc;
        }
        Q += Qc;
        __syncthreads();
    }
    double* p = b.part + (size_t)bid * (4 + 2 * k.r_pad);
    if (tid == 0) { p[0] = W; p[1] = Q; }
    // only partials with weight are merged, so a block
    // without weight -- most of them when the posterior is concentrated -- writes no moments
    if (W > 0.0) {
#pragma unroll
        for (int q = 0; q < kMomDims; ++q) {
            const int d = tid + 256 * q;
            if (d < k.r_pad) { p[4 + d] = mu[q]; p[4 + k.r_pad + d] = M2[q]; }
        }
    }
}

// The step's results from the nb (at most kNumPartBlocks) block partials, in blocks of two warps.
// The last block: weight sum W, sum of squares Q, ESS = W^2 / Q, Lambda = c_ref + lambda(c) +
// Lambda_rel, Z += Lambda, step k += 1 and the restart test.  The others, a warp per
// coordinate: mean and variance from the partials with weight (only those are written) in two
// reductions: the mean of the block means weighted by W_b (one division), then M2 = sum of M2_b +
// W_b (mu_b - mu)^2 about it (the parallel-axis identity: the same quantity as merging the partials
// pairwise, without a float64 division per partial); x_hat = c + mean.  A warp has all its loads
// of one kind in flight together, and two warps share a
// block because a float64 operation takes 64 clocks from one warp and 150 from eight: 11 + 5.5 us
// in two launches of 8 and 16 warps per block (r = 100), 8 us in one.
// rec != NULL (a shard of a row-split filter): the shard's record (its log-sum-exp, W, Q, merged
// mean and M2 of u) is written instead.  row != NULL: the step's row of the estimate history
// (x_hat[r], v_hat[r], ESS, Lambda, Z, restart test) is written too.
constexpr int kFinThreads = 64;
constexpr int kPartPerLane = (kNumPartBlocks + 31) / 32;
template <typename T>
__device__ __forceinline__ void finalize_body(const Consts<T>& k, const Bufs<T>& b, int nb, int restart_interval,
                                              double ess_frac, int bid, int dim_blocks, double* rec, double* row) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const size_t stride = 4 + 2 * (size_t)k.r_pad;
    if (bid == dim_blocks) {
        __shared__ double redw[kPartPerLane], redq[kPartPerLane];
        for (int g = w; 32 * g < nb; g += kFinThreads / 32) {   // groups of 32 partials
            const int t = 32 * g + lane;
            const double* p = b.part + (size_t)t * stride;
            const double p0 = t < nb ? p[0] : 0.0;
            double wv = p0 > 0.0 ? p0 : 0.0, qv = t < nb ? p[1] : 0.0;
            wv = warp_sum_u(wv);
            qv = warp_sum_u(qv);
            if (lane == 0) { redw[g] = wv; redq[g] = qv; }
        }
        __syncthreads();
        if (threadIdx.x != 0) return;
        double W = 0.0, Q = 0.0;
        for (int g = 0; 32 * g < nb; ++g) { W += redw[g]; Q += redq[g]; }
        DevStats* st = b.stats;
        if (rec) {
            rec[0] = st->lam_rel;
            rec[1] = W;
            rec[2] = Q;
            rec[3] = 0.0;
            return;
        }
        st->wsum = W;
        st->wsq = Q;
        const double ess = (Q > 0.0) ? W * W / Q : 0.0;
        st->ess = ess;
        const double lam = st->c_ref + st->lam_c + st->lam_rel;
        st->lam = lam;
        const double z = st->lognorm + lam;
        st->lognorm = z;
        if (!isfinite(lam)) atomicOr(&st->status, kStatusNonFinite);
        const long long step = st->step + 1;
        st->step = step;
        const bool by_ess = ess_frac > 0.0 && ess < ess_frac * (double)k.n;
        const bool by_int = restart_interval >= 2 && (step % restart_interval) == 0;
        const int flag = (by_ess || by_int) ? 1 : 0;
        st->restart_flag = flag;
        if (row) {
            row[2 * k.r] = ess;
            row[2 * k.r + 1] = lam;
            row[2 * k.r + 2] = z;
            row[2 * k.r + 3] = flag ? 1.0 : 0.0;
        }
        return;
    }
    const int d = bid * (kFinThreads / 32) + w;
    if (d >= k.r) return;
    // the partials with weight, listed in block order; lane l takes entries l, l + 32, ...
    __shared__ short s_list[kFinThreads / 32][kNumPartBlocks];
    __shared__ double s_wt[kFinThreads / 32][kNumPartBlocks];
    int np = 0;
    double p0[kPartPerLane];
#pragma unroll
    for (int q = 0; q < kPartPerLane; ++q) {
        const int t = lane + 32 * q;
        p0[q] = t < nb ? b.part[(size_t)t * stride] : 0.0;
    }
#pragma unroll
    for (int q = 0; q < kPartPerLane; ++q) {
        const uint32_t bal = __ballot_sync(0xffffffffu, p0[q] > 0.0);
        if (p0[q] > 0.0) {
            const int at = np + __popc(bal & ((1u << lane) - 1u));
            s_list[w][at] = (short)(lane + 32 * q);
            s_wt[w][at] = p0[q];
        }
        np += __popc(bal);
    }
    __syncwarp();
    double pm[kPartPerLane];
#pragma unroll
    for (int q = 0; q < kPartPerLane; ++q) {
        const int jj = lane + 32 * q;
        pm[q] = jj < np ? b.part[(size_t)s_list[w][jj] * stride + 4 + d] : 0.0;
    }
    double W = 0.0, WM = 0.0;
#pragma unroll
    for (int q = 0; q < kPartPerLane; ++q)
        if (lane + 32 * q < np) {
            const double pw = s_wt[w][lane + 32 * q];
            W += pw;
            WM = fma(pw, pm[q], WM);
        }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        W += __shfl_xor_sync(0xffffffffu, W, o);
        WM += __shfl_xor_sync(0xffffffffu, WM, o);
    }
    const double mu = (W > 0.0) ? WM / W : 0.0;
    double M2 = 0.0;
#pragma unroll
    for (int q = 0; q < kPartPerLane; ++q) {
        const int jj = lane + 32 * q;
        if (jj < np) {
            const double dm = pm[q] - mu;
            M2 += fma(s_wt[w][jj] * dm, dm, b.part[(size_t)s_list[w][jj] * stride + 4 + k.r_pad + d]);
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) M2 += __shfl_xor_sync(0xffffffffu, M2, o);
    if (lane != 0) return;
    if (rec) {
        rec[4 + d] = mu;
        rec[4 + k.r + d] = M2;
        return;
    }
    const double mean = b.centre[d] + mu;
    const double var = (W > 0.0) ? M2 / W : 0.0;
    b.mean[d] = mean;
    b.var[d] = var;
    if (row) {
        row[d] = mean;
        row[k.r + d] = var;
    }
    if (!isfinite(mean) || !isfinite(var)) atomicOr(&b.stats->status, kStatusNonFinite);
}

__device__ __forceinline__ void restart_begin_body(DevStats* st, int mode) {
    if (threadIdx.x != 0) return;
    if (mode == YY_RESTART_FORCE) st->restart_flag = 1;
    st->last_restarted = 0;
    st->norm_flag = 0;
}

// Box of the restart in progress.  Plain rule: centre x_hat, half-widths unchanged.
// Learned rule (out = network output [delta; lambda], or NULL): centre x_hat + delta,
// half-widths base_R exp(lambda), accepted only if every value is finite, every
// half-width lies in [base_R / 8, 8 base_R] and the box contains x_hat (|delta_d| <= half-
// width); the offset c_ref follows the box volume.
template <typename T>
__device__ __forceinline__ void restart_box_body(const Consts<T>& k, const Bufs<T>& b, const float* out,
                                                 double base_R) {
    __shared__ int s_ok;
    if (b.stats->restart_flag == 0) return;
    if (threadIdx.x == 0) s_ok = (out != nullptr) ? 1 : 0;
    __syncthreads();
    if (out) {
        for (int d = threadIdx.x; d < k.r; d += blockDim.x) {
            const double delta = (double)out[d], lam = (double)out[k.r + d];
            const double h = base_R * exp(lam);
            if (!isfinite(delta) || !isfinite(h) || h < base_R / 8.0 || h > 8.0 * base_R || fabs(delta) > h)
                atomicAnd(&s_ok, 0);
        }
        __syncthreads();
    }
    const bool learned = s_ok != 0;
    __shared__ double red[32];
    double dl = 0.0;
    int changed = 0;
    for (int d = threadIdx.x; d < k.r_pad; d += blockDim.x) {
        double c = 0.0, h = b.halfwidth[d];
        if (d < k.r) {
            c = b.mean[d];
            if (learned) {
                c += (double)out[d];
                h = base_R * exp((double)out[k.r + d]);
                dl += log(h / b.halfwidth[d]);
                changed |= (h != b.halfwidth[d]);
            }
        }
        b.next_centre[d] = c;
        b.next_half[d] = h;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) dl += __shfl_xor_sync(0xffffffffu, dl, o);
    changed = __any_sync(0xffffffffu, changed);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = dl;
    __shared__ int s_changed;
    if (threadIdx.x == 0) s_changed = 0;
    __syncthreads();
    if (changed && (threadIdx.x & 31) == 0) atomicOr(&s_changed, 1);
    __syncthreads();
    if (threadIdx.x == 0) {
        double tot = 0.0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) tot += red[w];
        b.stats->c_ref += tot;
        b.stats->scale_changed = s_changed;
    }
}

// End of a restart (one block): the log-normaliser of the new weights, the new box in force, and
// the request to normalise them (norm_flag; the restart flag itself is cleared here).
template <typename T>
__device__ __forceinline__ void restart_norm_body(const Consts<T>& k, const Bufs<T>& b, int nb) {
    if (b.stats->restart_flag == 0) return;
    for (int d = threadIdx.x; d < k.r_pad; d += blockDim.x) {
        b.centre[d] = b.next_centre[d];
        b.halfwidth[d] = b.next_half[d];
    }
    lse_merge_body<T>(b.part, nb, b.stats);
    __syncthreads();
    if (threadIdx.x == 0) {
        b.stats->restarts += 1;
        b.stats->restart_flag = 0;
        b.stats->norm_flag = 1;
        b.stats->last_restarted = 1;
        b.stats->op_stale = 1;   // the nodes moved: a materialised operator is rebuilt
    }
}

// ---------------------------------------------------------------------------------------
// single-filter wrappers
// ---------------------------------------------------------------------------------------

template <typename T>
__global__ void k_obs_prep(Consts<T> k, Bufs<T> b, const double* __restrict__ dy) { obs_prep_body<T>(k, b, dy); }
template <typename T, bool NOISE, int NQ>
__global__ void __launch_bounds__(256, sizeof(T) == 4 ? 4 : 2) k_loglik(const __grid_constant__ Consts<T> k,
                                                                        const __grid_constant__ Bufs<T> b) {
    loglik_body<T, NOISE, NQ>(k, b, blockIdx.x, gridDim.x);
}
template <typename T>
__global__ void __launch_bounds__(256) k_lse_partials(Consts<T> k, Bufs<T> b, int conditional) {
    lse_partials_body<T>(k, b, conditional, blockIdx.x, gridDim.x);
}
template <typename T>
__global__ void k_lse_merge(const double* __restrict__ part, int nb, DevStats* st, int report = 1) {
    lse_merge_body<T>(part, nb, st, report);
}
template <typename T>
__global__ void k_subtract(Consts<T> k, Bufs<T> b, int conditional) {
    subtract_body<T>(k, b, conditional, blockIdx.x, gridDim.x);
}
template <typename T>
__global__ void __launch_bounds__(256) k_moments(Consts<T> k, Bufs<T> b) { moments_body<T>(k, b, blockIdx.x, gridDim.x); }
template <typename T>
__global__ void __launch_bounds__(kFinThreads) k_finalize(Consts<T> k, Bufs<T> b, int nb, int restart_interval,
                                                          double ess_frac, double* rec, double* row) {
    finalize_body<T>(k, b, nb, restart_interval, ess_frac, blockIdx.x, (int)gridDim.x - 1, rec, row);
}
template <typename T>
__global__ void k_restart_begin(DevStats* st, int mode) { restart_begin_body(st, mode); }
// Float filters without a learned proposal: the restart decision, the box at x_hat and the
// restart pass's per-dimension constants in one block (the three steps of k_restart_begin,
// k_restart_box and k_prep_dims; each reads what the one before wrote).
template <typename T>
__global__ void __launch_bounds__(256) k_restart_head(Consts<T> k, Bufs<T> b, int mode, int init_kind,
                                                      double base_R) {
    restart_begin_body(b.stats, mode);
    __syncthreads();
    restart_box_body<T>(k, b, nullptr, base_R);
    __syncthreads();
    prep_dims_body<T>(k, b, kPrepRestart, init_kind, 0, 1);
}
template <typename T>
__global__ void __launch_bounds__(256) k_restart_norm(Consts<T> k, Bufs<T> b, int nb) { restart_norm_body<T>(k, b, nb); }
template <typename T>
__global__ void k_restart_box(Consts<T> k, Bufs<T> b, const float* out, double base_R) {
    restart_box_body<T>(k, b, out, base_R);
}

// ---------------------------------------------------------------------------------------
// batched wrappers: trajectory = blockIdx.y
// ---------------------------------------------------------------------------------------

template <typename T>
__global__ void kb_obs_prep(const Traj<T>* __restrict__ tr, const double* __restrict__ dy_row) {
    const Traj<T>& t = tr[blockIdx.y];
    obs_prep_body<T>(t.k, t.b, dy_row + t.dy_off);
}
template <typename T, int NQ>
__global__ void __launch_bounds__(256) kb_loglik(const Traj<T>* __restrict__ tr) {
    const Traj<T>& t = tr[blockIdx.y];
    loglik_body<T, false, NQ>(t.k, t.b, blockIdx.x, gridDim.x);
}
template <typename T>
__global__ void kb_lse_merge(const Traj<T>* __restrict__ tr, int nb) {
    const Traj<T>& t = tr[blockIdx.y];
    lse_merge_body<T>(t.b.part, nb, t.b.stats);
}
template <typename T>
__global__ void __launch_bounds__(256) kb_moments(const Traj<T>* __restrict__ tr) {
    const Traj<T>& t = tr[blockIdx.y];
    moments_body<T>(t.k, t.b, blockIdx.x, gridDim.x);
}
// grid.x = (coordinates of the longest member) / 2 + 1 blocks; each member uses its own share
template <typename T>
__global__ void __launch_bounds__(kFinThreads) kb_finalize(const Traj<T>* __restrict__ tr, int nb, double* __restrict__ hist_row) {
    const Traj<T>& t = tr[blockIdx.y];
    const int dim_blocks = (t.k.r + 1) / 2;
    if ((int)blockIdx.x > dim_blocks) return;
    finalize_body<T>(t.k, t.b, nb, t.restart_interval, t.ess_frac, blockIdx.x, dim_blocks, nullptr,
                     hist_row ? hist_row + t.hist_off : nullptr);
}
template <typename T>
__global__ void kb_reset(const Traj<T>* __restrict__ tr, int B) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= B) return;
    tr[i].b.stats->clamps = 0u;
    tr[i].b.stats->candidates = 0ull;
}
template <typename T>
__global__ void kb_restart_begin(const Traj<T>* __restrict__ tr) { restart_begin_body(tr[blockIdx.y].b.stats, YY_RESTART_AUTO); }
template <typename T>
__global__ void __launch_bounds__(256) kb_lse_partials(const Traj<T>* __restrict__ tr) {
    const Traj<T>& t = tr[blockIdx.y];
    lse_partials_body<T>(t.k, t.b, 1, blockIdx.x, gridDim.x);
}
template <typename T>
__global__ void kb_subtract(const Traj<T>* __restrict__ tr) {
    const Traj<T>& t = tr[blockIdx.y];
    subtract_body<T>(t.k, t.b, 1, blockIdx.x, gridDim.x);
}
template <typename T>
__global__ void kb_restart_box(const Traj<T>* __restrict__ tr) {
    const Traj<T>& t = tr[blockIdx.y];
    restart_box_body<T>(t.k, t.b, nullptr, 0.0);
}
template <typename T>
__global__ void __launch_bounds__(256) kb_restart_norm(const Traj<T>* __restrict__ tr, int nb) {
    const Traj<T>& t = tr[blockIdx.y];
    restart_norm_body<T>(t.k, t.b, nb);
}

// ---------------------------------------------------------------------------------------
// launchers
// ---------------------------------------------------------------------------------------

template <typename T>
void launch_loglik(const Consts<T>& k, const Bufs<T>& b, int nbl, cudaStream_t s) {
    const bool noise = k.noise == YY_NOISE_DIAG, small = k.r_pad <= 64 * kShortQ;
    if (noise && small) k_loglik<T, true, kShortQ><<<nbl, 256, 0, s>>>(k, b);
    else if (noise) k_loglik<T, true, kRowQ><<<nbl, 256, 0, s>>>(k, b);
    else if (small) k_loglik<T, false, kShortQ><<<nbl, 256, 0, s>>>(k, b);
    else k_loglik<T, false, kRowQ><<<nbl, 256, 0, s>>>(k, b);
}

template <typename T>
cudaError_t launch_update(const Consts<T>& k, const Bufs<T>& b, const double* dy,
                          int restart_interval, double ess_frac, double* hist_row, cudaStream_t s, int* launches) {
    const int nb = kNumPartBlocks;
    // the likelihood pass runs one wave of blocks: 4 per SM in float (64 registers a
    // thread), 2 in double (its partials are 2 doubles per block, well inside the moment
    // partials' space)
    const int nbl = (sizeof(T) == 4 ? 2 : 1) * kNumPartBlocks;
    k_obs_prep<T><<<1, 256, 0, s>>>(k, b, dy);
    launch_loglik<T>(k, b, nbl, s);
    k_lse_merge<T><<<1, 256, 0, s>>>(b.part, nbl, b.stats);
    k_moments<T><<<nb, 256, 0, s>>>(k, b);
    k_finalize<T><<<(k.r + 1) / 2 + 1, kFinThreads, 0, s>>>(k, b, nb, restart_interval, ess_frac, nullptr, hist_row);
    if (launches) *launches += 5;
    return cudaGetLastError();
}

// One shard of a row-split filter: the same passes over the shard's rows (k.row0..k.row1),
// its log-weights normalised by its own log-sum-exp, and its record written to rec
// (2r + 4 doubles, yy_shard.cuh) instead of the step's scalars and estimate.
template <typename T>
cudaError_t launch_update_shard(const Consts<T>& k, const Bufs<T>& b, const double* dy, double* rec, cudaStream_t s,
                                int* launches) {
    const int nb = kNumPartBlocks;
    const int nbl = (sizeof(T) == 4 ? 2 : 1) * kNumPartBlocks;
    k_obs_prep<T><<<1, 256, 0, s>>>(k, b, dy);
    launch_loglik<T>(k, b, nbl, s);
    k_lse_merge<T><<<1, 256, 0, s>>>(b.part, nbl, b.stats, 0);
    k_moments<T><<<nb, 256, 0, s>>>(k, b);
    k_finalize<T><<<(k.r + 1) / 2 + 1, kFinThreads, 0, s>>>(k, b, nb, 0, 0.0, rec, nullptr);
    if (launches) *launches += 5;
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_normalise_only(const Consts<T>& k, const Bufs<T>& b, cudaStream_t s,
                                  int* launches) {
    const int nb = kNumPartBlocks;
    k_lse_partials<T><<<nb, 256, 0, s>>>(k, b, 0);
    k_lse_merge<T><<<1, 256, 0, s>>>(b.part, nb, b.stats);
    k_subtract<T><<<nb, 256, 0, s>>>(k, b, 0);
    if (launches) *launches += 3;
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_prep_mode(const Consts<T>& k, const Bufs<T>& b, int mode, bool first,
                             double prior_mean, double prior_var, int init_kind, cudaStream_t s);
template <typename T>
cudaError_t launch_prep_rows(const Consts<T>& k, const Bufs<T>& b, int mode, cudaStream_t s);
template <typename T>
cudaError_t launch_prep_restart_batch(const Traj<T>* d_traj, int B, int r_max, long long n_pad_max, cudaStream_t s);

// Restart sequence (every kernel is a no-op unless the restart flag is set): begin, the
// learned proposal (network forward pass, if a network is attached), the box, re-mapping of
// the nodes when the half-widths change, preparation at the new box, weights, commit.
template <typename T>
cudaError_t launch_restart(const Consts<T>& k, const Bufs<T>& b, int mode, int init_kind, double base_R,
                           struct ::yy_mlp* net, cudaStream_t s, int* launches) {
    if (mode == YY_RESTART_NEVER) return cudaSuccess;
    const int nb = kNumPartBlocks;
    if (!net && sizeof(T) == 4) {   // float, plain or Gaussian restart: head, rows, weights, commit
        k_restart_head<T><<<1, 256, 0, s>>>(k, b, mode, init_kind, base_R);
        cudaError_t e = launch_prep_rows<T>(k, b, 2 /*restart*/, s);
        if (e != cudaSuccess) return e;
        k_restart_norm<T><<<1, 256, 0, s>>>(k, b, prep_grid(k.n_pad));
        k_subtract<T><<<nb, 256, 0, s>>>(k, b, 1);
        if (launches) *launches += 4;
        return cudaGetLastError();
    }
    int l = 0;
    k_restart_begin<T><<<1, 32, 0, s>>>(b.stats, mode);
    const float* out = nullptr;
    if (net) {
        cudaError_t e = mlp_propose(net, k.r, b.mean, b.var, b.dy_last, b.centre, (double)k.dt, &b.stats->restart_flag, s, &l);
        if (e != cudaSuccess) return e;
        out = mlp_output(net);
    }
    k_restart_box<T><<<1, 256, 0, s>>>(k, b, out, base_R);
    cudaError_t e = cudaSuccess;
    if (net) e = launch_sobol_points_restart(b.dirs, k.r, k.r_pad, k.n, b.u, b.next_half, b.stats, s);
    if (e != cudaSuccess) return e;
    e = launch_prep_mode<T>(k, b, 2 /*restart*/, false, 0.0, 1.0, init_kind, s);
    if (e != cudaSuccess) return e;
    // the preparation pass wrote the log-sum-exp partials of the new weights
    k_restart_norm<T><<<1, 256, 0, s>>>(k, b, prep_grid(k.n_pad));
    k_subtract<T><<<nb, 256, 0, s>>>(k, b, 1);
    if (launches) *launches += 6 + l + (net ? 1 : 0);
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_update_batch(const Traj<T>* d_traj, int B, int r_max, const double* dy_row, double* hist_row,
                                int nbu, cudaStream_t s, int* launches) {
    const dim3 one(1, B), many(nbu, B);
    kb_obs_prep<T><<<one, 256, 0, s>>>(d_traj, dy_row);
    if (r_max <= 64 * kShortQ) kb_loglik<T, kShortQ><<<many, 256, 0, s>>>(d_traj);
    else kb_loglik<T, kRowQ><<<many, 256, 0, s>>>(d_traj);
    kb_lse_merge<T><<<one, 256, 0, s>>>(d_traj, nbu);
    kb_moments<T><<<many, 256, 0, s>>>(d_traj);
    kb_finalize<T><<<dim3((r_max + 1) / 2 + 1, B), kFinThreads, 0, s>>>(d_traj, nbu, hist_row);
    if (launches) *launches += 5;
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_restart_batch(const Traj<T>* d_traj, int B, int r_max, long long n_pad_max,
                                 int nbu, cudaStream_t s, int* launches) {
    const dim3 one(1, B), many(nbu, B);
    kb_restart_begin<T><<<one, 32, 0, s>>>(d_traj);
    kb_restart_box<T><<<one, 256, 0, s>>>(d_traj);
    cudaError_t e = launch_prep_restart_batch<T>(d_traj, B, r_max, n_pad_max, s);
    if (e != cudaSuccess) return e;
    kb_lse_partials<T><<<many, 256, 0, s>>>(d_traj);
    kb_restart_norm<T><<<one, 256, 0, s>>>(d_traj, nbu);
    kb_subtract<T><<<many, 256, 0, s>>>(d_traj);
    if (launches) *launches += 7;
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_reset_batch(const Traj<T>* d_traj, int B, cudaStream_t s, int* launches) {
    kb_reset<T><<<(B + 127) / 128, 128, 0, s>>>(d_traj, B);
    if (launches) *launches += 1;
    return cudaGetLastError();
}

#define YY_INST(T)                                                                                      \
    template cudaError_t launch_update<T>(const Consts<T>&, const Bufs<T>&, const double*, int, double, \
                                          double*, cudaStream_t, int*);                                 \
    template cudaError_t launch_normalise_only<T>(const Consts<T>&, const Bufs<T>&, cudaStream_t, int*); \
    template cudaError_t launch_update_shard<T>(const Consts<T>&, const Bufs<T>&, const double*, double*,     \
                                                cudaStream_t, int*);                                            \
    template cudaError_t launch_restart<T>(const Consts<T>&, const Bufs<T>&, int, int, double, struct ::yy_mlp*, \
                                           cudaStream_t, int*);                                          \
    template cudaError_t launch_update_batch<T>(const Traj<T>*, int, int, const double*, double*, int,  \
                                                cudaStream_t, int*);                                    \
    template cudaError_t launch_restart_batch<T>(const Traj<T>*, int, int, long long, int, cudaStream_t,  \
                                                 int*);                                                 \
    template cudaError_t launch_reset_batch<T>(const Traj<T>*, int, cudaStream_t, int*);
YY_INST(float)
YY_INST(double)
#undef YY_INST

}  // namespace yy
