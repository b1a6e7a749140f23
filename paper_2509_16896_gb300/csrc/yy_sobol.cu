// Scrambled Sobol nodes on the device (Appendix A, "Sobol Sequence"; scrambling as in
// "Practical considerations" there).
//
// k_sobol_dirs: one warp per dimension turns the generator parameters (primitive
// polynomial x^s + a_1 x^{s-1} + ... + a_{s-1} x + 1 and initial m_1..m_s) into the 32
// direction integers V_k = m_k 2^{32-k}, continued for k > s by
//     V_k = V_{k-s} ^ (V_{k-s} >> s) ^ XOR_{i<s, a_i = 1} V_{k-i},
// and pre-multiplies them by the scramble matrix (the scramble y -> L y ^ e is linear in
// the XOR of direction integers, so L can be applied once per direction integer).
//
// k_sobol_points: XOR of the scrambled direction integers selected by the Gray code
// g = i ^ (i >> 1), XOR the digital shift, then the box map u = R (2 (y + 1/2) 2^-32 - 1) in float64
// rounded once more to float32 (box_coord).
#include "yy_internal.cuh"

namespace yy {

// One warp per dimension: lane l holds V_{l+1}; each step of the recurrence is one XOR
// reduction over the lanes (24 us with one thread per dimension).
__global__ void __launch_bounds__(128) k_sobol_dirs(const uint32_t* __restrict__ params, uint32_t* __restrict__ dirs,
                                                    int r) {
    const int d = blockIdx.x * 4 + (int)(threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (d >= r) return;
    const uint32_t* p = params + (size_t)d * (YY_SOBOL_POLY_WORDS + YY_SOBOL_SCRAMBLE_WORDS);
    const uint32_t* L = p + YY_SOBOL_POLY_WORDS;
    const int s = (int)p[0];
    const uint32_t a = p[1];
    uint32_t V = (s == 0) ? 1u << (31 - lane) : (lane < s ? p[2 + lane] << (31 - lane) : 0u);
    if (s > 0)
        for (int k = s + 1; k <= 32; ++k) {
            const int i = k - (lane + 1);   // this lane is V_{k-i}
            uint32_t t = 0u;
            if (i == s) t = V ^ (V >> s);
            else if (i >= 1 && i < s && ((a >> (s - 1 - i)) & 1u)) t = V;
            t = __reduce_xor_sync(0xffffffffu, t);
            if (lane == k - 1) V = t;
        }
    uint32_t w = 0;
#pragma unroll 8
    for (int k = 1; k <= 32; ++k) w |= (uint32_t)(__popc(L[k - 1] & V) & 1) << (32 - k);
    uint32_t* out = dirs + (size_t)d * 33;
    out[lane] = w;
    if (lane == 0) out[32] = L[32];
}

// Box coordinate of the scrambled integer y, as float32(float64(R t)), t = (2 y + 1) 2^-32 - 1: the
// float64 operations with explicit rounding ...
__device__ __noinline__ float box_coord_f64(uint32_t y, double R) {   // (out of line: not executed speculatively)
    double t = __dadd_rn((double)y, 0.5);
    t = __dmul_rn(t, 0x1p-31);      // 2 (y + 1/2) 2^-32, exact
    t = __dsub_rn(t, 1.0);          // exact
    return __double2float_rn(__dmul_rn(R, t));
}
// ... and the same value from float arithmetic, six float64 operations per point being what
// node generation would otherwise wait for (65.5 M points: 0.75 ms, 0.14 so).  With s = y - 2^31 as a
// signed integer, R t = R 2^-23 (a + c), a = floor(s / 256) and c = (s mod 256 + 1/2) / 256 both
// exact floats; rh + rl is R 2^-23 to 2^-48.  hi + lo below is R t with an error under 2^-21 rh
// (rounding of rh c and of the sum, the neglected rl c), and hi is its rounding to float
// unless lo lies within that error of half a unit in hi's last place -- there (and for small a or
// a power of two, where the unit changes) the float64 operations decide.
__device__ __forceinline__ float box_coord(uint32_t y, float rh, float rl, double R) {
    const int s = (int)(y ^ 0x80000000u);
    const float a = (float)(s >> 8), c = fmaf((float)(s & 255), 0.00390625f, 0.001953125f);
    const float p = rh * a;
    const float lo0 = fmaf(rh, a, -p) + fmaf(rl, a, rh * c);
    const float hi = p + lo0;
    const float lo = lo0 - (hi - p);
    const uint32_t hb = __float_as_uint(hi);
    const float half_ulp = __uint_as_float(max((hb & 0x7f800000u), 25u << 23) - (24u << 23));
    const bool sure = fabsf(fabsf(lo) - half_ulp) > 4.76837158e-7f * rh && fabsf(lo) < half_ulp && fabsf(a) >= 512.0f &&
                      (hb & 0x007fffffu) != 0u && rh > 1e-25f && rh < 1e25f;
    return sure ? hi : box_coord_f64(y, R);
}

// Points first .. first + count - 1 of 64 dimensions per block: a thread takes one dimension and
// kRun consecutive points, so that each point after the first is one XOR (consecutive Gray
// codes differ in one bit) with a direction integer from shared memory.
constexpr int kRun = 32;
__device__ __forceinline__ void sobol_points_body(const uint32_t* __restrict__ dirs, int r, int r_pad, long long first,
                                                  long long count, float* __restrict__ u, uint32_t* __restrict__ bits,
                                                  const double* __restrict__ halfwidth) {
    __shared__ uint32_t V[33][64];
    const int d0 = blockIdx.x * 64, dl = threadIdx.x & 63, d = d0 + dl;
    for (int e = threadIdx.x; e < 64 * 33; e += blockDim.x) {
        const int dd = e / 33, b = e - dd * 33;
        V[b][dd] = d0 + dd < r ? dirs[(size_t)(d0 + dd) * 33 + b] : 0u;
    }
    __syncthreads();
    if (d >= r) return;
    const double R = halfwidth ? halfwidth[d] : 0.0;
    const double Rs = R * 0x1p-23;
    const float rh = (float)Rs, rl = (float)(Rs - (double)rh);
    const int groups = blockDim.x / 64;
    for (long long i0 = ((long long)blockIdx.y * groups + threadIdx.x / 64) * kRun; i0 < count;
         i0 += (long long)gridDim.y * groups * kRun) {
        const unsigned long long idx = (unsigned long long)(first + i0);
        uint32_t g = (uint32_t)(idx ^ (idx >> 1));
        uint32_t y = V[32][dl];
        for (uint32_t m = g; m; m &= m - 1u) y ^= V[__ffs(m) - 1][dl];
        const int run = (int)min((long long)kRun, count - i0);
        for (int q = 0; q < run; ++q) {
            if (q) {
                const unsigned long long n = idx + q;   // Gray codes of n - 1 and n differ in bit ctz(n)
                const int z = __ffsll((long long)n) - 1;
                if (z < 32) y ^= V[z][dl];
            }
            if (bits) bits[(size_t)(i0 + q) * r + d] = y;
            if (u) u[(size_t)(first + i0 + q) * r_pad + d] = box_coord(y, rh, rl, R);
        }
    }
}

__global__ void __launch_bounds__(256) k_sobol_points(const uint32_t* __restrict__ dirs, int r, int r_pad,
                                                      long long first, long long count, float* __restrict__ u,
                                                      uint32_t* __restrict__ bits,
                                                      const double* __restrict__ halfwidth) {
    sobol_points_body(dirs, r, r_pad, first, count, u, bits, halfwidth);
}

// Re-mapping of the reference nodes to new half-widths during a restart (no-op unless the
// restart flag and the scale-changed flag are set).
__global__ void __launch_bounds__(256) k_sobol_points_restart(const uint32_t* __restrict__ dirs, int r, int r_pad,
                                                              long long n, float* __restrict__ u,
                                                              const double* __restrict__ half,
                                                              const DevStats* __restrict__ st) {
    if (st->restart_flag == 0 || st->scale_changed == 0) return;
    sobol_points_body(dirs, r, r_pad, 0, n, u, nullptr, half);
}

// Halton and Faure nodes (Appendix A, "Halton Sequence" and "Faure Sequence"): thread per
// (point, dimension), index k = first + i.  The fraction's base-p digits y_0, y_1, ... (most
// significant first) form the integer R = sum_i y_i p^(M-1-i) with M the largest digit count
// such that p^M <= 2^53, so R and p^M are exact in float64 and R / p^M is the correctly
// rounded fraction whatever M is.
//   Halton: p = the d-th prime, y_i = digit i of k (least significant first): the radical
//           inverse.
//   Faure:  p = the smallest prime >= r, y = C k mod p with C = P^(d-1), P_ij = binom(j, i);
//           the power of the Pascal matrix has the closed form
//           (P^c)_ij = binom(j, i) c^(j-i), used here (c = d - 1 mod p).
// Box map as for Sobol nodes: u = R_d (2 phi - 1), float64 with explicit rounding, then float32.
__device__ __forceinline__ int lds_digits(unsigned long long p, unsigned long long* pM) {
    int M = 0;
    unsigned long long v = 1;
    while (v <= (1ull << 53) / p) { v *= p; ++M; }
    *pM = v;
    return M;
}

__global__ void k_lds_points(int kind, const uint32_t* __restrict__ primes, uint32_t p_faure, int r, int r_pad,
                             long long first, long long count, float* __restrict__ u,
                             const double* __restrict__ halfwidth) {
    const int d = blockIdx.x * blockDim.x + threadIdx.x;
    if (d >= r) return;
    const unsigned long long p = (kind == YY_NODES_HALTON) ? primes[d] : p_faure;
    unsigned long long pM;
    const int M = lds_digits(p, &pM);
    const double R = halfwidth[d];
    const unsigned long long c = (unsigned long long)d % p;   // Faure: power of the Pascal matrix
    unsigned long long cp[64];                                  // c^t mod p
    if (kind == YY_NODES_FAURE) {
        cp[0] = 1 % p;
        for (int t = 1; t < M; ++t) cp[t] = (cp[t - 1] * c) % p;
    }
    for (long long i = blockIdx.y * (long long)blockDim.y + threadIdx.y; i < count; i += (long long)gridDim.y * blockDim.y) {
        unsigned long long kk = (unsigned long long)(first + i);
        unsigned long long dig[64];
        for (int t = 0; t < M; ++t) { dig[t] = kk % p; kk /= p; }
        unsigned long long Rn = 0;
        for (int a = 0; a < M; ++a) {
            unsigned long long y;
            if (kind == YY_NODES_HALTON) {
                y = dig[a];
            } else {
                // y_a = sum_{j >= a} binom(j, a) c^(j-a) k_j mod p
                unsigned long long acc = 0, binom = 1;   // binom(j, a), starting at j = a
                for (int j = a; j < M; ++j) {
                    if (j > a) binom = binom * (unsigned long long)j / (unsigned long long)(j - a);
                    acc += ((binom % p) * cp[j - a] % p) * dig[j];
                }
                y = acc % p;
            }
            Rn = Rn * p + y;
        }
        const double phi = __ddiv_rn((double)Rn, (double)pM);
        const double t = __dsub_rn(__dmul_rn(2.0, phi), 1.0);
        u[(size_t)i * r_pad + d] = __double2float_rn(__dmul_rn(R, t));
    }
}

cudaError_t launch_lds_points(int kind, const uint32_t* primes, uint32_t p_faure, int r, int r_pad, long long n,
                              float* u, const double* halfwidth, cudaStream_t s) {
    dim3 block(64, 4);
    long long gy = (n + 3) / 4;
    if (gy > 65535) gy = 65535;
    k_lds_points<<<dim3((r + 63) / 64, (unsigned)gy), block, 0, s>>>(kind, primes, p_faure, r, r_pad, 1, n, u, halfwidth);
    return cudaGetLastError();
}

// Blocks of 64 dimensions x 4 runs of points.
static dim3 points_grid(int r, long long count) {
    const long long gy = (count + 4 * kRun - 1) / (4 * kRun);
    return dim3((unsigned)((r + 63) / 64), (unsigned)(gy > 65535 ? 65535 : gy));
}

cudaError_t launch_sobol_points_restart(const uint32_t* dirs, int r, int r_pad, long long n, float* u,
                                        const double* next_half, const DevStats* st, cudaStream_t s) {
    k_sobol_points_restart<<<points_grid(r, n), 256, 0, s>>>(dirs, r, r_pad, n, u, next_half, st);
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_sobol_dirs(const uint32_t* params, uint32_t* dirs, int r, cudaStream_t s) {
    k_sobol_dirs<<<(r + 3) / 4, 128, 0, s>>>(params, dirs, r);
    return cudaGetLastError();
}
template cudaError_t launch_sobol_dirs<float>(const uint32_t*, uint32_t*, int, cudaStream_t);
template cudaError_t launch_sobol_dirs<double>(const uint32_t*, uint32_t*, int, cudaStream_t);

cudaError_t launch_sobol_points(const uint32_t* dirs, int r, int r_pad, long long first,
                                long long count, float* u, uint32_t* bits, const double* halfwidth,
                                cudaStream_t s) {
    if (count <= 0) return cudaSuccess;
    k_sobol_points<<<points_grid(r, count), 256, 0, s>>>(dirs, r, r_pad, first, count, u, bits, halfwidth);
    return cudaGetLastError();
}

}  // namespace yy
