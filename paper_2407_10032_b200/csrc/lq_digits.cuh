// Fixed-point digit slices of real matrices for the integer tensor-core path (tcgen05 kind::i8): x = 2^e sum_s d_s 2^-8s with
// balanced 8-bit digits d_1 .. d_S and one exponent e per row of an operand.  Used by stage 2 (fp64 matrices) and stage 4.
#pragma once

#include "lq_common.cuh"

constexpr int LQ_DIGIT_LD = 1024;        // digits per row of a slice

namespace {

// Exponent for the integer digits: the leading digit must not reach 128.
__device__ __forceinline__ int exp_for8(double mx) {
    if (!(mx > 0.0)) return 0;
    int e = ilogb(mx) + 2;                              // mx 2^(8 - e) < 128
    if (scalbn(mx, 8 - e) > 127.0) ++e;
    return e;
}

// Digits of x 2^sh, |x 2^sh| <= 127 256^(NS - 1) (exp_for8), leading digit first: the balanced digits in [-128, 127] of an integer
// are its bytes after 128 has been added to every byte.  (Unsigned lower digits would be simpler, but their mean of 127 puts a
// large common component into every lower level, and the fp32 rounding of that level's sum then costs five bits of the
// result: measured, 1e-7 instead of 4e-8 on U.)
template <int NS>
__device__ __forceinline__ void int_digits(double x, int sh, uint32_t (&d)[NS]) {
    constexpr long long BIAS = static_cast<long long>(0x8080808080808080ull >> (64 - 8 * NS));
    const long long y = __double2ll_rn(scalbn(x, sh)) + BIAS;
#pragma unroll
    for (int s = 0; s < NS; ++s) d[s] = static_cast<uint32_t>((y >> (8 * (NS - 1 - s))) & 0xff) ^ 0x80u;
}
// Four consecutive entries of a row: their digits, one 32-bit store per slice.
template <int NS>
__device__ __forceinline__ void store_digits(const double (&v)[4], int e, uint8_t* dst, int64_t slice_bytes) {
    uint32_t w[NS] = {};
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        uint32_t d[NS];
        int_digits<NS>(isfinite(v[u]) ? v[u] : 0.0, 8 * NS - e, d);
#pragma unroll
        for (int s = 0; s < NS; ++s) w[s] |= d[s] << (8 * u);
    }
#pragma unroll
    for (int s = 0; s < NS; ++s) LQ_AT(reinterpret_cast<uint32_t*>(dst + s * slice_bytes)) = w[s];
}
// The same for fp32 entries and up to four digits, in 32-bit arithmetic: scaling by a power of two is exact and
// |x 2^(8 NS - e)| <= 127 256^(NS - 1) < 2^31.  (Through fp64 the slices of one outer block of stage 4 took 40 us per 8000 columns.)
__device__ __forceinline__ int exp_for8(float mx) {
    if (!(mx > 0.0f)) return 0;
    int e = ilogbf(mx) + 2;
    if (scalbnf(mx, 8 - e) > 127.0f) ++e;
    return e;
}
template <int NS>
__device__ __forceinline__ void store_digits(const float (&v)[4], int e, uint8_t* dst, int64_t slice_bytes) {
    static_assert(NS <= 4, "32-bit digits");
    uint32_t y[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        const int x = isfinite(v[u]) ? __float2int_rn(scalbnf(v[u], 8 * NS - e)) : 0;
        y[u] = (static_cast<uint32_t>(x) + (0x80808080u >> (32 - 8 * NS))) ^ (0x80808080u >> (32 - 8 * NS));
    }
#pragma unroll
    for (int s = 0; s < NS; ++s) {
        const int b = 8 * (NS - 1 - s);
        const uint32_t w = ((y[0] >> b) & 0xffu) | ((y[1] >> b) & 0xffu) << 8 | ((y[2] >> b) & 0xffu) << 16 | ((y[3] >> b) & 0xffu) << 24;
        LQ_AT(reinterpret_cast<uint32_t*>(dst + s * slice_bytes)) = w;
    }
}
__device__ __forceinline__ float digit_mag(float x) { return isfinite(x) ? fabsf(x) : INFINITY; }
__device__ __forceinline__ float digit_shift(float x, int n) { return scalbnf(x, n); }
__device__ __forceinline__ double digit_shift(double x, int n) { return scalbn(x, n); }
__device__ __forceinline__ float digit_max(float a, float b) { return fmaxf(a, b); }
__device__ __forceinline__ double digit_max(double a, double b) { return fmax(a, b); }

// Magnitude for the choice of an exponent: a NaN must not hide behind fmax.
__device__ __forceinline__ double digit_mag(double x) { return isfinite(x) ? fabs(x) : INFINITY; }
__device__ __forceinline__ double cta_max256(double mx, double* red) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = mx;
    __syncthreads();
    mx = red[0];
#pragma unroll
    for (int w = 1; w < 8; ++w) mx = fmax(mx, red[w]);
    return mx;
}

// Columns [col0, col0 + gridDim.x * 32) below col1 of the K rows src[0..K): exponent ex[j - col0] and NS digits of entry t times
// 2^(-f(t)) (f may be null), transposed (scale, if given, gets 2^e as a float, NaN for a column that is not finite): slice row j - col0 holds the column.  32 columns per CTA: their largest entries
// first, then the digits (the second read comes out of the L2).  1024 threads, because there may be 32 CTAs only: with 256 the
// digits of 1024 columns took 118 us.
constexpr int SC_THREADS = 1024;
template <int NS, typename T>
__global__ void __launch_bounds__(SC_THREADS)
slice_cols_wide_kernel(const T* __restrict__ src, int64_t ld, int K, int64_t col0, int64_t col1, const int* __restrict__ f,
                       int* __restrict__ ex, float* __restrict__ scale, uint8_t* __restrict__ SL, int64_t slice_bytes) {
    __shared__ T tile[128][33];
    __shared__ T part[32][33];
    __shared__ int sh_e[32];
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    const int64_t j0 = col0 + blockIdx.x * 32LL, j = j0 + tx;
    T mx = T(0);
    if (j < col1) {
#pragma unroll 8
        for (int t = ty; t < K; t += 32) {
            const T x = LQ_AT(src + t * ld + j);
            mx = digit_max(mx, digit_mag(f ? digit_shift(x, -LQ_AT(f + t)) : x));
        }
    }
    part[ty][tx] = mx;
    __syncthreads();
    mx = part[tx][ty];                                   // warp ty: column ty
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) mx = digit_max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    if (tx == 0) {
        const int e = isfinite(mx) ? exp_for8(mx) : 0;
        sh_e[ty] = e;
        if (ex && j0 + ty < col1) LQ_AT(ex + (j0 + ty - col0)) = e;
        if (scale && j0 + ty < col1) LQ_AT(scale + (j0 + ty - col0)) = isfinite(mx) ? ldexpf(1.0f, e) : __int_as_float(0x7fc00000);
    }
    for (int t0 = 0; t0 < K; t0 += 128) {                // K is a multiple of 128
        __syncthreads();
#pragma unroll
        for (int a = ty; a < 128; a += 32) {
            T x = j < col1 ? LQ_AT(src + (t0 + a) * ld + j) : T(0);
            if (f) x = digit_shift(x, -LQ_AT(f + t0 + a));
            tile[a][tx] = x;
        }
        __syncthreads();
        const int b = threadIdx.x >> 5, a = (threadIdx.x & 31) * 4;      // column j0 + b, entries t0 + a ..
        if (j0 + b < col1) {
            const T v[4] = {tile[a][b], tile[a + 1][b], tile[a + 2][b], tile[a + 3][b]};
            store_digits<NS>(v, sh_e[b], SL + (j0 + b - col0) * LQ_DIGIT_LD + t0 + a, slice_bytes);
        }
    }
}

}  // namespace
