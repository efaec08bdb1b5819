// FP64 numbers as eight base-128 digits for exact tensor-core products: the
// fixed-point form under a power of two, its digits as bf16 numbers, and the sum
// of the level accumulators.
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

namespace ftq {

// bias that makes the digits of a signed integer non-negative: 64 (1 + 128 + .. + 128^6)
constexpr long long DIGIT_BIAS = 64LL * (((1LL << 49) - 1) / 127);

// 64-bit integer round(|v| 2^s) with the sign of v, for a row, column or table
// whose largest exponent field is E: s = 1075 - E + up puts its values below
// 2^(53 + up).
__device__ __forceinline__ long long fixed_point(double v, int E, int up) {
    const long long b = __double_as_longlong(v);
    const int e = (int)((b >> 52) & 0x7ff);
    const unsigned long long m = e > 0 ? (((unsigned long long)b & 0xfffffffffffffULL) | (1ULL << 52)) : 0ULL;
    int rs = E - e;
    rs = rs < 0 ? 0 : (rs > 62 ? 62 : rs);
    const unsigned long long half = rs > 0 ? (1ULL << (rs - 1)) : 0ULL;
    const long long f = (long long)(((m << up) + half) >> rs);
    return b < 0 ? -f : f;
}

// The digits d_0 .. d_7 of f = sum d_j 128^(7 - j), |d_j| <= 64 for j >= 1, as
// FP32 numbers whose upper halves are their bf16 form.
__device__ __forceinline__ void digits8(long long f, float (&d)[8]) {
    const long long g = f + DIGIT_BIAS;
    const uint32_t lo = (uint32_t)g;
    const int hi = (int)(g >> 32);
    const uint32_t mid = __funnelshift_r(lo, (uint32_t)hi, 28);
    d[0] = (float)(hi >> 17);
    const uint32_t u[7] = {(uint32_t)hi >> 10, (uint32_t)hi >> 3, mid, lo >> 21, lo >> 14, lo >> 7, lo};
#pragma unroll
    for (int j = 0; j < 7; ++j) d[j + 1] = __uint_as_float((u[j] & 127u) | 0x4B000000u) - 8388672.0f;
}

__device__ __forceinline__ uint32_t pack_hi(float a, float b) {
    return __byte_perm(__float_as_uint(a), __float_as_uint(b), 0x7632);
}

// v 2^n, in one multiplication where 2^n is a normal number.
__device__ __forceinline__ double scale_pow2(double v, int n) {
    return n > -1000 && n < 1000 ? v * __hiloint2double((1023 + n) << 20, 0) : scalbn(v, n);
}

// sum_l lv[l] 128^(7 - l) of eight exact integers |lv[l]| < 2^25, rounded once.
__device__ __forceinline__ double level_sum(const float (&lv)[8]) {
    auto i = [&](int l) { return (long long)__float2int_rn(lv[l]); };
    const long long h = (i(0) << 21) + (i(1) << 14) + (i(2) << 7) + i(3);
    const long long m = (i(4) << 21) + (i(5) << 14) + (i(6) << 7) + i(7);
    // |h|, |m| < 2^47: exact in FP64, by adding 1.5 2^52 in the integer domain
    const double magic = 6755399441055744.0;
    const double hd = __longlong_as_double(__double_as_longlong(magic) + h) - magic;
    const double md = __longlong_as_double(__double_as_longlong(magic) + m) - magic;
    return fma(hd, 268435456.0, md);                       // levels 0..3 weigh 2^28 more
}

}  // namespace ftq
