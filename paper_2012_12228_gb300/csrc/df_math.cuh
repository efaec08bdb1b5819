// Double-FP32 arithmetic: a value as an unevaluated sum of two floats (48
// significand bits).  Products are split exactly with FMA (Dekker / Knuth
// two-product, two-sum; the lo * lo term, 2^-48 relative, is dropped).
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

namespace ftq {

struct df2 { float h, l; };

__device__ __forceinline__ df2 df_split(double v) {
    df2 r;
    r.h = (float)v;
    r.l = (float)(v - (double)r.h);
    return r;
}

// acc -= x * u  (x, u double-FP32; acc.l collects the rounding errors)
__device__ __forceinline__ void df_msub(df2& acc, float xh, float xl, float uh, float ul) {
    const float p = xh * uh;
    float e = fmaf(xh, uh, -p);
    e = fmaf(xh, ul, e);
    e = fmaf(xl, uh, e);
    const float t = acc.h - p;
    const float bb = t - acc.h;
    const float err = (acc.h - (t - bb)) + (-p - bb);
    acc.h = t;
    acc.l += err - e;
}

// acc += x * u
__device__ __forceinline__ void df_madd(df2& acc, float xh, float xl, float uh, float ul) {
    df_msub(acc, -xh, -xl, uh, ul);
}

__device__ __forceinline__ df2 df_norm(df2 a) {
    df2 r;
    r.h = a.h + a.l;
    r.l = a.l - (r.h - a.h);
    return r;
}

// The split of v by its bits (upper 24 bits of the significand, then the rest): no
// FP64 instruction for |v| in [2^-70, 2^127) and 0.
__device__ __forceinline__ df2 df_split_int(double v) {
    const int hi = __double2hiint(v);
    const uint32_t lo = (uint32_t)__double2loint(v);
    const int e = ((hi >> 20) & 0x7ff) - 1023;
    if ((((uint32_t)hi << 1) | lo) == 0u) return df2{0.f, 0.f};
    if (e < -70 || e > 126) return df_split(v);
    const uint32_t sign = (uint32_t)hi & 0x80000000u;
    df2 r;
    r.h = __uint_as_float(sign | (uint32_t)(e + 127) << 23 | ((uint32_t)hi & 0xfffffu) << 3 | lo >> 29);
    r.l = (float)(int)(lo & 0x1fffffffu) * __uint_as_float(sign | (uint32_t)(e - 52 + 127) << 23);
    return df_norm(r);
}

}  // namespace ftq
