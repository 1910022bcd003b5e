// Counter-based start vectors: splitmix64 (Steele, Lea & Flood 2014) as a
// counter-based generator, Box-Muller for Gaussian entries.  The definition is the
// one stated for ftlm_lanczos in include/ftlm.h.
#pragma once

#include <cstdint>

#include "ftlm.h"
#include "start_tables.cuh"

namespace ftlm {

constexpr uint64_t kGamma = 0x9E3779B97F4A7C15ull;

__host__ __device__ __forceinline__ uint64_t sm64_mix(uint64_t z)
{
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

__host__ __device__ __forceinline__ uint64_t chain_key(uint64_t seed, int N, int K, uint32_t r)
{
    const uint64_t tag = ((uint64_t)N << 48) | ((uint64_t)K << 32) | (uint64_t)r;
    return sm64_mix(sm64_mix(seed + kGamma) + tag + kGamma);
}

// Entry of a Gaussian start vector from its two 64-bit words.
__device__ __forceinline__ double gaussian_value(uint64_t u1, uint64_t u2)
{
    const double U1 = ((double)(u1 >> 11) + 1.0) * 0x1p-53;
    const double U2 = (double)(u2 >> 11) * 0x1p-53;
    const double two_pi = 2.0 * 3.14159265358979323846;
    return sqrt(-2.0 * log(U1)) * cos(two_pi * U2);
}

__device__ __forceinline__ double start_value(uint64_t key, uint64_t t, int dist)
{
    if (dist == FTLM_VEC_RADEMACHER) {
        const uint64_t u = sm64_mix(key + (t + 1) * kGamma);
        return (u >> 63) ? -1.0 : 1.0;
    }
    return gaussian_value(sm64_mix(key + (2 * t + 1) * kGamma), sm64_mix(key + (2 * t + 2) * kGamma));
}

// ---- Gaussian values of FP32 chains ------------------------------------------
// gaussian_value takes about sixty FP64 instructions, and an SM starts one FP64 warp
// instruction per 16 cycles.  Below, the value is a sum of two floats; its rounding to
// FP32 is checked against the bound of its error, and the few values in doubt (one in
// 2^13) take the FP64 expression, so the stored float is (float)gaussian_value always.
// The explicitly rounded operations keep the compiler from contracting them.
// Issue-bound at about 130 FP32 and integer instructions a value: 2^27 values take 1.11 ms,
// the FP64 expression 16.5 ms.  The tables stay in L1.

struct TwoFloat {
    float h, l;
};

// |a| >= |b| or a == 0; exact.
__device__ __forceinline__ TwoFloat two_sum(float a, float b)
{
    const float s = __fadd_rn(a, b);
    return {s, __fsub_rn(b, __fsub_rn(s, a))};
}

// d 2^-22 for |d| <= 2^44; exact.
__device__ __forceinline__ TwoFloat two_float(int64_t d)
{
    return two_sum((float)(int)(d >> 22), __fmul_rn((float)(int)((uint32_t)d & 0x3FFFFFu), 0x1p-22f));
}

// Relative error below 2^-45.
__device__ __forceinline__ TwoFloat two_mul(TwoFloat a, TwoFloat b)
{
    const float p = __fmul_rn(a.h, b.h);
    return {p, __fadd_rn(__fmaf_rn(a.h, b.h, -p), __fmaf_rn(a.h, b.l, __fmul_rn(a.l, b.h)))};
}

static __device__ __noinline__ float gaussian_rounded(uint64_t u1, uint64_t u2)
{
    return (float)gaussian_value(u1, u2);
}

__device__ __forceinline__ float gaussian_f32(uint64_t u1, uint64_t u2)
{
    // ln U1: U1 = m 2^e, m = (i / 256) (1 + z), i in [181, 362].  z i is a whole number of 2^-45
    // below 2^44 of them, so z keeps its relative accuracy where U1 is close to 1.
    const uint64_t a = (u1 >> 11) + 1;
    const int lead = __clzll((long long)a);  // >= 10
    const uint64_t an = a << lead;           // 11 zero bits at the end
    const uint32_t top = (uint32_t)(an >> 54);
    int i = (int)((top + 1) >> 1), half = 0;
    if (i > 362) {
        half = 1;
        i = (int)(((top >> 1) + 1) >> 1);
    }
    const float e = (float)(10 + half - lead);
    const int64_t d = (int64_t)(an - ((uint64_t)i << (55 + half))) >> (10 + half);
    const float4 lt = __ldg(&kLogTable[i - kLogFirst]);
    const TwoFloat z = two_mul(two_float(d), {lt.x, lt.y});
    // ln(1 + z) = z - z^2 / 2 + z^3 (1/3 - z/4 + z^2/5)
    const float hz = __fmul_rn(0.5f, z.h), qh = __fmul_rn(hz, z.h);
    const float ql = __fmaf_rn(z.h, z.l, __fmaf_rn(hz, z.h, -qh));
    const float poly = __fmaf_rn(z.h, __fmaf_rn(z.h, 0.2f, -0.25f), 0x1.555556p-2f);
    const float cub = __fmul_rn(__fmul_rn(z.h, z.h), __fmul_rn(z.h, poly));
    // e ln 2 = e (16 bits, exact products) + e (rest)
    const TwoFloat s1 = two_sum(__fmul_rn(e, 0x1.62e4p-1f), lt.z);
    const TwoFloat s2 = two_sum(s1.h, z.h);
    const TwoFloat s3 = two_sum(s2.h, -qh);
    const float small = __fadd_rn(__fadd_rn(__fsub_rn(z.l, ql), cub),
                                  __fadd_rn(__fmaf_rn(e, 0x1.7f7d1cp-20f, lt.w), __fadd_rn(s1.l, __fadd_rn(s2.l, s3.l))));
    const TwoFloat ln = two_sum(s3.h, small);
    const float yh = __fmul_rn(-2.0f, ln.h), yl = __fmul_rn(-2.0f, ln.l);
    // sqrt: one Newton correction of yh / sqrt(yh)
    const float rs = rsqrtf(yh), rh = __fmul_rn(yh, rs);
    const float rl = __fmul_rn(__fadd_rn(__fmaf_rn(-rh, rh, yh), yl), __fmul_rn(0.5f, rs));
    // cos(2 pi U2): quadrant n, angle +-(i pi / 512 + delta) from it, |delta| <= pi / 1024
    const uint64_t b = (u2 >> 11) + (1ull << 50);
    const int n = (int)(b >> 51) & 3;
    const int64_t f = (int64_t)(b & ((1ull << 51) - 1)) - (1ll << 50);
    const int64_t fa = f < 0 ? -f : f;
    const int k = (int)((fa + (1ll << 42)) >> 43);
    const float4 tt = __ldg(&kTrigTable[k]);
    const TwoFloat dl = two_mul(two_float(fa - ((int64_t)k << 43)), {0x1.921fb6p-29f, -0x1.777a5cp-54f});
    // A cos(delta) + B sin(delta): cosine (C, -S) of the even quadrants, sine (S, C) of the odd ones
    const bool odd = n & 1;
    const TwoFloat A = {odd ? tt.x : tt.z, odd ? tt.y : tt.w};
    const TwoFloat B = {odd ? tt.z : -tt.x, odd ? tt.w : -tt.y};
    const TwoFloat bd = two_mul(B, dl);
    const float d2 = __fmul_rn(dl.h, dl.h);
    const float d2l = __fmaf_rn(2.0f * dl.h, dl.l, __fmaf_rn(dl.h, dl.h, -d2));
    // cos - 1 = -d2 / 2 + d2^2 / 24; sin = d - d^3 / 6 + d^5 / 120
    const float ah = __fmul_rn(__fmul_rn(-0.5f, A.h), d2);
    const float al = __fmaf_rn(__fmul_rn(-0.5f, A.h), d2, -ah);
    const float a4 = __fmul_rn(__fmul_rn(A.h, d2), __fmul_rn(d2, 0x1.555556p-5f));
    const float b3 = __fmul_rn(__fmul_rn(bd.h, d2), __fmaf_rn(d2, 0x1.111112p-7f, -0x1.555556p-3f));
    const TwoFloat c1 = two_sum(A.h, bd.h);
    const TwoFloat c2 = two_sum(c1.h, ah);
    const float csmall =
        __fadd_rn(__fadd_rn(__fadd_rn(c1.l, c2.l), __fadd_rn(A.l, bd.l)),
                  __fadd_rn(__fmaf_rn(__fmul_rn(-0.5f, A.h), d2l, al), __fadd_rn(a4, b3)));
    const TwoFloat c = two_sum(c2.h, csmall);
    const TwoFloat v = two_mul({rh, rl}, c);
    const TwoFloat w = two_sum(v.h, v.l);
    // Relative error of w below 2^-39; the FP64 argument 2 pi U2 itself is off by up to 2^-51.
    const float tol = __fmaf_rn(fabsf(w.h), 0x1p-39f, __fmul_rn(rh, 0x1p-50f));
    const float lo = __fadd_rn(w.h, __fsub_rn(w.l, tol)), hi = __fadd_rn(w.h, __fadd_rn(w.l, tol));
    const bool negative = n == 2 || (odd && (f < 0) == (n == 3));
    float out = negative ? -lo : lo;
    if (!(lo == hi)) out = gaussian_rounded(u1, u2);  // also for U1 == 1, where lo is not a number
    return out;
}

// Entry t of a start vector as the type of the chain stores it.
template <typename V> __device__ __forceinline__ V start_entry(uint64_t key, uint64_t t, int dist)
{
    if (sizeof(V) == 4 && dist != FTLM_VEC_RADEMACHER)
        return gaussian_f32(sm64_mix(key + (2 * t + 1) * kGamma), sm64_mix(key + (2 * t + 2) * kGamma));
    return (V)start_value(key, t, dist);
}

}  // namespace ftlm
