// Sums of doubles as whole numbers of two words, for terms that are added in any order:
// hi counts the unit of the sum (1 / scale) and lo its 2^-40th part, so every term is taken
// to 2^-40 units and whole numbers add to the same total in every order.  Plain C++, so that the
// arithmetic can be checked on the host.
//
// Range.  Terms of at most 2^50 units in magnitude, with a total of the magnitudes below
// 2^62 units, as hi never leaves 64 bits then.  The rounded rest of a term is at most 2^39
// in magnitude and may have the same sign in every term (tiles with equal sums), so lo
// is carried into hi after every term: 0 <= lo < 2^40, whatever the number of terms (without
// the carry 2^24 terms overflow it).  Pairs are added word by word, up to 2^23 of them.
#pragma once

#include <cstring>
#ifndef __CUDACC__
#include <cmath>
#endif

namespace ftlm {

#ifdef __CUDACC__
#define FTLM_TWO_WORD __host__ __device__ __forceinline__
#else
#define FTLM_TWO_WORD inline
#endif

FTLM_TWO_WORD long long two_word_bits(double x)
{
#ifdef __CUDA_ARCH__
    return __double_as_longlong(x);
#else
    long long b;
    std::memcpy(&b, &x, 8);
    return b;
#endif
}

// hi + lo 2^-40 unchanged, with 0 <= lo < 2^40.
FTLM_TWO_WORD void two_word_carry(long long &hi, long long &lo)
{
    hi += lo >> 40;
    lo &= (1ll << 40) - 1;
}

// Adds a (a * scale units) to w = {hi, lo}; false when a is too large or not a number, and
// the sum is void.  Through the mantissa of 1.5 2^52 + v: four FP64 instructions (conversions to 64-bit
// integers and back would be four more).
FTLM_TWO_WORD bool two_word_add(long long *w, double a, double scale)
{
    constexpr double kOne = 0x1.8p52;
    const double m = fma(a, scale, kOne), h = m - kOne;
    const double f = fma(fma(a, scale, -h), 0x1p40, kOne);
    long long hi = w[0] + (two_word_bits(m) - two_word_bits(kOne));
    long long lo = w[1] + (two_word_bits(f) - two_word_bits(kOne));
    two_word_carry(hi, lo);
    w[0] = hi;
    w[1] = lo;
    return fabs(h) < 0x1p51;
}

// The sum, rounded once (|hi| <= 2^53): a function of hi + lo 2^-40 only.
FTLM_TWO_WORD double two_word_value(long long hi, long long lo, double unscale)
{
    two_word_carry(hi, lo);
    return ((double)hi + (double)lo * 0x1p-40) * unscale;
}

}  // namespace ftlm
