// Arithmetic on the bit patterns of doubles, for kernels that spare GB300's narrow FP64
// unit.  Compiles for the host as well (plain C++).
#pragma once

#include <cmath>
#include <cstring>

#ifdef __CUDACC__
#define PDHG_HD __host__ __device__ __forceinline__
#else
#define PDHG_HD inline
#endif

namespace pdhg {

PDHG_HD long long double_bits(double v)
{
#ifdef __CUDA_ARCH__
    return __double_as_longlong(v);
#else
    long long b;
    std::memcpy(&b, &v, sizeof(b));
    return b;
#endif
}

PDHG_HD double bits_double(long long b)
{
#ifdef __CUDA_ARCH__
    return __longlong_as_double(b);
#else
    double v;
    std::memcpy(&v, &b, sizeof(v));
    return v;
#endif
}

// A value that is not negative as an integer that orders like it: -0 counts as 0 and, as
// for fmax, a NaN as no value (0).
PDHG_HD unsigned long long nonneg_key(double v)
{
    const unsigned long long b = (unsigned long long)double_bits(v) & 0x7fffffffffffffffull;
    return b > 0x7ff0000000000000ull ? 0ull : b;
}

PDHG_HD float float_recip(float v)   // rounded to nearest
{
#ifdef __CUDA_ARCH__
    return __frcp_rn(v);
#else
    return 1.0f / v;
#endif
}

// The bit pattern of a value as an integer that orders like it (a sign bit turns
// the order of the rest round; NaNs lie beyond the infinities).
PDHG_HD long long order_key(double a)
{
    const long long b = double_bits(a);
    return b ^ (long long)((unsigned long long)(b >> 63) >> 1);
}

// v clamped to [lo, hi] (l <= u; a NaN stays).  FP64: on the bit patterns as
// integers, which order like the values (a sign bit turns the order round): an
// FP64 comparison would take the FP64 unit.
PDHG_HD double res_clamp(double v, double lo, double hi)
{
    const long long k = order_key(v);
    const bool nan = (unsigned long long)(double_bits(v) & 0x7fffffffffffffffll) >
                     0x7ff0000000000000ull;
    double r = v;
    if (k < order_key(lo)) r = lo;
    if (k > order_key(hi)) r = hi;
    return nan ? v : r;
}
PDHG_HD float res_clamp(float v, float lo, float hi)
{
    if (v < lo) v = lo;
    if (v > hi) v = hi;
    return v;
}
// v where it is not negative, else 0 (a NaN stays)
PDHG_HD double res_pos(double v)
{
    const unsigned long long b = (unsigned long long)double_bits(v);
    return b > 0x8000000000000000ull && b <= 0xfff0000000000000ull ? 0.0 : v;
}
PDHG_HD float res_pos(float v) { return v < 0.0f ? 0.0f : v; }

// v > 0, and lo < v < hi (NaNs: false; the zeros are equal), on the bit patterns as well
PDHG_HD bool res_positive(double v)
{
    const long long b = double_bits(v);
    return b > 0 && b <= 0x7ff0000000000000ll;
}
PDHG_HD bool res_positive(float v) { return v > 0.0f; }
PDHG_HD bool res_inside(double v, double lo, double hi)
{
    long long k = order_key(v), a = order_key(lo), b = order_key(hi);
    k += k == -1;    // -0
    a += a == -1;
    b += b == -1;
    return a < k && k < b;   // a NaN lies beyond the infinities: no bound is
}
PDHG_HD bool res_inside(float v, float lo, float hi) { return lo < v && v < hi; }

// n / d for rd = 1 / d (correctly rounded): the product with rd corrected by its residual
// (Markstein, 1990).  Three fused multiply-adds (200 cycles of GB300's FP64 unit) instead of
// a division (1,500).  As quotient below: the bits of the division in all of 200M pairs, 12M of
// them with a quotient next to the middle of two doubles, 132M next to powers of two.
PDHG_HD double div_by(double n, double d, double rd)
{
    const double q = n * rd;
    return std::fma(std::fma(-d, q, n), rd, q);
}

// n / d where both are of ordinary size (and n may be 0): an FP32 reciprocal refined by two
// Newton steps, the quotient corrected by its residual as above (a divisor whose mantissa is
// all ones, the method's exception, is divided by: 2^52 / (2^53 - 1) came out one unit off).
// About 600 cycles of the
// deciding thread, on every attempt's critical path, instead of the 1,500 of a division.
PDHG_HD double quotient(double n, double d)
{
    const int en = (int)((unsigned long long)double_bits(n) >> 52) & 2047;
    const int ed = (int)((unsigned long long)double_bits(d) >> 52) & 2047;
    const bool ones = (~double_bits(d) & 0xfffffffffffffll) == 0;
    if (ed < 923 || ed > 1123 || ones || (n != 0.0 && (en < 523 || en > 1523))) return n / d;
    double r = (double)float_recip((float)d);
    r = std::fma(r, std::fma(-d, r, 1.0), r);
    r = std::fma(r, std::fma(-d, r, 1.0), r);
    const double q = n * r;
    return std::fma(std::fma(-d, q, n), r, q);
}

}  // namespace pdhg
