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

}  // namespace pdhg
