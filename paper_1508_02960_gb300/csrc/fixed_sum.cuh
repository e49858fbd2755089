// fixed_sum.cuh -- integer sums in fixed point (noalloc.cu).  Compiles for the host, too.
#pragma once

namespace lbm {

struct FixedSum {           // sum = hi 2^32 + lo, as the sums of the halves of the terms
    long long hi;
    unsigned long long lo;
    __host__ __device__ __forceinline__ void add(long long x)
    {
        lo += (unsigned long long)(unsigned)x;
        hi += x >> 32;
    }
};

// t in FP64: exact below 2^53.  By its magnitude: the low word of a small negative t is close to
// 2^64, where FP64 holds multiples of 2^11 only.
__host__ __device__ __forceinline__ double to_double(__int128 t)
{
    const unsigned __int128 m = t < 0 ? -(unsigned __int128)t : (unsigned __int128)t;
    const double d =
        (double)(unsigned long long)(m >> 64) * 18446744073709551616.0 + (double)(unsigned long long)m;
    return t < 0 ? -d : d;
}

}  // namespace lbm
