// storage.cuh -- storage types of the propagated fields, shared by the moment-propagation kernels
// of libmp (not part of the C ABI).
#pragma once

#include <cuda_fp16.h>
#include <stdint.h>

#include <type_traits>

#include "lattice.cuh"

namespace mp {

// ---------------------------------------------------------------------------------------
// Storage type TS of the fields: float or double (the arithmetic type T itself), or IEEE
// binary16 with FP32 arithmetic. A record is widened to T on load and narrowed on store.
// Binary16 rounding is to nearest or stochastic: the magnitude is rounded up with
// probability equal to the dropped fraction of the binary16 spacing, compared against
// random bits from a counter-based hash of (step, element). Stochastic rounding is
// unbiased, so per-step changes below half a spacing still move a field on average.
// ---------------------------------------------------------------------------------------
__device__ __forceinline__ float widen1(float v) { return v; }
__device__ __forceinline__ double widen1(double v) { return v; }
__device__ __forceinline__ float widen1(__half v) { return __half2float(v); }

// 32-bit integer hash "lowbias32" (C. Wellons, "Prospecting for hash functions", 2018)
__device__ __forceinline__ uint32_t hash32(uint32_t x)
{
    x ^= x >> 16;
    x *= 0x7feb352du;
    x ^= x >> 15;
    x *= 0x846ca68bu;
    x ^= x >> 16;
    return x;
}

__device__ __forceinline__ __half half_stochastic(float x, uint32_t r)
{
    if (fabsf(x) < 6.103515625e-05f) {
        // below the smallest normal binary16 the spacing is 2^-24: round q = x 2^24 to an
        // integer, up with probability q - floor(q); the result is exact in binary16
        const float q = x * 16777216.0f;
        const float lo = floorf(q);
        const float u = (float)(r >> 8) * 5.9604644775390625e-08f;  // uniform in [0, 1)
        return __float2half_rz((u < q - lo ? lo + 1.0f : lo) * 5.9604644775390625e-08f);
    }
    // normal range: binary16 keeps 10 of the 23 FP32 mantissa bits; adding 13 random bits
    // below the kept ones carries into them with the probability of the dropped fraction
    const uint32_t b = (__float_as_uint(x) + (r & 0x1fffu)) & ~0x1fffu;
    return __float2half_rz(__uint_as_float(b));
}

template <typename TS>
struct Narrow;
template <>
struct Narrow<float> {
    __device__ static float one(float v, uint32_t, bool) { return v; }
};
template <>
struct Narrow<double> {
    __device__ static double one(double v, uint32_t, bool) { return v; }
};
template <>
struct Narrow<__half> {
    __device__ static __half one(float v, uint32_t key, bool stochastic)
    {
        return stochastic ? half_stochastic(v, hash32(key)) : __float2half_rn(v);
    }
};

template <typename T, typename TS, int W>
__device__ __forceinline__ FieldVec<T, W> ld_wide(const FieldVec<TS, W>* p)
{
    if constexpr (std::is_same<T, TS>::value) {
        return ld_rec(p);
    } else {
        const FieldVec<TS, W> h = *p;
        FieldVec<T, W> r;
#pragma unroll
        for (int j = 0; j < W; ++j) r.v[j] = widen1(h.v[j]);
        return r;
    }
}

// key: distinct per stored element and step (see step_body)
template <typename T, typename TS, int W>
__device__ __forceinline__ void st_narrow(FieldVec<TS, W>* p, const FieldVec<T, W>& v, uint32_t key, bool stochastic)
{
    if constexpr (std::is_same<T, TS>::value) {
        st_rec(p, v);
    } else {
        FieldVec<TS, W> h;
#pragma unroll
        for (int j = 0; j < W; ++j) h.v[j] = Narrow<TS>::one(v.v[j], key + (uint32_t)j, stochastic);
        *p = h;
    }
}

}  // namespace mp
