// solve_word.cuh -- values of the solve as words, one of which means "not yet".
#pragma once

#include <cstdint>

namespace bk {

// A word of ones is no value yet.  As a number it is a NaN that arithmetic does not
// make; a result with these bits is stored as the plain NaN.
template <typename V> struct SvWord;
template <> struct SvWord<double> {
    typedef unsigned long long U;
    static constexpr U none = ~0ull, plain_nan = 0x7ff8000000000000ull;
    static __device__ __forceinline__ U bits(double v) { return (U)__double_as_longlong(v); }
    static __device__ __forceinline__ double value(U b) { return __longlong_as_double((long long)b); }
    static __device__ __forceinline__ U load(const U *p)
    {
        U v;
        asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
        return v;
    }
    static __device__ __forceinline__ void store(U *p, U v)
    {
        asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
    }
};
template <> struct SvWord<float> {
    typedef uint32_t U;
    static constexpr U none = ~0u, plain_nan = 0x7fc00000u;
    static __device__ __forceinline__ U bits(float v) { return __float_as_uint(v); }
    static __device__ __forceinline__ float value(U b) { return __uint_as_float(b); }
    static __device__ __forceinline__ U load(const U *p)
    {
        U v;
        asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
        return v;
    }
    static __device__ __forceinline__ void store(U *p, U v)
    {
        asm volatile("st.relaxed.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
    }
};

}  // namespace bk
