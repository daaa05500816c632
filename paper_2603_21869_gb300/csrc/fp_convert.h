// FP32 to FP64 and back by integer operations (the IEEE 754 layouts), for kernels that sum FP32 values in
// FP64: the conversion instructions run at a fraction of the FP64 rate, itself two lanes a clock and SM
// here (the FP64 residual of 430,080 cells 44 us a launch with them, 32 us without; the flexible-CG
// pair 51 and 35 us).  Denormal, infinite and NaN values take the instruction.  Plain C++ as well as CUDA.
#pragma once
#include <cstdint>
#include <cstring>

#ifdef __CUDACC__
#define FVM_HD __host__ __device__ __forceinline__
#define FVM_HD_RARE __host__ __device__ __noinline__   // (out of line: not predicated into the common path)
#else
#define FVM_HD inline
#define FVM_HD_RARE inline
#endif

template <class To, class From>
FVM_HD To same_bits(From x) {
    static_assert(sizeof(To) == sizeof(From), "sizes");
    To y;
    memcpy(&y, &x, sizeof(y));
    return y;
}

FVM_HD_RARE static double widened_rare(float x) { return (double)x; }
FVM_HD_RARE static float narrowed_rare(double x) { return (float)x; }

// (double)x of several values: one test for all of them, so that their chains overlap
template <int N>
FVM_HD void widened(const float (&x)[N], double (&y)[N]) {
    bool rare = false;
#ifdef __CUDACC__
#pragma unroll
#endif
    for (int i = 0; i < N; ++i) {
        const uint32_t u = same_bits<uint32_t>(x[i]), t = u & 0x7fffffffu;
        rare |= t != 0u && t - 0x00800000u >= 0x7f000000u;
        const uint32_t hi = (u & 0x80000000u) | (t != 0u ? (t >> 3) + (896u << 20) : 0u);
        y[i] = same_bits<double>(((uint64_t)hi << 32) | (uint64_t)(u << 29));
    }
    if (rare) {
#ifdef __CUDACC__
#pragma unroll
#endif
        for (int i = 0; i < N; ++i) y[i] = widened_rare(x[i]);
    }
}

// (float)x, to nearest even
template <int N>
FVM_HD void narrowed(const double (&x)[N], float (&y)[N]) {
    bool rare = false;
#ifdef __CUDACC__
#pragma unroll
#endif
    for (int i = 0; i < N; ++i) {
        const uint64_t u = same_bits<uint64_t>(x[i]), t = u & 0x7fffffffffffffffull;
        const uint64_t q = (t + 0x0fffffffull + ((t >> 29) & 1ull)) >> 29;   // rounded: FP64's exponent, FP32's mantissa
        rare |= t != 0ull && q - ((uint64_t)897 << 23) >= ((uint64_t)254 << 23);
        const uint32_t f = (uint32_t)(q - ((uint64_t)896 << 23));
        y[i] = same_bits<float>(((uint32_t)(u >> 32) & 0x80000000u) | (t != 0ull ? f : 0u));
    }
    if (rare) {
#ifdef __CUDACC__
#pragma unroll
#endif
        for (int i = 0; i < N; ++i) y[i] = narrowed_rare(x[i]);
    }
}
// values that are of the type already
template <class T, int N>
FVM_HD void widened(const T (&x)[N], T (&y)[N]) {
    for (int i = 0; i < N; ++i) y[i] = x[i];
}
template <class T, int N>
FVM_HD void narrowed(const T (&x)[N], T (&y)[N]) {
    for (int i = 0; i < N; ++i) y[i] = x[i];
}
