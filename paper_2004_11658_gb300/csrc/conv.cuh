// conv.cuh -- conversions between FP32 and FP64 on the integer pipe (the FP64 pipe
// takes 16 cycles per warp instruction, conversions included): exact, and rounded
// to nearest even, for normal FP32 results; zero, subnormal and non-finite values
// take the instruction.  Bit for bit the values of the casts (a NaN stays a NaN).
#pragma once

#include <cstdint>
#include <cstring>

#include <cuda_runtime.h>

template <class TO, class FROM>
static __host__ __device__ __forceinline__ TO dp_bits(FROM v)
{
    static_assert(sizeof(TO) == sizeof(FROM), "bits of the same size");
    TO r;
    memcpy(&r, &v, sizeof(r));
    return r;
}

static __host__ __device__ __forceinline__ double f2d(float v)
{
    const uint32_t u = dp_bits<uint32_t>(v), e = (u >> 23) & 0xff;
    if (e == 0 || e == 0xff) return (u << 1) == 0 ? dp_bits<double>((uint64_t)u << 32) : (double)v;
    const uint32_t hi = (u & 0x80000000u) | (((u >> 3) & 0x0fffffffu) + 0x38000000u);
    return dp_bits<double>(((uint64_t)hi << 32) | (u << 29));
}

static __host__ __device__ __forceinline__ float d2f(double v)
{
    const uint64_t b = dp_bits<uint64_t>(v), r = b + 0x0fffffffull + ((b >> 29) & 1ull);
    const uint32_t e = (uint32_t)(r >> 52) & 0x7ff;
    if (e < 897 || e > 1150) return (b << 1) == 0 ? dp_bits<float>((uint32_t)(b >> 32)) : (float)v;
    return dp_bits<float>(((uint32_t)(b >> 32) & 0x80000000u) | ((e - 896) << 23) | ((uint32_t)(r >> 29) & 0x7fffffu));
}
