// Packed FP32 pairs (two lanes per instruction on the device), rounded once
// per operation; on the host the same operations one lane after the other, for
// code whose roundings are checked there.
#pragma once
#include <cuda_runtime.h>

#include <cmath>
#include <cstdint>
#include <cstring>

#ifdef __CUDACC__
#define DVM_HD __host__ __device__ __forceinline__
#else
#define DVM_HD inline
#endif

namespace dvm {

DVM_HD float f_mul(float a, float b)
{
#ifdef __CUDA_ARCH__
    return __fmul_rn(a, b);  // never contracted with a following addition
#else
    return a * b;
#endif
}

DVM_HD uint32_t f_bits(float a)
{
#ifdef __CUDA_ARCH__
    return __float_as_uint(a);
#else
    uint32_t u;
    std::memcpy(&u, &a, 4);
    return u;
#endif
}

DVM_HD float bits_f(uint32_t u)
{
#ifdef __CUDA_ARCH__
    return __uint_as_float(u);
#else
    float a;
    std::memcpy(&a, &u, 4);
    return a;
#endif
}

DVM_HD float2 f2_add(float2 a, float2 b)
{
#ifdef __CUDA_ARCH__
    return __fadd2_rn(a, b);
#else
    return make_float2(a.x + b.x, a.y + b.y);
#endif
}

DVM_HD float2 f2_mul(float2 a, float2 b)
{
#ifdef __CUDA_ARCH__
    return __fmul2_rn(a, b);
#else
    return make_float2(a.x * b.x, a.y * b.y);
#endif
}

DVM_HD float2 f2_fma(float2 a, float2 b, float2 c)
{
#ifdef __CUDA_ARCH__
    return __ffma2_rn(a, b, c);
#else
    return make_float2(std::fma(a.x, b.x, c.x), std::fma(a.y, b.y, c.y));
#endif
}

// b - a, rounded once
DVM_HD float2 f2_sub(float2 b, float2 a) { return f2_fma(a, make_float2(-1.0f, -1.0f), b); }

}  // namespace dvm
