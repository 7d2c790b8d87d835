// Quads: the values one thread handles per sign group (four FP32 or BF16, or
// two FP64, consecutive along z), their packed arithmetic and storage access,
// the signed sums over the eight groups and the warp reduction of the seven
// moment sums.  Shared by the step kernel and the moments of a stored f.
#pragma once
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <cstdint>

#include "f2.cuh"

namespace dvm {

// The values one thread handles per group: four FP32 values as two packed
// pairs (FFMA2/FADD2/FMUL2, two lanes per instruction), or two FP64 values.
template <typename TC> struct QV;
template <> struct QV<float> { float2 a, b; };
template <> struct QV<double> { double a, b; };

__device__ inline QV<float> q_splat(float s) { return {make_float2(s, s), make_float2(s, s)}; }
__device__ inline QV<double> q_splat(double s) { return {s, s}; }
__device__ inline QV<float> q_fma(QV<float> x, QV<float> y, QV<float> z)
{
    return {__ffma2_rn(x.a, y.a, z.a), __ffma2_rn(x.b, y.b, z.b)};
}
__device__ inline QV<double> q_fma(QV<double> x, QV<double> y, QV<double> z)
{
    return {fma(x.a, y.a, z.a), fma(x.b, y.b, z.b)};
}
__device__ inline QV<float> q_mul(QV<float> x, QV<float> y) { return {__fmul2_rn(x.a, y.a), __fmul2_rn(x.b, y.b)}; }
__device__ inline QV<double> q_mul(QV<double> x, QV<double> y) { return {x.a * y.a, x.b * y.b}; }
__device__ inline QV<float> q_add(QV<float> x, QV<float> y) { return {__fadd2_rn(x.a, y.a), __fadd2_rn(x.b, y.b)}; }
__device__ inline QV<double> q_add(QV<double> x, QV<double> y) { return {x.a + y.a, x.b + y.b}; }
__device__ inline QV<float> q_neg(QV<float> x) { return {make_float2(-x.a.x, -x.a.y), make_float2(-x.b.x, -x.b.y)}; }
__device__ inline QV<double> q_neg(QV<double> x) { return {-x.a, -x.b}; }
__device__ inline float q_sum(QV<float> x)
{
    const float2 t = __fadd2_rn(x.a, x.b);
    return t.x + t.y;
}
__device__ inline double q_sum(QV<double> x) { return x.a + x.b; }
__device__ inline QV<float> q_make(const float v[4]) { return {make_float2(v[0], v[1]), make_float2(v[2], v[3])}; }
__device__ inline QV<double> q_make(const double v[2]) { return {v[0], v[1]}; }

// storage <-> quads
template <typename TS> struct QIO;
template <> struct QIO<float> {
    __device__ static inline QV<float> ldg(const float *p)
    {
        const float4 t = __ldg(reinterpret_cast<const float4 *>(p));
        return {make_float2(t.x, t.y), make_float2(t.z, t.w)};
    }
    __device__ static inline QV<float> lds(const float *p)
    {
        const float4 t = *reinterpret_cast<const float4 *>(p);
        return {make_float2(t.x, t.y), make_float2(t.z, t.w)};
    }
    __device__ static inline void stg(float *p, QV<float> q)
    {
        __stcs(reinterpret_cast<float4 *>(p), make_float4(q.a.x, q.a.y, q.b.x, q.b.y));
    }
    __device__ static inline void sts(float *p, QV<float> q)
    {
        *reinterpret_cast<float4 *>(p) = make_float4(q.a.x, q.a.y, q.b.x, q.b.y);
    }
};
template <> struct QIO<double> {
    __device__ static inline QV<double> ldg(const double *p)
    {
        const double2 t = __ldg(reinterpret_cast<const double2 *>(p));
        return {t.x, t.y};
    }
    __device__ static inline QV<double> lds(const double *p)
    {
        const double2 t = *reinterpret_cast<const double2 *>(p);
        return {t.x, t.y};
    }
    __device__ static inline void stg(double *p, QV<double> q)
    {
        __stcs(reinterpret_cast<double2 *>(p), make_double2(q.a, q.b));
    }
    __device__ static inline void sts(double *p, QV<double> q) { *reinterpret_cast<double2 *>(p) = make_double2(q.a, q.b); }
};
template <> struct QIO<__nv_bfloat16> {
    __device__ static inline QV<float> cvt(uint2 raw)
    {
        const float2 fa = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&raw.x));
        const float2 fb = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&raw.y));
        return {fa, fb};
    }
    __device__ static inline QV<float> ldg(const __nv_bfloat16 *p) { return cvt(__ldg(reinterpret_cast<const uint2 *>(p))); }
    __device__ static inline QV<float> lds(const __nv_bfloat16 *p) { return cvt(*reinterpret_cast<const uint2 *>(p)); }
    __device__ static inline uint2 pack(QV<float> q)
    {
        const __nv_bfloat162 a = __floats2bfloat162_rn(q.a.x, q.a.y), b = __floats2bfloat162_rn(q.b.x, q.b.y);
        uint2 raw;
        raw.x = *reinterpret_cast<const uint32_t *>(&a);
        raw.y = *reinterpret_cast<const uint32_t *>(&b);
        return raw;
    }
    __device__ static inline void stg(__nv_bfloat16 *p, QV<float> q) { __stcs(reinterpret_cast<uint2 *>(p), pack(q)); }
    __device__ static inline void sts(__nv_bfloat16 *p, QV<float> q) { *reinterpret_cast<uint2 *>(p) = pack(q); }
};

// Warp totals of seven per-lane sums by reduce-scatter: each butterfly level
// sends only the half of the sums that the partner keeps, so that three
// levels leave lane l with the sum (l >> 2) over the eight lanes that differ
// from it in bits 2-4, and two full levels finish it.  9 shuffles instead of
// 35.  Returns, in lane l, the warp total of sum l >> 2 (l < 28).
template <typename TC> __device__ inline TC warp_reduce7(const TC (&m)[7], int lane)
{
    TC a[4], b[2];
    const bool h4 = lane & 16, h3 = lane & 8, h2 = lane & 4;
#pragma unroll
    for (int i = 0; i < 4; i++) {
        const TC lo = m[i], hi = i < 3 ? m[4 + i] : (TC)0;
        a[i] = (h4 ? hi : lo) + __shfl_xor_sync(0xffffffffu, h4 ? lo : hi, 16);
    }
#pragma unroll
    for (int i = 0; i < 2; i++)
        b[i] = (h3 ? a[2 + i] : a[i]) + __shfl_xor_sync(0xffffffffu, h3 ? a[i] : a[2 + i], 8);
    TC c = (h2 ? b[1] : b[0]) + __shfl_xor_sync(0xffffffffu, h2 ? b[0] : b[1], 4);
    c += __shfl_xor_sync(0xffffffffu, c, 2);
    c += __shfl_xor_sync(0xffffffffu, c, 1);
    return c;
}

// Signed sums over the eight sign groups, per position (packed pairs):
// S = sum_o x_o and X, Y, Z = sum_o s_d(o) x_o with s_d = +1 in the groups of
// positive xi_d (group o = 4[xi_x > 0] + 2[xi_y > 0] + [xi_z > 0]).
__device__ inline void group_sums(const float2 (&x)[8], float2 &S, float2 &X, float2 &Y, float2 &Z)
{
    float2 pz[4], mz[4];
#pragma unroll
    for (int k = 0; k < 4; k++) {
        pz[k] = f2_add(x[2 * k], x[2 * k + 1]);
        mz[k] = f2_sub(x[2 * k + 1], x[2 * k]);
    }
    Z = f2_add(f2_add(mz[0], mz[1]), f2_add(mz[2], mz[3]));
    const float2 pp0 = f2_add(pz[0], pz[1]), pm0 = f2_sub(pz[1], pz[0]);
    const float2 pp1 = f2_add(pz[2], pz[3]), pm1 = f2_sub(pz[3], pz[2]);
    Y = f2_add(pm0, pm1);
    S = f2_add(pp0, pp1);
    X = f2_sub(pp1, pp0);
}

}  // namespace dvm
