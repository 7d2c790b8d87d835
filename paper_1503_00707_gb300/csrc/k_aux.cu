// Auxiliary kernels outside the timed step: Maxwellian initialisation,
// moments of the stored f, and precision conversions for host transfers.
#include <algorithm>
#include <cmath>

#include "../../include/dvm.h"
#include "async.cuh"
#include "common.cuh"
#include "kernels.hpp"
#include "quads.cuh"

namespace dvm {

void count_launch();

namespace {

template <typename TS> __device__ inline TS from_double(double v);
template <> __device__ inline double from_double<double>(double v) { return v; }
template <> __device__ inline float from_double<float>(double v) { return (float)v; }
template <> __device__ inline __nv_bfloat16 from_double<__nv_bfloat16>(double v) { return __double2bfloat16(v); }

template <typename TS> __device__ inline double to_double(TS v);
template <> __device__ inline double to_double<double>(double v) { return v; }
template <> __device__ inline double to_double<float>(float v) { return (double)v; }
template <> __device__ inline double to_double<__nv_bfloat16>(__nv_bfloat16 v) { return (double)__bfloat162float(v); }

// M(rho, u, T; xi) = rho (2 pi T)^(-3/2) exp(-|xi - u|^2 / (2T)), FP64
template <typename TS>
__global__ void k_init(TS *f, int64_t ncells, int nv, int nmix, const double *w, const double *rho,
                       const double *u, const double *T, const double *xi)
{
    const int64_t total = ncells * (int64_t)nv;
    for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < total;
         q += (int64_t)gridDim.x * blockDim.x) {
        const int64_t c = q / nv;
        const int v = (int)(q - c * nv);
        double s = 0.0;
        for (int m = 0; m < nmix; m++) {
            const int64_t k = c * nmix + m;
            double d2 = 0.0;
            for (int d = 0; d < 3; d++) {
                const double t = xi[3 * v + d] - u[3 * k + d];
                d2 += t * t;
            }
            const double tp = 2.0 * 3.14159265358979323846 * T[k];
            s += w[k] * rho[k] / (tp * sqrt(tp)) * exp(-d2 / (2.0 * T[k]));
        }
        f[q] = from_double<TS>(s);
    }
}

// Moments of a stored f: rho, u, T of every cell in FP64, one CTA per cell.
//
// A value enters only through the seven integer-weighted sums sum f,
// sum j_d f, sum j_d^2 f (xi_d = (h_d/2) j_d, j_d odd).  FP64 runs at 1/64 of
// the FP32 rate here and thirteen FP64 operations a value bound the kernel at
// 57 GB/s of its read of f, so FP32 and BF16 storage sum exactly in fixed
// point instead: with M the cell's largest |f| and sigma = 2^k >= 512 M, each
// value splits without error (the extraction of Rump, Ogita and Oishi, 2008)
// into a multiple of 2^(k-24), a multiple of 2^(k-39) and a rest of at most
// 2^(k-39).  A thread's sums of its 32 values of either multiple, with the
// weights that k_step's partials use (total size below 16 against the split's
// margin), are exact in FP32 and go into 64-bit integers; the rests are summed
// in FP32.  What is lost is below 2^-60 of sum |f|, less than FP64 summation
// loses.  A cell with non-finite values or M outside [2^-86, 2^115] takes FP64
// sums.
//
// f is read once from HBM and twice by its thread, for M and for the sums.
// Cells of up to 56 KB go through shared memory (PIPE): a CTA takes every
// gridDim-th cell, and each thread copies its own pieces of the next one with
// cp.async while it sums this one, so that the stream does not stop for the
// barriers and the FP64 tail of a cell.  Larger cells are read from memory
// twice.  17,680 cells x 24^3, FP32 (0.98 GB): 4,110 us with FP64 sums, 319 us
// with the cell held in registers (one cell per CTA), 283 us through
// shared memory; what bounds it now is the arithmetic of the split at 14 warps
// an SM.
constexpr int MOM_T = 256;
constexpr size_t MOM_ROW = 56 * 1024;

__device__ inline uint32_t abs_bits(float2 v) { return max(__float_as_uint(v.x) & 0x7fffffffu, __float_as_uint(v.y) & 0x7fffffffu); }

// the seven base sums of a quad at one level of the split, times 2^-quantum
// as integers: S, X, Y, Z over the four positions, sum e Z_e, sum e S_e,
// sum e^2 S_e (e = 0..3)
__device__ inline void base_sums(const float2 (&a)[8], const float2 (&b)[8], float (&s)[7])
{
    float2 Sa, Xa, Ya, Za, Sb, Xb, Yb, Zb;
    group_sums(a, Sa, Xa, Ya, Za);
    group_sums(b, Sb, Xb, Yb, Zb);
    s[0] = (Sa.x + Sa.y) + (Sb.x + Sb.y);
    s[1] = (Xa.x + Xa.y) + (Xb.x + Xb.y);
    s[2] = (Ya.x + Ya.y) + (Yb.x + Yb.y);
    s[3] = (Za.x + Za.y) + (Zb.x + Zb.y);
    s[4] = (Za.y + 2.0f * Zb.x) + 3.0f * Zb.y;
    s[5] = (Sa.y + 2.0f * Sb.x) + 3.0f * Sb.y;
    s[6] = (Sa.y + 4.0f * Sb.x) + 9.0f * Sb.y;
}

// the seven weighted sums from the base sums (j = j0 + 2 e along z)
template <typename T, typename J> __device__ inline void weighted_sums(const T (&s)[7], J jx, J jy, J jz, T (&m)[7])
{
    m[0] += s[0];
    m[1] += s[1] * jx;
    m[2] += s[2] * jy;
    m[3] += s[3] * jz + s[4] * (J)2;
    m[4] += s[0] * (jx * jx);
    m[5] += s[0] * (jy * jy);
    m[6] += s[0] * (jz * jz) + s[5] * (J)(4 * jz) + s[6] * (J)4;
}

// split a thread's 32 values at one level: x = q + r, q a multiple of
// sigma 2^-24
__device__ inline void extract8(float2 (&x)[8], float sigma, float2 (&q)[8])
{
    const float2 s2 = make_float2(sigma, sigma);
#pragma unroll
    for (int o = 0; o < 8; o++) {
        q[o] = f2_sub(f2_add(x[o], s2), s2);
        x[o] = f2_sub(x[o], q[o]);
    }
}

struct MomSum {
    int64_t I[7];  // in units of 2^(k-39)
    float R[7];
};

__device__ inline void add_quad(const QV<float> (&x)[8], int ex, int jx, int jy, int jz, MomSum &m)
{
    const float sg1 = __int_as_float((ex + 10) << 23), sg2 = __int_as_float((ex - 5) << 23);  // 2^k, 2^(k-15)
    const float c1 = __int_as_float((268 - ex) << 23), c2 = __int_as_float((283 - ex) << 23);  // 2^(24-k), 2^(39-k)
    float2 ra[8], rb[8], qa[8], qb[8];
#pragma unroll
    for (int o = 0; o < 8; o++) {
        ra[o] = x[o].a;
        rb[o] = x[o].b;
    }
    float s1[7], s2[7], s3[7];
    extract8(ra, sg1, qa);
    extract8(rb, sg1, qb);
    base_sums(qa, qb, s1);
    extract8(ra, sg2, qa);
    extract8(rb, sg2, qb);
    base_sums(qa, qb, s2);
    base_sums(ra, rb, s3);
    int64_t v[7];
#pragma unroll
    for (int k = 0; k < 7; k++)
        v[k] = (int64_t)__float2int_rn(s1[k] * c1) * 32768 + (int64_t)__float2int_rn(s2[k] * c2);
    weighted_sums<int64_t, int>(v, jx, jy, jz, m.I);
    weighted_sums<float, float>(s3, (float)jx, (float)jy, (float)jz, m.R);
}

// the same sums in FP64
template <typename TC> __device__ inline void add_quad_f64(const QV<TC> (&x)[8], int jx, int jy, int jz, double (&m)[7])
{
    constexpr int VEC = sizeof(TC) == 8 ? 2 : 4;
    double s[7] = {0, 0, 0, 0, 0, 0, 0};
#pragma unroll 1
    for (int e = 0; e < VEC; e++) {
        double S = 0, X = 0, Y = 0, Z = 0;
#pragma unroll
        for (int o = 0; o < 8; o++) {
            double v;
            if constexpr (sizeof(TC) == 8) v = e ? x[o].b : x[o].a;
            else v = (double)(e == 0 ? x[o].a.x : e == 1 ? x[o].a.y : e == 2 ? x[o].b.x : x[o].b.y);
            S += v;
            X += (o & 4) ? v : -v;
            Y += (o & 2) ? v : -v;
            Z += (o & 1) ? v : -v;
        }
        s[0] += S;
        s[1] += X;
        s[2] += Y;
        s[3] += Z;
        s[4] += e * Z;
        s[5] += e * S;
        s[6] += e * e * S;
    }
    weighted_sums<double, double>(s, (double)jx, (double)jy, (double)jz, m);
}

template <typename TS, bool PIPE>
__global__ void __launch_bounds__(MOM_T, 2)
    k_moments(const TS *__restrict__ f, int64_t ncells, int P, int3 half, double3 hh, double dV, double *__restrict__ out)
{
    using IO = QIO<TS>;
    using TC = typename Store<TS>::TC;
    constexpr int VEC = Store<TS>::VEC;
    extern __shared__ __align__(16) unsigned char mom_tile[];  // PIPE: [2][8 P]
    __shared__ uint32_t wmax[MOM_T / 32];
    __shared__ double red[MOM_T / 32][7];
    __shared__ int64_t redI[MOM_T / 32][7];
    __shared__ float redR[MOM_T / 32][7];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, T = blockDim.x, nw = T >> 5, Q = P / VEC;
    TS *tile = reinterpret_cast<TS *>(mom_tile);
    // the thread's pieces of cell c into buffer b (each thread reads back only
    // what it copied)
    auto copy = [&](int64_t c, int b) {
        if (c < ncells)
            for (int q = tid; q < Q; q += T)
#pragma unroll
                for (int o = 0; o < 8; o++) {
                    const TS *src = f + (c * 8 + o) * (int64_t)P + q * VEC;
                    TS *dst = tile + (size_t)(b * 8 + o) * P + q * VEC;
                    if constexpr (sizeof(TS) == 2) cp_async8(dst, src, 0u);
                    else cp_async16(dst, src, 0u);
                }
        cp_async_commit();
    };
    auto nodes = [&](int q, int &jx, int &jy, int &jz) {
        const int p = q * VEC, t = p / half.z;
        jz = 2 * (p - t * half.z) + 1;
        jy = 2 * (t % half.y) + 1;
        jx = 2 * (t / half.y) + 1;
    };
    if constexpr (PIPE) copy(blockIdx.x, 0);
    int buf = 0;
    for (int64_t c = blockIdx.x; c < ncells; c += gridDim.x, buf ^= 1) {
        if constexpr (PIPE) {
            // the other buffer's values were all used before this cell's
            // predecessor reached its barriers
            copy(c + gridDim.x, buf ^ 1);
            cp_async_wait<1>();
        }
        auto load = [&](int q, QV<TC> (&x)[8]) {
#pragma unroll
            for (int o = 0; o < 8; o++) {
                if constexpr (PIPE) x[o] = IO::lds(tile + (size_t)(buf * 8 + o) * P + q * VEC);
                else x[o] = IO::ldg(f + (c * 8 + o) * (int64_t)P + q * VEC);
            }
        };
        int jx, jy, jz;
        bool wide = true;  // FP64 sums
        int ex = 0;
        if constexpr (sizeof(TC) == 4) {
            uint32_t mx = 0;
            for (int q = tid; q < Q; q += T) {
                QV<float> x[8];
                load(q, x);
#pragma unroll
                for (int o = 0; o < 8; o++) mx = max(mx, max(abs_bits(x[o].a), abs_bits(x[o].b)));
            }
            mx = __reduce_max_sync(0xffffffffu, mx);
            if (lane == 0) wmax[warp] = mx;
            __syncthreads();
            for (int w = 0; w < nw; w++) mx = max(mx, wmax[w]);
            ex = (int)(mx >> 23);  // M < 2^(ex - 126)
            wide = ex < 40 || ex > 240;
            if (!wide) {
                MomSum m{};
#pragma unroll 1
                for (int q = tid; q < Q; q += T) {
                    QV<float> x[8];
                    load(q, x);
                    nodes(q, jx, jy, jz);
                    add_quad(x, ex, jx, jy, jz, m);
                }
                const int64_t I = warp_reduce7<int64_t>(m.I, lane);
                const float R = warp_reduce7<float>(m.R, lane);
                if ((lane & 3) == 0 && lane < 28) {
                    redI[warp][lane >> 2] = I;
                    redR[warp][lane >> 2] = R;
                }
            }
        }
        if (wide) {
            double m[7] = {0, 0, 0, 0, 0, 0, 0};
#pragma unroll 1
            for (int q = tid; q < Q; q += T) {
                QV<TC> x[8];
                load(q, x);
                nodes(q, jx, jy, jz);
                add_quad_f64<TC>(x, jx, jy, jz, m);
            }
            const double t = warp_reduce7<double>(m, lane);
            if ((lane & 3) == 0 && lane < 28) red[warp][lane >> 2] = t;
        }
        __syncthreads();
        if (warp == 0) {
            double s = 0.0;
            if (lane < 7) {
                if (wide) {
                    for (int w = 0; w < nw; w++) s += red[w][lane];
                } else {
                    int64_t I = 0;
                    float R = 0.0f;
                    for (int w = 0; w < nw; w++) {
                        I += redI[w][lane];
                        R += redR[w][lane];
                    }
                    s = (double)I * __longlong_as_double((long long)(1023 + ex - 156) << 52) + (double)R;  // 2^(k-39)
                }
            }
            // lane 0: sum f; 1..3: u_d; 4..6: sum xi_d^2 f / sum f
            const double s0 = __shfl_sync(0xffffffffu, s, 0);
            const int d = (lane + 2) % 3;
            const double h1 = d == 0 ? hh.x : (d == 1 ? hh.y : hh.z);
            const double v = s / s0 * (lane < 4 ? h1 : h1 * h1);
            const double u2 = v * v, e2 = __shfl_down_sync(0xffffffffu, v, 3);
            const double ux2 = __shfl_sync(0xffffffffu, u2, 1), uy2 = __shfl_sync(0xffffffffu, u2, 2),
                         uz2 = __shfl_sync(0xffffffffu, u2, 3);
            const double ex2 = __shfl_sync(0xffffffffu, e2, 1), ey2 = __shfl_sync(0xffffffffu, e2, 2),
                         ez2 = __shfl_sync(0xffffffffu, e2, 3);
            double *o = out + c * 5;
            if (lane == 0) {
                o[0] = s0 * dV;
                o[4] = (ex2 + ey2 + ez2 - (ux2 + uy2 + uz2)) / 3.0;
            } else if (lane < 4) {
                o[lane] = v;
            }
        }
        if (sizeof(TC) == 8) __syncthreads();  // red is read above (FP32: the next cell's first barrier)
    }
    if constexpr (PIPE) cp_async_wait_all();
}

template <typename TS>
__global__ void k_to_f64(const TS *src, double *dst, int64_t n)
{
    for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < n; q += (int64_t)gridDim.x * blockDim.x)
        dst[q] = to_double<TS>(src[q]);
}

template <typename TS>
__global__ void k_from_f64(const double *src, TS *dst, int64_t n)
{
    for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < n; q += (int64_t)gridDim.x * blockDim.x)
        dst[q] = from_double<TS>(src[q]);
}

inline unsigned blocks_for(int64_t n, int threads)
{
    int64_t b = (n + threads - 1) / threads;
    if (b > 152 * 64) b = 152 * 64;
    if (b < 1) b = 1;
    return (unsigned)b;
}

int last_status()
{
    count_launch();
    return cudaGetLastError() == cudaSuccess ? DVM_OK : DVM_ECUDA;
}

template <typename TS> int moments_t(const void *f, int64_t ncells, const MomGrid &g, double *out, cudaStream_t s)
{
    const int P = g.half[0] * g.half[1] * g.half[2], Q = P / Store<TS>::VEC;
    // one quad a thread up to 256 quads, then two or more, evenly (24^3: 432
    // quads on 224 threads)
    const int rounds = (Q + MOM_T - 1) / MOM_T, t = ((Q + rounds - 1) / rounds + 31) / 32 * 32;
    const int3 half = make_int3(g.half[0], g.half[1], g.half[2]);
    const double3 hh = make_double3(0.5 * g.hv[0], 0.5 * g.hv[1], 0.5 * g.hv[2]);
    const TS *ft = static_cast<const TS *>(f);
    const size_t row = (size_t)8 * P * sizeof(TS);
    if (row > MOM_ROW) {
        k_moments<TS, false><<<(unsigned)ncells, t, 0, s>>>(ft, ncells, P, half, hh, g.dV, out);
        return last_status();
    }
    auto kern = k_moments<TS, true>;
    int dev = 0, nsm = 0, occ = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(2 * MOM_ROW)) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, t, 2 * row) != cudaSuccess || occ < 1)
        return DVM_ECUDA;
    kern<<<(unsigned)std::min<int64_t>(ncells, (int64_t)nsm * occ), t, 2 * row, s>>>(ft, ncells, P, half, hh, g.dV, out);
    return last_status();
}

// Row copies between buffers: entry r of rows is {destination buffer, row,
// source buffer, row}; rows are row_bytes long (a multiple of 16).
__global__ void k_copy_rows(void *const *bufs, const int64_t *rows, int64_t n, int64_t row_bytes)
{
    const int64_t n16 = row_bytes / 16;
    for (int64_t r = blockIdx.x; r < n; r += gridDim.x) {
        const int64_t *e = rows + 4 * r;
        const uint4 *src = reinterpret_cast<const uint4 *>(static_cast<const char *>(bufs[e[2]]) + e[3] * row_bytes);
        uint4 *dst = reinterpret_cast<uint4 *>(static_cast<char *>(bufs[e[0]]) + e[1] * row_bytes);
        for (int64_t i = threadIdx.x; i < n16; i += blockDim.x) dst[i] = src[i];
    }
}

// Halo pack and unpack: dst row r = src row idx[r] (gather), or dst row
// idx[r] = src row r (scatter); rows are row_bytes long (a multiple of 16).
template <bool GATHER>
__global__ void k_rows_indexed(char *dst, const char *src, const int64_t *idx, int64_t n, int64_t row_bytes)
{
    const int64_t n16 = row_bytes / 16;
    for (int64_t r = blockIdx.x; r < n; r += gridDim.x) {
        const int64_t rd = GATHER ? r : idx[r], rs = GATHER ? idx[r] : r;
        const uint4 *a = reinterpret_cast<const uint4 *>(src + rs * row_bytes);
        uint4 *b = reinterpret_cast<uint4 *>(dst + rd * row_bytes);
        for (int64_t i = threadIdx.x; i < n16; i += blockDim.x) b[i] = a[i];
    }
}

// Row means: destination row r of dst is the mean of source rows
// idx[start[r] .. start[r+1]) of src (nv values each, storage precision;
// the sum in FP64 for FP64 storage, FP32 otherwise).
template <typename T, typename A>
__global__ void k_mean_rows(T *dst, const T *src, const int64_t *start, const int64_t *idx, int64_t nrows, int nv)
{
    for (int64_t r = blockIdx.x; r < nrows; r += gridDim.x) {
        const int64_t b = start[r], e = start[r + 1];
        const A inv = A(1) / A(e - b);
        for (int v = threadIdx.x; v < nv; v += blockDim.x) {
            A acc = A(0);
            for (int64_t k = b; k < e; k++) acc += (A)src[idx[k] * nv + v];
            dst[r * nv + v] = (T)(acc * inv);
        }
    }
}

}  // namespace

int launch_mean_rows(int prec, void *dst, const void *src, const int64_t *start, const int64_t *idx, int64_t nrows,
                     int nv, cudaStream_t s)
{
    if (nrows <= 0) return DVM_OK;
    const unsigned grid = (unsigned)std::min<int64_t>(nrows, 1 << 16);
    switch (prec) {
    case DVM_F64: k_mean_rows<double, double><<<grid, 256, 0, s>>>((double *)dst, (const double *)src, start, idx, nrows, nv); break;
    case DVM_F32: k_mean_rows<float, float><<<grid, 256, 0, s>>>((float *)dst, (const float *)src, start, idx, nrows, nv); break;
    case DVM_BF16:
        k_mean_rows<__nv_bfloat16, float><<<grid, 256, 0, s>>>((__nv_bfloat16 *)dst, (const __nv_bfloat16 *)src, start,
                                                               idx, nrows, nv);
        break;
    default: return DVM_EINVAL;
    }
    count_launch();
    return cudaGetLastError() == cudaSuccess ? DVM_OK : DVM_ECUDA;
}

int launch_copy_rows(void *const *bufs, const int64_t *rows, int64_t n, int64_t row_bytes, cudaStream_t s)
{
    if (n <= 0) return DVM_OK;
    if (row_bytes % 16 != 0) return DVM_EINVAL;
    const unsigned grid = (unsigned)std::min<int64_t>(n, 1 << 16);
    k_copy_rows<<<grid, 256, 0, s>>>(bufs, rows, n, row_bytes);
    count_launch();
    return cudaGetLastError() == cudaSuccess ? DVM_OK : DVM_ECUDA;
}

int launch_rows_indexed(bool gather, void *dst, const void *src, const int64_t *idx, int64_t n, int64_t row_bytes,
                        cudaStream_t s)
{
    if (n <= 0) return DVM_OK;
    if (row_bytes % 16 != 0) return DVM_EINVAL;
    const unsigned grid = (unsigned)std::min<int64_t>(n, 1 << 16);
    if (gather)
        k_rows_indexed<true><<<grid, 256, 0, s>>>(static_cast<char *>(dst), static_cast<const char *>(src), idx, n,
                                                  row_bytes);
    else
        k_rows_indexed<false><<<grid, 256, 0, s>>>(static_cast<char *>(dst), static_cast<const char *>(src), idx, n,
                                                   row_bytes);
    count_launch();
    return cudaGetLastError() == cudaSuccess ? DVM_OK : DVM_ECUDA;
}

int launch_init_maxwellian(int prec, void *f, int64_t ncells, int nv, int nmix, const double *w,
                           const double *rho, const double *u, const double *T, const double *xi,
                           cudaStream_t s)
{
    const int64_t n = ncells * (int64_t)nv;
    const unsigned b = blocks_for(n, 256);
    switch (prec) {
    case DVM_F64: k_init<double><<<b, 256, 0, s>>>((double *)f, ncells, nv, nmix, w, rho, u, T, xi); break;
    case DVM_F32: k_init<float><<<b, 256, 0, s>>>((float *)f, ncells, nv, nmix, w, rho, u, T, xi); break;
    case DVM_BF16: k_init<__nv_bfloat16><<<b, 256, 0, s>>>((__nv_bfloat16 *)f, ncells, nv, nmix, w, rho, u, T, xi); break;
    default: return DVM_EINVAL;
    }
    return last_status();
}

int launch_moments(int prec, const void *f, int64_t ncells, const MomGrid &g, double *out, cudaStream_t s)
{
    if (ncells <= 0) return DVM_OK;
    switch (prec) {
    case DVM_F64: return moments_t<double>(f, ncells, g, out, s);
    case DVM_F32: return moments_t<float>(f, ncells, g, out, s);
    case DVM_BF16: return moments_t<__nv_bfloat16>(f, ncells, g, out, s);
    default: return DVM_EINVAL;
    }
}

int launch_to_f64(int prec, const void *src, double *dst, int64_t n, cudaStream_t s)
{
    const unsigned b = blocks_for(n, 256);
    switch (prec) {
    case DVM_F64: k_to_f64<double><<<b, 256, 0, s>>>((const double *)src, dst, n); break;
    case DVM_F32: k_to_f64<float><<<b, 256, 0, s>>>((const float *)src, dst, n); break;
    case DVM_BF16: k_to_f64<__nv_bfloat16><<<b, 256, 0, s>>>((const __nv_bfloat16 *)src, dst, n); break;
    default: return DVM_EINVAL;
    }
    return last_status();
}

int launch_from_f64(int prec, const double *src, void *dst, int64_t n, cudaStream_t s)
{
    const unsigned b = blocks_for(n, 256);
    switch (prec) {
    case DVM_F64: k_from_f64<double><<<b, 256, 0, s>>>(src, (double *)dst, n); break;
    case DVM_F32: k_from_f64<float><<<b, 256, 0, s>>>(src, (float *)dst, n); break;
    case DVM_BF16: k_from_f64<__nv_bfloat16><<<b, 256, 0, s>>>(src, (__nv_bfloat16 *)dst, n); break;
    default: return DVM_EINVAL;
    }
    return last_status();
}

}  // namespace dvm
