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
// point instead: with 2^m above a warp's largest |f|, each of its values splits
// without error (the extraction of Rump, Ogita and Oishi, 2008) into multiples
// of u1 = 2^(m-17), u2 = 2^(m-35) and u3 = 2^(m-53) and a rest of at most u3/2.
// A thread's sums of its 32 values of each multiple, with the weights that
// k_step's partials use (total size at most 112), stay below 2^24 units, hence
// exact in FP32, and go into 64-bit integers; the rests (of values below
// 2^(m-30)) are summed in FP32, in at most 60 additions a value: off by less
// than 60 2^-24 2^-54 2^m a value, 2^-60 of the warp's sum of |f| at 24^3, and
// their total is rounded to u3.  The warps' sums are added in FP64.  Two
// multiples and the rests in FP32 instead (rests of 2^-30 of the cell's largest
// value) took 283 us where this takes 282, but were up to 9.5e-13 of sum |f| off
// on values of that size, FP64 sums 1.1e-15.  A warp with non-finite values or
// its largest above 2^115 takes FP64 sums; one with its largest below 2^-71
// scales its values by 2^96.
//
// f is read once from HBM and twice by its thread, for m and for the sums.
// Cells of up to 56 KB go through shared memory (PIPE): a CTA takes every
// gridDim-th cell by bulk copies, two at a time.  With SPLIT a last warp
// finishes the cells (FP64, a long serial chain) and refills their buffers while
// the others go on (17,680 cells, calls of 16^3 184 -> 167 us, 24^3 376 -> 357);
// a CTA of one working warp does it itself (8^3 115 us, 128 with SPLIT).  Larger
// cells are read from memory twice.  17,680 cells x 24^3, FP32 (0.98 GB): 4,110
// us with FP64 sums, 282 us now; what bounds it is the arithmetic of the split,
// about 800 instructions for a warp's 1,024 values at 54% of the issue slots.
constexpr int MOM_T = 224, MOM_FP64 = 1 << 20;
constexpr size_t MOM_ROW = 56 * 1024;

// the largest of |a|, |b|, |c|, NaN if one is
__device__ inline float max_abs(float a, float b, float c)
{
    float m;
    asm("max.NaN.abs.f32 %0, %1, %2, %3;" : "=f"(m) : "f"(a), "f"(b), "f"(c));
    return m;
}

// the seven base sums of a quad at one level of the split, times 2^-quantum
// as integers: S, X, Y, Z over the four positions, sum e Z_e, sum e S_e,
// sum e^2 S_e (e = 0..3)
__device__ inline void base_sums(const float2 (&a)[8], const float2 (&b)[8], float (&s)[7])
{
    float2 Sa, Xa, Ya, Za, Sb, Xb, Yb, Zb;
    group_sums(a, Sa, Xa, Ya, Za);
    group_sums(b, Sb, Xb, Yb, Zb);
    const float2 St = f2_add(Sa, Sb), Xt = f2_add(Xa, Xb), Yt = f2_add(Ya, Yb), Zt = f2_add(Za, Zb);
    s[0] = St.x + St.y;
    s[1] = Xt.x + Xt.y;
    s[2] = Yt.x + Yt.y;
    s[3] = Zt.x + Zt.y;
    s[4] = (Za.y + 2.0f * Zb.x) + 3.0f * Zb.y;
    s[5] = (Sa.y + 2.0f * Sb.x) + 3.0f * Sb.y;
    s[6] = (Sa.y + 4.0f * Sb.x) + 9.0f * Sb.y;
}

// the seven weighted sums from the base sums (j = j0 + 2 e along z)
template <typename T> __device__ inline void weighted_sums(const T (&s)[7], T jx, T jy, T jz, T (&m)[7])
{
    using J = T;
    m[0] += s[0];
    m[1] += s[1] * jx;
    m[2] += s[2] * jy;
    m[3] += s[3] * jz + s[4] * (J)2;
    m[4] += s[0] * (jx * jx);
    m[5] += s[0] * (jy * jy);
    m[6] += s[0] * (jz * jz) + s[5] * (J)(4 * jz) + s[6] * (J)4;
}

// 1.5 2^(e - 127): an x of at most 2^(e - 128) splits against it into a multiple
// of 2^(e - 150) and a rest of at most half of that
__device__ inline float sigma_of(int e) { return __int_as_float((e << 23) | 0x400000); }

// the same in integers, times k: one 32 x 32 + 64 bit multiply-add a term (left
// to the compiler the call of 17,680 cells x 24^3 takes 750 us, so 737)
__device__ inline void weighted_sums(const int (&s)[7], int jx, int jy, int jz, int k, int64_t (&m)[7])
{
    auto add = [&](int i, int v, int w) {
        asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(m[i]) : "r"(v), "r"(w * k));
    };
    add(0, s[0], 1);
    add(1, s[1], jx);
    add(2, s[2], jy);
    add(3, s[3], jz);
    add(3, s[4], 2);
    add(4, s[0], jx * jx);
    add(5, s[0], jy * jy);
    add(6, s[0], jz * jz);
    add(6, s[5], 4 * jz);
    add(6, s[6], 4);
}

// split a thread's 32 values at one level: x = q + r
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
    int64_t hi[7], lo[7];  // in units of u1 and u3
    float R[7];
};

__device__ inline uint32_t any_bits(const float2 (&a)[8], const float2 (&b)[8])
{
    uint32_t v = 0;
#pragma unroll
    for (int o = 0; o < 8; o++)
        v |= __float_as_uint(a[o].x) | __float_as_uint(a[o].y) | __float_as_uint(b[o].x) | __float_as_uint(b[o].y);
    return v & 0x7fffffffu;
}

// m = ex - 126; COARSE: values of 8 significant bits (BF16)
template <bool COARSE> __device__ inline void add_quad(const QV<float> (&x)[8], int ex, int jx, int jy, int jz, MomSum &m)
{
    float2 ra[8], rb[8], qa[8], qb[8];
#pragma unroll
    for (int o = 0; o < 8; o++) {
        ra[o] = x[o].a;
        rb[o] = x[o].b;
    }
    float s[7];
    int v[7];
    // the sums of the multiples of 2^(e - 150), in those units
    auto level = [&](int e) {
        const float sg = sigma_of(e), c = __int_as_float((277 - e) << 23);
        extract8(ra, sg, qa);
        extract8(rb, sg, qb);
        base_sums(qa, qb, s);
#pragma unroll
        for (int k = 0; k < 7; k++) v[k] = __float2int_rn(s[k] * c);
    };
    level(ex + 7);
    weighted_sums(v, jx, jy, jz, 1, m.hi);
    level(ex - 11);
    weighted_sums(v, jx, jy, jz, 1 << 18, m.lo);
    if (COARSE && !any_bits(ra, rb)) return;
    level(ex - 29);
    weighted_sums(v, jx, jy, jz, 1, m.lo);
    if (!COARSE || any_bits(ra, rb)) {
        base_sums(ra, rb, s);
        weighted_sums<float>(s, (float)jx, (float)jy, (float)jz, m.R);
    }
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
    weighted_sums<double>(s, (double)jx, (double)jy, (double)jz, m);
}

// The thread's values of a cell in shared memory times 2^96.  A call: inlined,
// these few instructions that most warps never run slow the others (fields of
// 17,680 cells x 24^3 727 us, 709 so).
template <typename TS> __device__ __noinline__ void scale_tile(TS *tile, int P, int Q, int T)
{
    using IO = QIO<TS>;
    constexpr int VEC = Store<TS>::VEC;
    if constexpr (sizeof(TS) < 8) {
        for (int q = threadIdx.x; q < Q; q += T)
            for (int o = 0; o < 8; o++) {
                TS *at = tile + (size_t)o * P + q * VEC;
                IO::sts(at, q_mul(IO::lds(at), q_splat(0x1p96f)));
            }
        fence_proxy_async();  // before the copy that takes the place
    }
}

// barriers of k_moments: the sums of buffer 0 or 1 are ready
constexpr int BAR_READY = 1;

template <typename TS, bool PIPE, bool SPLIT>
__global__ void __launch_bounds__(256, 2)
    k_moments(const TS *__restrict__ f, int64_t ncells, int P, int3 half, double3 hh, double dV, double *__restrict__ out)
{
    using IO = QIO<TS>;
    using TC = typename Store<TS>::TC;
    constexpr int VEC = Store<TS>::VEC;
    // a cell's sums by warp, in one of two buffers
    union Red {
        struct {
            int64_t hi, lo;
        } fx;
        double d;
    };
    extern __shared__ __align__(128) unsigned char mom_tile[];  // PIPE: [2][8 P]
    __shared__ Red red[2][MOM_T / 32][7];
    __shared__ int rexp[2][MOM_T / 32];  // exponent of the warp's largest value, or MOM_FP64
    __shared__ __align__(8) uint64_t full[2], taken[2];  // the cell has arrived; its sums have been read
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, T = blockDim.x - (SPLIT ? 32 : 0), nw = T >> 5,
              Q = P / VEC;
    TS *tile = reinterpret_cast<TS *>(mom_tile);
    auto copy = [&](int64_t c, int b) {
        if (PIPE && c < ncells) {
            const uint32_t bytes = 8u * (uint32_t)P * (uint32_t)sizeof(TS);
            mbar_expect_tx(&full[b], bytes);
            bulk_g2s(tile + (size_t)b * 8 * P, f + c * 8 * (int64_t)P, bytes, &full[b]);
        }
    };
    const double h1 = lane % 3 == 1 ? hh.x : (lane % 3 == 2 ? hh.y : hh.z), hd = lane < 4 ? h1 : h1 * h1;
    // one warp: the moments of cell c from the warps' sums
    auto finish = [&](int64_t c, int b) {
        // all are through with the cell: the one after next takes its place
        if (lane == 0) copy(c + 2 * (int64_t)gridDim.x, b);
        const int k = lane % 7;  // lane: sum k of every fourth warp (lanes 28..31: spare)
        double s = 0.0;
        for (int w = lane < 28 ? lane / 7 : nw; w < nw; w += 4) {
            const int ex = rexp[b][w];
            const Red &r = red[b][w][k];
            double v = r.d;
            if (ex != MOM_FP64) {
                const double u1 = __longlong_as_double((long long)(1023 + ex - 143) << 52),
                             u3 = __longlong_as_double((long long)(1023 + ex - 179) << 52);
                v = fma((double)r.fx.hi, u1, (double)r.fx.lo * u3);
            }
            s = w < 4 ? v : s + v;
        }
        __syncwarp();
        if (SPLIT && lane == 0) mbar_arrive(&taken[b]);
        if (nw > 2) s += __shfl_down_sync(0xffffffffu, s, 14);
        if (nw > 1) s += __shfl_down_sync(0xffffffffu, s, 7);
        // lane 0: sum f; 1..3: u_d; 4..6: sum xi_d^2 f / sum f
        const double s0 = __shfl_sync(0xffffffffu, s, 0), v = s / s0 * hd;
        const double u2 = v * v, e2 = __shfl_down_sync(0xffffffffu, v, 3);
        const double ux2 = __shfl_sync(0xffffffffu, u2, 1), uy2 = __shfl_sync(0xffffffffu, u2, 2),
                     uz2 = __shfl_sync(0xffffffffu, u2, 3);
        const double ex2 = __shfl_sync(0xffffffffu, e2, 1), ey2 = __shfl_sync(0xffffffffu, e2, 2),
                     ez2 = __shfl_sync(0xffffffffu, e2, 3);
        double *o = out + c * 5;
        if (lane == 0) {
            // a third of x: the product with 1/3, corrected by its remainder (Markstein, 1990)
            const double x = ex2 + ey2 + ez2 - (ux2 + uy2 + uz2), third = 1.0 / 3.0, t = x * third;
            o[0] = s0 * dV;
            o[4] = fma(fma(-3.0, t, x), third, t);
        } else if (lane < 4) {
            o[lane] = v;
        }
    };
    if (tid == 0) {
        mbar_init(&taken[0], 1);
        mbar_init(&taken[1], 1);
        mbar_init(&full[0], 1);
        mbar_init(&full[1], 1);
        mbar_fence_init();
        copy(blockIdx.x, 0);
        copy((int64_t)blockIdx.x + gridDim.x, 1);
    }
    __syncthreads();
    if (SPLIT && warp == nw) {
        int buf = 0;
        for (int64_t c = blockIdx.x; c < ncells; c += gridDim.x, buf ^= 1) {
            bar_sync_n(BAR_READY + buf, T + 32);
            finish(c, buf);
        }
        return;
    }
    auto node = [&](int q) {
        const int p = q * VEC, t = p / half.z;
        return make_int3(2 * (t / half.y) + 1, 2 * (t % half.y) + 1, 2 * (p - t * half.z) + 1);
    };
    const int3 j0 = node(tid), j1 = node(tid + T);  // most grids have no more quads a thread
    int buf = 0, done = 0;
    for (int64_t c = blockIdx.x; c < ncells; c += gridDim.x, buf ^= 1, done++) {
        bool here = true;
        // (waited for twice at most, to leave no copy in flight behind)
        if constexpr (PIPE)
            here = mbar_wait(&full[buf], (uint32_t)(done >> 1) & 1u) || mbar_wait(&full[buf], (uint32_t)(done >> 1) & 1u);
        auto load = [&](int q, QV<TC> (&x)[8]) {
#pragma unroll
            for (int o = 0; o < 8; o++) {
                if constexpr (PIPE) x[o] = IO::lds(tile + (size_t)(buf * 8 + o) * P + q * VEC);
                else x[o] = IO::ldg(f + (c * 8 + o) * (int64_t)P + q * VEC);
            }
        };
        auto place = [&](int q) {
            if (PIPE && q < 2 * T) return q == tid ? j0 : j1;
            return node(q);
        };
        int ex = 0;  // exponent of the warp's largest value, + 256 where scaled; 0: FP64 sums
        MomSum m{};
        if constexpr (sizeof(TC) == 4) {
            float top = 0.0f;
            for (int q = tid; q < Q; q += T) {
                QV<float> x[8];
                load(q, x);
#pragma unroll
                for (int o = 0; o < 8; o++)
                    top = max_abs(max_abs(top, x[o].a.x, x[o].a.y), x[o].b.x, x[o].b.y);
            }
            const float most = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(top)));
            ex = (int)(__float_as_uint(most) >> 23);
            if (ex < 56) {
                // the far corner of a grid: values scaled, no FP64 sums
                ex = 256 + max(56, (int)(__float_as_uint(most * 0x1p96f) >> 23));
                if constexpr (PIPE) scale_tile<TS>(tile + (size_t)buf * 8 * P, P, Q, T);
            }
            if ((ex & 255) > 240) ex = 0;
            if (ex) {
#pragma unroll 1
                for (int q = tid; q < Q; q += T) {
                    QV<float> x[8];
                    load(q, x);
                    if (!PIPE && ex >= 256)
#pragma unroll
                        for (int o = 0; o < 8; o++) x[o] = q_mul(x[o], q_splat(0x1p96f));
                    const int3 j = place(q);
                    add_quad<sizeof(TS) == 2>(x, ex & 255, j.x, j.y, j.z, m);
                }
            }
        }
        double md[7] = {0, 0, 0, 0, 0, 0, 0};
        if (!ex) {
#pragma unroll 1
            for (int q = tid; q < Q; q += T) {
                QV<TC> x[8];
                load(q, x);
                const int3 j = place(q);
                add_quad_f64<TC>(x, j.x, j.y, j.z, md);
            }
        }
        // the buffer's last sums, of two cells ago, have been taken (a wait that
        // gave up, here or on the copy, leaves NaN)
        if (SPLIT && done >= 2) here = mbar_wait(&taken[buf], (uint32_t)((done >> 1) - 1) & 1u) && here;
        if (!here) {
            ex = 0;
            md[0] = nan("");
        }
        const bool mine = (lane & 3) == 0 && lane < 28;
        if (ex) {
            const int64_t hi = warp_reduce7<int64_t>(m.hi, lane), lo = warp_reduce7<int64_t>(m.lo, lane);
            // the warp's rests, below 2^27 u3, rounded to u3
            const float R = warp_reduce7<float>(m.R, lane) * __int_as_float((306 - (ex & 255)) << 23);
            if (mine) red[buf][warp][lane >> 2].fx = {hi, lo + __float2int_rn(R)};
        } else {
            const double t = warp_reduce7<double>(md, lane);
            if (mine) red[buf][warp][lane >> 2].d = t;
        }
        if (lane == 0) rexp[buf][warp] = ex == 0 ? MOM_FP64 : ex < 256 ? ex : ex - 256 - 96;
        __syncwarp();
        if constexpr (SPLIT) {
            bar_arrive_n(BAR_READY + buf, T + 32);
        } else {
            __syncthreads();
            if (warp == 0) finish(c, buf);
        }
    }
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

template <typename TS, bool PIPE, bool SPLIT>
int moments_k(const TS *f, int64_t ncells, const MomGrid &g, int t, double *out, cudaStream_t s)
{
    const int P = g.half[0] * g.half[1] * g.half[2];
    const int3 half = make_int3(g.half[0], g.half[1], g.half[2]);
    const double3 hh = make_double3(0.5 * g.hv[0], 0.5 * g.hv[1], 0.5 * g.hv[2]);
    auto kern = k_moments<TS, PIPE, SPLIT>;
    const size_t dyn = PIPE ? 16 * (size_t)P * sizeof(TS) : 0;
    int64_t grid = ncells;
    t += SPLIT ? 32 : 0;
    if (PIPE) {
        int dev = 0, nsm = 0, occ = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
        if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(2 * MOM_ROW)) != cudaSuccess ||
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, t, dyn) != cudaSuccess || occ < 1)
            return DVM_ECUDA;
        grid = std::min<int64_t>(ncells, (int64_t)nsm * occ);
    }
    kern<<<(unsigned)grid, t, dyn, s>>>(f, ncells, P, half, hh, g.dV, out);
    return last_status();
}

template <typename TS> int moments_t(const void *f, int64_t ncells, const MomGrid &g, double *out, cudaStream_t s)
{
    const int P = g.half[0] * g.half[1] * g.half[2], Q = P / Store<TS>::VEC;
    const TS *ft = static_cast<const TS *>(f);
    // up to two quads a thread on one warp (24 x 8 x 8 with 48 quads: 122 us the
    // call, 137 on two warps); else one up to MOM_T quads, then two or more, evenly
    // (24^3: 432 quads on 224 threads).  Five or six warps and the last one spread
    // unevenly over an SM's four schedulers, and two such CTAs fit it: three warps
    // take their place where shared memory holds four CTAs (11,632 cells x 20 x 16 x
    // 16 FP32 156 -> 129 us, 20 x 20 x 24 BF16 243 -> 200; 20 x 20 x 24 FP32, where it does
    // not, 223 -> 240).
    const int rounds = (Q + MOM_T - 1) / MOM_T, even = ((Q + rounds - 1) / rounds + 31) / 32 * 32;
    const bool four = (size_t)8 * 8 * P * sizeof(TS) <= 216 * 1024;
    const int t = Q <= 64 ? 32 : four && (even == 160 || even == 192) ? 96 : even;
    if ((size_t)8 * P * sizeof(TS) > MOM_ROW) return moments_k<TS, false, false>(ft, ncells, g, t, out, s);
    if (t > 32) return moments_k<TS, true, true>(ft, ncells, g, t, out, s);
    return moments_k<TS, true, false>(ft, ncells, g, t, out, s);
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
