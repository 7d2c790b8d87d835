// The learned collision operator's network: 64 -> 256 -> 256 -> 256 -> 64 with
// SiLU hidden activations, BF16 weights and activations, FP32 accumulation,
// run and trained on the 5th-generation tensor cores.
//
// Every contraction is C[M x N] = A[M x K] . B[N x K]^T with both operands BF16
// and K contiguous in global memory: a CTA owns 128 rows of C, stages 64-wide K
// chunks of A and B into a four-deep shared-memory ring with cp.async in the
// 128-byte swizzled K-major layout, one thread issues tcgen05.mma (M = 128,
// N <= 256, K = 16 per instruction) into a tensor-memory accumulator, and the
// eight warps read it back with tcgen05.ld for a fused epilogue: bias, SiLU and
// the transposed copies of the forward pass; the output gradient with loss and
// bias-gradient sums; the SiLU derivative of the backward pass.  The weight
// gradients (C = dZ^T . activation, long K) of all four layers are one launch,
// split over K up to 12,000 rows.  Forward, backward and the Adam update all run on the device.
//
// Bound by the latency of a few dependent chunks per launch (the network is
// 3.1 GFLOP a pass at 24k rows): with 16-byte loads through registers, two
// stages and 128 threads a 256 x 256 layer took 52 us on 24,032 rows, 38 us on
// 8,192, and the weight gradients, on two CTAs each, most of a gradient's
// 2.9 ms.  Now 14 us (24,032 rows, inference), 20 to 23 us with the transposed copies of
// training (8,192 rows), and 15 us for all their weight gradients; the whole gradient
// takes 9 launches instead of 24.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <vector>

#include "../../include/dvm.h"
#include "async.cuh"
#include "common.cuh"
#include "kernels.hpp"
#include "mlp.hpp"
#include "tc.cuh"

namespace dvm {

void count_launch();

namespace {

constexpr int GT = 256;             // threads per GEMM CTA
constexpr int NSTAGE = 4;
constexpr uint32_t STAGE_A = 16384; // 128 rows x 128 bytes
constexpr uint32_t STAGE_BYTES = STAGE_A + 32768;

// what the epilogue makes of the accumulator v
enum {
    EP_FORWARD,  // z = v + bias: Cf = z, H = act(z) and its transposed copy
    EP_OUT,      // r = v + bias - T: H = d = scale r and its transposed copy, sums of d and of r^2
    EP_BACK,     // H = d = v silu'(Z) and its transposed copy, sums of d
    EP_PLAIN,    // Cf = v
};

struct GemmArgs {
    const __nv_bfloat16 *A;
    int64_t lda;
    const __nv_bfloat16 *B;
    int64_t ldb;
    int64_t M;
    int N;                  // multiple of 32, at most 256
    int64_t K;              // multiple of 64
    const float *bias;      // [N]
    float *Cf;              // FP32 output, [M][N], or null
    __nv_bfloat16 *H;       // BF16 output, [M][N], or null
    __nv_bfloat16 *HT;      // its transpose, [N][ldt], zero in columns M .. M rounded up to 64, or null
    int64_t ldt;
    const float *X;         // T [M][N] (EP_OUT), Z [M][N] (EP_BACK)
    float scale;            // EP_OUT
    float *colsum;          // [tiles][ldsum]: column sums of d over each tile's rows, or null
    int64_t ldsum;
    double *loss;           // [tiles]: sum of r^2 (EP_OUT)
    int act;                // EP_FORWARD: 0 none, 1 SiLU
    int *status;
};

__device__ inline float silu(float x) { return x / (1.0f + __expf(-x)); }

// Sums over the warp's lanes of 16 values each by reduce-scatter: lanes 2c and
// 2c + 1 end with the sum of value c.
__device__ inline float warp_colsum16(const float (&d)[16], int lane)
{
    float v[16];
#pragma unroll
    for (int i = 0; i < 16; i++) v[i] = d[i];
#pragma unroll
    for (int s = 0; s < 4; s++) {
        const int off = 16 >> s, half = 8 >> s;
        const bool up = lane & off;
#pragma unroll
        for (int i = 0; i < half; i++) {
            const float send = up ? v[i] : v[half + i], keep = up ? v[half + i] : v[i];
            v[i] = keep + __shfl_xor_sync(0xffffffffu, send, off);
        }
    }
    return v[0] + __shfl_xor_sync(0xffffffffu, v[0], 1);
}

// Rows m0 .. m0 + 127 of C over the K chunks [k0, k1).
template <int EP> __device__ __forceinline__ void gemm_tile(const GemmArgs &g, int64_t m0, int k0, int k1, int tile)
{
    extern __shared__ unsigned char sraw[];
    __shared__ __align__(8) uint64_t bar[NSTAGE];
    __shared__ uint32_t tmem_slot;
    __shared__ float csum[4][256];
    __shared__ double lsum[GT / 32];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    // operand tiles must start on 1024-byte boundaries (swizzle atoms)
    const uint32_t base = (smem_u32(sraw) + 1023u) & ~1023u;
    const uint32_t ncols = g.N <= 32 ? 32u : g.N <= 64 ? 64u : g.N <= 128 ? 128u : 256u;
    const uint32_t idesc = idesc_bf16(128, g.N);
    if (warp == 0) tmem_alloc(&tmem_slot, ncols);
    if (tid == 0) {
        for (int s = 0; s < NSTAGE; s++) mbar_init(&bar[s], 1);
        mbar_fence_init();
    }
    const int nk = k1 - k0;
    auto load = [&](int c) {
        if (c < nk) {
            const uint32_t sa = base + (uint32_t)(c % NSTAGE) * STAGE_BYTES, sb = sa + STAGE_A;
            const int64_t kk = (int64_t)(k0 + c) * 64;
#pragma unroll
            for (int i = 0; i < 4; i++) {
                const int r = (i * GT + tid) >> 3, q = tid & 7;
                const bool on = m0 + r < g.M;
                cp_async16_zfill(sa + sw128_offset(r, q), g.A + (on ? m0 + r : 0) * g.lda + kk + q * 8, on ? 16u : 0u);
            }
            for (int i = tid; i < g.N * 8; i += GT)
                cp_async16_zfill(sb + sw128_offset(i >> 3, i & 7), g.B + (int64_t)(i >> 3) * g.ldb + kk + (i & 7) * 8, 16u);
        }
        cp_async_commit();
    };
    for (int c = 0; c < NSTAGE - 1; c++) load(c);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_slot;
    bool bad = false;
    for (int c = 0; c < nk && !bad; c++) {
        // the ring slot of chunk c + NSTAGE - 1 was read by the MMAs of chunk c - 1
        bool late = false;
        if (c >= 1 && c + NSTAGE - 1 < nk) late = !mbar_wait(&bar[(c - 1) % NSTAGE], (uint32_t)((c - 1) / NSTAGE) & 1u);
        cp_async_wait<NSTAGE - 2>();
        fence_proxy_async();
        bad = __syncthreads_or(late);
        if (bad) break;
        if (tid == 0) {
            tc_fence_after();
            const uint32_t a = base + (uint32_t)(c % NSTAGE) * STAGE_BYTES, b = a + STAGE_A;
#pragma unroll
            for (int ks = 0; ks < 4; ks++)
                tc_mma_bf16(tmem, sw128_desc(a + ks * 32), sw128_desc(b + ks * 32), idesc, c > 0 || ks > 0);
            tc_commit(&bar[c % NSTAGE]);
        }
        load(c + NSTAGE - 1);
    }
    cp_async_wait_all();
    bool late = false;
    if (!bad) late = !mbar_wait(&bar[(nk - 1) % NSTAGE], (uint32_t)((nk - 1) / NSTAGE) & 1u);
    bad = __syncthreads_or(late || bad);
    tc_fence_after();
    if (bad) {
        if (tid == 0) atomicOr(g.status, ST_TIMEOUT);
    } else {
        // warp w reads lanes 32 (w mod 4) .. + 31 of the accumulator, warps 0-3
        // the first half of the columns, warps 4-7 the second
        const int quad = warp & 3;
        const int64_t row = m0 + 32 * quad + lane, Mt = (g.M + 63) / 64 * 64;
        const bool on = row < g.M;
        double acc = 0.0;
#pragma unroll 1
        for (int col = (warp >> 2) * (g.N / 2), end = col + g.N / 2; col < end; col += 16) {
            float v[16];
            tmem_ld16(tmem + ((uint32_t)(32 * quad) << 16) + (uint32_t)col, v);
            if constexpr (EP == EP_PLAIN || EP == EP_FORWARD) {
                if constexpr (EP == EP_FORWARD)
#pragma unroll
                    for (int j = 0; j < 16; j++) v[j] += g.bias[col + j];
                if (g.Cf && on) {
                    float4 *d = reinterpret_cast<float4 *>(g.Cf + row * g.N + col);
#pragma unroll
                    for (int q = 0; q < 4; q++) d[q] = make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
                }
                if (EP == EP_FORWARD && g.act)
#pragma unroll
                    for (int j = 0; j < 16; j++) v[j] = silu(v[j]);
            } else {
                float x[16];
#pragma unroll
                for (int q = 0; q < 4; q++) {
                    const float4 t = on ? __ldg(reinterpret_cast<const float4 *>(g.X + row * g.N + col) + q)
                                        : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
                    x[4 * q] = t.x;
                    x[4 * q + 1] = t.y;
                    x[4 * q + 2] = t.z;
                    x[4 * q + 3] = t.w;
                }
#pragma unroll
                for (int j = 0; j < 16; j++) {
                    if constexpr (EP == EP_OUT) {
                        const float r = (v[j] + g.bias[col + j]) - x[j];
                        if (on) acc += (double)r * r;
                        v[j] = g.scale * r;
                    } else {
                        const float sg = 1.0f / (1.0f + __expf(-x[j]));
                        v[j] = v[j] * sg * (1.0f + x[j] * (1.0f - sg));
                    }
                    if (!on) v[j] = 0.0f;
                }
                const float cs = warp_colsum16(v, lane);
                if ((lane & 1) == 0) csum[quad][col + (lane >> 1)] = cs;
            }
            if constexpr (EP != EP_PLAIN) {
                uint32_t hp[8];
#pragma unroll
                for (int j = 0; j < 16; j += 2) {
                    const __nv_bfloat162 p2 = __floats2bfloat162_rn(on ? v[j] : 0.0f, on ? v[j + 1] : 0.0f);
                    hp[j / 2] = *reinterpret_cast<const uint32_t *>(&p2);
                    if (g.HT && row < Mt) {
                        g.HT[(int64_t)(col + j) * g.ldt + row] = p2.x;
                        g.HT[(int64_t)(col + j + 1) * g.ldt + row] = p2.y;
                    }
                }
                if (g.H && on) {
                    uint4 *d = reinterpret_cast<uint4 *>(g.H + row * g.N + col);
                    d[0] = make_uint4(hp[0], hp[1], hp[2], hp[3]);
                    d[1] = make_uint4(hp[4], hp[5], hp[6], hp[7]);
                }
            }
        }
        if constexpr (EP == EP_OUT || EP == EP_BACK) {
            if (EP == EP_OUT) {
                acc = warp_allsum(acc);
                if (lane == 0) lsum[warp] = acc;
            }
            __syncthreads();
            if (tid < g.N) g.colsum[tile * g.ldsum + tid] = (csum[0][tid] + csum[1][tid]) + (csum[2][tid] + csum[3][tid]);
            if (EP == EP_OUT && tid == 0) {
                double s = 0.0;
                for (int w = 0; w < GT / 32; w++) s += lsum[w];
                g.loss[tile] = s;
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) tmem_dealloc(tmem, ncols);
}

template <int EP> __global__ void __launch_bounds__(GT) k_gemm(const GemmArgs g)
{
    gemm_tile<EP>(g, (int64_t)blockIdx.x * 128, 0, (int)(g.K / 64), blockIdx.x);
}

// Partial weight gradients of all four layers: CTA (tile, split), tiles 0-1,
// 2-3, 4-5 and 6 the rows of gW1, gW2, gW3 and gW4; part [splits][MLP_NPARAM]
// in the parameters' order.
struct WgradArgs {
    const __nv_bfloat16 *A[4], *B[4];  // dZ^T [out][ld], activation^T [in][ld]
    int64_t ld;
    int chunks;                        // of 64 rows of the batch
    int64_t off[4];
    float *part;
    int *status;
};
constexpr int WG_TILES = 7;

__global__ void __launch_bounds__(GT) k_wgrad(const WgradArgs a)
{
    const int l = blockIdx.x >> 1, per = (a.chunks + gridDim.y - 1) / gridDim.y;
    const int k0 = blockIdx.y * per, k1 = min(a.chunks, k0 + per);
    GemmArgs g{};
    g.A = a.A[l];
    g.B = a.B[l];
    g.lda = g.ldb = a.ld;
    g.M = l == 3 ? 64 : 256;
    g.N = l == 0 ? 64 : 256;
    g.Cf = a.part + (int64_t)blockIdx.y * MLP_NPARAM + a.off[l];
    g.status = a.status;
    gemm_tile<EP_PLAIN>(g, (int64_t)(blockIdx.x & 1) * 128, k0, k1, 0);
}

// g = sum over splits of the partial weight gradients, and over tiles of the
// partial bias gradients; loss = sum over tiles
struct ReduceArgs {
    const float *part, *bias;  // [splits][MLP_NPARAM], [tiles][832]
    const double *lossp;       // [tiles]
    int splits, tiles;
    float *g;
    double *loss;
};
__global__ void __launch_bounds__(256) k_grad_reduce(const ReduceArgs r)
{
    const int q = blockIdx.x * 256 + threadIdx.x;
    // the flat order: W1 (16384) b1 (256) W2 (65536) b2 (256) W3 b3 W4 (16384) b4 (64)
    if (q < MLP_NPARAM) {
        int b = -1;
        if (q >= 16384 && q < 16640) b = q - 16384;
        else if (q >= 82176 && q < 82432) b = 256 + q - 82176;
        else if (q >= 147968 && q < 148224) b = 512 + q - 147968;
        else if (q >= 164608) b = 768 + q - 164608;
        float s = 0.0f;
        if (b < 0) {
#pragma unroll 8
            for (int k = 0; k < r.splits; k++) s += __ldg(r.part + (int64_t)k * MLP_NPARAM + q);
        } else {
#pragma unroll 16
            for (int k = 0; k < r.tiles; k++) s += __ldg(r.bias + (int64_t)k * 832 + b);
        }
        r.g[q] = s;
    }
    if (blockIdx.x == 0 && threadIdx.x < 32) {
        double s = 0.0;
        for (int k = threadIdx.x; k < r.tiles; k += 32) s += r.lossp[k];
        s = warp_allsum(s);
        if (threadIdx.x == 0) *r.loss = s;
    }
}

constexpr size_t GEMM_DYN = (size_t)NSTAGE * STAGE_BYTES + 1024;

template <typename Kern> int gemm_shape(Kern *kern)
{
    return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)GEMM_DYN) == cudaSuccess
               ? DVM_OK
               : DVM_ECUDA;
}

template <int EP> int gemm(const GemmArgs &g, cudaStream_t s)
{
    if (g.M <= 0) return DVM_OK;
    if (g.K % 64 || g.K < 64 || g.N % 32 || g.N < 32 || g.N > 256) return DVM_EINVAL;
    if (gemm_shape(k_gemm<EP>)) return DVM_ECUDA;
    k_gemm<EP><<<(unsigned)((g.M + 127) / 128), GT, GEMM_DYN, s>>>(g);
    count_launch();
    return cudaGetLastError() == cudaSuccess ? DVM_OK : DVM_ECUDA;
}

// ---- elementwise kernels ------------------------------------------------------
// 64 rows of x [n][64] to BF16 rows y and, if yt is given, columns of yt
// [64][ldt] (zero in rows n .. n rounded up to 64)
__global__ void __launch_bounds__(256) k_to_bf16(const float *x, __nv_bfloat16 *y, __nv_bfloat16 *yt, int64_t n, int64_t ldt)
{
    __shared__ __nv_bfloat16 t[64][66];
    const int64_t r0 = (int64_t)blockIdx.x * 64;
    for (int q = threadIdx.x; q < 64 * 16; q += 256) {
        const int r = q >> 4, c = (q & 15) * 4;
        float4 v = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        if (r0 + r < n) v = __ldg(reinterpret_cast<const float4 *>(x + (r0 + r) * 64 + c));
        const __nv_bfloat162 a = __floats2bfloat162_rn(v.x, v.y), b = __floats2bfloat162_rn(v.z, v.w);
        if (r0 + r < n) {
            uint2 w;
            w.x = *reinterpret_cast<const uint32_t *>(&a);
            w.y = *reinterpret_cast<const uint32_t *>(&b);
            *reinterpret_cast<uint2 *>(y + (r0 + r) * 64 + c) = w;
        }
        t[r][c] = a.x;
        t[r][c + 1] = a.y;
        t[r][c + 2] = b.x;
        t[r][c + 3] = b.y;
    }
    if (!yt) return;
    __syncthreads();
    for (int q = threadIdx.x; q < 64 * 64; q += 256) yt[(int64_t)(q >> 6) * ldt + r0 + (q & 63)] = t[q & 63][q >> 6];
}

// FP32 master weights -> BF16 W[out][in] and W^T[in][out]; biases stay FP32
__global__ void k_cast_weights(const float *w, int rows, int cols, __nv_bfloat16 *W, __nv_bfloat16 *WT)
{
    for (int q = blockIdx.x * blockDim.x + threadIdx.x; q < rows * cols; q += gridDim.x * blockDim.x) {
        const int r = q / cols, c = q - r * cols;
        const __nv_bfloat16 b = __float2bfloat16_rn(w[q]);
        W[q] = b;
        WT[c * rows + r] = b;
    }
}

// Adam (Kingma & Ba) on the flat FP32 parameter vector
__global__ void k_adam(float *w, float *m, float *v, const float *g, int64_t n, float lr, float b1, float b2,
                       float eps, float c1, float c2)
{
    for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < n; q += (int64_t)gridDim.x * blockDim.x) {
        const float gq = g[q];
        const float mq = b1 * m[q] + (1.0f - b1) * gq;
        const float vq = b2 * v[q] + (1.0f - b2) * gq * gq;
        m[q] = mq;
        v[q] = vq;
        w[q] -= lr * (mq / c1) / (sqrtf(vq / c2) + eps);
    }
}

unsigned blocks(int64_t n) { return (unsigned)std::min<int64_t>(std::max<int64_t>((n + 255) / 256, 1), 152 * 16); }

}  // namespace

// ---------------------------------------------------------------- MLP object
static const int L_IN[4] = {64, 256, 256, 256};
static const int L_OUT[4] = {256, 256, 256, 64};

static size_t param_offset(int l)
{
    size_t off = 0;
    for (int k = 0; k < l; k++) off += (size_t)L_IN[k] * L_OUT[k] + L_OUT[k];
    return off;
}

int mlp_init(Mlp &m, const DevAllocF &alloc)
{
    if (m.ready) return DVM_OK;
    const size_t n = MLP_NPARAM;
    m.w = static_cast<float *>(alloc(n * 4));
    m.m = static_cast<float *>(alloc(n * 4));
    m.v = static_cast<float *>(alloc(n * 4));
    m.g = static_cast<float *>(alloc(n * 4));
    m.loss = static_cast<double *>(alloc(8));
    for (int l = 0; l < 4; l++) {
        m.W[l] = static_cast<__nv_bfloat16 *>(alloc((size_t)L_IN[l] * L_OUT[l] * 2));
        m.WT[l] = static_cast<__nv_bfloat16 *>(alloc((size_t)L_IN[l] * L_OUT[l] * 2));
    }
    if (!m.w || !m.m || !m.v || !m.g || !m.loss) return DVM_ENOMEM;
    for (int l = 0; l < 4; l++)
        if (!m.W[l] || !m.WT[l]) return DVM_ENOMEM;
    cudaMemset(m.m, 0, n * 4);
    cudaMemset(m.v, 0, n * 4);
    m.steps = 0;
    m.ready = true;
    return cudaGetLastError() == cudaSuccess ? DVM_OK : DVM_ECUDA;
}

void mlp_free(Mlp &m, const DevFreeF &dfree)
{
    void *ps[] = {m.w, m.m, m.v, m.g, m.loss};
    for (void *p : ps)
        if (p) dfree(p);
    for (int l = 0; l < 4; l++) {
        if (m.W[l]) dfree(m.W[l]);
        if (m.WT[l]) dfree(m.WT[l]);
    }
    for (int l = 0; l < 4; l++) m.W[l] = m.WT[l] = nullptr;
    m.w = m.m = m.v = m.g = nullptr;
    m.loss = nullptr;
    m.ready = false;
    for (auto &b : m.work) b.reset(dfree);
    for (auto &c : m.cap) c = 0;
}

int mlp_cast(Mlp &m, cudaStream_t s)
{
    for (int l = 0; l < 4; l++) {
        k_cast_weights<<<blocks((int64_t)L_IN[l] * L_OUT[l]), 256, 0, s>>>(m.w + param_offset(l), L_OUT[l], L_IN[l],
                                                                            m.W[l], m.WT[l]);
        count_launch();
    }
    return cudaGetLastError() == cudaSuccess ? DVM_OK : DVM_ECUDA;
}

const float *mlp_bias(const Mlp &m, int l) { return m.w + param_offset(l) + (size_t)L_IN[l] * L_OUT[l]; }

// K splits of the weight gradients: the seven tiles on about all 152 SMs for
// batches up to 12,000 rows, one chain for larger ones.  The line is no line of
// speed or of precision, split sums are better on either side of it: the tensor
// core truncates as it accumulates, so that a sum drifts from the exact one with
// the length of its chain (relative to the gradient's norm, one chain 1.1e-5 at
// 12,008 rows, 3.4e-5 at 30,000, 7.6e-5 at 60,000; 21 splits 3e-7, 8e-7, 1.7e-6),
// and a whole gradient takes 401, 757 and 1,380 us with one chain, 294, 479 and 850
// with splits.  It keeps a gradient within 2e-5 of the one-chain value, which
// gradients of every size had before there were splits, so that runs can be
// compared with older ones to FP32 rounding.
static int wgrad_splits(int64_t n) { return n <= 12000 ? (int)std::min<int64_t>(21, (n + 63) / 64) : 1; }

// one set of working buffers for a batch of n rows (n padded to a multiple of 64)
int mlp_reserve(Mlp &m, int set, int64_t n, const DevAllocF &alloc, const DevFreeF &dfree)
{
    const int64_t np = (n + 63) / 64 * 64;
    if (np <= m.cap[set]) return DVM_OK;
    const size_t tiles = (size_t)(np + 127) / 128;
    const size_t sz[] = {(size_t)np * 64 * 2, (size_t)np * 256 * 2 * 3,      // X, H
                         (size_t)np * 64 * 2,                                // Xt
                         (size_t)np * 256 * 4 * 3,                           // Z1..Z3
                         (size_t)np * 256 * 2 * 3,                           // Ht
                         (size_t)np * 64 * 2, (size_t)np * 64 * 2,           // dO, dOt
                         (size_t)np * 256 * 2 * 2, (size_t)np * 256 * 2 * 3, // dZ (two in turn), dZt of each layer
                         (size_t)21 * MLP_NPARAM * 4,                        // partial weight gradients (at most 21 splits)
                         tiles * 832 * 4, tiles * 8,                         // partial bias gradients and losses
                         (size_t)np * 256, (size_t)np * 256};                // a host call's rows
    static_assert(sizeof(sz) / sizeof(sz[0]) == MLP_NWORK, "work buffer count");
    const int first[MLP_NSETS + 1] = {W_X, W_XT, W_R0, MLP_NWORK};
    for (int i = first[set]; i < first[set + 1]; i++) m.work[i].reset(dfree);
    m.cap[set] = 0;
    for (int i = first[set]; i < first[set + 1]; i++) {
        m.work[i].p = alloc(sz[i]);
        m.work[i].bytes = sz[i];
        if (!m.work[i].p) return DVM_ENOMEM;
    }
    m.cap[set] = np;
    return DVM_OK;
}

// layers 1 to 3 on rows X (BF16 [n][64] in work X); with train = true also
// keeps pre-activations and transposed activations for the backward pass
static int forward3(Mlp &m, int64_t n, bool train, int *status, cudaStream_t s)
{
    const int64_t np = m.cap[MLP_FORWARD], nt = m.cap[MLP_GRAD];
    auto *Z = static_cast<float *>(m.work[W_Z].p);
    auto *H = static_cast<__nv_bfloat16 *>(m.work[W_H].p);
    auto *Ht = static_cast<__nv_bfloat16 *>(m.work[W_HT].p);
    const __nv_bfloat16 *in = static_cast<__nv_bfloat16 *>(m.work[W_X].p);
    for (int l = 0; l < 3; l++) {
        GemmArgs g{};
        g.A = in;
        g.lda = g.ldb = g.K = L_IN[l];
        g.B = m.W[l];
        g.M = n;
        g.N = 256;
        g.bias = mlp_bias(m, l);
        g.status = status;
        g.act = 1;
        g.Cf = train ? Z + (size_t)l * nt * 256 : nullptr;
        g.H = H + (size_t)l * np * 256;
        g.HT = train ? Ht + (size_t)l * nt * 256 : nullptr;
        g.ldt = nt;
        in = g.H;
        int rc = gemm<EP_FORWARD>(g, s);
        if (rc) return rc;
    }
    return DVM_OK;
}

static GemmArgs layer4(Mlp &m, int64_t n, int *status)
{
    GemmArgs g{};
    g.A = static_cast<__nv_bfloat16 *>(m.work[W_H].p) + (size_t)2 * m.cap[MLP_FORWARD] * 256;
    g.B = m.W[3];
    g.lda = g.ldb = g.K = 256;
    g.M = n;
    g.N = 64;
    g.bias = mlp_bias(m, 3);
    g.status = status;
    return g;
}

int mlp_forward(Mlp &m, const float *x_dev, int64_t n, float *y_dev, int *status, cudaStream_t s)
{
    if (n > m.cap[MLP_FORWARD]) return DVM_EINVAL;
    k_to_bf16<<<(unsigned)((n + 63) / 64), 256, 0, s>>>(x_dev, static_cast<__nv_bfloat16 *>(m.work[W_X].p), nullptr, n, 0);
    count_launch();
    int rc = forward3(m, n, false, status, s);
    if (rc) return rc;
    GemmArgs g = layer4(m, n, status);
    g.Cf = y_dev;
    return gemm<EP_FORWARD>(g, s);
}

// loss and gradient (m.g) for rows x_dev / targets t_dev (FP32 [n][64])
int mlp_grad(Mlp &m, const float *x_dev, const float *t_dev, int64_t n, int *status, cudaStream_t s)
{
    if (n > m.cap[MLP_FORWARD] || n > m.cap[MLP_GRAD]) return DVM_EINVAL;
    const int64_t np = m.cap[MLP_GRAD];
    const int tiles = (int)((n + 127) / 128), splits = wgrad_splits(n);
    auto *X = static_cast<__nv_bfloat16 *>(m.work[W_X].p);
    auto *Xt = static_cast<__nv_bfloat16 *>(m.work[W_XT].p);
    auto *Z = static_cast<float *>(m.work[W_Z].p);
    auto *Ht = static_cast<__nv_bfloat16 *>(m.work[W_HT].p);
    auto *dO = static_cast<__nv_bfloat16 *>(m.work[W_DO].p);
    auto *dOt = static_cast<__nv_bfloat16 *>(m.work[W_DOT].p);
    auto *dZ = static_cast<__nv_bfloat16 *>(m.work[W_DZ].p);
    auto *dZt = static_cast<__nv_bfloat16 *>(m.work[W_DZT].p);
    auto *bias = static_cast<float *>(m.work[W_BIAS].p);
    auto *lossp = static_cast<double *>(m.work[W_LOSS].p);
    k_to_bf16<<<(unsigned)((n + 63) / 64), 256, 0, s>>>(x_dev, X, Xt, n, np);
    count_launch();
    int rc = forward3(m, n, true, status, s);
    if (rc) return rc;
    // dO = 2 (O - T) / (64 n)
    GemmArgs g = layer4(m, n, status);
    g.X = t_dev;
    g.scale = 2.0f / ((float)n * 64.0f);
    g.H = dO;
    g.HT = dOt;
    g.ldt = np;
    g.colsum = bias + 768;
    g.ldsum = 832;
    g.loss = lossp;
    if ((rc = gemm<EP_OUT>(g, s))) return rc;
    // dZ_l = (dZ_{l+1} . W_{l+1}) silu'(Z_l)
    for (int l = 2; l >= 0; l--) {
        GemmArgs h{};
        h.A = l == 2 ? dO : dZ + (size_t)((l + 1) & 1) * np * 256;
        h.B = m.WT[l + 1];
        h.lda = h.ldb = h.K = L_OUT[l + 1];
        h.M = n;
        h.N = 256;
        h.X = Z + (size_t)l * np * 256;
        h.H = l > 0 ? dZ + (size_t)(l & 1) * np * 256 : nullptr;
        h.HT = dZt + (size_t)l * np * 256;
        h.ldt = np;
        h.colsum = bias + 256 * l;
        h.ldsum = 832;
        h.status = status;
        if ((rc = gemm<EP_BACK>(h, s))) return rc;
    }
    // gW_l[out][in] = dZ_l^T . (input of layer l)
    WgradArgs w{};
    for (int l = 0; l < 4; l++) {
        w.A[l] = l < 3 ? dZt + (size_t)l * np * 256 : dOt;
        w.B[l] = l > 0 ? Ht + (size_t)(l - 1) * np * 256 : Xt;
        w.off[l] = (int64_t)param_offset(l);
    }
    w.ld = np;
    w.chunks = (int)((n + 63) / 64);
    w.part = static_cast<float *>(m.work[W_PART].p);
    w.status = status;
    // every split holds at least one chunk
    const int per = (w.chunks + splits - 1) / splits, used = (w.chunks + per - 1) / per;
    if (gemm_shape(k_wgrad)) return DVM_ECUDA;
    k_wgrad<<<dim3(WG_TILES, used), GT, GEMM_DYN, s>>>(w);
    count_launch();
    const ReduceArgs r{w.part, bias, lossp, used, tiles, m.g, m.loss};
    k_grad_reduce<<<(unsigned)((MLP_NPARAM + 255) / 256), 256, 0, s>>>(r);
    count_launch();
    return cudaGetLastError() == cudaSuccess ? DVM_OK : DVM_ECUDA;
}

int mlp_adam(Mlp &m, double lr, cudaStream_t s)
{
    m.steps++;
    const float b1 = 0.9f, b2 = 0.999f;
    const float c1 = 1.0f - powf(b1, (float)m.steps), c2 = 1.0f - powf(b2, (float)m.steps);
    k_adam<<<blocks(MLP_NPARAM), 256, 0, s>>>(m.w, m.m, m.v, m.g, MLP_NPARAM, (float)lr, b1, b2, 1e-8f, c1, c2);
    count_launch();
    return mlp_cast(m, s);
}

}  // namespace dvm
