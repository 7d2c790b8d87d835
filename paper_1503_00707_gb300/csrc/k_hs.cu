// Hard-sphere discrete collision integral (paper Sec. 3.2, Eqs. 3-6).
//
// The trial table (gamma, l, m, b for every node i and trial k) is the same
// for all cells (Sec. 3.2), and each trial needs three random gathers from a
// cell's f.  The paper's kernel keeps one node's table in shared memory and
// gathers f across cells from a velocity-major copy; here the roles are
// swapped to keep every gather on chip:
//
//  k_hs_pairs   interleaves the f of two cells, so that one 64-bit gather
//            serves both;
//  k_hs_gather  table-stationary: a CTA of 512 threads holds the weighted
//            trials of some nodes in registers (64 or 48 per thread) and
//            streams pairs of cells through two shared-memory tiles, each a
//            single bulk copy (cp.async.bulk, completion on an mbarrier).  It
//            writes B_i = sum_k b f_gamma (Eq. 4) or C_i = sum_k c f_l f_m
//            (Eq. 5) for its nodes to per-cell scratch arrays.
//  k_hs_bc   the same sums one cell at a time, for grids whose pair tiles do
//            not fit in shared memory twice (more than 14,336 nodes).
//  k_hs_corr per cell: the five coefficients of P (Eq. 6) from the moment
//            system, its sums formed in an integer basis to about twice
//            FP32 precision (hs_sums.cuh), solved in the centred basis
//            (1, c, |c|^2 - 3), c = (xi - u)/sqrt(T), and refined against
//            those sums in FP64; then I = -f P B + C and f <- f + dt/Kn I in
//            place.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <mutex>

#include "../../include/dvm.h"
#include "async.cuh"
#include "common.cuh"
#include "hs.hpp"
#include "hs_sums.cuh"

namespace dvm {

void count_launch();

namespace {

constexpr int HE = 32;    // trials held per thread of k_hs_bc
constexpr int HT = 512;   // threads per CTA of k_hs_bc
constexpr int CT = 128;   // threads per CTA of k_hs_corr (at most)

// The rows of a batch: rows r0, r0 + 1, .. (at most nb) of the cells, or of
// a device list of cells.
struct Rows {
    int64_t r0, nb, ncells;
    const int32_t *list;  // may be null
    const int *n;         // entries of the list
    __device__ int64_t count() const
    {
        const int64_t left = (list ? (int64_t)*n : ncells) - r0;
        return left < 0 ? 0 : left < nb ? left : nb;
    }
    __device__ int64_t cell(int64_t r) const { return list ? (int64_t)list[r0 + r] : r0 + r; }
};

// f of the batch's rows as pairs: out [row / 2][nv][2]; the missing partner
// of an odd last row is zero.  HBM-bound: 12,016 cells x 24^3 (1.33 GB read
// and written) in 199 us, 3% of the gather kernel's time.
__global__ void __launch_bounds__(256) k_hs_pairs(const float *__restrict__ f, float4 *__restrict__ out, Rows rw, int nv)
{
    const int64_t n = rw.count(), r = 2 * (int64_t)blockIdx.x;
    if (r >= n) return;
    const bool two = r + 1 < n;
    const float4 *a = reinterpret_cast<const float4 *>(f + rw.cell(r) * nv);
    const float4 *b = reinterpret_cast<const float4 *>(f + rw.cell(two ? r + 1 : r) * nv);
    float4 *o = out + (int64_t)blockIdx.x * (nv / 2);
    for (int q = threadIdx.x; q < nv / 4; q += blockDim.x) {
        const float4 x = __ldg(a + q);
        float4 y = __ldg(b + q);
        if (!two) y = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        o[2 * q] = make_float4(x.x, y.x, x.y, y.y);
        o[2 * q + 1] = make_float4(x.z, y.z, x.w, y.w);
    }
}

// ---------------------------------------------------------------- pairs of cells
// What bounds it: the shared-memory pipe.  A trial costs one (B) or two (C)
// 64-bit gathers for two cells; a warp's gather takes two wavefronts without
// conflicts and about 2.6 with the order that hs_pack finds, against 1.5
// instruction issue cycles, and each pair's tile costs its own write into
// shared memory.  The 96 registers a thread holds of the table set how many
// nodes a tile serves.
constexpr int GT = 32 * HS_WARPS;                 // threads of k_hs_gather
constexpr uint32_t STAGE = 8u * HS_PAIR_MAX_NV;  // distance of the two tiles

struct GatherArgs {
    const float2 *pairs;
    float *out[2];  // B and C planes, [rows][nv]
    Rows rw;
    int nv, chunks;
    const uint32_t *tab, *lane;
    const uint8_t *desc;
    int *status;
};

__device__ inline float2 lds_pair(uint32_t addr)
{
    float2 v;
    asm volatile("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(addr));
    return v;
}

// The pairs p0 .. p1 - 1 on one warp of kind KIND with 8 NG slots.  The last
// warp to leave a tile refills it with the pair after next, so no warp waits
// for another but through the tiles.
template <int KIND, int NG>
__device__ __forceinline__ void gather_pairs(const GatherArgs &g, int warp, int p0, int np, bool odd, uint32_t tile,
                                             uint64_t *full, int *left)
{
    constexpr int SL = 8 * NG, BROW = HS_ROWS - hs_slots(KIND);
    constexpr uint32_t MASK = 0x1fff8u;
    const int lane = threadIdx.x & 31;
    const uint32_t *tb = g.tab + (int64_t)warp * (HS_ROWS * 32) + lane;
    uint32_t w[KIND ? SL : SL / 2];
    float b[SL];
#pragma unroll
    for (int e = 0; e < (KIND ? SL : SL / 2); e++) w[e] = __ldg(tb + 32 * e);
#pragma unroll
    for (int e = 0; e < SL; e++) b[e] = __uint_as_float(__ldg(tb + 32 * (BROW + e)));
    const uint32_t lt = __ldg(g.lane + (int64_t)warp * 32 + lane);
    const uint32_t node = lt & 0xfffffu;
    const int t = 1 << (lt >> 20);
    const bool writes = node != HS_NO_NODE && (lane & (t - 1)) == 0;
    float *out = g.out[KIND] + 2 * (int64_t)p0 * g.nv + node;
    for (int p = 0; p < np; p++) {
        const int s = p & 1;
        const uint32_t base = tile + (s ? STAGE : 0u);
        if (!mbar_wait(&full[s], (uint32_t)(p >> 1) & 1u)) {
            // a tile never arrived: report, and leave no copy in flight behind
            // (the other tile's is the next pair's, if there is one)
            if (lane == 0) atomicOr(g.status, ST_TIMEOUT);
            mbar_wait(&full[s], (uint32_t)(p >> 1) & 1u);
            if (p + 1 < np) mbar_wait(&full[s ^ 1], (uint32_t)((p + 1) >> 1) & 1u);
            return;
        }
        float2 acc = make_float2(0.0f, 0.0f);
#pragma unroll
        for (int e = 0; e < SL; e++) {
            // keep the offsets' extraction inside the loop (hoisted, the
            // extracted offsets would need another 32 to 48 registers)
            if (KIND == 1 || (e & 1) == 0) asm volatile("" : "+r"(w[KIND ? e : e / 2]));
            if constexpr (KIND == 0) {
                const uint32_t at = (e & 1) ? (w[e / 2] >> 14) & MASK : w[e / 2] & MASK;
                const float2 v = lds_pair(base + at);
                acc.x = fmaf(b[e], v.x, acc.x);
                acc.y = fmaf(b[e], v.y, acc.y);
            } else {
                const float2 l = lds_pair(base + (w[e] & MASK)), m = lds_pair(base + ((w[e] >> 14) & MASK));
                const float2 v = __fmul2_rn(l, m);
                acc.x = fmaf(b[e], v.x, acc.x);
                acc.y = fmaf(b[e], v.y, acc.y);
            }
        }
        __syncwarp();
        if (lane == 0) {
            __threadfence_block();
            if (atomicAdd(&left[s], 1) == HS_WARPS - 1) {
                __threadfence_block();
                left[s] = 0;
                if (p + 2 < np) {
                    mbar_expect_tx(&full[s], 8u * (uint32_t)g.nv);
                    bulk_g2s_addr(base, g.pairs + (int64_t)(p0 + p + 2) * g.nv, 8u * (uint32_t)g.nv, &full[s]);
                }
            }
        }
        for (int m = 1; m < t; m <<= 1) {
            acc.x += __shfl_xor_sync(0xffffffffu, acc.x, m);
            acc.y += __shfl_xor_sync(0xffffffffu, acc.y, m);
        }
        if (writes) {
            out[0] = acc.x;
            if (p + 1 < np || !odd) out[g.nv] = acc.y;
        }
        out += 2 * (int64_t)g.nv;
    }
}

// CTA (segment, chunk): the nodes of a chunk of the tables for a segment of
// the batch's pairs.
__global__ void __launch_bounds__(GT, 1) k_hs_gather(const GatherArgs g)
{
    extern __shared__ __align__(128) unsigned char gtile[];  // two tiles, STAGE apart
    __shared__ __align__(8) uint64_t full[2];
    __shared__ int left[2];
    const int nrows = (int)g.rw.count(), npairs = (nrows + 1) / 2;  // a batch is below 2^31 rows
    const int nseg = gridDim.x / g.chunks, per = (npairs + nseg - 1) / nseg;
    const int p0 = (int)(blockIdx.x / g.chunks) * per, np = min(per, npairs - p0);
    if (np <= 0) return;
    const bool odd = (nrows & 1) && p0 + np == npairs;  // the last pair has one cell
    const int chunk = blockIdx.x % g.chunks;
    const uint32_t tile = smem_u32(gtile);
    if (threadIdx.x == 0) {
        mbar_init(&full[0], 1);
        mbar_init(&full[1], 1);
        left[0] = left[1] = 0;
        mbar_fence_init();
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        const uint32_t bytes = 8u * (uint32_t)g.nv;
        for (int s = 0; s < 2 && s < np; s++) {
            mbar_expect_tx(&full[s], bytes);
            bulk_g2s_addr(tile + (s ? STAGE : 0u), g.pairs + (int64_t)(p0 + s) * g.nv, bytes, &full[s]);
        }
    }
    const int warp = chunk * HS_WARPS + (threadIdx.x >> 5);
#define DVM_RUN(K, N) \
    case (K << 7 | N): gather_pairs<K, N>(g, warp, p0, np, odd, tile, full, left); break;
    switch (g.desc[chunk]) {
        DVM_RUN(0, 1) DVM_RUN(0, 2) DVM_RUN(0, 3) DVM_RUN(0, 4)
        DVM_RUN(0, 5) DVM_RUN(0, 6) DVM_RUN(0, 7) DVM_RUN(0, 8)
        DVM_RUN(1, 1) DVM_RUN(1, 2) DVM_RUN(1, 3) DVM_RUN(1, 4) DVM_RUN(1, 5) DVM_RUN(1, 6)
    }
#undef DVM_RUN
    // the copies issued ahead have all been waited for (or given up on) above
}

// ---------------------------------------------------------------- one cell at a time
__global__ void __launch_bounds__(HT, 1)
    k_hs_bc(const float *__restrict__ fs, float *__restrict__ Bp, float *__restrict__ Cp, Rows rw, int nv, int M,
            const uint2 *__restrict__ idx, const float *__restrict__ bw, int *status)
{
    extern __shared__ __align__(128) float tile[];  // [2][nv]
    __shared__ __align__(8) uint64_t bar[2];
    __shared__ int abort_flag;

    const int tid = threadIdx.x;
    const int tpn = M / HE;  // threads per node (power of two, <= 32)
    const int npc = HT / tpn;
    const int node = blockIdx.x * npc + tid / tpn;
    const bool valid = node < nv;
    const int64_t e0 = (int64_t)(valid ? node : 0) * M + (tid % tpn) * HE;
    uint32_t w0[HE], w1[HE];
    float b[HE];
#pragma unroll
    for (int e = 0; e < HE; e++) {
        const uint2 t = idx[e0 + e];
        w0[e] = t.x;
        w1[e] = t.y;
        b[e] = valid ? bw[e0 + e] : 0.0f;
    }
    // rows c0..c1-1 of the batch for this CTA
    const int64_t nrows = rw.count();
    const int64_t per = (nrows + gridDim.y - 1) / gridDim.y;
    const int64_t c0 = (int64_t)blockIdx.y * per;
    const int64_t c1 = c0 + per < nrows ? c0 + per : nrows;
    auto src = [&](int64_t r) { return fs + rw.cell(r) * nv; };
    const uint32_t bytes = (uint32_t)nv * 4u;
    if (tid == 0) {
        mbar_init(&bar[0], 1);
        mbar_init(&bar[1], 1);
        abort_flag = 0;
        mbar_fence_init();
    }
    __syncthreads();
    // copies issued into / completions seen on each buffer (uniform over the CTA)
    int issued[2] = {0, 0}, done[2] = {0, 0};
    if (c0 < c1) {
        if (tid == 0) {
            mbar_expect_tx(&bar[0], bytes);
            bulk_g2s(tile, src(c0), bytes, &bar[0]);
        }
        issued[0]++;
    }
    for (int64_t c = c0; c < c1; c++) {
        const int j = (int)(c - c0), s = j & 1;
        if (c + 1 < c1) {
            // buffer s^1 was last read in the previous iteration, which ended
            // with a barrier
            if (tid == 0) {
                mbar_expect_tx(&bar[s ^ 1], bytes);
                bulk_g2s(tile + (size_t)(s ^ 1) * nv, src(c + 1), bytes, &bar[s ^ 1]);
            }
            issued[s ^ 1]++;
        }
        if (mbar_wait(&bar[s], (uint32_t)done[s] & 1u)) done[s]++;
        else abort_flag = 1;
        const float *t = tile + (size_t)s * nv;
        float B = 0.0f, C = 0.0f;
#pragma unroll
        for (int e = 0; e < HE; e++) {
            const float fg = t[w0[e] & 0xffffu];
            const float fl = t[w0[e] >> 16];
            const float fm = t[w1[e]];
            B = fmaf(b[e], fg, B);
            C = fmaf(b[e], fl * fm, C);
        }
        for (int m = 1; m < tpn; m <<= 1) {
            B += __shfl_xor_sync(0xffffffffu, B, m);
            C += __shfl_xor_sync(0xffffffffu, C, m);
        }
        if (valid && tid % tpn == 0) {
            Bp[c * nv + node] = B;
            Cp[c * nv + node] = C;
        }
        __syncthreads();
        if (abort_flag) {
            // a tile never arrived: report, give the copies in flight a bounded
            // time to land, and stop
            if (tid == 0) {
                atomicOr(status, ST_TIMEOUT);
                for (int q = 0; q < 2; q++)
                    while (done[q] < issued[q] && mbar_wait(&bar[q], (uint32_t)done[q] & 1u)) done[q]++;
            }
            return;
        }
    }
}

// k_hs_corr: one CTA per cell.  The correction polynomial of Eq. 6,
// P = 1 + d.phi, phi = (1, c, |c|^2 - 3), c = (xi - u)/sqrt(T), makes
// I = C - f P B conserve mass, momentum and energy.  With xi_d = (h/2) j_d
// (j_d odd integers, the same h on every axis) the integer basis psi^ = (1,
// j_x, j_y, j_z, |j|^2) spans the same polynomials, so the 15 sums A^_rs =
// sum_i psi^_r psi^_s f_i B_i and the 5 sums c^_r = sum_i psi^_r C_i have
// integer weights.  A thread takes two z nodes at one position of all eight
// sign groups (hs_sums.cuh): about 30 operations a node where a node at a time
// takes 72, at the same precision (3e-15 of the terms' sizes at worst, rms 6e-16).
// The lanes of warp 0 solve A^ e = c^, e = (1, 0, 0, 0, 0) + L^T d (L the map
// psi^ -> phi), through the well-conditioned L A^ L^T, refined against FP64
// residuals of the sums.  The last residual, sum_i psi_r I_i dV with
// psi = (1, xi, |xi|^2), goes to res (may be null).  Then I_i is evaluated in
// FP32 with the FP32 copy of d and f <- f + dt/Kn I (or I to q_out).
// Bound by HBM at best (f, B, C in, f out); 12,016 cells x 24^3 (2.66 GB):
// 1.81 -> 0.87 ms, 16,584 x 16^3 0.94 -> 0.53 ms (a node at a time, FP64 factor,
// 256 threads before); what is left is the serial solve and the sums' reduction
// per cell.
// five CTAs of 128 threads per SM (96 registers): four other cells' passes
// overlap one cell's serial solve (whole steps at 16^3 / 24^3: 3.42 / 7.65 ms;
// 4 x 128 without spills 3.48 / 7.66)
__global__ void __launch_bounds__(CT, 5)
    k_hs_corr(float *__restrict__ f, const float *__restrict__ Bp, const float *__restrict__ Cp,
              const float *__restrict__ xi3, double hh, double dV, const double *__restrict__ mom, int nv, int3 half,
              float dtkn, Rows rw, float *__restrict__ q_out, double *__restrict__ res, int *status)
{
    __shared__ ffn part[NSUM][CT];
    __shared__ double S[NSUM], Lm[25];
    __shared__ float sd[5];
    // row blockIdx.x of B and C belongs to this cell (an entry of the list, if any)
    const int64_t row = blockIdx.x;
    if (row >= rw.count()) return;
    const int64_t cell = rw.cell(row);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, T = blockDim.x;
    const double *mo = mom + cell * 5;
    const double rho = mo[0], Td = mo[4];
    if (!(rho > 0.0) || !(Td > 0.0) || !isfinite(rho + Td + mo[1] + mo[2] + mo[3])) {
        // no correction exists: report, leave f as it is
        if (tid == 0) {
            atomicOr(status, ST_NONPOS);
            if (res)
                for (int r = 0; r < 5; r++) res[cell * 5 + r] = 0.0;
        }
        return;
    }
    const int P = nv / 8, hz = half.z;
    float *fc = f + cell * (int64_t)nv;
    const float *Bc = Bp + row * (int64_t)nv, *Cc = Cp + row * (int64_t)nv;
    auto ld2 = [](const float *p) { return __ldg(reinterpret_cast<const float2 *>(p)); };
    auto node = [&](int p, float &a, float &b, float &c) {
        const int t = p / hz;
        a = (float)(2 * (t / half.y) + 1);
        b = (float)(2 * (t % half.y) + 1);
        c = (float)(2 * (p - t * hz) + 1);
    };
    Acc2 acc[NSUM];
#pragma unroll
    for (int k = 0; k < NSUM; k++) acc[k] = Acc2{0.0f, 0.0f};
#pragma unroll 1
    for (int p = 2 * tid; p < P; p += 2 * T) {
        float a, b, c0;
        node(p, a, b, c0);
        float2 w[8], wl[8];
#pragma unroll
        for (int o = 0; o < 8; o++) {
            w[o] = *reinterpret_cast<const float2 *>(fc + o * P + p);
            wl[o] = ld2(Bc + o * P + p);
        }
        add_losses(acc, w, wl, a, b, c0);
    }
    // (a loop of its own: fewer accumulators at a time in registers)
#pragma unroll 1
    for (int p = 2 * tid; p < P; p += 2 * T) {
        float a, b, c0;
        node(p, a, b, c0);
        float2 w[8];
#pragma unroll
        for (int o = 0; o < 8; o++) w[o] = ld2(Cc + o * P + p);
        add_gains(acc, w, a, b, c0);
    }
#pragma unroll
    for (int k = 0; k < NSUM; k++) {
        float lo;
        const float hi = two_sum(acc[k].s, acc[k].e, lo);
        part[k][tid] = ffn{hi, lo};
    }
    __syncthreads();
    // the warps take the sums in turn and add each over the CTA in double-float
    for (int k = warp; k < NSUM; k += T / 32) {
        ffn a = part[k][lane];
#pragma unroll 4
        for (int t = lane + 32; t < T; t += 32) a = a + part[k][t];
#pragma unroll
        for (int m = 16; m > 0; m >>= 1)
            a = a + ffn{__shfl_xor_sync(0xffffffffu, a.hi, m), __shfl_xor_sync(0xffffffffu, a.lo, m)};
        if (lane == 0) S[k] = (double)a.hi + (double)a.lo;
    }
    __syncthreads();
    if (warp == 0) {
        // The 5x5 solve on the lanes of warp 0.  phi = L psi^ with
        //   phi_0 = 1, phi_d = be_d + al j_d, phi_4 = |be|^2 - 3 + 2 al be.j + al^2 |j|^2,
        // al = (h/2)/sqrt(T), be = -u/sqrt(T); the system A^ e = c^ with
        // e = (1, 0, 0, 0, 0) + L^T d is factored through the well-conditioned
        // centred-basis matrix L A^ L^T (an LDL^T on lane 0) and refined
        // against the FP64 residual of the sums.  The factor is FP32
        // with four rounds (each gains at least three digits; FP64 runs at
        // 1/64 of the FP32 rate, and an FP64 factor with two rounds took a
        // third of this kernel's time at 16^3); where it does not converge
        // to 1e-12, or a pivot fails, the FP64 factor follows.  Lane 5 r + s
        // holds entry (r, s) of the 5x5 products; lanes 0..4 hold the vectors.
        const double isT = 1.0 / sqrt(Td), al = hh * isT;
        if (lane < 25) {
            const int r = lane / 5, k = lane % 5;
            const double be0 = -mo[1] * isT, be1 = -mo[2] * isT, be2 = -mo[3] * isT;
            const double bk = k == 1 ? be0 : (k == 2 ? be1 : be2), br = r == 1 ? be0 : (r == 2 ? be1 : be2);
            double v = r == k ? (r == 0 ? 1.0 : al) : 0.0;
            if (r >= 1 && r < 4 && k == 0) v = br;
            if (r == 4) v = k == 0 ? be0 * be0 + be1 * be1 + be2 * be2 - 3.0 : (k < 4 ? 2.0 * al * bk : al * al);
            Lm[lane] = v;
        }
        __syncwarp();
        // entry (r, s) of A^ (index of the upper-triangle sum)
        auto Aj = [&](int r, int q) -> double {
            const int lo = r < q ? r : q, hi = r < q ? q : r;
            return S[lo * 5 - (lo * (lo - 1)) / 2 + (hi - lo)];
        };
        auto bcast = [](auto v, int src) { return __shfl_sync(0xffffffffu, v, src); };
        const int r5 = lane < 25 ? lane / 5 : 0, s5 = lane < 25 ? lane % 5 : 0;
        // T1 = L A^ (lane 5 r + s), then Ap = T1 L^T
        double t1 = 0.0;
#pragma unroll
        for (int k = 0; k < 5; k++) t1 = fma(Lm[r5 * 5 + k], Aj(k, s5), t1);
        double ap = 0.0;
#pragma unroll
        for (int k = 0; k < 5; k++) ap = fma(bcast(t1, r5 * 5 + k), Lm[s5 * 5 + k], ap);
        const int rv = lane < 5 ? lane : 0;
        double Arow[5], Lrow[5], Lcol[5];  // row rv of A^ and of L, column rv of L
#pragma unroll
        for (int k = 0; k < 5; k++) {
            Arow[k] = Aj(rv, k);
            Lrow[k] = Lm[rv * 5 + k];
            Lcol[k] = Lm[k * 5 + rv];
        }
        double d[5] = {0.0, 0.0, 0.0, 0.0, 0.0}, R = 0.0;  // every lane: d; lane r < 5: the residual's row r
        // R_r = c^_r - sum_s A^_rs e_s on lane r, e_s = (s == 0) + sum_k L_ks d_k
        auto residual = [&]() {
            double e = rv == 0 ? 1.0 : 0.0;
#pragma unroll
            for (int k = 0; k < 5; k++) e = fma(Lcol[k], d[k], e);
            R = S[15 + rv];
#pragma unroll
            for (int q = 0; q < 5; q++) R = fma(-Arow[q], bcast(e, q), R);
        };
        // `rounds` solves with a factor of type F, and the residual after them
        auto solve = [&](auto one, int rounds) -> bool {
            using F = decltype(one);
            F Ap[25], Lf[5][5], Di[5];
            const F av = (F)ap;
#pragma unroll
            for (int k = 0; k < 25; k++) Ap[k] = bcast(av, k);
            bool ok = true;
            if (lane == 0) ok = ldl5<F>(Ap, Lf, Di);
            ok = bcast(ok ? 1 : 0, 0) != 0;
            bool still = false;  // the last correction still moved d
#pragma unroll
            for (int k = 0; k < 5; k++) d[k] = 0.0;
            residual();
            for (int it = 0; it < rounds && ok; it++) {
                // LR = L R on lane r, then the LDL^T solve on lane 0
                double lr = 0.0;
#pragma unroll
                for (int k = 0; k < 5; k++) lr = fma(Lrow[k], bcast(R, k), lr);
                const F lf = (F)lr;
                F LR[5], dl[5] = {0, 0, 0, 0, 0};
#pragma unroll
                for (int k = 0; k < 5; k++) LR[k] = bcast(lf, k);
                if (lane == 0) ldl5_solve<F>(Lf, Di, LR, dl);
                still = false;
#pragma unroll
                for (int k = 0; k < 5; k++) {
                    const F x = bcast(dl[k], 0);
                    d[k] += (double)x;
                    still = still || !(fabsf((float)x) <= 1e-12f * (1.0f + fabsf((float)d[k])));
                }
                residual();
            }
            return ok && (sizeof(F) == 8 || !still);
        };
        bool ok = solve(0.0f, 4);
        if (!ok) ok = solve(0.0, 2);
        bool fin = ok;
#pragma unroll
        for (int k = 0; k < 5; k++) fin = fin && isfinite(d[k]);
        if (lane == 0 && !fin) atomicOr(status, ST_SINGULAR);
        if (lane < 5) {
            double dv = d[0];
#pragma unroll
            for (int k = 1; k < 5; k++) dv = lane == k ? d[k] : dv;
            sd[lane] = fin ? (float)dv : 0.0f;
            if (res) {
                const double sc = lane == 0 ? dV : (lane < 4 ? dV * hh : dV * hh * hh);
                res[cell * 5 + lane] = fin ? sc * R : 0.0;
            }
        }
    }
    __syncthreads();
    const float ux = (float)mo[1], uy = (float)mo[2], uz = (float)mo[3];
    const float ist = rsqrtf((float)Td);
    const float d0 = sd[0], dx = sd[1], dy = sd[2], dz = sd[3], d4 = sd[4];
    // P at node = (1 + d0 - 3 d4) + sum over the axes of c (d_axis + d4 c)
    auto axis = [&](float x, float u, float da) {
        const float cc = (x - u) * ist;
        return cc * fmaf(d4, cc, da);
    };
    const float k0 = 1.0f + d0 - 3.0f * d4;
    float *qc = q_out ? q_out + cell * (int64_t)nv : nullptr;
    float worst = 0.0f;
#pragma unroll 1
    for (int p = 2 * tid; p < P; p += 2 * T) {
        const int v = 7 * P + p;  // the node with every component positive
        const float x = xi3[v], y = xi3[nv + v];
        const float2 z = ld2(xi3 + 2 * nv + v);
        const float px[2] = {axis(-x, ux, dx), axis(x, ux, dx)}, py[2] = {axis(-y, uy, dy), axis(y, uy, dy)};
        const float2 pz[2] = {make_float2(axis(-z.x, uz, dz), axis(-z.y, uz, dz)),
                              make_float2(axis(z.x, uz, dz), axis(z.y, uz, dz))};
        float2 fv[8], bv[8], cv[8];
#pragma unroll
        for (int o = 0; o < 8; o++) {
            fv[o] = *reinterpret_cast<const float2 *>(fc + o * P + p);
            bv[o] = ld2(Bc + o * P + p);
            cv[o] = ld2(Cc + o * P + p);
        }
#pragma unroll
        for (int o = 0; o < 8; o++) {
            const float kxy = k0 + (px[o >> 2] + py[(o >> 1) & 1]);
            const float2 loss = __fmul2_rn(f2_add(make_float2(kxy, kxy), pz[o & 1]), bv[o]);
            worst = fmaxf(worst, dtkn * fmaxf(loss.x, loss.y));
            const float2 I = __ffma2_rn(make_float2(-fv[o].x, -fv[o].y), loss, cv[o]);
            if (qc) *reinterpret_cast<float2 *>(qc + o * P + p) = I;  // the term alone, f kept
            else
                *reinterpret_cast<float2 *>(fc + o * P + p) =
                    __ffma2_rn(make_float2(dtkn, dtkn), I, fv[o]);
        }
    }
    if (worst > 1.0f) atomicOr(status, ST_NUDT);
}

}  // namespace

bool hs_trials_supported(int trials)
{
    if (trials < HE || trials % HE) return false;
    const int tpn = trials / HE;
    return tpn <= 32 && (tpn & (tpn - 1)) == 0;
}

// Rows of one batch: scratch of 8 nv bytes a row for B and C and, for the
// pair kernel, 4 nv for f as pairs, 4 GB at most (24k cells at 24^3, enough to
// fill the GPU many times over; the scratch of a whole mesh would be three
// times its f).
static int64_t batch_rows(int64_t ncells, int nv, size_t bytes)
{
    const int64_t cap = std::max<int64_t>(2, (int64_t)(bytes / ((size_t)nv * 12)) & ~(int64_t)1);
    return std::min(cap, (ncells + 1) & ~(int64_t)1);
}

int hs_prepare(HsTables &t, int64_t ncells, const DevAlloc &alloc, const DevFree &dfree)
{
    if (!t.ready) return DVM_ESTATE;
    if (t.d_bc && t.prep_cells == ncells) return DVM_OK;
    if (t.d_bc) dfree(t.d_bc);
    t.prep_cells = 0;
    t.bc_cells = batch_rows(ncells, t.nv, (size_t)4 << 30);
    // one block (an allocation can cost a first step more than a small mesh's
    // kernels): B, C and, for the pair kernel, f as pairs
    t.d_bc = static_cast<float *>(alloc((size_t)t.bc_cells * t.nv * (t.chunks ? 3 : 2) * sizeof(float)));
    if (!t.d_bc) return DVM_ENOMEM;
    t.prep_cells = ncells;
    return DVM_OK;
}

// Cell splits of the k_hs_bc grid (node chunks x cell ranges): at least two
// waves of resident CTAs, and a total that fills its last wave as far as
// possible.  Every CTA streams the same number of cells, so a last wave that
// is only partly full leaves the rest of the GPU idle for a whole CTA's time
// (64 chunks x 10 ranges on 304 resident CTAs ran as 304 + 304 + 32).
static int64_t hs_splits(int chunks, int slots, int64_t ncells)
{
    const int64_t s0 = std::max<int64_t>(1, (2 * (int64_t)slots + chunks - 1) / chunks);
    int64_t best = s0;
    double best_eff = -1.0;
    for (int64_t sp = s0; sp <= 4 * s0; sp++) {
        const int64_t per = (ncells + sp - 1) / sp, used = (ncells + per - 1) / per;
        const int64_t total = (int64_t)chunks * used, waves = (total + slots - 1) / slots;
        const double eff = (double)total / (double)(waves * slots);
        if (eff > best_eff + 1e-9) {
            best_eff = eff;
            best = sp;
        }
    }
    return std::max<int64_t>(1, std::min<int64_t>(best, ncells));
}

// The launch of the B and C sums for batches of nb rows (the last may be
// shorter).  Every check that can refuse it is made here, before anything is
// queued.  Pair kernel: each CTA takes one chunk of the tables and a segment
// of the pairs; loading its tables costs about as much as three pairs, and
// CTAs are handed out as SMs come free, so that with W pair steps an SM a
// segment of sqrt(6 W) pairs balances the two (3 W / L against half a segment
// at the end).
struct BcLaunch {
    dim3 grid;
    size_t dyn = 0;
    int64_t nb = 0;
};

static int bc_plan(const HsTables &t, int nv, int64_t nb, BcLaunch &L)
{
    int dev = 0, nsm = 0, occ = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    L.nb = nb;
    if (t.chunks) {
        L.dyn = STAGE + 8 * (size_t)nv;
        if (cudaFuncSetAttribute(k_hs_gather, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(2 * STAGE)) !=
            cudaSuccess)
            return DVM_ECUDA;
        const int64_t pairs = (nb + 1) / 2;
        const double W = (double)pairs * t.chunks / nsm;
        int64_t len = std::max<int64_t>(1, (int64_t)std::sqrt(6.0 * W));
        len = std::min(len, std::max<int64_t>(1, pairs * t.chunks / nsm));
        L.grid = dim3((unsigned)(t.chunks * ((pairs + len - 1) / len)));
        return DVM_OK;
    }
    const int tpn = t.trials / HE, npc = HT / tpn;
    const int chunks = (nv + npc - 1) / npc;
    L.dyn = 2 * (size_t)nv * sizeof(float);
    if (L.dyn > 200 * 1024) return DVM_ENOTIMPL;
    if (cudaFuncSetAttribute(k_hs_bc, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024) != cudaSuccess)
        return DVM_ECUDA;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_hs_bc, HT, L.dyn) != cudaSuccess || occ < 1)
        return DVM_ENOTIMPL;
    L.grid = dim3((unsigned)chunks, (unsigned)hs_splits(chunks, nsm * occ, nb));
    return DVM_OK;
}

// What an update needs beside its rows.
struct CorrArgs {
    double dV;
    const double *mom;
    float dtkn;
    float *q_out;
    double *res;
};

// B, C and the correction, batch by batch.
static int run_batches(const BcLaunch &L, const HsTables &t, float *f, float *bc, float *pair, int nv, int64_t ncells,
                       const int32_t *list, const int *count, const CorrArgs &c, cudaStream_t s, int *status)
{
    float *Bp = bc, *Cp = bc + L.nb * nv;
    for (int64_t r0 = 0; r0 < ncells; r0 += L.nb) {
        const Rows rw{r0, L.nb, ncells, list, count};
        const unsigned rows = (unsigned)std::min(L.nb, ncells - r0);
        if (t.chunks) {
            k_hs_pairs<<<(rows + 1) / 2, 256, 0, s>>>(f, reinterpret_cast<float4 *>(pair), rw, nv);
            count_launch();
            const GatherArgs g{reinterpret_cast<const float2 *>(pair), {Bp, Cp}, rw, nv, t.chunks, t.d_tab, t.d_lane,
                               t.d_desc, status};
            k_hs_gather<<<L.grid, GT, L.dyn, s>>>(g);
        } else {
            k_hs_bc<<<L.grid, HT, L.dyn, s>>>(f, Bp, Cp, rw, nv, t.trials, reinterpret_cast<const uint2 *>(t.d_idx),
                                              t.d_b, status);
        }
        count_launch();
        // pairs of z nodes per sign group over rounds of at most CT threads,
        // evenly (24^3: 864 in 7 rounds of 124, on 128 threads)
        static_assert(CT % 32 == 0, "the rounding below stays within k_hs_corr's part[][CT]");
        const int units = nv / 16, rounds = (units + CT - 1) / CT, per = (units + rounds - 1) / rounds;
        k_hs_corr<<<rows, (per + 31) / 32 * 32, 0, s>>>(f, Bp, Cp, t.d_xi, t.hh, c.dV, c.mom, nv,
                                                        make_int3(t.half[0], t.half[1], t.half[2]), c.dtkn, rw,
                                                        c.q_out, c.res, status);
        count_launch();
        if (cudaGetLastError() != cudaSuccess) return DVM_ECUDA;
    }
    return DVM_OK;
}

int launch_hs_collide(HsTables &t, const StepParams &p, void *f, double kn, double dt)
{
    return launch_hs_general(t, p, static_cast<float *>(f), nullptr, nullptr, nullptr, kn, dt);
}

// The update on the cells of a device list only (*count entries, at most
// p.ncells), or, with q_out, the term I of every cell without the update.
int launch_hs_general(HsTables &t, const StepParams &p, float *f, const int32_t *list, const int *count,
                      float *q_out, double kn, double dt)
{
    if (p.prec != DVM_F32) return DVM_ENOTIMPL;
    if (!t.ready || t.nv != p.nv || !t.d_bc || t.prep_cells < p.ncells) return DVM_ESTATE;
    if (p.ncells <= 0) return DVM_OK;
    BcLaunch L;
    const int rc = bc_plan(t, p.nv, t.bc_cells, L);
    if (rc) return rc;
    const CorrArgs c{p.dV, p.mom_out, q_out ? 0.0f : (float)(dt / kn), q_out, q_out ? nullptr : p.res_out};
    return run_batches(L, t, f, t.d_bc, t.d_bc + 2 * t.bc_cells * p.nv, p.nv, p.ncells, list, count, c, p.stream, p.status);
}

// ---------------------------------------------------------------- allocation-free variant
namespace {

// Fixed scratch for dvm_hs_collide_noalloc.  It is part of the library's
// device image, so every GPU that loads the library holds it until the
// process exits; all calls share it.
constexpr size_t NOALLOC_BYTES = (size_t)DVM_HS_NOALLOC_SCRATCH_BYTES;
static __device__ __align__(256) unsigned char g_noalloc_scratch[NOALLOC_BYTES];

std::mutex g_noalloc_mu;
struct NoallocSlot {
    void *ctx = nullptr;  // the context the address belongs to
    void *ptr = nullptr;
};
NoallocSlot g_noalloc[256];

// The calling thread's current context (a CUcontext), through the driver
// entry point that the runtime hands out; null if it cannot be had.  Called
// with g_noalloc_mu held.
void *current_context()
{
    using Fn = int (*)(void **);
    static Fn fn = nullptr;
    static bool tried = false;
    if (!tried) {
        tried = true;
        void *f = nullptr;
        cudaDriverEntryPointQueryResult q = cudaDriverEntryPointSymbolNotFound;
        if (cudaGetDriverEntryPointByVersion("cuCtxGetCurrent", &f, 12000, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<Fn>(f);
        else
            cudaGetLastError();
    }
    void *ctx = nullptr;
    if (!fn || fn(&ctx) != 0) return nullptr;
    return ctx;
}

// Device address of the fixed scratch on the current device.  In host code
// g_noalloc_scratch names a host-side stand-in, so the address is looked up
// with the device current: once per device, and again if the device's
// context has been re-created since (after cudaDeviceReset the old address
// is stale).
int noalloc_scratch(void **ptr)
{
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 256) {
        cudaGetLastError();
        return DVM_ECUDA;
    }
    std::lock_guard<std::mutex> lock(g_noalloc_mu);
    NoallocSlot &slot = g_noalloc[dev];
    void *ctx = current_context();
    if (!slot.ptr || !ctx || slot.ctx != ctx) {
        void *p = nullptr;
        if (cudaGetSymbolAddress(&p, g_noalloc_scratch) != cudaSuccess || !p) {
            cudaGetLastError();
            return DVM_ECUDA;
        }
        slot.ptr = p;
        slot.ctx = current_context();  // the lookup has made the context current
    }
    *ptr = slot.ptr;
    return DVM_OK;
}

}  // namespace

int launch_hs_collide_noalloc(HsTables &t, const StepParams &p, float *f, const MomGrid &g, double kn, double dt)
{
    if (p.prec != DVM_F32) return DVM_ENOTIMPL;
    if (!t.ready || t.nv != p.nv) return DVM_ESTATE;
    const size_t mom_bytes = (size_t)p.ncells * 5 * sizeof(double);
    if ((size_t)p.ncells * p.nv * 2 * sizeof(float) + mom_bytes > NOALLOC_BYTES) return DVM_EINVAL;
    // every check comes before the first launch, so that a refusal queues no
    // work.  At the scratch limit the pairs of f leave room for two thirds of
    // the rows: two batches.
    BcLaunch L;
    int rc = bc_plan(t, p.nv, batch_rows(p.ncells, p.nv, NOALLOC_BYTES - mom_bytes - 64), L);
    if (rc) return rc;
    void *base = nullptr;
    rc = noalloc_scratch(&base);
    if (rc) return rc;
    float *bc = static_cast<float *>(base), *pair = bc + (size_t)L.nb * p.nv * 2;
    double *mom = reinterpret_cast<double *>(static_cast<unsigned char *>(base) + (NOALLOC_BYTES - mom_bytes) / 64 * 64);
    rc = launch_moments(DVM_F32, f, p.ncells, g, mom, p.stream);
    if (rc) return rc;
    const CorrArgs c{g.dV, mom, (float)(dt / kn), nullptr, nullptr};
    return run_batches(L, t, f, bc, pair, p.nv, p.ncells, nullptr, nullptr, c, p.stream, p.status);
}

}  // namespace dvm
