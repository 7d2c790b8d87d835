// Lattice Boltzmann step on the tree (paper Sec. 4): finite-volume upwind
// transport of Eq. 2 on the lattice velocities, then the lattice BGK
// relaxation towards the second-order equilibrium, fused in one pass over f.
//
// Layout: f is [q][ld] (structure of arrays: velocity i of every cell is one
// contiguous row; column ncells holds the inflow ghost), so one thread per
// cell reads and writes each of its q values with fully coalesced warp
// accesses.  The upwind codes are [2 dim][ncells], also coalesced.  Upwind
// neighbours are gathered from the same rows: cells near in Morton order
// are near in the rows, so the gathers hit L1/L2.
#include <cuda_runtime.h>

#include <type_traits>

#include "../../include/dvm.h"
#include "lbm.hpp"

namespace dvm {

void count_launch();

namespace {

// The velocity set as compile-time tables (same rule as lbm_lattice: order
// by |c|^2, then lexicographic in (c_x, c_y, c_z)).
struct LatTab {
    int q = 0;
    int c[27][3] = {};
    int r2[27] = {};
    int mirror[27][3] = {};  // index of the velocity with component d negated
};

__host__ __device__ constexpr LatTab make_tab(int Q)
{
    LatTab t{};
    for (int r2 = 0; r2 <= 3; r2++)
        for (int x = -1; x <= 1; x++)
            for (int y = -1; y <= 1; y++)
                for (int z = -1; z <= 1; z++) {
                    if (x * x + y * y + z * z != r2) continue;
                    if (Q == 9 && z != 0) continue;
                    if (Q == 19 && r2 == 3) continue;
                    t.c[t.q][0] = x;
                    t.c[t.q][1] = y;
                    t.c[t.q][2] = z;
                    t.r2[t.q] = r2;
                    t.q++;
                }
    for (int i = 0; i < t.q; i++)
        for (int d = 0; d < 3; d++)
            for (int j = 0; j < t.q; j++) {
                bool same = true;
                for (int e = 0; e < 3; e++)
                    same = same && t.c[j][e] == (e == d ? -t.c[i][e] : t.c[i][e]);
                if (same) t.mirror[i][d] = j;
            }
    return t;
}

template <int Q> struct Lat {
    static constexpr LatTab t = make_tab(Q);
};

// every mirror exists, is an involution and negates exactly one component
__host__ __device__ constexpr bool tab_ok(int Q)
{
    const LatTab t = make_tab(Q);
    if (t.q != Q) return false;
    for (int i = 0; i < t.q; i++)
        for (int d = 0; d < 3; d++) {
            const int j = t.mirror[i][d];
            if (t.mirror[j][d] != i) return false;
            for (int e = 0; e < 3; e++)
                if (t.c[j][e] != (e == d ? -t.c[i][e] : t.c[i][e])) return false;
        }
    return true;
}
static_assert(tab_ok(9) && tab_ok(19) && tab_ok(27), "lattice tables");

// weight of |c|^2 class r2, exact quotients of small integers
template <typename T, int Q> __device__ constexpr T lat_w(int r2)
{
    if (Q == 9) return r2 == 0 ? T(4) / T(9) : r2 == 1 ? T(1) / T(9) : T(1) / T(36);
    if (Q == 19) return r2 == 0 ? T(1) / T(3) : r2 == 1 ? T(1) / T(18) : T(1) / T(36);
    return r2 == 0 ? T(8) / T(27) : r2 == 1 ? T(2) / T(27) : r2 == 2 ? T(1) / T(54) : T(1) / T(216);
}

// compile-time loop over velocities
template <int I, int Q> struct ForV {
    template <typename F> __device__ __forceinline__ static void run(F &&f)
    {
        f(std::integral_constant<int, I>{});
        ForV<I + 1, Q>::run(f);
    }
};
template <int Q> struct ForV<Q, Q> {
    template <typename F> __device__ __forceinline__ static void run(F &&) {}
};

// the side list (2d + s) whose sources velocity i takes along axis d: the
// minus side for c_d > 0, the plus side for c_d < 0
template <int Q> __host__ __device__ constexpr int side_of(int i, int d)
{
    return Lat<Q>::t.c[i][d] > 0 ? 2 * d : 2 * d + 1;
}

// compile-time loop over the 2 dim sides
template <int K, int NS> struct ForS {
    template <typename F> __device__ __forceinline__ static void run(F &&f)
    {
        f(std::integral_constant<int, K>{});
        ForS<K + 1, NS>::run(f);
    }
};
template <int NS> struct ForS<NS, NS> {
    template <typename F> __device__ __forceinline__ static void run(F &&) {}
};

// a value of f: overlapped steps are resident while f is still written, so
// theirs is no read-only load
template <bool OVL, typename T> __device__ __forceinline__ T ld_f(const T *a)
{
    if constexpr (OVL) return *a;
    else return __ldg(a);
}

// g_i += w f_e for every velocity i that takes side K, f_e the source's
// value of velocity i (or of its mirror along the side's axis for a wall;
// WALLS: the side may be one)
template <typename T, int Q, int K, bool WALLS, bool OVL>
__device__ __forceinline__ void add_side(T (&g)[Q], const T *fin, int64_t ld, uint32_t src, bool wall, T w)
{
    constexpr int d = K / 2;
    ForV<0, Q>::run([&](auto II) {
        constexpr int i = decltype(II)::value;
        if constexpr (Lat<Q>::t.c[i][d] != 0 && side_of<Q>(i, d) == K) {
            if constexpr (WALLS) {
                constexpr int jm = Lat<Q>::t.mirror[i][d];
                g[i] += w * ld_f<OVL>(fin + (int64_t)(wall ? jm : i) * ld + src);
            } else {
                g[i] += w * ld_f<OVL>(fin + (int64_t)i * ld + src);
            }
        }
    });
}

// Fused step.  Every side's first source is decoded once (a side with
// several finer sources starts from its first overflow entry), and all
// first-source gathers are issued without branches, so a thread keeps its
// gathers in flight together; the remaining entries of sides with 2 or 4
// finer sources are added in a second pass that few threads take.
// CTAs of 256 threads per SM that the register budget is sized for: more
// registers keep more of a thread's gathers in flight, more CTAs hide more
// latency
__host__ __device__ constexpr int lbm_min_blocks(int Q, int tsize)
{
    return tsize == 8 ? 2 : Q == 27 ? 3 : Q == 19 ? 4 : 4;
}

template <typename T, int DIM, int Q, bool OVL>
__global__ void __launch_bounds__(256, lbm_min_blocks(Q, sizeof(T))) k_lbm(const LbmParams p)
{
    const int64_t cell = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const unsigned lanes = __ballot_sync(0xffffffffu, cell < p.ncells);
    if (cell >= p.ncells) return;
    const T *fin = static_cast<const T *>(p.f_in);
    T *fout = static_cast<T *>(p.f_out);
    const int64_t ld = p.ld, nc = p.ncells;
    constexpr int NS = 2 * DIM;
    uint32_t code[NS];
#pragma unroll
    for (int k = 0; k < NS; k++) code[k] = __ldg(p.codes + (int64_t)k * nc + cell);
    // dt / h and dt / (2^(dim-1) h), h = 2^-level
    const T dth = T(p.dt) * T(1ull << __ldg(p.lev + cell));
    const T dtq = dth * (T(1) / T(1 << (DIM - 1)));
    // Overlapped steps: the tree's codes above are the same for every step and
    // are read while the step before still runs; f, the status word and every
    // store wait for its end.  The trigger comes after the wait, so that a
    // grid is resident only beside the one right before it.
    if constexpr (OVL) {
        asm volatile("griddepcontrol.wait;" ::: "memory");
        asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    }
    // f_i (1 - dt n_i / h), n_i the number of non-zero components of c_i
    T g[Q];
    ForV<0, Q>::run([&](auto II) {
        constexpr int i = decltype(II)::value;
        constexpr int cx = Lat<Q>::t.c[i][0], cy = Lat<Q>::t.c[i][1], cz = Lat<Q>::t.c[i][2];
        constexpr int na = (cx != 0) + (cy != 0) + (DIM == 3 && cz != 0);
        const T v = ld_f<OVL>(fin + (int64_t)i * ld + cell);
        g[i] = v - dth * T(na) * v;
    });
    // transport, Eq. 2: add dt m_e f_e / (2^(dim-1) h) over each upwind
    // side's sources, first sources for all sides at once.  Warps without a
    // wall or a side with several sources, most of them, take the copy without
    // the choice of a mirrored row per gather (602k cells D3Q19 FP32, 0.19 GB
    // a step and its codes: 31.9 -> 25.0 us; the kernel waits on its gathers
    // and issues 59% of the cycles; 3, 5 and 6 CTAs an SM 28.4, 30.1, 32.8 us).
    uint32_t any = 0;
#pragma unroll
    for (int k = 0; k < NS; k++) any |= code[k];
    if (!__any_sync(lanes, any & (LBM_OVF | LBM_WALL))) {
        ForS<0, NS>::run([&](auto KK) {
            constexpr int k = decltype(KK)::value;
            add_side<T, Q, k, false, OVL>(g, fin, ld, code[k] & LBM_CELL, false,
                                     dtq * T((int)((code[k] >> LBM_M_SHIFT) & 3u) + 1));
        });
    } else {
        bool any_ovf = false;
        ForS<0, NS>::run([&](auto KK) {
            constexpr int k = decltype(KK)::value;
            uint32_t e = code[k];
            if (e & LBM_OVF) {
                any_ovf = true;
                e = __ldg(p.ovf + (e & LBM_CELL));
            }
            add_side<T, Q, k, true, OVL>(g, fin, ld, e & LBM_CELL, (e & LBM_WALL) != 0,
                                    dtq * T((int)((e >> LBM_M_SHIFT) & 3u) + 1));
        });
        if (any_ovf) {
            ForS<0, NS>::run([&](auto KK) {
                constexpr int k = decltype(KK)::value;
                if (code[k] & LBM_OVF) {
                    const uint32_t base = code[k] & LBM_CELL;
                    const int n = (int)((code[k] >> LBM_M_SHIFT) & 3u) + 1;
                    for (int j = 1; j < n; j++) {
                        const uint32_t e = __ldg(p.ovf + base + j);
                        add_side<T, Q, k, true, OVL>(g, fin, ld, e & LBM_CELL, (e & LBM_WALL) != 0,
                                                dtq * T((int)((e >> LBM_M_SHIFT) & 3u) + 1));
                    }
                }
            });
        }
    }
    // moments of f*
    T rho = T(0), jx = T(0), jy = T(0), jz = T(0);
    ForV<0, Q>::run([&](auto II) {
        constexpr int i = decltype(II)::value;
        constexpr int cx = Lat<Q>::t.c[i][0], cy = Lat<Q>::t.c[i][1], cz = Lat<Q>::t.c[i][2];
        rho += g[i];
        if constexpr (cx > 0) jx += g[i];
        if constexpr (cx < 0) jx -= g[i];
        if constexpr (cy > 0) jy += g[i];
        if constexpr (cy < 0) jy -= g[i];
        if constexpr (cz > 0) jz += g[i];
        if constexpr (cz < 0) jz -= g[i];
    });
    const T irho = T(1) / rho;
    const T ux = jx * irho, uy = jy * irho, uz = jz * irho;
    if (!(rho > T(0)) || !isfinite(ux + uy + uz)) atomicOr(p.status, 1);
    const T om = T(p.omega);
    const T q0 = T(1) - T(1.5) * (ux * ux + uy * uy + uz * uz);
    // BGK towards feq_i = w_i rho (1 + 3 c.u + 4.5 (c.u)^2 - 1.5 |u|^2)
    ForV<0, Q>::run([&](auto II) {
        constexpr int i = decltype(II)::value;
        constexpr int cx = Lat<Q>::t.c[i][0], cy = Lat<Q>::t.c[i][1], cz = Lat<Q>::t.c[i][2];
        constexpr int r2 = Lat<Q>::t.r2[i];
        const T cu = T(cx) * ux + T(cy) * uy + T(cz) * uz;
        const T feq = lat_w<T, Q>(r2) * rho * (q0 + cu * (T(3) + T(4.5) * cu));
        fout[(int64_t)i * ld + cell] = g[i] - om * (g[i] - feq);
    });
}

// rho [ncells] and u [ncells][3] of the stored f in FP64.  FP32 values are
// summed exactly on the FP32 pipe (FP64 runs at 1/64 of its rate): each splits
// without error against 2^k > 32 max|f| into a multiple of 2^(k-24), a multiple
// of 2^(k-42) and a rest, and the sums of either multiple over a cell are exact
// in FP32 (the extraction of Rump, Ogita and Oishi, 2008).  602k cells
// D3Q19: the FP64 sums took 136 us.
template <typename T, int Q>
__global__ void __launch_bounds__(256) k_lbm_moments(const T *__restrict__ f, int64_t ncells, int64_t ld,
                                                     double *__restrict__ out)
{
    const int64_t cell = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (cell >= ncells) return;
    T v[Q];
    ForV<0, Q>::run([&](auto II) {
        constexpr int i = decltype(II)::value;
        v[i] = __ldg(f + (int64_t)i * ld + cell);
    });
    // s[0] = sum x_i, s[1 + d] = sum c_id x_i
    auto sums = [&](const T(&x)[Q], auto &s) {
        ForV<0, Q>::run([&](auto II) {
            constexpr int i = decltype(II)::value;
            constexpr int cx = Lat<Q>::t.c[i][0], cy = Lat<Q>::t.c[i][1], cz = Lat<Q>::t.c[i][2];
            s[0] += x[i];
            if constexpr (cx > 0) s[1] += x[i];
            if constexpr (cx < 0) s[1] -= x[i];
            if constexpr (cy > 0) s[2] += x[i];
            if constexpr (cy < 0) s[2] -= x[i];
            if constexpr (cz > 0) s[3] += x[i];
            if constexpr (cz < 0) s[3] -= x[i];
        });
    };
    double m[4] = {0, 0, 0, 0};
    bool wide = true;
    if constexpr (sizeof(T) == 4) {
        uint32_t mx = 0;
#pragma unroll
        for (int i = 0; i < Q; i++) mx = max(mx, __float_as_uint(v[i]) & 0x7fffffffu);
        const int ex = (int)(mx >> 23);  // max|f| < 2^(ex - 126)
        wide = ex < 48 || ex > 240;
        if (!wide) {
            const float sg1 = __int_as_float((ex + 7) << 23), sg2 = __int_as_float((ex - 11) << 23);
            float q[Q], s1[4] = {0, 0, 0, 0}, s2[4] = {0, 0, 0, 0}, s3[4] = {0, 0, 0, 0};
#pragma unroll
            for (int i = 0; i < Q; i++) {
                q[i] = __fadd_rn(__fadd_rn(v[i], sg1), -sg1);
                v[i] -= q[i];
            }
            sums(q, s1);
#pragma unroll
            for (int i = 0; i < Q; i++) {
                q[i] = __fadd_rn(__fadd_rn(v[i], sg2), -sg2);
                v[i] -= q[i];
            }
            sums(q, s2);
            sums(v, s3);
#pragma unroll
            for (int k = 0; k < 4; k++) m[k] = (double)s1[k] + ((double)s2[k] + (double)s3[k]);
        }
    }
    if (wide) sums(v, m);
    out[cell] = m[0];
#pragma unroll
    for (int d = 0; d < 3; d++) out[ncells + 3 * cell + d] = m[1 + d] / m[0];
}

template <typename T, int DIM, int Q> int launch_t(const LbmParams &p)
{
    const unsigned grid = (unsigned)((p.ncells + p.threads - 1) / p.threads);
    if (p.overlap) {
        cudaLaunchAttribute at{};
        at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
        at.val.programmaticStreamSerializationAllowed = 1;
        cudaLaunchConfig_t lc{};
        lc.gridDim = dim3(grid);
        lc.blockDim = dim3(p.threads);
        lc.stream = p.stream;
        lc.attrs = &at;
        lc.numAttrs = p.follows ? 1 : 0;
        if (cudaLaunchKernelEx(&lc, k_lbm<T, DIM, Q, true>, p) != cudaSuccess) return DVM_ECUDA;
    } else {
        k_lbm<T, DIM, Q, false><<<grid, p.threads, 0, p.stream>>>(p);
    }
    count_launch();
    return cudaGetLastError() == cudaSuccess ? DVM_OK : DVM_ECUDA;
}

template <typename T> int launch_prec(const LbmParams &p)
{
    if (p.dim == 2 && p.q == 9) return launch_t<T, 2, 9>(p);
    if (p.dim == 3 && p.q == 19) return launch_t<T, 3, 19>(p);
    if (p.dim == 3 && p.q == 27) return launch_t<T, 3, 27>(p);
    return DVM_EINVAL;
}

template <typename T>
int launch_mom_t(int q, const void *f, int64_t ncells, int64_t ld, double *out, cudaStream_t s)
{
    const unsigned blocks = (unsigned)((ncells + 255) / 256);
    const T *ft = static_cast<const T *>(f);
    if (q == 9) k_lbm_moments<T, 9><<<blocks, 256, 0, s>>>(ft, ncells, ld, out);
    else if (q == 19) k_lbm_moments<T, 19><<<blocks, 256, 0, s>>>(ft, ncells, ld, out);
    else if (q == 27) k_lbm_moments<T, 27><<<blocks, 256, 0, s>>>(ft, ncells, ld, out);
    else return DVM_EINVAL;
    count_launch();
    return cudaGetLastError() == cudaSuccess ? DVM_OK : DVM_ECUDA;
}

}  // namespace

// Threads per CTA: 256, fewer where that leaves SMs without a CTA (1,388
// cells D2Q9 FP64 ran on six SMs, each bound by its FP64 pipe:
// 14.5 -> 8.4 us a step).
int lbm_threads(int64_t ncells, int nsm)
{
    int t = 256;
    while (t > 32 && (ncells + t - 1) / t < nsm) t /= 2;
    return t;
}

// Steps that overlap the one before (their launch and the codes' latency), by
// the cells an SM has.  FP32, at most as many as threads fit on an SM: 1.15 to
// 1.9 times faster from 476 to 284k cells (D2Q9 5,508 cells: 4.2 -> 2.9 us;
// D3Q19 68,880 8.3 -> 5.6, 283,640 12.2 -> 9.7), 1.07 to 1.2 at 355k; larger grids
// hide both behind their own CTAs and keep the read-only loads (602k D3Q19
// within 1%; 3.34M 0.120 -> 0.123 ms D3Q19, 0.178 -> 0.199 D3Q27).  FP64 is bound by
// its pipe, and CTAs that become resident early spread unevenly over the SMs
// once they are large (D2Q9 63,480 cells on 256 threads: 20.6 -> 28.2 us), so
// only grids on CTAs of up to 128 threads: 1.06 to 1.36 times faster up to 20k
// cells (D2Q9 1,388 cells: 8.3 -> 6.8 us).
bool lbm_overlap(int prec, int64_t ncells, int nsm)
{
    return ncells <= (int64_t)nsm * (prec == DVM_F64 ? 128 : 2048);
}

int launch_lbm(const LbmParams &p)
{
    if (p.ncells <= 0) return DVM_OK;
    if (p.prec == DVM_F64) return launch_prec<double>(p);
    if (p.prec == DVM_F32) return launch_prec<float>(p);
    return DVM_ENOTIMPL;
}

int launch_lbm_moments(int prec, int q, const void *f, int64_t ncells, int64_t ld, double *out, cudaStream_t s)
{
    if (ncells <= 0) return DVM_OK;
    if (prec == DVM_F64) return launch_mom_t<double>(q, f, ncells, ld, out, s);
    if (prec == DVM_F32) return launch_mom_t<float>(q, f, ncells, ld, out, s);
    return DVM_ENOTIMPL;
}

}  // namespace dvm
