// Hard-sphere discrete collision integral (paper Sec. 3.2, Eqs. 3-6):
// seeded trial tables built on the host, collision kernel on the device.
#pragma once
#include <cstdint>
#include <functional>
#include <string>
#include <vector>

#include "../../include/dvm.h"
#include "kernels.hpp"

namespace dvm {

struct HsTables {
    bool ready = false;
    int trials = 0;
    uint64_t seed = 0;
    int nv = 0;
    int64_t discarded = 0;
    // Node-major tables, entry e = i*trials + k: idx {gamma | l << 16, m},
    // weight b (= c).  A discarded trial keeps b = 0 and points at node i.
    std::vector<uint32_t> host_idx;   // [nv*trials][2]
    std::vector<float> host_b;        // [nv*trials]
    // gather tables: packed by warps for pairs of cells (chunks > 0), or in
    // node order (idx, b)
    int chunks = 0;                   // CTAs that hold the packed tables
    uint32_t *d_tab = nullptr, *d_lane = nullptr;
    uint8_t *d_desc = nullptr;
    uint32_t *d_idx = nullptr;
    float *d_b = nullptr;
    float *d_xi = nullptr;            // node velocities [3][nv], FP32
    double hh = 0.0;                  // half the velocity spacing (the same on every axis)
    int half[3] = {0, 0, 0};          // nodes per axis / 2 (the grid's sign-group shape)
    // scratch for bc_cells cells at a time: B and C, [2][bc_cells][nv], then f
    // as pairs of cells, [bc_cells / 2][nv][2] (packed tables)
    float *d_bc = nullptr;
    int64_t prep_cells = 0;           // the mesh size the scratch was made for
    int64_t bc_cells = 0;
};

using DevAlloc = std::function<void *(size_t)>;
using DevFree = std::function<void(void *)>;

// Output n (0-based) of the SplitMix64 stream seeded with `seed`.
uint64_t splitmix64_at(uint64_t seed, uint64_t n);

// lattice = false: seeded random trials; true: trials on a shifted 5D
// Korobov lattice (partner by axis indices, omega from the last two
// coordinates).
int hs_build(HsTables &t, const int n[3], const double lo[3], const double h[3],
             const std::vector<double> &xi, int trials, uint64_t seed, bool lattice, std::string &err,
             const DevAlloc &alloc, const DevFree &dfree);

// Korobov multiplier of an M-point rank-1 lattice in five dimensions.
int64_t korobov_multiplier(int64_t M);
void hs_free(HsTables &t, const DevFree &dfree);

// The weighted trials packed for the gather kernel on pairs of cells.  Two
// kinds of warp: kind 0 holds the partners gamma for the sums B (Eq. 4), kind
// 1 the post-collision nodes l, m for the sums C (Eq. 5).  A warp's 96 rows of
// 32 words (one word per lane):
//   kind 0: 32 rows of two partners (slots 2r, 2r + 1), then 64 rows of b;
//   kind 1: 48 rows of (l, m), then 48 rows of b;
// two nodes x, y in a word as x << 3 | y << 17 (x << 3 is the byte offset in a
// tile of 8-byte pairs).
constexpr int HS_WARPS = 16;          // warps per CTA of the gather kernel
constexpr int HS_ROWS = 96;
constexpr uint32_t HS_NO_NODE = 0xfffffu;
constexpr int hs_slots(int kind) { return kind == 0 ? 64 : 48; }
struct HsPacked {
    int chunks = 0;                // CTAs
    std::vector<uint32_t> tab;     // [chunks * HS_WARPS][HS_ROWS][32]
    std::vector<uint32_t> lane;    // [chunks * HS_WARPS][32]: node (HS_NO_NODE: none) | log2(lanes of the node) << 20
    std::vector<uint8_t> desc;     // [chunks]: groups of eight slots that its warps run | kind << 7
};
void hs_pack(const std::vector<uint32_t> &idx, const std::vector<float> &b, int nv, int M, HsPacked &out);

// Largest grid of the pair kernel: two stages of 8 nv bytes beside its own
// few bytes of shared memory, and node offsets of 17 bits.  Larger grids (up
// to 25,600 nodes) run one cell at a time: a pair's tile would fill shared
// memory alone, and its copy could not overlap the gathers.
constexpr int HS_PAIR_MAX_NV = 14336;

// Scratch for batches of cells (B, C and the cells' f as pairs), at most 4 GB.
int hs_prepare(HsTables &t, int64_t ncells, const DevAlloc &alloc, const DevFree &dfree);

// f (storage precision, already holding f* from the transport launch) is
// updated in place: f <- f* + dt/Kn * I(f*).
int launch_hs_collide(HsTables &t, const StepParams &p, void *f, double kn, double dt);

// The update restricted to the cells list[0 .. *count-1] (device list and
// count, count <= p.ncells), or, if q_out is not NULL, the term I(f) of every
// cell written to q_out [ncells][nv] with f left unchanged.  p.mom_out holds
// the moments of f per cell.
int launch_hs_general(HsTables &t, const StepParams &p, float *f, const int32_t *list, const int *count,
                      float *q_out, double kn, double dt);

// The same update on caller-owned f with a fixed, statically allocated
// device scratch (no allocation).  Needs p.ncells * (8 nv + 40) bytes of
// scratch at most DVM_HS_NOALLOC_SCRATCH_BYTES (else DVM_EINVAL).
int launch_hs_collide_noalloc(HsTables &t, const StepParams &p, float *f, const MomGrid &g, double kn, double dt);

// Trials per node that the register-resident table layout supports.
bool hs_trials_supported(int trials);

}  // namespace dvm
