// Host check of the packed hard-sphere trials (the library's own code,
// compiled in).  Builds seeded random tables for nv nodes with M trials, of
// which a share carries no weight, packs them, reads the packed tables the way
// the gather kernel does and checks that every node occurs once per kind, in
// lanes of one warp, and that its trials (b with gamma; b with l and m in
// either order) come back as the multiset put in; that every offset lies
// inside the grid, and every trial inside the slots that its CTA runs.
// Prints the faults and the gathered values per 32-value wavefront.
// Usage: hs_pack_check nv M
namespace dvm {
bool hs_trials_supported(int) { return true; }
}
#include "../paper_1503_00707_gb300/csrc/hs.cpp"

#include <cstdio>
#include <map>

using namespace dvm;

int main(int argc, char **argv)
{
    if (argc != 3) return 2;
    const int nv = std::atoi(argv[1]), M = std::atoi(argv[2]);
    std::vector<uint32_t> idx((size_t)nv * M * 2);
    std::vector<float> b((size_t)nv * M);
    for (int i = 0; i < nv; i++)
        for (int k = 0; k < M; k++) {
            const size_t q = (size_t)i * M + k;
            const uint32_t g = (uint32_t)(splitmix64_at(1, 4 * q) % nv), l = (uint32_t)(splitmix64_at(1, 4 * q + 1) % nv),
                           m = (uint32_t)(splitmix64_at(1, 4 * q + 2) % nv);
            // from no weighted trial to all of them
            const bool on = (int)(splitmix64_at(1, 4 * q + 3) % 1000) < 1000 * i / std::max(1, nv - 1);
            idx[2 * q] = g | l << 16;
            idx[2 * q + 1] = m;
            b[q] = on ? 1.0f + (float)k : 0.0f;
        }
    HsPacked p;
    hs_pack(idx, b, nv, M, p);
    using Trial = std::vector<float>;
    std::vector<std::vector<Trial>> want[2] = {std::vector<std::vector<Trial>>(nv), std::vector<std::vector<Trial>>(nv)};
    for (int i = 0; i < nv; i++)
        for (int k = 0; k < M; k++) {
            const size_t q = (size_t)i * M + k;
            if (b[q] == 0.0f) continue;
            const float g = (float)(idx[2 * q] & 0xffffu), l = (float)(idx[2 * q] >> 16), m = (float)idx[2 * q + 1];
            want[0][i].push_back({b[q], g});
            want[1][i].push_back({b[q], std::min(l, m), std::max(l, m)});
        }
    std::vector<std::vector<Trial>> got[2] = {std::vector<std::vector<Trial>>(nv), std::vector<std::vector<Trial>>(nv)};
    std::vector<int> seen[2] = {std::vector<int>(nv, 0), std::vector<int>(nv, 0)};
    int bad = 0;
    double waves[2] = {0, 0}, values[2] = {0, 0};
    for (int w = 0; w < p.chunks * HS_WARPS; w++) {
        const int kind = p.desc[w / HS_WARPS] >> 7, SL = 8 * (p.desc[w / HS_WARPS] & 0x7f);
        if (SL < 8 || SL > hs_slots(kind)) bad++;
        const uint32_t *tab = &p.tab[(size_t)w * HS_ROWS * 32];
        for (int e = 0; e < hs_slots(kind); e++)
            for (int hf = 0; hf < 2; hf++) {
                int cnt[2][16] = {};
                uint32_t ad[2][16][16];
                for (int lane = 16 * hf; lane < 16 * hf + 16; lane++) {
                    uint32_t a[2] = {0, 0};
                    if (kind == 0) a[0] = (e & 1) ? (tab[32 * (e / 2) + lane] >> 14) & 0x1fff8u : tab[32 * (e / 2) + lane] & 0x1fff8u;
                    else {
                        a[0] = tab[32 * e + lane] & 0x1fff8u;
                        a[1] = (tab[32 * e + lane] >> 14) & 0x1fff8u;
                    }
                    float bw;
                    std::memcpy(&bw, &tab[32 * (HS_ROWS - hs_slots(kind) + e) + lane], 4);
                    const uint32_t lt = p.lane[(size_t)w * 32 + lane], node = lt & 0xfffffu;
                    const int t = 1 << (lt >> 20);
                    if (t > 32) bad++;
                    if (node != HS_NO_NODE && node >= (uint32_t)nv) bad++;
                    if (e == 0 && node != HS_NO_NODE && lane % t == 0) seen[kind][node]++;
                    if (node != HS_NO_NODE && (p.lane[(size_t)w * 32 + lane / t * t] & 0xfffffu) != node) bad++;
                    for (int g = 0; g <= kind; g++) {
                        if (a[g] / 8 >= (uint32_t)nv) bad++;
                        bool dup = false;
                        for (int q = 0; q < cnt[g][a[g] / 8 % 16]; q++) dup |= ad[g][a[g] / 8 % 16][q] == a[g];
                        if (!dup) ad[g][a[g] / 8 % 16][cnt[g][a[g] / 8 % 16]++] = a[g];
                    }
                    if (bw == 0.0f) continue;
                    if (e >= SL || node == HS_NO_NODE) {
                        bad++;
                        continue;
                    }
                    values[kind] += kind + 1;
                    const float x = (float)(a[0] / 8), y = (float)(a[1] / 8);
                    if (kind == 0) got[0][node].push_back({bw, x});
                    else got[1][node].push_back({bw, std::min(x, y), std::max(x, y)});
                }
                if (e < SL)
                    for (int g = 0; g <= kind; g++) {
                        int mx = 1;
                        for (int k = 0; k < 16; k++) mx = std::max(mx, cnt[g][k]);
                        waves[kind] += mx;
                    }
            }
    }
    for (int kind = 0; kind < 2; kind++)
        for (int i = 0; i < nv; i++) {
            std::sort(want[kind][i].begin(), want[kind][i].end());
            std::sort(got[kind][i].begin(), got[kind][i].end());
            bad += want[kind][i] != got[kind][i];
            bad += seen[kind][i] != 1;
        }
    std::printf("%d %.3f %.3f %d\n", bad, 2.0 * values[0] / waves[0], 2.0 * values[1] / waves[1], p.chunks);
    return 0;
}
