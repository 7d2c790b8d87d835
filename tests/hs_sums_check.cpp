// Host check of the sums of the hard-sphere correction's moment system (the
// library's own header, whose packed operations run lane by lane on the host).
// Seeded cells of a grid of hx x hy x hz nodes per sign group: Maxwellians of
// several drifts and temperatures, two beams, and values spread over 40 binary
// orders.  Prints, for the matrix entries and for the gain moments, the largest
// and the root-mean-square error against extended precision, relative to the
// sum of the terms' sizes, and then the same for every node added by itself
// (exact product, Sum2), node after node of a thread.
// Usage: hs_sums_check hx hy hz threads
#include <cstdio>
#include <cstdlib>
#include <vector>

#include "../paper_1503_00707_gb300/csrc/hs_sums.cuh"

using namespace dvm;

static uint64_t state = 20150303;
static double uniform()
{
    state += 0x9E3779B97F4A7C15ull;
    uint64_t x = state;
    x = (x ^ (x >> 30)) * 0xBF58476D1CE4E5B9ull;
    x = (x ^ (x >> 27)) * 0x94D049BB133111EBull;
    return (double)((x ^ (x >> 31)) >> 11) * 0x1p-53;
}

int main(int argc, char **argv)
{
    if (argc != 5) return 2;
    const int hx = std::atoi(argv[1]), hy = std::atoi(argv[2]), hz = std::atoi(argv[3]), T = std::atoi(argv[4]);
    const int P = hx * hy * hz, nv = 8 * P;
    std::vector<float> f(nv), B(nv), C(nv);
    double worst[2][2] = {{0, 0}, {0, 0}}, sq[2][2] = {{0, 0}, {0, 0}};
    const int ncell = 24;
    for (int cell = 0; cell < ncell; cell++) {
        const double u = 3.0 * uniform(), Tm = 1.0 + 3.0 * uniform();
        for (int o = 0; o < 8; o++)
            for (int p = 0; p < P; p++) {
                const int t = p / hz, jx = 2 * (t / hy) + 1, jy = 2 * (t % hy) + 1, jz = 2 * (p % hz) + 1;
                const double x = (o & 4) ? jx : -jx, y = (o & 2) ? jy : -jy, z = (o & 1) ? jz : -jz;
                double v = std::exp(-((x - u) * (x - u) + y * y + z * z) / (4 * Tm));
                if (cell % 3 == 1) v += 0.7 * std::exp(-((x + u) * (x + u) + (y - 1) * (y - 1) + z * z) / (4 * Tm));
                if (cell % 6 == 5) v = std::exp2(-40.0 * uniform());
                const int q = o * P + p;
                f[q] = (float)(v * (1 + 0.02 * uniform()));
                B[q] = (float)((1 + std::sqrt(x * x + y * y + z * z)) * (1 + 0.1 * uniform()));
                C[q] = (float)((double)f[q] * B[q] * (0.5 + uniform()));
            }

        std::vector<long double> sum(NSUM, 0.0L), size(NSUM, 0.0L), part[2] = {sum, sum};
        for (int tid = 0; tid < T; tid++) {
            Acc2 acc[NSUM] = {}, one[NSUM] = {};
            for (int p = 2 * tid; p < P; p += 2 * T) {
                const int t = p / hz;
                const float a = (float)(2 * (t / hy) + 1), b = (float)(2 * (t % hy) + 1), c = (float)(2 * (p % hz) + 1);
                float2 x[8], y[8], z[8];
                for (int o = 0; o < 8; o++) {
                    const int q = o * P + p;
                    x[o] = make_float2(f[q], f[q + 1]);
                    y[o] = make_float2(B[q], B[q + 1]);
                    z[o] = make_float2(C[q], C[q + 1]);
                    for (int e = 0; e < 2; e++) {
                        const float jx = (o & 4) ? a : -a, jy = (o & 2) ? b : -b, jz = (o & 1) ? c + 2 * e : -(c + 2 * e);
                        const float psi[5] = {1, jx, jy, jz, a * a + b * b + jz * jz};
                        const long double w = (long double)f[q + e] * B[q + e], g = C[q + e];
                        const float wh = f[q + e] * B[q + e], wl = std::fma(f[q + e], B[q + e], -wh);
                        int k = 0;
                        for (int r = 0; r < 5; r++)
                            for (int s = r; s < 5; s++, k++) {
                                sum[k] += w * psi[r] * psi[s];
                                size[k] += std::fabs((double)(w * psi[r] * psi[s]));
                                acc2_prod(one[k], wh, wl, psi[r] * psi[s]);
                            }
                        for (int r = 0; r < 5; r++, k++) {
                            sum[k] += g * psi[r];
                            size[k] += std::fabs((double)(g * psi[r]));
                            acc2_prod(one[k], C[q + e], 0.0f, psi[r]);
                        }
                    }
                }
                add_losses(acc, x, y, a, b, c);
                add_gains(acc, z, a, b, c);
            }
            for (int k = 0; k < NSUM; k++) {
                part[0][k] += (long double)acc[k].s + acc[k].e;
                part[1][k] += (long double)one[k].s + one[k].e;
            }
        }
        for (int m = 0; m < 2; m++)
            for (int k = 0; k < NSUM; k++) {
                const double e = std::fabs((double)((part[m][k] - sum[k]) / size[k]));
                const int kind = k < 15 ? 0 : 1;
                worst[m][kind] = std::fmax(worst[m][kind], e);
                sq[m][kind] += e * e / (ncell * (kind ? 5 : 15));
            }
    }
    for (int m = 0; m < 2; m++)
        std::printf("%.3e %.3e %.3e %.3e\n", worst[m][0], std::sqrt(sq[m][0]), worst[m][1], std::sqrt(sq[m][1]));
    return 0;
}
