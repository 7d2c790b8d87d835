// The sums of the hard-sphere correction's moment system over a cell's nodes:
// the 15 distinct entries sum psi_r psi_s f B (numbered as the upper triangle
// of the 5x5 matrix) and the 5 gain moments sum psi_r C over the integer basis
// psi = (1, j_x, j_y, j_z, |j|^2), to about twice FP32 precision with FP32
// operations.  Used by k_hs_corr; compiles on the host too, where its rounding
// is checked against extended precision.
#pragma once
#include "f2.cuh"

namespace dvm {

constexpr int NSUM = 20;

// s + e = a + b exactly, s rounded (Knuth's TwoSum)
DVM_HD float two_sum(float a, float b, float &e)
{
    const float s = a + b, bb = s - a;
    e = (a - (s - bb)) + (b - bb);
    return s;
}

// Sum2 accumulation (Ogita, Rump and Oishi, 2005) of exact products: s + e
// carries the running sum to about twice the FP32 precision.
struct Acc2 {
    float s, e;
};
// a += (x + xl) k, with x k split exactly (FMA) and xl k a correction of at
// most about 2^-24 x k
DVM_HD void acc2_prod(Acc2 &a, float x, float xl, float k)
{
    const float p = f_mul(x, k);
    float se;
    a.s = two_sum(a.s, p, se);
    a.e += se + std::fma(xl, k, std::fma(x, k, -p));
}

// The signed sums over the eight sign groups that the moment system needs, per
// position (packed pairs of z nodes), from the sums p and differences m of the
// groups' pairs along z: S, X, Y, Z as group_sums, and XY = sum s_x s_y x, XZ,
// YZ.
DVM_HD void group_sums7(const float2 (&p)[4], const float2 (&m)[4], float2 (&v)[7])
{
    const float2 pp0 = f2_add(p[0], p[1]), pm0 = f2_sub(p[1], p[0]);
    const float2 pp1 = f2_add(p[2], p[3]), pm1 = f2_sub(p[3], p[2]);
    v[0] = f2_add(pp0, pp1);
    v[1] = f2_sub(pp1, pp0);
    v[2] = f2_add(pm0, pm1);
    v[4] = f2_sub(pm1, pm0);
    const float2 mp0 = f2_add(m[0], m[1]), mm0 = f2_sub(m[1], m[0]);
    const float2 mp1 = f2_add(m[2], m[3]), mm1 = f2_sub(m[3], m[2]);
    v[3] = f2_add(mp0, mp1);
    v[5] = f2_sub(mp1, mp0);
    v[6] = f2_add(mm0, mm1);
}

// 2^k > 16 max |x|
DVM_HD float2 split_sigma(const float2 (&x)[8])
{
    uint32_t mx = 0;
#pragma unroll
    for (int o = 0; o < 8; o++) {
        const uint32_t a = f_bits(x[o].x) & 0x7fffffffu, b = f_bits(x[o].y) & 0x7fffffffu;
        mx = mx > a ? mx : a;
        mx = mx > b ? mx : b;
    }
    const uint32_t ex = (mx >> 23) < 249u ? mx >> 23 : 249u;
    const float sg = bits_f((ex + 5u) << 23);
    return make_float2(sg, sg);
}

// The seven signed sums over the groups of x + xl (xl may be null), as V + Vr
// with |Vr| at most about 2^-24 |V|: x splits against sigma = 2^k > 16 max |x|
// into a multiple of 2^(k-24), and the rest against 2^-19 sigma into a multiple
// of 2^(k-43); the sums of either multiple are exact in FP32, and what is left,
// 2^-38 of x and xl, is summed in FP32.  One multiple alone leaves rests of
// 2^-19, whose roundings made the sums of a cell 10 to 20 times less exact than
// node-by-node Sum2 (3e-14 against 3e-15).
DVM_HD void sign_sums(const float2 (&x)[8], const float2 *xl, float2 (&V)[7], float2 (&Vr)[7])
{
    float2 r[8], U[7];
#pragma unroll
    for (int o = 0; o < 8; o++) r[o] = x[o];
    auto level = [&](float2 sg, float2 (&v)[7]) {
        float2 qp[4], qm[4];
#pragma unroll
        for (int k = 0; k < 4; k++) {
            const float2 q0 = f2_sub(f2_add(r[2 * k], sg), sg), q1 = f2_sub(f2_add(r[2 * k + 1], sg), sg);
            r[2 * k] = f2_sub(r[2 * k], q0);
            r[2 * k + 1] = f2_sub(r[2 * k + 1], q1);
            qp[k] = f2_add(q0, q1);
            qm[k] = f2_sub(q1, q0);
        }
        group_sums7(qp, qm, v);
    };
    const float2 sg = split_sigma(x);
    level(sg, V);
    level(f2_mul(sg, make_float2(0x1p-19f, 0x1p-19f)), U);
#pragma unroll
    for (int k = 0; k < 7; k++) {
        const float2 t = f2_add(V[k], U[k]), z = f2_sub(t, V[k]);
        Vr[k] = f2_add(f2_sub(V[k], f2_sub(t, z)), f2_sub(U[k], z));
        V[k] = t;
    }
    float2 rp[4], rm[4];
#pragma unroll
    for (int k = 0; k < 4; k++) {
        const float2 r0 = xl ? f2_add(r[2 * k], xl[2 * k]) : r[2 * k];
        const float2 r1 = xl ? f2_add(r[2 * k + 1], xl[2 * k + 1]) : r[2 * k + 1];
        rp[k] = f2_add(r0, r1);
        rm[k] = f2_sub(r1, r0);
    }
    group_sums7(rp, rm, U);
#pragma unroll
    for (int k = 0; k < 7; k++) Vr[k] = f2_add(Vr[k], U[k]);
}

// The matrix entries' share of two nodes next to each other along z (j = a, b,
// c and c + 2) in all eight sign groups, from f and B.
DVM_HD void add_losses(Acc2 (&acc)[NSUM], float2 (&f)[8], float2 (&B)[8], float a, float b, float c)
{
    float2 V[7], Vr[7];
#pragma unroll
    for (int o = 0; o < 8; o++) {
        // f B = f + B exactly
        const float2 m = f2_mul(f[o], B[o]);
        B[o] = f2_fma(f[o], B[o], make_float2(-m.x, -m.y));
        f[o] = m;
    }
    sign_sums(f, B, V, Vr);
#pragma unroll
    for (int e = 0; e < 2; e++) {
        const float cz = c + 2.0f * e, j2 = a * a + b * b + cz * cz;
        auto put = [&](int k, int v, float coef) { acc2_prod(acc[k], e ? V[v].y : V[v].x, e ? Vr[v].y : Vr[v].x, coef); };
        put(0, 0, 1.0f);          // (1, 1)
        put(1, 1, a);             // (1, j_x)
        put(2, 2, b);             // (1, j_y)
        put(3, 3, cz);            // (1, j_z)
        put(4, 0, j2);            // (1, |j|^2)
        put(5, 0, a * a);         // (j_x, j_x)
        put(6, 4, a * b);         // (j_x, j_y)
        put(7, 5, a * cz);        // (j_x, j_z)
        put(8, 1, a * j2);        // (j_x, |j|^2)
        put(9, 0, b * b);         // (j_y, j_y)
        put(10, 6, b * cz);       // (j_y, j_z)
        put(11, 2, b * j2);       // (j_y, |j|^2)
        put(12, 0, cz * cz);      // (j_z, j_z)
        put(13, 3, cz * j2);      // (j_z, |j|^2)
        put(14, 0, j2 * j2);      // (|j|^2, |j|^2): below 2^23 (at most 32 nodes an axis)
    }
}

// the same for the gain moments, from C
DVM_HD void add_gains(Acc2 (&acc)[NSUM], const float2 (&C)[8], float a, float b, float c)
{
    float2 V[7], Vr[7];
    sign_sums(C, nullptr, V, Vr);
#pragma unroll
    for (int e = 0; e < 2; e++) {
        const float cz = c + 2.0f * e, j2 = a * a + b * b + cz * cz;
        auto put = [&](int k, int v, float coef) { acc2_prod(acc[k], e ? V[v].y : V[v].x, e ? Vr[v].y : Vr[v].x, coef); };
        put(15, 0, 1.0f);
        put(16, 1, a);
        put(17, 2, b);
        put(18, 3, cz);
        put(19, 0, j2);
    }
}

}  // namespace dvm
