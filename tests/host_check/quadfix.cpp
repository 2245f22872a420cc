// The fixed-point quadrupole part (csrc/quadfix.h) against long double, term by
// term and in sums, over magnitudes of the lengths, softenings and moments.
#include <cmath>
#include <cstdio>
#include <random>

#include "quadfix.h"

using namespace otoo;
typedef long double ld;

// a[0..2], a[3] = phi of one cell from the given FP64 values
static void exact(const float v[7], ld x, ld y, ld z, ld q, ld et, ld a[4])
{
    const ld ux = x * q, uy = y * q, uz = z * q;
    const ld n0 = v[0] * ux + v[3] * uy + v[4] * uz, n1 = v[3] * ux + v[1] * uy + v[5] * uz;
    const ld n2 = v[4] * ux + v[5] * uy + v[2] * uz;
    const ld w = ux * n0 + uy * n1 + uz * n2 - v[6] * et, q4 = q * q * q * q;
    a[0] = q4 * (2.5L * w * ux - n0);
    a[1] = q4 * (2.5L * w * uy - n1);
    a[2] = q4 * (2.5L * w * uz - n2);
    a[3] = -0.5L * w * q * q * q;
}

// the same in FP64
static void fp64(const float v[7], double x, double y, double z, double q, double eps2, double a[4])
{
    const double n0 = std::fma(v[0], x, std::fma(v[3], y, v[4] * z)), n1 = std::fma(v[3], x, std::fma(v[1], y, v[5] * z));
    const double n2 = std::fma(v[4], x, std::fma(v[5], y, v[2] * z));
    const double w = std::fma(x, n0, std::fma(y, n1, std::fma(z, n2, -v[6] * eps2)));
    const double q2 = q * q, q5 = q * (q2 * q2), t = w * q5, cr = q2 * 2.5 * t;
    a[0] = std::fma(cr, x, -q5 * n0);
    a[1] = std::fma(cr, y, -q5 * n1);
    a[2] = std::fma(cr, z, -q5 * n2);
    a[3] = -0.5 * t;
}

int main()
{
    std::mt19937_64 g(3);
    std::normal_distribution<double> N;
    std::uniform_real_distribution<double> U(0, 1);
    int failed = 0;
    double worst[2] = {0, 0}, sum2[2] = {0, 0};  // fixed point, FP64
    for (int k = 0; k < 200000; ++k) {
        const double s = std::pow(10.0, 40 * U(g) - 20);
        double rx = N(g) * s, ry = N(g) * s, rz = N(g) * s, eps2 = std::pow(s * std::pow(10.0, 0.5 - 4 * U(g)), 2);
        if (k % 7 == 0) ry *= 1e-9, rz *= 1e-12, eps2 = s * s * 1e-40;  // |u| = 1 on an axis
        if (k % 11 == 0) rx = ry = rz = 0.0;                            // all softening
        const double q = 1 / std::sqrt(std::fma(rx, rx, std::fma(ry, ry, std::fma(rz, rz, eps2)))), et = eps2 * q * q;
        float v[7];
        const double qs = std::pow(10.0, 55 * U(g) - 40);  // some subnormal
        for (int i = 0; i < 6; ++i) v[i] = (float)(N(g) * qs * (k % 3 ? 1.0 : std::pow(10.0, -6 * U(g))));
        v[2] = -v[0] - v[1];
        v[6] = (float)(std::fabs(N(g)) * qs);
        float top = 0;
        for (int i = 0; i < 7; ++i) top = std::fmax(top, std::fabs(v[i]));
        const QuadFix c = quad_fix(v);
        failed += (c.kind == 1) != (top > 0) || (c.kind == 0) != (top == 0);
        if (c.kind != 1) continue;
        QuadSum Q;
        Q.zero();
        double p[4] = {0, 0, 0, 0};
        quad_fix_pair(c, rx, ry, rz, q, et, Q, p);
        Q.fold(p);
        ld a[4];
        exact(v, rx, ry, rz, q, et, a);
        // the errors of u (12 units of 2^-60), n (31), w (142), the bracket (232) and q^4
        // (15), where the cell's scale is 2^-7 of the fixed point's or more: below 2^-44
        double d[4];
        fp64(v, rx, ry, rz, q, eps2, d);
        const ld sa = (ld)top * q * q * q * q, sp = (ld)top * q * q * q;
        const bool normal = sa > 1e-290L && sp > 1e-290L && top > 1e-30f;  // (else FP64 itself underflows)
        for (int i = 0; i < 4; ++i) {
            const ld sc = i < 3 ? sa : sp;
            failed += !(std::fabs(p[i] - a[i]) <= 0x1p-44L * sc + 1e-320L);
            if (!normal) continue;
            const double e[2] = {(double)(std::fabs(p[i] - a[i]) / sc), (double)(std::fabs(d[i] - a[i]) / sc)};
            for (int f = 0; f < 2; ++f) worst[f] = std::fmax(worst[f], e[f]), sum2[f] += e[f] * e[f];
        }
    }
    printf("terms: %d failed; worst %.3g (FP64 %.3g), rms ratio %.3f\n", failed, worst[0], worst[1],
           std::sqrt(sum2[0] / sum2[1]));
    failed += !(worst[0] <= worst[1]) || !(sum2[0] <= sum2[1]);
    // sums of as many terms as fit between two folds, some cells far beyond the others
    for (int rep = 0; rep < 100; ++rep) {
        QuadSum Q;
        Q.zero();
        double p[4] = {0, 0, 0, 0};
        ld s[4] = {0, 0, 0, 0}, mag[4] = {0, 0, 0, 0};
        for (int k = 0; k < kQuadTerms; ++k) {
            const double d = std::pow(10.0, 3 * U(g)), eps2 = 1e-4;
            const double rx = N(g) * d, ry = N(g) * d, rz = N(g) * d;
            const double q = 1 / std::sqrt(std::fma(rx, rx, std::fma(ry, ry, std::fma(rz, rz, eps2)))), et = eps2 * q * q;
            float v[7];
            for (int i = 0; i < 6; ++i) v[i] = (float)(N(g) * (rep % 2 && k % 100 == 50 ? 1e10 : 1.0));
            if (rep == 0) v[0] = v[1] = v[3] = v[4] = v[5] = 1.99f;  // one sign throughout, near the limit
            v[2] = -v[0] - v[1];
            v[6] = 1.f;
            quad_fix_pair(quad_fix(v), rep == 0 ? 1.0 : rx, rep == 0 ? 1.0 : ry, rep == 0 ? 1.0 : rz,
                          rep == 0 ? 1 / std::sqrt(3.0001) : q, rep == 0 ? 1e-4 / 3.0001 : et, Q, p);
            ld a[4];
            exact(v, rep == 0 ? 1.0 : rx, rep == 0 ? 1.0 : ry, rep == 0 ? 1.0 : rz, rep == 0 ? 1 / std::sqrt(3.0001) : q,
                  rep == 0 ? 1e-4 / 3.0001 : et, a);
            float top = 0;
            for (int i = 0; i < 7; ++i) top = std::fmax(top, std::fabs(v[i]));
            const ld qq = rep == 0 ? 1 / std::sqrt(3.0001) : q, sp = top * qq * qq * qq;
            for (int i = 0; i < 4; ++i) s[i] += a[i], mag[i] += i < 3 ? sp * qq : sp;
        }
        Q.fold(p);
        // every term within its bound; the folds' roundings are far below that
        for (int i = 0; i < 4; ++i) failed += !(std::fabs(p[i] - s[i]) <= 0x1p-44L * mag[i]);
    }
    // not finite and all zero
    float bad[7] = {1, 2, 3, 4, 5, INFINITY, 7}, zero[7] = {0, -0.f, 0, 0, 0, 0, 0}, nan[7] = {NAN, 0, 0, 0, 0, 0, 0};
    failed += quad_fix(bad).kind != 2 || quad_fix(zero).kind != 0 || quad_fix(nan).kind != 2;
    printf("%d failed\n", failed);
    return failed != 0;
}
