// The quadrupole part of a cell pair in 62-bit fixed point, for the FP64 form of
// the force.
//
// GB300 runs FP64 at 1/76 of its FP32 rate, so the 20 FP64 operations of the
// quadrupole part would take as long as 1500 of other kinds.  All its factors are
// bounded: with q = (r^2 + eps^2)^(-1/2), u = r q has length below 1, and a cell's
// Q and B_2 divided by a power of two are below 1/2.  So the part is evaluated in
// integers of 2^-60 (two limbs of 31 bits, products of limbs in 64 bits), about
// 330 integer operations that the FP64 operations of the monopole part hide, and the
// terms are summed in 128 bits.  Error of a term over 200000 random cells, relative to
// the cell's largest |Q| q^4: 2^-53.1 rms, 2^-50.4 at worst (FP64: 2^-52.2 and 2^-48.9).
// Builds for the host too.
#pragma once
#include <stdint.h>
#include <string.h>
#include <math.h>

#ifdef __CUDACC__
#define OTOO_QHD __host__ __device__ __forceinline__
#else
#define OTOO_QHD inline
#endif

namespace otoo {

// A cell's Q (xx, yy, zz, xy, xz, yz) and B_2 as h 2^31 + l (0 <= l < 2^31) in units
// of 2^(e - 60), all below 2^(e - 1); 64 bytes.
struct alignas(16) QuadFix {
    int32_t h[7], l[7];
    int32_t e;
    int32_t kind;  // 0: all zero, 1: these integers, 2: not finite (h: the fields' bits)
};

// v: the seven fields of an otoo_quad.
OTOO_QHD QuadFix quad_fix(const float v[7])
{
    QuadFix q;
    uint32_t b[7], most = 0;
    for (int k = 0; k < 7; ++k) {
        memcpy(&b[k], &v[k], 4);
        const uint32_t a = b[k] & 0x7fffffffu;
        most = a > most ? a : most;
    }
    const uint32_t top = most >> 23 ? most >> 23 : 1u;  // (subnormals have the field 1's unit)
    // (all subnormal: their leading zeros)
#ifdef __CUDA_ARCH__
    const int z = most < 0x800000u && most ? __clz((int)most) - 8 : 0;
#else
    const int z = most < 0x800000u && most ? __builtin_clz(most) - 8 : 0;
#endif
    q.kind = top == 255u ? 2 : most ? 1 : 0;
    q.e = (int)top - 125 - z;  // every |v| < 2^(e - 1)
    if (q.kind == 2) {
        for (int k = 0; k < 7; ++k) q.h[k] = (int32_t)b[k], q.l[k] = 0;
        return q;
    }
    for (int k = 0; k < 7; ++k) {
        const uint32_t a = b[k] & 0x7fffffffu;
        const uint32_t f = a >> 23;
        const uint64_t m = (a & 0x7fffffu) | (f ? 0x800000u : 0u);
        const uint32_t s = top - (f ? f : 1u);
        int64_t x = s < 64u ? (int64_t)((m << (35 + z)) >> s) : 0;
        if (b[k] >> 31) x = -x;
        q.h[k] = (int32_t)(x >> 31);
        q.l[k] = (int32_t)(x & 0x7fffffff);
    }
    return q;
}

// Fixed point: h 2^31 + l in units of 2^-60.
struct Fix {
    int32_t h, l;
};
OTOO_QHD Fix fix_limbs(int64_t x)
{
    return Fix{(int32_t)(x >> 31), (int32_t)(x & 0x7fffffff)};
}
// The sums of the products' high and middle parts (the low limbs' products, below
// 2^-60, are left out).
struct FixProd {
    int64_t hh, x;
    OTOO_QHD void set(Fix a, Fix b)
    {
        hh = (int64_t)a.h * b.h;
        x = (int64_t)a.h * b.l + (int64_t)a.l * b.h;
    }
    OTOO_QHD void add(Fix a, Fix b)
    {
        hh += (int64_t)a.h * b.h;
        x += (int64_t)a.h * b.l + (int64_t)a.l * b.h;
    }
    OTOO_QHD int64_t value() const { return hh * 4 + (x >> 29); }  // |value| < 8
};
OTOO_QHD int64_t fix_mul(Fix a, Fix b)
{
    FixProd p;
    p.set(a, b);
    return p.value();
}

OTOO_QHD uint64_t quad_bits(double x)
{
#ifdef __CUDA_ARCH__
    return (uint64_t)__double_as_longlong(x);
#else
    uint64_t b;
    memcpy(&b, &x, 8);
    return b;
#endif
}

// x 2^k cut off to units of 2^-60; |x 2^k| < 2.
OTOO_QHD int64_t fix_of(double x, int k)
{
    const uint64_t b = quad_bits(x);
    const int f = (int)(b >> 52) & 2047;
    const uint64_t m = (b & 0xfffffffffffffull) | (f ? 1ull << 52 : 0);
    const int s = 1023 - (f ? f : 1) - k;  // m 2^8 2^-s
    const int64_t v = (int64_t)((m << 8) >> (s < 0 ? 0 : s > 63 ? 63 : s));
    return (int64_t)b < 0 ? -v : v;
}

// One sum in 128 bits, units of 2^(u - 51) of the high word.
struct QuadAcc {
    int64_t hi;
    uint64_t lo;
    // adds t 2^-60 2^(u - s), s >= 0; below 2^53 units, so 1024 terms fit
    OTOO_QHD void add(int64_t t, int s)
    {
        const int64_t h = t >> (s < 54 ? s + 9 : 63);
        const int r = s - 55;
        const uint64_t l = r <= 0 ? (uint64_t)t << -r : (uint64_t)(t >> (r < 63 ? r : 63));
        lo += l;
        hi += h + (lo < l ? 1 : 0);
    }
    OTOO_QHD double value(int u) const { return scalbn((double)hi, u - 51) + scalbn((double)lo, u - 115); }
};
constexpr int kQuadTerms = 1024;  // terms between two folds at most

// The sums of one target's quadrupole terms in units of 2^ua (accelerations) and
// 2^up (potential): a cell beyond the units folds the sums and gives the next
// ones, 2^24 times its own (the sums keep 2^-91 of it).
struct QuadSum {
    QuadAcc s[4];
    int ua, up;
    static constexpr int kOff = -100000;
    OTOO_QHD void zero()
    {
        for (int c = 0; c < 4; ++c) s[c].hi = 0, s[c].lo = 0;
        ua = up = kOff;
    }
    // adds the sums to p in the caller's units and clears them
    OTOO_QHD void fold(double p[4])
    {
        if (ua == kOff) return;
        for (int c = 0; c < 4; ++c) {
            p[c] = c < 3 ? p[c] + s[c].value(ua) : p[c] - s[c].value(up);
            s[c].hi = 0, s[c].lo = 0;
        }
    }
};

// The quadrupole terms of cell c on one target at difference (rx, ry, rz) from it:
// with n = Q u and w = u.n - B_2 eps^2 q^2,
//   phi -= (1/2) w q^3,  a += q^4 ((5/2) w u - n)
// (q = r^-1, e2q2 = eps^2 q^2; c.kind 1; q normal).
OTOO_QHD void quad_fix_pair(const QuadFix& c, double rx, double ry, double rz, double q, double e2q2, QuadSum& Q,
                            double p[4])
{
    const uint64_t qb = quad_bits(q);
    const int eq = ((int)(qb >> 52) & 2047) - 1022;  // q = qf 2^eq, 1/2 <= qf < 1
    const Fix qf = fix_limbs((int64_t)((qb & 0xfffffffffffffull) | 1ull << 52) << 7);
    // (r 2^(eq - 1) is below 1 but for rounding)
    const Fix ux = fix_limbs(2 * fix_mul(fix_limbs(fix_of(rx, eq - 1)), qf));
    const Fix uy = fix_limbs(2 * fix_mul(fix_limbs(fix_of(ry, eq - 1)), qf));
    const Fix uz = fix_limbs(2 * fix_mul(fix_limbs(fix_of(rz, eq - 1)), qf));
    const Fix xx = {c.h[0], c.l[0]}, yy = {c.h[1], c.l[1]}, zz = {c.h[2], c.l[2]};
    const Fix xy = {c.h[3], c.l[3]}, xz = {c.h[4], c.l[4]}, yz = {c.h[5], c.l[5]}, b2 = {c.h[6], c.l[6]};
    FixProd m;
    m.set(xx, ux), m.add(xy, uy), m.add(xz, uz);
    const int64_t n0 = m.value();
    m.set(xy, ux), m.add(yy, uy), m.add(yz, uz);
    const int64_t n1 = m.value();
    m.set(xz, ux), m.add(yz, uy), m.add(zz, uz);
    const int64_t n2 = m.value();  // |n| < 3/2
    const Fix et = fix_limbs(-fix_of(e2q2, 0));
    m.set(ux, fix_limbs(n0)), m.add(uy, fix_limbs(n1)), m.add(uz, fix_limbs(n2)), m.add(b2, et);
    const Fix w = fix_limbs(m.value());  // |w| < 2
    const Fix q2 = fix_limbs(fix_mul(qf, qf));
    const Fix q4 = fix_limbs(fix_mul(q2, q2));
    // half the acceleration's bracket, below 13/4
    const int64_t wx = fix_mul(w, ux), wy = fix_mul(w, uy), wz = fix_mul(w, uz);
    const int64_t ax = fix_mul(fix_limbs(wx + (wx >> 2) - (n0 >> 1)), q4);
    const int64_t ay = fix_mul(fix_limbs(wy + (wy >> 2) - (n1 >> 1)), q4);
    const int64_t az = fix_mul(fix_limbs(wz + (wz >> 2) - (n2 >> 1)), q4);
    const int64_t ph = fix_mul(w, fix_limbs(fix_mul(q2, qf)));
    const int ea = c.e + 4 * eq + 1, ep = c.e + 3 * eq - 1;
    if (ea > Q.ua || ep > Q.up) {
        Q.fold(p);
        Q.ua = ea > Q.ua ? ea + 24 : Q.ua;
        Q.up = ep > Q.up ? ep + 24 : Q.up;
    }
    Q.s[0].add(ax, Q.ua - ea);
    Q.s[1].add(ay, Q.ua - ea);
    Q.s[2].add(az, Q.ua - ea);
    Q.s[3].add(ph, Q.up - ep);
}

}  // namespace otoo
