// Pairs in two-float arithmetic: the FP64 forms' pair law on the FP32 pipe.
//
// GB300 runs FP64 at 1/80 of its FP32 rate (1.6 against 128 operations per
// clock and SM; conversions to and from FP64 at the same 1.6, measured), so an
// FP64 pair of 19 operations costs as much pipe time as 1500 FP32 operations.
// Here a value is an unevaluated sum of two floats (48 bits; Dekker 1971, Knuth
// TAOCP 2 4.2.2: error-free sums and products), a pair takes about 195 FP32
// operations, and two targets share every packed two-wide instruction.  A
// pair's relative error is about 2^-47 and unbiased, and sums are kept in three
// floats, so the error of a sum over many pairs is below that of FP64 pairs
// summed one after another; each use states its measurement.
//
// Coordinates enter as 64-bit integers on a grid of 2^-62 of the system's
// largest coordinate (a power of two above it), so a difference is exact; the
// difference becomes a float pair through three exact pieces.  Included after
// pair.cuh inside each translation unit's anonymous namespace.
#pragma once

// Power-of-two scales of one system, from the largest coordinate and mass.
struct TfScale {
    int ex;       // every |coordinate| < 2^ex
    int em;       // every mass < 2^em
    bool ok;      // the two-float form holds (else the FP64 form runs)
};

// xmax, mmax: bit patterns of the largest |coordinate| (FP64) and mass (FP32
// widened).  The form needs finite values, exponents that leave room for
// r^2 and r^-3, masses whose power of two has a reciprocal in FP32's normal range
// (below 2^126), and a softening of at least 2^-30 of the largest coordinate (r^-3
// stays far inside the FP32 range).
__device__ __forceinline__ TfScale tf_scale(unsigned long long xmax, uint32_t mmax, double eps2)
{
    TfScale s;
    const int xe = (int)(xmax >> 52), me = (int)(mmax >> 23);
    s.ex = xe - 1022;
    s.em = me - 126;
    const int ee = (int)(((unsigned long long)__double_as_longlong(eps2) >> 52) & 2047) - 1023;  // eps2 >= 2^ee
    s.ok = xe > 0 && me > 0 && s.em <= 126 && s.ex > -300 && s.ex < 300 && ee - 2 * s.ex >= -60 && ee - 2 * s.ex < 60;
    return s;
}

// x on the grid: x 2^(62 - ex) rounded to an integer (|x| < 2^ex).
__device__ __forceinline__ long long tf_fixed(double x, int ex)
{
    const unsigned long long b = (unsigned long long)__double_as_longlong(x);
    const int e = (int)((b >> 52) & 2047);
    unsigned long long m = b & 0xfffffffffffffull;
    if (e > 0) m |= 1ull << 52;
    const int sh = (e > 0 ? e : 1) - 1075 + 62 - ex;  // x = m 2^(sh - 62 + ex)
    unsigned long long v;
    if (sh >= 0)
        v = sh < 11 ? m << sh : 0ull;
    else
        v = sh > -55 ? ((m >> (-sh - 1)) + 1ull) >> 1 : 0ull;
    return (long long)b < 0 ? -(long long)v : (long long)v;
}

// 2^k as a double, -1022 <= k <= 1023.
__device__ __forceinline__ double tf_pow2(int k) { return __longlong_as_double((long long)(k + 1023) << 52); }

__device__ __forceinline__ f2 f2neg(f2 a) { return a ^ 0x8000000080000000ull; }
__device__ __forceinline__ f2 f2dup(float a) { return f2pack(a, a); }

struct F2x2 {
    f2 h, l;
};

// s + e = a + b exactly
__device__ __forceinline__ F2x2 two_sum(f2 a, f2 b)
{
    F2x2 r;
    r.h = f2add(a, b);
    const f2 bb = f2sub(r.h, a);
    r.l = f2add(f2sub(a, f2sub(r.h, bb)), f2sub(b, bb));
    return r;
}

// p + e = a b exactly
__device__ __forceinline__ F2x2 two_prod(f2 a, f2 b)
{
    F2x2 r;
    r.h = f2mul(a, b);
    r.l = f2fma(a, b, f2neg(r.h));
    return r;
}

// The differences d0, d1 of two targets (in units of 2^-62) as float pairs:
// 24, 24 and 16 bits of the integer, each exact.
__device__ __forceinline__ F2x2 tf_diff(long long d0, long long d1)
{
    const f2 ca = f2dup(0x1p-30f), cb = f2dup(0x1p-46f), cc = f2dup(0x1p-62f);
    const int h0 = (int)(d0 >> 32), h1 = (int)(d1 >> 32);
    const unsigned l0 = (unsigned)d0, l1 = (unsigned)d1;
    const f2 a = f2mul(f2pack((float)(h0 & ~0xff), (float)(h1 & ~0xff)), ca);
    const f2 b = f2mul(f2pack((float)(int)(((h0 & 0xff) << 16) | (l0 >> 16)), (float)(int)(((h1 & 0xff) << 16) | (l1 >> 16))),
                       cb);
    const f2 c = f2pack((float)(int)(l0 & 0xffffu), (float)(int)(l1 & 0xffffu));
    F2x2 r;
    r.h = f2add(a, b);
    r.l = f2fma(c, cc, f2sub(b, f2sub(r.h, a)));
    return r;
}

// r^2 + eps^2 of two targets from the difference's float pairs.
__device__ __forceinline__ F2x2 tf_r2(const F2x2& x, const F2x2& y, const F2x2& z, const F2x2& e2)
{
    F2x2 px = two_prod(x.h, x.h), py = two_prod(y.h, y.h), pz = two_prod(z.h, z.h);
    // (the squares of the low parts too: they are small but never negative)
    px.l = f2fma(f2add(x.h, x.h), x.l, f2fma(x.l, x.l, px.l));
    py.l = f2fma(f2add(y.h, y.h), y.l, f2fma(y.l, y.l, py.l));
    pz.l = f2fma(f2add(z.h, z.h), z.l, f2fma(z.l, z.l, pz.l));
    const F2x2 s1 = two_sum(px.h, py.h), s2 = two_sum(s1.h, pz.h), s3 = two_sum(s2.h, e2.h);
    const f2 low = f2add(f2add(f2add(px.l, py.l), f2add(pz.l, e2.l)), f2add(f2add(s1.l, s2.l), s3.l));
    F2x2 r;
    r.h = f2add(s3.h, low);
    r.l = f2sub(low, f2sub(r.h, s3.h));
    return r;
}

// q = r2^(-1/2): the hardware approximation y (relative error 2^-22) and one
// step of third order, y + y (e / 2 + 3 e^2 / 8) with e = 1 - r2 y^2 kept as an
// exact part eh and a remainder, renormalised: relative error about 2^-48.
__device__ __forceinline__ F2x2 tf_rsqrt(const F2x2& r2)
{
    const f2 one = f2dup(1.f);
    const f2 y = f2rsqrt(r2.h);
    const F2x2 t = two_prod(y, y);
    F2x2 p = two_prod(r2.h, t.h);
    p.l = f2fma(r2.h, t.l, p.l);
    p.l = f2fma(r2.l, t.h, p.l);
    const f2 eh = f2sub(one, p.h);  // exact
    const f2 hy = f2mul(y, f2dup(0.5f));
    const F2x2 c = two_prod(hy, eh);
    const f2 e = f2sub(eh, p.l);
    f2 low = f2fma(hy, f2neg(p.l), c.l);
    low = f2fma(f2mul(e, e), f2mul(hy, f2dup(0.75f)), low);
    F2x2 q;
    q.h = f2add(y, c.h);
    const f2 x = f2sub(c.h, f2sub(q.h, y));
    q.l = f2add(x, low);
    return q;
}

// the same value with a low part of at most half an ulp of the high one
__device__ __forceinline__ F2x2 tf_norm(const F2x2& a)
{
    F2x2 r;
    r.h = f2add(a.h, a.l);
    r.l = f2sub(a.l, f2sub(r.h, a.h));
    return r;
}

// a b of two-floats with low parts of at most about 2^-23 of the high ones
__device__ __forceinline__ F2x2 tf_mul(const F2x2& a, const F2x2& b)
{
    F2x2 r = two_prod(a.h, b.h);
    r.l = f2fma(a.h, b.l, r.l);
    r.l = f2fma(a.l, b.h, r.l);
    return r;
}

// A running sum of three floats: the additions of the high and the middle part
// are exact (their errors go to the next part), so the sum's error over
// thousands of terms stays far below the terms' own.
struct F2x3 {
    f2 h, m, l;
    __device__ __forceinline__ void zero() { h = m = l = 0ull; }
    __device__ __forceinline__ void add(const F2x2& p)
    {
        const F2x2 t = two_sum(h, p.h), u = two_sum(m, t.l), v = two_sum(u.h, p.l);
        h = t.h;
        m = v.h;
        l = f2add(l, f2add(u.l, v.l));
    }
    // the two targets' sums in FP64
    __device__ __forceinline__ void value(double& a, double& b) const
    {
        float h0, h1, m0, m1, l0, l1;
        f2unpack(h, h0, h1);
        f2unpack(m, m0, m1);
        f2unpack(l, l0, l1);
        a = (double)h0 + ((double)m0 + (double)l0);
        b = (double)h1 + ((double)m1 + (double)l1);
    }
};

// One source of mass m (per target) at difference (x, y, z) from two targets:
// A[0..2] += m q^3 r, A[3] += m q.  Returns m q^2 (single floats), the pair's
// weight in the acceleration.
__device__ __forceinline__ f2 tf_pair_mono(const F2x2& x, const F2x2& y, const F2x2& z, f2 m, const F2x2& e2,
                                           F2x3 A[4])
{
    const F2x2 q = tf_rsqrt(tf_r2(x, y, z, e2));
    F2x2 t = two_prod(q.h, q.h);
    t.l = f2fma(q.l, q.l, t.l);
    t.l = f2fma(f2add(q.h, q.h), q.l, t.l);
    t = tf_norm(t);
    F2x2 mq = two_prod(m, q.h);
    mq.l = f2fma(m, q.l, mq.l);
    A[3].add(mq);
    F2x2 g = tf_mul(mq, t);
    g.l = f2fma(mq.l, t.l, g.l);
    g = tf_norm(g);
    A[0].add(tf_mul(g, x));
    A[1].add(tf_mul(g, y));
    A[2].add(tf_mul(g, z));
    return f2mul(mq.h, q.h);
}

// ---- one value per operand (the quadrupole part of the FP64 form) ------------

struct F2s {
    float h, l;
};

__device__ __forceinline__ F2s sum2(float a, float b)
{
    F2s r;
    r.h = __fadd_rn(a, b);
    const float bb = __fsub_rn(r.h, a);
    r.l = __fadd_rn(__fsub_rn(a, __fsub_rn(r.h, bb)), __fsub_rn(b, bb));
    return r;
}
__device__ __forceinline__ F2s prod2(float a, float b)
{
    F2s r;
    r.h = __fmul_rn(a, b);
    r.l = __fmaf_rn(a, b, -r.h);
    return r;
}
__device__ __forceinline__ F2s mul2(const F2s& a, const F2s& b)
{
    F2s r = prod2(a.h, b.h);
    r.l = __fmaf_rn(a.h, b.l, r.l);
    r.l = __fmaf_rn(a.l, b.h, r.l);
    return r;
}
__device__ __forceinline__ F2s mul2(float a, const F2s& b)
{
    F2s r = prod2(a, b.h);
    r.l = __fmaf_rn(a, b.l, r.l);
    return r;
}
// the same value with a low part of at most half an ulp of the high one
__device__ __forceinline__ F2s norm2(const F2s& a)
{
    F2s r;
    r.h = __fadd_rn(a.h, a.l);
    r.l = __fsub_rn(a.l, __fsub_rn(r.h, a.h));
    return r;
}
__device__ __forceinline__ F2s add2(const F2s& a, const F2s& b)
{
    F2s r = sum2(a.h, b.h);
    r.l = __fadd_rn(r.l, __fadd_rn(a.l, b.l));
    return r;
}

// x 2^k as a float pair by integer operations on x's bits (the FP64 pipe, which
// a conversion would occupy, bounds the kernels that use this): the top 24
// bits of the mantissa, truncated, and the rest, then renormalised (a low part
// of one sign would bias the products that leave out the low parts' product).
// |x 2^k| below 2^-73 gives 0; it must stay below 2^127.
__device__ __forceinline__ F2s split2(double x, int k)
{
    const int hi = __double2hiint(x), lo = __double2loint(x);
    const int a = (hi & 0x7fffffff) + ((k - 896) << 20);  // float exponent field above 20 mantissa bits
    const unsigned sign = (unsigned)hi & 0x80000000u;
    const bool tiny = a < (54 << 20);
    const float h = tiny ? 0.f : __uint_as_float(__funnelshift_l((unsigned)lo, (unsigned)a, 3) | sign);
    const float ulp = tiny ? 0.f : __uint_as_float(((((unsigned)a >> 20) - 52u) << 23) | sign);
    const float l = __fmul_rn((float)(lo & 0x1fffffff), ulp);
    F2s r;
    r.h = __fadd_rn(h, l);
    r.l = __fsub_rn(l, __fsub_rn(r.h, h));
    return r;
}

// A running sum of three floats (F2x3 for one value).
struct F3s {
    float h, m, l;
    __device__ __forceinline__ void zero() { h = m = l = 0.f; }
    __device__ __forceinline__ void add(const F2s& p)
    {
        const F2s t = sum2(h, p.h), u = sum2(m, t.l), v = sum2(u.h, p.l);
        h = t.h;
        m = v.h;
        l = __fadd_rn(l, __fadd_rn(u.l, v.l));
    }
    __device__ __forceinline__ double value() const { return (double)h + ((double)m + (double)l); }
};

// The quadrupole terms of one target: sums of three floats in units of powers
// of two taken from a cell of the list (mass 2^km, q = 2^kq), in which the
// terms that matter stay far inside the FP32 range: a cell whose acceleration is
// beyond 2^24 times the unit folds the sums and gives the next units, and a
// term far below the unit is as far below the cell that gave it.
struct QuadSum {
    F3s s[4];
    int km, kq;  // km + 2 kq: the unit of the acceleration
    __device__ __forceinline__ void zero()
    {
#pragma unroll
        for (int c = 0; c < 4; ++c) s[c].zero();
        km = kq = kOff;
    }
    static constexpr int kOff = -4096;
    // adds the sums to p in the caller's units, and clears them
    __device__ __forceinline__ void fold(double p[4])
    {
        if (km == kOff) return;
        const double sa = scalbn(1.0, km + 2 * kq), sp = scalbn(1.0, km + kq);
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            p[c] = fma(s[c].value(), c < 3 ? sa : -sp, p[c]);
            s[c].zero();
        }
    }
};

// A quadrupole cell (pair_quad2's law) with the monopole part in FP64 and the
// quadrupole part, a few percent of it, in two-float arithmetic (relative error
// 2^-47, so 2^-50 or less of the pair): with u = r q, n = Q u and w = u.n - B_2 eps^2 q^2,
//   phi -= m q + (1/2) w q^3,  a += m q^3 r + q^4 ((5/2) w u - n).
// 18 FP64 operations and about 340 FP32 and integer ones, which the FP64 pipe's
// time (80 FP32 operations each) hides; all in FP64 it is 38.
__device__ __forceinline__ void pair_quad_mixed(const V4<double>& s, const float4 qa, const float4 qb, double xi,
                                                double yi, double zi, double eps2, double p[4], QuadSum& Q)
{
    const double rx = s.x - xi, ry = s.y - yi, rz = s.z - zi;
    const double r2 = fma(rx, rx, fma(ry, ry, fma(rz, rz, eps2)));
    const double q = rsqrt(r2);
    const double q2 = q * q;
    const double mq = s.w * q;
    const double mq3 = mq * q2;
    p[3] -= mq;
    p[0] = fma(mq3, rx, p[0]);
    p[1] = fma(mq3, ry, p[1]);
    p[2] = fma(mq3, rz, p[2]);
    const int em = (__double2hiint(s.w) >> 20) & 2047, eq = (__double2hiint(q) >> 20) & 2047;
    if (em == 0 || eq == 0) return;  // no mass, or r^2 past the FP64 range
    if (em + 2 * eq - 3 * 1023 > Q.km + 2 * Q.kq + 24) {
        Q.fold(p);
        Q.km = em - 1023;
        Q.kq = eq - 1023;
    }
    const F2s qs = split2(q, -Q.kq);
    const F2s ux = norm2(mul2(split2(rx, Q.kq), qs)), uy = norm2(mul2(split2(ry, Q.kq), qs));
    const F2s uz = norm2(mul2(split2(rz, Q.kq), qs));
    const F2s et = split2(eps2 * q2, 0);  // (eps q)^2 <= 1
    // Q and B_2 in units of 2^(km - 2 kq), the power applied in two exact halves
    const int kk = 2 * Q.kq - Q.km, k1 = max(-126, min(126, kk / 2)), k2 = max(-126, min(126, kk - k1));
    const float f1 = __int_as_float((127 + k1) << 23), f2_ = __int_as_float((127 + k2) << 23);
    const float xx = qa.x * f1 * f2_, yy = qa.y * f1 * f2_, zz = qa.z * f1 * f2_, xy = qa.w * f1 * f2_;
    const float xz = qb.x * f1 * f2_, yz = qb.y * f1 * f2_, bb = qb.z * f1 * f2_;
    const F2s n0 = norm2(add2(add2(mul2(xx, ux), mul2(xy, uy)), mul2(xz, uz)));
    const F2s n1 = norm2(add2(add2(mul2(xy, ux), mul2(yy, uy)), mul2(yz, uz)));
    const F2s n2 = norm2(add2(add2(mul2(xz, ux), mul2(yz, uy)), mul2(zz, uz)));
    const F2s w = norm2(add2(add2(mul2(ux, n0), mul2(uy, n1)), add2(mul2(uz, n2), mul2(-bb, et))));
    F2s qq = mul2(qs, qs);
    qq.l = __fmaf_rn(qs.l, qs.l, qq.l);
    qq = norm2(qq);
    const F2s q3 = norm2(mul2(qq, qs)), q4 = norm2(mul2(qq, qq));
    const F2s hw = {0.5f * w.h, 0.5f * w.l}, cw = mul2(2.5f, w);
    Q.s[3].add(mul2(hw, q3));
    const F2s m0 = {-n0.h, -n0.l}, m1 = {-n1.h, -n1.l}, m2 = {-n2.h, -n2.l};
    Q.s[0].add(mul2(norm2(add2(mul2(cw, ux), m0)), q4));
    Q.s[1].add(mul2(norm2(add2(mul2(cw, uy), m1)), q4));
    Q.s[2].add(mul2(norm2(add2(mul2(cw, uz), m2)), q4));
}
