// Pairs in two-float arithmetic: the FP64 forms' pair law on the FP32 pipe.
//
// GB300 runs FP64 at 1/80 of its FP32 rate (1.6 against 128 operations per
// clock and SM; conversions to and from FP64 at the same 1.6, measured), so an
// FP64 pair of 19 operations costs as much pipe time as 1500 FP32 operations.
// Here a value is an unevaluated sum of two floats (48 bits; Dekker 1971, Knuth
// TAOCP 2 4.2.2: error-free sums and products) and two targets share every packed
// two-wide instruction.  Differences of coordinates and r^2 + eps^2 are exact to
// 2^-60, r^-3 comes from one correction of m y^3 (y the approximate reciprocal
// root), and sums are kept in three floats: a pair's relative error is 2^-48
// (rms), without bias.  Included after pair.cuh inside each translation unit's
// anonymous namespace.
#pragma once

// Power-of-two scales of one system, from the largest coordinate and mass.
struct TfScale {
    int ex;       // every |coordinate| < 2^ex
    int em;       // every mass < 2^em
    bool ok;      // the two-float form holds (else the FP64 form runs)
};

// xmax, mmax, mmin: bit patterns of the largest |coordinate| (FP64), the largest
// and the smallest positive mass (FP32).  The form needs finite values, exponents
// that leave room for r^2 and r^-3, masses whose power of two has a reciprocal in
// FP32's normal range (below 2^126), a softening of at least 2^-30 of the largest
// coordinate (r^-3 stays far inside the FP32 range), and of the lightest source a
// smallest m r^-3 of 2^-90 in these units (its low parts stay above 2^-149).
__device__ __forceinline__ TfScale tf_scale(unsigned long long xmax, uint32_t mmax, uint32_t mmin, double eps2)
{
    TfScale s;
    const int xe = (int)(xmax >> 52), me = (int)(mmax >> 23), ml = (int)(mmin >> 23);
    s.ex = xe - 1022;
    s.em = me - 126;
    const int ee = (int)(((unsigned long long)__double_as_longlong(eps2) >> 52) & 2047) - 1023;  // eps2 >= 2^ee
    const int eo = ee - 2 * s.ex;
    s.ok = xe > 0 && me > 0 && ml > 0 && s.em <= 126 && s.ex > -300 && s.ex < 300 && eo >= -60 && eo < 60 &&
           2 * (me - ml) + 3 * max(4, eo + 2) <= 180;
    return s;
}

// A coordinate in units of 2^ex as a sum of four floats on fixed grids: |x| 2^-ex
// cut off at 2^-92, its fields of 22, 23, 23 and 24 bits.  Equal fields of two
// coordinates differ by at most 24 bits, so their difference is exact whatever the
// coordinates are: one particle far out, which makes the units large, takes
// nothing from pairs near the origin (2^-92 of the extent is 2^-62 of the smallest
// softening the form takes).
struct TfCoord {
    float a, b, c, d;
};
__device__ __forceinline__ TfCoord tf_split(double x, int ex)
{
    const unsigned long long u = (unsigned long long)__double_as_longlong(x);
    const int e = (int)((u >> 52) & 2047);
    unsigned long long m = u & 0xfffffffffffffull;
    if (e > 0) m |= 1ull << 52;
    const int sh = (e > 0 ? e : 1) - 1075 + 92 - ex;  // |x| 2^(92 - ex) = m 2^sh; below 2^92: sh <= 39
    unsigned long long lo = 0, hi = 0;
    if (sh >= 0) {
        lo = m << (sh & 63);
        hi = (m >> 1) >> ((63 - sh) & 63);
    } else if (sh > -64) {
        lo = m >> -sh;
    }
    const unsigned sign = (unsigned)(u >> 32) & 0x80000000u;
    auto field = [&](unsigned v, float unit) {  // +- v unit, exact (v below 2^24)
        return __uint_as_float(__float_as_uint(__fmul_rn((float)(int)v, unit)) ^ sign);
    };
    TfCoord r;
    r.a = field((unsigned)(hi >> 6) & 0x3fffffu, 0x1p-22f);
    r.b = field(((unsigned)hi & 63u) << 17 | (unsigned)(lo >> 47), 0x1p-45f);
    r.c = field((unsigned)(lo >> 24) & 0x7fffffu, 0x1p-68f);
    r.d = field((unsigned)lo & 0xffffffu, 0x1p-92f);
    return r;
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

// s + e = a + b exactly, for |a| >= |b| or a = 0
__device__ __forceinline__ F2x2 fast_two_sum(f2 a, f2 b)
{
    F2x2 r;
    r.h = f2add(a, b);
    r.l = f2sub(b, f2sub(r.h, a));
    return r;
}

// The difference of two coordinates from its fields' differences (exact), the low
// part cut at 2^-48 of the high one.
__device__ __forceinline__ F2x2 tf_diff(f2 a, f2 b, f2 c, f2 d)
{
    const F2x2 u = fast_two_sum(a, b);
    F2x2 r = fast_two_sum(u.h, f2add(u.l, c));
    r.l = f2add(r.l, d);
    return r;
}

// A value as a sum of three floats, each at most about 2^-23 of the one before.
struct F2v3 {
    f2 h, l, t;
};

// r^2 + eps^2 of two targets from the difference's float pairs, exact to 2^-60:
// the squares' high parts by exact sums, then the ten terms of 2^-24 (their errors,
// the squares' and the cross products' low parts) added to a constant of 2^-18 that
// takes their bits down to 2^-41 without rounding, and what is left below in plain
// floats.  (Added in plain floats those ten terms left an error of 2^-48.5, and a
// bias up to 2^-50: squares end in few bit patterns, so that their sums meet ties
// which all round the same way.)
__device__ __forceinline__ F2v3 tf_r2(const F2x2& x, const F2x2& y, const F2x2& z, const F2v3& e2)
{
    const F2x2 px = two_prod(x.h, x.h), py = two_prod(y.h, y.h), pz = two_prod(z.h, z.h);
    const F2x2 bx = two_prod(f2add(x.h, x.h), x.l), by = two_prod(f2add(y.h, y.h), y.l),
               bz = two_prod(f2add(z.h, z.h), z.l);
    f2 t = f2fma(x.l, x.l, f2fma(y.l, y.l, f2fma(z.l, z.l, e2.t)));
    t = f2add(t, f2add(f2add(bx.l, by.l), bz.l));
    const F2x2 s1 = two_sum(px.h, py.h), s2 = two_sum(s1.h, pz.h), s3 = two_sum(s2.h, e2.h);
    // 1.5 x 2^-18 of each half's power of two (r^2 >= 2^-60: no borrow between the halves)
    const f2 big = ((s3.h & 0x7f8000007f800000ull) - 0x0900000009000000ull) | 0x0040000000400000ull;
    f2 T = big;
    const f2 v[10] = {px.l, py.l, pz.l, bx.h, by.h, bz.h, s1.l, s2.l, s3.l, e2.l};
#pragma unroll
    for (int k = 0; k < 10; ++k) {
        const f2 u = f2add(T, v[k]);
        t = f2add(t, f2sub(v[k], f2sub(u, T)));
        T = u;
    }
    const F2x2 u = fast_two_sum(s3.h, f2sub(T, big));
    F2v3 r;
    r.h = u.h;
    r.l = f2add(u.l, t);
    r.t = f2sub(t, f2sub(r.l, u.l));
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

// w (1 + c), c = (ch, cl) small, of the float pair w
__device__ __forceinline__ F2x2 tf_corrected(const F2x2& w, f2 ch, f2 cl)
{
    const F2x2 k = two_prod(w.h, ch);
    F2x2 r = fast_two_sum(w.h, k.h);
    r.l = f2add(r.l, f2add(w.l, f2fma(w.l, ch, f2fma(w.h, cl, k.l))));
    return r;
}

// One source of mass m (per target) at difference (x, y, z) from two targets:
// A[0..2] += m r^-3 (x, y, z), A[3] += m r^-1.  With y the hardware's approximate
// r^-1 (relative error 2^-22) and e = 1 - r^2 y^2 as a float pair, m r^-1 =
// m y (1 + e / 2 + 3 e^2 / 8) and m r^-3 = m y^3 (1 + 3 e / 2 + 15 e^2 / 8), which rounds
// once where a cube of r^-1 has its error three times.  Returns m r^-2 (single
// floats), the pair's weight in the acceleration.
__device__ __forceinline__ f2 tf_pair_mono(const F2x2& x, const F2x2& y, const F2x2& z, f2 m, const F2v3& e2,
                                           F2x3 A[4])
{
    const F2v3 R = tf_r2(x, y, z, e2);
    const f2 iy = f2rsqrt(R.h);
    const F2x2 t = two_prod(iy, iy), p = two_prod(R.h, t.h);
    const f2 low = f2fma(R.l, t.h, f2fma(R.h, t.l, p.l));
    F2x2 e = fast_two_sum(f2sub(f2dup(1.f), p.h), f2neg(low));
    e.l = f2fma(f2neg(R.t), t.h, e.l);
    const f2 ee = f2mul(e.h, e.h);
    const F2x2 u = two_prod(m, iy);
    const F2x2 mq = tf_corrected(u, f2mul(e.h, f2dup(0.5f)), f2fma(ee, f2dup(0.375f), f2mul(e.l, f2dup(0.5f))));
    A[3].add(mq);
    F2x2 v = two_prod(u.h, t.h);
    v.l = f2fma(u.l, t.h, f2fma(u.h, t.l, v.l));
    const f2 c15 = f2dup(1.5f), ch = f2mul(e.h, c15);
    const f2 cl = f2fma(ee, f2dup(1.875f), f2fma(e.l, c15, f2fma(e.h, c15, f2neg(ch))));
    F2x2 g = tf_corrected(v, ch, cl);
    g = fast_two_sum(g.h, g.l);
    A[0].add(tf_mul(g, x));
    A[1].add(tf_mul(g, y));
    A[2].add(tf_mul(g, z));
    return f2mul(mq.h, iy);
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
