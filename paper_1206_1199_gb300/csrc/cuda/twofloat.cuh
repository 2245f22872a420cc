// Pairs in two-float arithmetic: the FP64 forms' pair law on the FP32 pipe.
//
// GB300 runs FP64 at 1/76 of its FP32 rate (1.7 against 128 operations per
// clock and SM; conversions to and from FP64 at the same rate, measured), so an
// FP64 pair of 19 operations costs as much pipe time as 1450 FP32 operations.
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
