// FP64 to FP32 and back by integer operations on the device.  GB300 converts at
// its FP64 rate, 1.7 per clock and SM: one conversion takes the time of about
// fifty integer operations (128 per clock and SM for two instructions of three),
// and the kernels that turn coordinates into float pairs are bound by it.  The
// results are those of the conversions, bit for bit; values outside FP32's
// normal range take the conversions themselves.  On the host: plain casts.
#pragma once
#include <stdint.h>

#ifdef __CUDACC__
#define OTOO_NHD __host__ __device__ __forceinline__
#else
#define OTOO_NHD inline
#endif

namespace otoo {

// x rounded to FP32 (nearest, ties to even).
OTOO_NHD float narrow(double x)
{
#ifdef __CUDA_ARCH__
    const int hi = __double2hiint(x);
    const unsigned lo = (unsigned)__double2loint(x);
    const int ex = (hi >> 20) & 2047;
    if (ex >= 897 && ex <= 1150) {
        unsigned f = __funnelshift_l(lo, (unsigned)((hi & 0x7fffffff) - (896 << 20)), 3);
        const unsigned rem = lo & 0x1fffffffu;
        f += rem + (f & 1u) > 0x10000000u ? 1u : 0u;  // (the carry may pass into the exponent)
        return __uint_as_float(f | ((unsigned)hi & 0x80000000u));
    }
    if (((hi & 0x7fffffff) | (int)lo) == 0) return __uint_as_float((unsigned)hi);
    return __double2float_rn(x);
#else
    return (float)x;
#endif
}

// x as a float pair: h = x rounded to FP32, l = x - h rounded to FP32.
OTOO_NHD void narrow2(double x, float& h, float& l)
{
#ifdef __CUDA_ARCH__
    const int hi = __double2hiint(x);
    const unsigned lo = (unsigned)__double2loint(x);
    const int ex = (hi >> 20) & 2047;
    if (ex >= 949 && ex <= 1149) {
        unsigned f = __funnelshift_l(lo, (unsigned)((hi & 0x7fffffff) - (896 << 20)), 3);
        int rem = (int)(lo & 0x1fffffffu);
        const bool up = (unsigned)rem + (f & 1u) > 0x10000000u;
        f += up ? 1u : 0u;
        rem -= up ? 0x20000000 : 0;
        rem = hi < 0 ? -rem : rem;
        h = __uint_as_float(f | ((unsigned)hi & 0x80000000u));
        l = __fmul_rn((float)rem, __uint_as_float((unsigned)(ex - 948) << 23));  // rem 2^(ex - 1075)
        return;
    }
    if (((hi & 0x7fffffff) | (int)lo) == 0) {
        h = __uint_as_float((unsigned)hi);
        l = 0.f;
        return;
    }
    h = __double2float_rn(x);
    l = __double2float_rn(__dsub_rn(x, (double)h));
#else
    h = (float)x;
    l = (float)(x - (double)h);
#endif
}

// An integer 0 <= k < 2^24 as FP64.
OTOO_NHD double small_int(uint32_t k)
{
#ifdef __CUDA_ARCH__
    const unsigned f = __float_as_uint((float)k);
    return __hiloint2double(k ? (int)((f >> 3) + (896u << 20)) : 0, (int)(f << 29));
#else
    return (double)k;
#endif
}

// 2^k, |k| < 1023.
OTOO_NHD double pow2(int k)
{
#ifdef __CUDA_ARCH__
    return __hiloint2double((1023 + k) << 20, 0);
#else
    return k >= 0 ? (double)((uint64_t)1 << k) : 1.0 / (double)((uint64_t)1 << -k);
#endif
}

}  // namespace otoo
