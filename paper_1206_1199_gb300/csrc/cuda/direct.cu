// Direct summation on the device: chosen targets against every particle of
// a system, in FP64 -- the exact reference the learned opening angle is
// trained against (the measured group errors are this sum's, the paper's
// O(N^2) brute force of Section II), and a check of the tree force.
//
// Kernels
//   k_direct_range, k_direct_tf  at least kTfMinSources sources: the system's
//                  scale, then the pairs in two-float arithmetic
//                  (twofloat.cuh), 256 targets per block.
//   k_direct_part  fewer sources, or a scale the two-float form does not take
//                  (k_direct_tf then returns at once, else this one does): block (target tile of 128, source chunk): the chunk's
//                  sources staged through shared memory, FP64 pairs, one
//                  partial sum per (chunk, target).
//   k_direct_sum   the chunk partials of each target summed in chunk order.
#include <cuda_runtime.h>

#include <cstdint>

#include "../common.h"

using namespace otoo;

namespace {

#include "pair.cuh"
#include "twofloat.cuh"

constexpr int kTgt = 128;     // targets per block
constexpr int kTile = 128;    // sources staged per tile

// Largest |coordinate| and mass of the sources (order-preserving bit
// patterns; range is zero before the launch): the scales of the two-float
// form.  An infinite or NaN coordinate gives the largest pattern.
struct DirectRange {
    unsigned long long xmax;
    uint32_t mmax, pad;
};

__global__ void __launch_bounds__(256) k_direct_range(const otoo_src* __restrict__ src, int64_t n,
                                                      DirectRange* __restrict__ range)
{
    unsigned long long x = 0;
    uint32_t m = 0;
    for (int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x; i < n; i += (int64_t)gridDim.x * 256) {
        const otoo_src q = src[i];  // (8-byte loads: the sources may start on any 8-byte boundary)
        const double v[3] = {q.x, q.y, q.z};
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const unsigned long long u = (unsigned long long)__double_as_longlong(v[k]) & 0x7fffffffffffffffull;
            x = u > x ? u : x;
        }
        const uint32_t w = __float_as_uint(q.m) & 0x7fffffffu;
        m = w > m ? w : m;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long u = __shfl_xor_sync(kFull, x, o);
        x = u > x ? u : x;
    }
    m = __reduce_max_sync(kFull, m);
    if ((threadIdx.x & 31) == 0) {
        atomicMax(&range->xmax, x);
        atomicMax(&range->mmax, m);
    }
}

// The two-float form: 256 targets per block, two per thread; the block's
// halves of 128 threads take the halves of every staged tile, and the second
// half's sums join the first's at the end.  The float sums are moved into FP64
// every kTfFold tiles.  Bound by the FP32 pipe: about 195 packed operations per
// source and two targets.
// N = 2^19, 5003 targets: 25.1 ms (1.05e11 pairs/s) against 110 ms for the FP64
// form.  Relative error (2-norm over 40 targets, against extended precision) over
// N = 66000, 90000, 130000 and 400000, four models and softenings 1e-4 and 1e-2,
// two-float / FP64 form: accelerations 3.3e-16 to 1.2e-15 / 8.0e-16 to 5.8e-15,
// potentials 0.9e-16 to 2.5e-16 / 3.9e-16 to 1.7e-15, for each input the
// two-float form's no larger (one of 32 equal, 8.3e-16 / 8.0e-16): the FP64 form's
// sums of a chunk's pairs lose more the longer they are.  N = 20000 1.2e-15 / 7.0e-16:
// the line is where the two-float form is no less exact.
constexpr int64_t kTfMinSources = 65536;
constexpr int kTfTile = 256;
constexpr int kTfFold = 8;  // the longest run (1024 sources) the float sums take before FP64

constexpr unsigned kTfPos = kTfFold * kTfTile - 1;  // position in a run
static_assert(((kTfPos + 1) & kTfPos) == 0, "a run's length is a power of two");

// What the heaviest pair of each target of a run (run0 + the low bits of top)
// lacks: its FP64 value less the two-float one.  A close pair at a small
// softening can be most of a target's acceleration, and its 2^-47, or the grid's
// spacing against its distance, would then be the sum's error (Hernquist, eps
// 1e-4, N = 130000: 6.4e-15 without this, 3.8e-16 with it, all FP64 1.6e-15).
__device__ __forceinline__ void tf_refine(const otoo_src* __restrict__ src, int64_t run0, int64_t j1,
                                          const unsigned top[2], const int64_t ti[2], const long long x[2],
                                          const long long y[2], const long long z[2], const TfScale& sc, float ms,
                                          double eps2, const F2x2& e2, double fix[4][2])
{
    long long d[3][2];
    float m[2];
    const double es = eps2 * tf_pow2(-2 * sc.ex), sx = tf_pow2(-sc.ex);
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        int64_t j = run0 + (top[k] & kTfPos);
        j = j < j1 ? j : j1 - 1;
        const otoo_src q = src[j];
        d[0][k] = tf_fixed(q.x, sc.ex) - x[k];
        d[1][k] = tf_fixed(q.y, sc.ex) - y[k];
        d[2][k] = tf_fixed(q.z, sc.ex) - z[k];
        m[k] = j == ti[k] || top[k] == 0u ? 0.f : q.m * ms;  // (0: no pair)
        // (from the coordinates themselves: near the origin they are finer than the grid)
        const otoo_src t = src[ti[k] < 0 ? j : ti[k]];
        const double rx = (q.x - t.x) * sx, ry = (q.y - t.y) * sx, rz = (q.z - t.z) * sx;
        const double inv = rsqrt(fma(rx, rx, fma(ry, ry, fma(rz, rz, es))));
        const double mi = (double)m[k] * inv, mi3 = mi * inv * inv;
        fix[0][k] = mi3 * rx;
        fix[1][k] = mi3 * ry;
        fix[2][k] = mi3 * rz;
        fix[3][k] = mi;
    }
    F2x3 A[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) A[c].zero();
    tf_pair_mono(tf_diff(d[0][0], d[0][1]), tf_diff(d[1][0], d[1][1]), tf_diff(d[2][0], d[2][1]), f2pack(m[0], m[1]), e2,
                 A);
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        double v0, v1;
        A[c].value(v0, v1);
        fix[c][0] -= v0;
        fix[c][1] -= v1;
    }
}

__global__ void __launch_bounds__(256, 2) k_direct_tf(const otoo_src* __restrict__ src, int64_t n_src,
                                                      const int64_t* __restrict__ tgt, int64_t n_tgt, double eps2,
                                                      int64_t chunk, double* __restrict__ part,
                                                      const DirectRange* __restrict__ range,
                                                      uint32_t* __restrict__ status)
{
    __shared__ longlong2 s_xy[kTfTile];
    __shared__ longlong2 s_zm[kTfTile];
    __shared__ double s_sum[128][9];
    const TfScale sc = tf_scale(range->xmax, range->mmax, eps2);
    if (!sc.ok) return;  // k_direct_part runs
    const int lt = threadIdx.x & 127, half = threadIdx.x >> 7;
    const int64_t j0 = (int64_t)blockIdx.y * chunk;
    const int64_t j1 = j0 + chunk < n_src ? j0 + chunk : n_src;
    int64_t ti[2];
    long long x[2] = {0, 0}, y[2] = {0, 0}, z[2] = {0, 0};
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        const int64_t t = (int64_t)blockIdx.x * 256 + 128 * k + lt;
        ti[k] = -1;
        if (t < n_tgt) {
            ti[k] = tgt[t];
            if (ti[k] < 0 || ti[k] >= n_src) {
                atomicOr(status, 2u);
                ti[k] = -1;
            } else {
                x[k] = tf_fixed(src[ti[k]].x, sc.ex);
                y[k] = tf_fixed(src[ti[k]].y, sc.ex);
                z[k] = tf_fixed(src[ti[k]].z, sc.ex);
            }
        }
    }
    F2x2 e2;
    {
        const double e = eps2 * tf_pow2(-2 * sc.ex);  // exact
        const float eh = __double2float_rn(e);
        e2.h = f2dup(eh);
        e2.l = f2dup(__double2float_rn(e - (double)eh));
    }
    const float ms = __int_as_float((127 - sc.em) << 23);  // 2^-em (em from -125 to 126)
    F2x3 A[4];
    double sum[4][2];
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        A[c].zero();
        sum[c][0] = sum[c][1] = 0.0;
    }
    int fold = 0;
    int64_t run0 = j0;            // first source of the run being summed
    unsigned top[2] = {0u, 0u};   // the run's heaviest pair: m q^2's bits above its position in the run
    for (int64_t b = j0; b < j1; b += kTfTile) {
        const int64_t j = b + threadIdx.x;
        if (j < j1) {
            const otoo_src q = src[j];
            s_xy[threadIdx.x] = make_longlong2(tf_fixed(q.x, sc.ex), tf_fixed(q.y, sc.ex));
            s_zm[threadIdx.x] = make_longlong2(tf_fixed(q.z, sc.ex), (long long)__float_as_uint(q.m * ms));
        }
        __syncthreads();
        const int cnt = j1 - b < kTfTile ? (int)(j1 - b) : kTfTile;
        const int k0 = half * (kTfTile / 2), k1 = half ? cnt : (cnt < kTfTile / 2 ? cnt : kTfTile / 2);
        const int self0 = ti[0] >= b && ti[0] < b + cnt ? (int)(ti[0] - b) : -1;  // j != i
        const int self1 = ti[1] >= b && ti[1] < b + cnt ? (int)(ti[1] - b) : -1;
#pragma unroll 1
        for (int k = k0; k < k1; ++k) {
            const longlong2 xy = s_xy[k], zm = s_zm[k];
            const float m = __uint_as_float((unsigned)zm.y);
            const F2x2 dx = tf_diff(xy.x - x[0], xy.x - x[1]);
            const F2x2 dy = tf_diff(xy.y - y[0], xy.y - y[1]);
            const F2x2 dz = tf_diff(zm.x - z[0], zm.x - z[1]);
            float w0, w1;
            f2unpack(tf_pair_mono(dx, dy, dz, f2pack(k == self0 ? 0.f : m, k == self1 ? 0.f : m), e2, A), w0, w1);
            const unsigned at = (unsigned)(fold * kTfTile + k);
            top[0] = max(top[0], (__float_as_uint(w0) & ~kTfPos) | at);
            top[1] = max(top[1], (__float_as_uint(w1) & ~kTfPos) | at);
        }
        if (++fold == kTfFold || b + kTfTile >= j1) {
            fold = 0;
            // the heaviest pair of the run again in FP64, less what was added for it
            double fix[4][2];
            tf_refine(src, run0, j1, top, ti, x, y, z, sc, ms, eps2, e2, fix);
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                double v0, v1;
                A[c].value(v0, v1);
                sum[c][0] += v0 + fix[c][0];
                sum[c][1] += v1 + fix[c][1];
                A[c].zero();
            }
            top[0] = top[1] = 0u;
            run0 = b + kTfTile;
        }
        __syncthreads();
    }
    if (half) {
#pragma unroll
        for (int c = 0; c < 4; ++c) s_sum[lt][c] = sum[c][0], s_sum[lt][4 + c] = sum[c][1];
    }
    __syncthreads();
    if (half) return;
    // back to the caller's units: powers of two, exact
    const double sa = tf_pow2(sc.em - 2 * sc.ex), sp = -tf_pow2(sc.em - sc.ex);
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        const int64_t t = (int64_t)blockIdx.x * 256 + 128 * k + lt;
        if (t >= n_tgt) continue;
        double* d = part + ((int64_t)blockIdx.y * n_tgt + t) * 4;
#pragma unroll
        for (int c = 0; c < 4; ++c) d[c] = (sum[c][k] + s_sum[lt][4 * k + c]) * (c < 3 ? sa : sp);
    }
}

// kAfterTf: launched behind k_direct_tf, returns when that one did the work.
template <bool kAfterTf>
__global__ void __launch_bounds__(kTgt) k_direct_part(const otoo_src* __restrict__ src, int64_t n_src,
                                                      const int64_t* __restrict__ tgt, int64_t n_tgt, double eps2,
                                                      int64_t chunk, double* __restrict__ part,
                                                      const DirectRange* __restrict__ range,
                                                      uint32_t* __restrict__ status)
{
    __shared__ double4 s[kTile];
    if (kAfterTf && tf_scale(range->xmax, range->mmax, eps2).ok) return;
    const int64_t t = (int64_t)blockIdx.x * kTgt + threadIdx.x;
    const int64_t j0 = (int64_t)blockIdx.y * chunk;
    const int64_t j1 = j0 + chunk < n_src ? j0 + chunk : n_src;
    int64_t ti = -1;
    double xi = 0, yi = 0, zi = 0;
    if (t < n_tgt) {
        ti = tgt[t];
        if (ti < 0 || ti >= n_src) {
            atomicOr(status, 2u);
            ti = -1;
        } else {
            xi = src[ti].x;
            yi = src[ti].y;
            zi = src[ti].z;
        }
    }
    double ax = 0, ay = 0, az = 0, ph = 0;
    for (int64_t b = j0; b < j1; b += kTile) {
        const int64_t j = b + threadIdx.x;
        if (j < j1) {
            const otoo_src q = src[j];
            s[threadIdx.x] = make_double4(q.x, q.y, q.z, (double)q.m);
        }
        __syncthreads();
        const int cnt = j1 - b < kTile ? (int)(j1 - b) : kTile;
        const int kself = (ti >= b && ti < b + cnt) ? (int)(ti - b) : -1;  // j != i
        for (int k = 0; k < cnt; ++k) {
            const double4 q = s[k];
            const double rx = q.x - xi, ry = q.y - yi, rz = q.z - zi;
            // (18 FP64 operations per pair, rsqrt 5 of them: 1.6 per clock and SM bound this kernel)
            const double r2 = fma(rx, rx, fma(ry, ry, fma(rz, rz, eps2)));
            const double inv = rsqrt(r2);
            const double mi = (k == kself ? 0.0 : q.w) * inv;
            const double mi3 = mi * inv * inv;
            ax += mi3 * rx;
            ay += mi3 * ry;
            az += mi3 * rz;
            ph -= mi;
        }
        __syncthreads();
    }
    if (t < n_tgt) {
        double* d = part + ((int64_t)blockIdx.y * n_tgt + t) * 4;
        d[0] = ax;
        d[1] = ay;
        d[2] = az;
        d[3] = ph;
    }
}

__global__ void k_direct_sum(const double* __restrict__ part, int64_t n_tgt, int n_chunk, double* __restrict__ accel,
                             double* __restrict__ pot)
{
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= n_tgt) return;
    double a[4] = {0, 0, 0, 0};
    for (int c = 0; c < n_chunk; ++c)
        for (int k = 0; k < 4; ++k) a[k] += part[((int64_t)c * n_tgt + t) * 4 + k];
    accel[3 * t] = a[0];
    accel[3 * t + 1] = a[1];
    accel[3 * t + 2] = a[2];
    pot[t] = a[3];
}

#define CUDA_TRY(expr)                                                                                 \
    do {                                                                                               \
        cudaError_t e_ = (expr);                                                                       \
        if (e_ != cudaSuccess) return set_error(OTOO_ECUDA, "%s: %s", #expr, cudaGetErrorString(e_));  \
    } while (0)

}  // namespace

extern "C" {

int64_t otoo_direct_chunks(int64_t n_src, int64_t n_tgt)
{
    if (n_src < 1 || n_tgt < 1) return 0;
    // enough blocks to fill the GPU several times over
    const int64_t tblocks = (n_tgt + kTgt - 1) / kTgt;
    int64_t chunks = (4 * 152 + tblocks - 1) / tblocks;
    if (chunks < 1) chunks = 1;
    const int64_t maxc = (n_src + kTile - 1) / kTile;
    return chunks < maxc ? chunks : maxc;
}

int otoo_direct(const otoo_src* src, int64_t n_src, const int64_t* targets, int64_t n_tgt, double eps2, double* accel,
                double* pot, double* scratch, uint32_t* status, void* stream)
{
    otoo::Range range_("otoo_direct");
    OTOO_REQUIRE(src && targets && accel && pot && scratch && status, OTOO_EINVAL, "otoo_direct: NULL pointer");
    OTOO_REQUIRE(n_src >= 1 && n_tgt >= 1 && n_tgt <= ((int64_t)1 << 31), OTOO_EINVAL, "otoo_direct: bad sizes");
    OTOO_REQUIRE(eps2 > 0.0, OTOO_EINVAL, "otoo_direct: eps2 must be > 0");
    const int64_t nc = otoo_direct_chunks(n_src, n_tgt);
    const int64_t chunk = ((n_src + nc - 1) / nc + kTile - 1) / kTile * kTile;
    const int64_t nch = (n_src + chunk - 1) / chunk;
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    CUDA_TRY(cudaMemsetAsync(status, 0, sizeof(uint32_t), s));
    dim3 grid((unsigned)((n_tgt + kTgt - 1) / kTgt), (unsigned)nch);
    if (n_src >= kTfMinSources) {
        // the range lives in accel until the last kernel writes it
        static_assert(sizeof(DirectRange) <= 3 * sizeof(double), "accel of one target holds the range");
        DirectRange* range = reinterpret_cast<DirectRange*>(accel);
        CUDA_TRY(cudaMemsetAsync(range, 0, sizeof(DirectRange), s));
        k_direct_range<<<(unsigned)((n_src + 2047) / 2048 < 608 ? (n_src + 2047) / 2048 : 608), 256, 0, s>>>(src, n_src,
                                                                                                        range);
        dim3 gtf((unsigned)((n_tgt + 255) / 256), (unsigned)nch);
        k_direct_tf<<<gtf, 256, 0, s>>>(src, n_src, targets, n_tgt, eps2, chunk, scratch, range, status);
        CUDA_TRY(cudaGetLastError());
        k_direct_part<true><<<grid, kTgt, 0, s>>>(src, n_src, targets, n_tgt, eps2, chunk, scratch, range, status);
    } else {
        k_direct_part<false><<<grid, kTgt, 0, s>>>(src, n_src, targets, n_tgt, eps2, chunk, scratch, nullptr, status);
    }
    CUDA_TRY(cudaGetLastError());
    k_direct_sum<<<(unsigned)((n_tgt + 127) / 128), 128, 0, s>>>(scratch, n_tgt, (int)nch, accel, pot);
    CUDA_TRY(cudaGetLastError());
    return OTOO_OK;
}

}  // extern "C"
