// Direct summation on the device: chosen targets against every particle of
// a system, to FP64's accuracy -- the exact reference the learned opening angle is
// trained against (the measured group errors are this sum's, the paper's
// O(N^2) brute force of Section II), and a check of the tree force.
//
// Kernels
//   k_direct_range, k_direct_tf  at least kTfMinSources sources: the system's
//                  scale, then the pairs in two-float arithmetic
//                  (twofloat.cuh), 256 targets per block.
//   k_direct_part  fewer sources, or a scale the two-float form does not take
//                  (k_direct_tf then returns at once, else this one does): block
//                  (target tile of 128, source chunk): the chunk's sources staged
//                  through shared memory, FP64 pairs, one partial sum per (chunk,
//                  target).
//   k_direct_sum / k_direct_tree  the chunk partials of each target, in chunk
//                  order or by the lanes of a warp.
#include <cuda_runtime.h>

#include <cstdint>

#include "../common.h"

using namespace otoo;

namespace {

#include "pair.cuh"
#include "twofloat.cuh"

constexpr int kTgt = 128;     // targets per block
constexpr int kTile = 128;    // sources staged per tile

// Largest |coordinate|, largest and smallest mass of the sources
// (order-preserving bit patterns; range is zero before the launch): the scales of
// the two-float form.  An infinite or NaN coordinate gives the largest pattern.
struct DirectRange {
    unsigned long long xmax;
    uint32_t mmax;
    uint32_t mlow;  // 0x7f800000 less the smallest positive mass's pattern
};

__device__ __forceinline__ TfScale direct_scale(const DirectRange* __restrict__ r, double eps2)
{
    return tf_scale(r->xmax, r->mmax, 0x7f800000u - r->mlow, eps2);
}

__global__ void __launch_bounds__(256) k_direct_range(const otoo_src* __restrict__ src, int64_t n,
                                                      DirectRange* __restrict__ range)
{
    unsigned long long x = 0;
    uint32_t m = 0, ml = 0;
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
        if (w - 1u < 0x7f7fffffu) ml = max(ml, 0x7f800000u - w);  // (neither zero, infinite nor NaN)
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long u = __shfl_xor_sync(kFull, x, o);
        x = u > x ? u : x;
    }
    m = __reduce_max_sync(kFull, m);
    ml = __reduce_max_sync(kFull, ml);
    if ((threadIdx.x & 31) == 0) {
        atomicMax(&range->xmax, x);
        atomicMax(&range->mmax, m);
        atomicMax(&range->mlow, ml);
    }
}

// The two-float form: 256 targets per block, two per thread; the block's
// halves of 128 threads take the halves of every staged tile, and the second
// half's sums join the first's at the end.  The float sums are moved into FP64
// every kTfFold tiles.  Bound by the FP32 pipe: about 260 packed operations per
// source and two targets.
// N = 2^19, 5003 targets: 24.0 ms (1.09e11 pairs/s) against 110 ms for the FP64
// form.  Relative error (2-norm over 40 targets, against extended precision) over
// N = 66000 and 130000, four models, softenings 1e-4 and 1e-2, and 40, 600 and 5000
// targets, two-float / FP64 form: accelerations 0.6e-16 to 1.2e-16 / 2.5e-16 to
// 9.2e-16, potentials 0.5e-16 to 1.2e-16 / 1.9e-16 to 7.4e-16; with one particle 1e3
// to 1e7 core radii out 0.8e-16 to 2.1e-16 / 2.5e-16 to 6.7e-16; with a fifth of the
// system in close groups of 2 to 1000, 1.5e-16 to 8.0e-16 / 7.8e-16 to 3.0e-15.
// (Before, with coordinates on one grid of 2^-62 of the extent, r^2 summed in plain
// floats and one pair of a run again in FP64, 25.1 ms in a wave and a twentieth: 2.9e-16 to 1.3e-15, 4e-16 to
// 7e-13 and 3e-16 to 2e-13, larger than the FP64 form's in most of them.)
// Below 65536 sources the FP64 form stays: the line is not a matter of accuracy.
constexpr int64_t kTfMinSources = 65536;
constexpr int kTfTile = 256;
constexpr int kTfFold = 8;  // the longest run (1024 sources of each half) the float sums take before FP64

constexpr unsigned kTfPos = kTfFold * kTfTile - 1;  // position in a run
static_assert(((kTfPos + 1) & kTfPos) == 0, "a run's length is a power of two");

// The pairs of a run that are evaluated again in FP64: the four heaviest of its even
// and the four of its odd positions (two lists of four cost half the comparisons of
// one of eight).
constexpr int kTfTop = 4;
constexpr int kTfLists = 2;

// A target's coordinates, negated, and another's, one field per operand.
struct TfTargets {
    f2 n[3][4];
};
__device__ __forceinline__ f2 tf_pack_neg(float a, float b) { return f2pack(-a, -b); }
__device__ __forceinline__ void tf_targets(const TfCoord c0[3], const TfCoord c1[3], TfTargets& t)
{
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        t.n[a][0] = tf_pack_neg(c0[a].a, c1[a].a);
        t.n[a][1] = tf_pack_neg(c0[a].b, c1[a].b);
        t.n[a][2] = tf_pack_neg(c0[a].c, c1[a].c);
        t.n[a][3] = tf_pack_neg(c0[a].d, c1[a].d);
    }
}

// What one heavy pair of each target of a run (run0 + the low bits of top) lacks:
// its FP64 value less the two-float one, added to sum.  A few close pairs at a
// small softening can be most of a target's acceleration, and their 2^-48 would
// then be the sum's error.
__device__ __forceinline__ void tf_refine(const otoo_src* __restrict__ src, int64_t run0, int64_t j1, unsigned top0,
                                          unsigned top1, const int64_t ti[2], const TfTargets& tg, const TfScale& sc,
                                          float ms, double eps2, const F2v3& e2, double sum[4][2])
{
    const double es = eps2 * tf_pow2(-2 * sc.ex), sx = tf_pow2(-sc.ex);
    TfCoord c[2][3];
    float m[2];
    double fix[4][2];
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        const unsigned top = k ? top1 : top0;
        int64_t j = run0 + (top & kTfPos);
        j = j < j1 ? j : j1 - 1;
        const otoo_src q = src[j];
        c[k][0] = tf_split(q.x, sc.ex);
        c[k][1] = tf_split(q.y, sc.ex);
        c[k][2] = tf_split(q.z, sc.ex);
        m[k] = j == ti[k] || top == 0u ? 0.f : q.m * ms;  // (0: no pair)
        const otoo_src t = src[ti[k] < 0 ? j : ti[k]];
        const double rx = (q.x - t.x) * sx, ry = (q.y - t.y) * sx, rz = (q.z - t.z) * sx;
        const double r2 = fma(rx, rx, fma(ry, ry, fma(rz, rz, es)));
        // (the library's rsqrt is within an ulp, three of them in its cube: corrected
        // by its residual e = 1 - r^2 y^2)
        const double y = rsqrt(r2), yy = y * y, e = fma(-r2, fma(y, y, -yy), fma(-r2, yy, 1.0));
        const double my = (double)m[k] * y, myyy = my * yy, mi3 = fma(1.5 * myyy, e, myyy);
        fix[0][k] = mi3 * rx;
        fix[1][k] = mi3 * ry;
        fix[2][k] = mi3 * rz;
        fix[3][k] = fma(0.5 * my, e, my);
    }
    F2x2 d[3];
#pragma unroll
    for (int a = 0; a < 3; ++a)
        d[a] = tf_diff(f2add(f2pack(c[0][a].a, c[1][a].a), tg.n[a][0]), f2add(f2pack(c[0][a].b, c[1][a].b), tg.n[a][1]),
                       f2add(f2pack(c[0][a].c, c[1][a].c), tg.n[a][2]), f2add(f2pack(c[0][a].d, c[1][a].d), tg.n[a][3]));
    F2x3 A[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) A[k].zero();
    tf_pair_mono(d[0], d[1], d[2], f2pack(m[0], m[1]), e2, A);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        double v0, v1;
        A[k].value(v0, v1);
        sum[k][0] += fix[k][0] - v0;
        sum[k][1] += fix[k][1] - v1;
    }
}

// Keeps the kTfTop largest of the values w has taken, in order.
__device__ __forceinline__ void tf_keep(unsigned top[kTfTop], unsigned w)
{
#pragma unroll
    for (int r = 0; r < kTfTop; ++r) {
        const unsigned hi = max(top[r], w);
        w = min(top[r], w);
        top[r] = hi;
    }
}

__global__ void __launch_bounds__(256, 2) k_direct_tf(const otoo_src* __restrict__ src, int64_t n_src,
                                                      const int64_t* __restrict__ tgt, int64_t n_tgt, double eps2,
                                                      int64_t chunk, double* __restrict__ part,
                                                      const DirectRange* __restrict__ range,
                                                      uint32_t* __restrict__ status)
{
    __shared__ ulonglong2 s_c[6][kTfTile];  // the fields (a, b) and (c, d) of x, y, z, each twice
    __shared__ float s_m[kTfTile];
    __shared__ double s_sum[128][9];
    const TfScale sc = direct_scale(range, eps2);
    if (!sc.ok) return;  // k_direct_part runs
    const int lt = threadIdx.x & 127, half = threadIdx.x >> 7;
    const int64_t j0 = (int64_t)blockIdx.y * chunk;
    const int64_t j1 = j0 + chunk < n_src ? j0 + chunk : n_src;
    int64_t ti[2];
    TfTargets tg;
    {
        TfCoord c[2][3];
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            const int64_t t = (int64_t)blockIdx.x * 256 + 128 * k + lt;
            ti[k] = -1;
            c[k][0] = c[k][1] = c[k][2] = TfCoord{0.f, 0.f, 0.f, 0.f};
            if (t < n_tgt) {
                ti[k] = tgt[t];
                if (ti[k] < 0 || ti[k] >= n_src) {
                    atomicOr(status, 2u);
                    ti[k] = -1;
                } else {
                    const otoo_src q = src[ti[k]];
                    c[k][0] = tf_split(q.x, sc.ex);
                    c[k][1] = tf_split(q.y, sc.ex);
                    c[k][2] = tf_split(q.z, sc.ex);
                }
            }
        }
        tf_targets(c[0], c[1], tg);
    }
    F2v3 e2;
    {
        const double e = eps2 * tf_pow2(-2 * sc.ex);  // exact
        const float eh = __double2float_rn(e), el = __double2float_rn(e - (double)eh);
        e2.h = f2dup(eh);
        e2.l = f2dup(el);
        // (in two floats it would be off by the same 2^-50 in every pair)
        e2.t = f2dup(__double2float_rn((e - (double)eh) - (double)el));
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
    // the run's heaviest pairs per list and target: m r^-2's bits above the position in the run
    unsigned top[kTfLists][2][kTfTop];
#pragma unroll
    for (int r = 0; r < kTfTop; ++r)
#pragma unroll
        for (int u = 0; u < kTfLists; ++u) top[u][0][r] = top[u][1][r] = 0u;
    for (int64_t b = j0; b < j1; b += kTfTile) {
        const int64_t j = b + threadIdx.x;
        if (j < j1) {
            const otoo_src q = src[j];
            const double x[3] = {q.x, q.y, q.z};
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                const TfCoord c = tf_split(x[a], sc.ex);
                s_c[2 * a][threadIdx.x] = make_ulonglong2(f2dup(c.a), f2dup(c.b));
                s_c[2 * a + 1][threadIdx.x] = make_ulonglong2(f2dup(c.c), f2dup(c.d));
            }
            s_m[threadIdx.x] = q.m * ms;
        }
        __syncthreads();
        const int cnt = j1 - b < kTfTile ? (int)(j1 - b) : kTfTile;
        const int k0 = half * (kTfTile / 2), k1 = half ? cnt : (cnt < kTfTile / 2 ? cnt : kTfTile / 2);
        const int self0 = ti[0] >= b && ti[0] < b + cnt ? (int)(ti[0] - b) : -1;  // j != i
        const int self1 = ti[1] >= b && ti[1] < b + cnt ? (int)(ti[1] - b) : -1;
#pragma unroll 1
        for (int k2 = k0; k2 < k1; k2 += kTfLists) {
#pragma unroll
            for (int u = 0; u < kTfLists; ++u) {
                const int k = k2 + u;
                if (k >= k1) break;
                const float m = s_m[k];
                F2x2 d[3];
#pragma unroll
                for (int a = 0; a < 3; ++a) {
                    const ulonglong2 p = s_c[2 * a][k], q = s_c[2 * a + 1][k];
                    d[a] = tf_diff(f2add(p.x, tg.n[a][0]), f2add(p.y, tg.n[a][1]), f2add(q.x, tg.n[a][2]),
                                   f2add(q.y, tg.n[a][3]));
                }
                float w0, w1;
                f2unpack(tf_pair_mono(d[0], d[1], d[2], f2pack(k == self0 ? 0.f : m, k == self1 ? 0.f : m), e2, A), w0,
                         w1);
                const unsigned at = (unsigned)(fold * kTfTile + k);
                tf_keep(top[u][0], (__float_as_uint(w0) & ~kTfPos) | at);
                tf_keep(top[u][1], (__float_as_uint(w1) & ~kTfPos) | at);
            }
        }
        if (++fold == kTfFold || b + kTfTile >= j1) {
            fold = 0;
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                double v0, v1;
                A[c].value(v0, v1);
                sum[c][0] += v0;
                sum[c][1] += v1;
                A[c].zero();
            }
            // the heaviest pairs of the run again in FP64, less what was added for them
#pragma unroll 1
            for (int r = 0; r < kTfTop; ++r)
#pragma unroll
                for (int u = 0; u < kTfLists; ++u) {
                    tf_refine(src, run0, j1, top[u][0][0], top[u][1][0], ti, tg, sc, ms, eps2, e2, sum);
#pragma unroll
                    for (int k = 0; k < 2; ++k) {
#pragma unroll
                        for (int q = 0; q + 1 < kTfTop; ++q) top[u][k][q] = top[u][k][q + 1];
                        top[u][k][kTfTop - 1] = 0u;
                    }
                }
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
    if (kAfterTf && direct_scale(range, eps2).ok) return;
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
            // (18 FP64 operations per pair, rsqrt 5 of them: 1.7 per clock and SM bound this kernel)
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

// The same by a warp per target (at least kTfMinSources sources): lane l the chunks
// l, l + 32, ..., then the lanes pairwise.  One after another, the up to 608 partials of
// a few targets lose more digits than the pairs (N = 66000, 40 targets: 8.2e-16 of the
// acceleration).
__global__ void __launch_bounds__(128) k_direct_tree(const double* __restrict__ part, int64_t n_tgt, int n_chunk,
                                                     double* __restrict__ accel, double* __restrict__ pot)
{
    const int lane = threadIdx.x & 31;
    const int64_t t = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (t >= n_tgt) return;
    double a[4] = {0, 0, 0, 0};
    for (int c = lane; c < n_chunk; c += 32)
#pragma unroll
        for (int k = 0; k < 4; ++k) a[k] += part[((int64_t)c * n_tgt + t) * 4 + k];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
        for (int k = 0; k < 4; ++k) a[k] += __shfl_xor_sync(kFull, a[k], o);
    if (lane < 3) accel[3 * t + lane] = lane == 0 ? a[0] : lane == 1 ? a[1] : a[2];
    if (lane == 3) pot[t] = a[3];
}

// Sources per chunk of the two-float form: as many chunks (nc at most) as fill one to
// four waves of its blocks (256 targets each, two resident per SM), or the FP64
// form's number, whichever takes the least time.  A wave takes its chunk's sources
// and about 128 more for a block's start and the pairs evaluated again, one of a few
// blocks half of that (140 blocks took as long as 304: they are not spread over the
// SMs one by one).  N = 2^19, 5003 targets: 24.0 ms in one wave of 300 blocks, 32.9 ms
// with the 320 that the FP64 form's rule gives.
int64_t direct_tf_chunk(int64_t n_src, int64_t n_tgt, int64_t nc, int nsm)
{
    const int64_t tb = (n_tgt + 255) / 256, resident = 2 * (int64_t)nsm;
    int64_t best = 0;
    double cost = 1e300;
    for (int w = 0; w <= 4; ++w) {
        const int64_t c = w == 0 ? nc : w * resident / tb;
        if (c < 1 || c > nc) continue;
        const int64_t chunk = ((n_src + c - 1) / c + kTile - 1) / kTile * kTile;
        const int64_t blocks = tb * ((n_src + chunk - 1) / chunk), rest = blocks % resident;
        const double waves = (double)(blocks / resident) + (rest == 0 ? 0.0 : rest > resident / 8 ? 1.0 : 0.5);
        const double t = waves * (double)(chunk + 128);
        if (t < cost) cost = t, best = chunk;
    }
    return best;
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
    int64_t chunk = ((n_src + nc - 1) / nc + kTile - 1) / kTile * kTile;
    if (n_src >= kTfMinSources) {
        int dev = 0, nsm = 0;
        CUDA_TRY(cudaGetDevice(&dev));
        CUDA_TRY(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
        chunk = direct_tf_chunk(n_src, n_tgt, nc, nsm);
    }
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
    if (n_src >= kTfMinSources)
        k_direct_tree<<<(unsigned)((n_tgt + 3) / 4), 128, 0, s>>>(scratch, n_tgt, (int)nch, accel, pot);
    else
        k_direct_sum<<<(unsigned)((n_tgt + 127) / 128), 128, 0, s>>>(scratch, n_tgt, (int)nch, accel, pot);
    CUDA_TRY(cudaGetLastError());
    return OTOO_OK;
}

}  // extern "C"
