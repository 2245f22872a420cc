// Learned opening angle: a 6-32-32-1 multilayer perceptron that predicts a
// group's log10 RMS relative force error from statistics of its interaction
// list and a candidate opening angle.  The paper controls accuracy with the
// absolute MAC parameter Delta (Section II-B, Eq. SW_MAC; Section III-F); this
// network replaces that control by choosing an angle per group.
//
// Kernels
//   k_mlp_forward   one thread per row, bf16 weights widened to FP32 in shared
//                   memory, FP32 accumulation, tanhf activations.
//   k_mlp_backward  one CTA per 128 rows: four threads run a row forward and
//                   backward, the per-row deltas go to shared memory, then the
//                   threads sum the rows' outer products in fixed row order
//                   into a per-CTA gradient partial (deterministic).
//   k_mlp_adam      eight threads per parameter sum the CTA partials in a
//                   fixed order, one applies Adam to the FP32 master weight and rounds
//                   the bf16 copy (round to nearest even).
//   k_select_theta  one thread per group: the largest grid angle whose
//                   predicted error meets the target.
//   k_theta_weights, k_theta_lambda, k_theta_choose
//                   the whole per-group selection from raw list statistics
//                   (otoo_learned_theta): range check, standardisation,
//                   budgeted per-group targets normalised to the global RMS
//                   target, the choice over the angle grid.
//   k_group_rms     per-group RMS relative acceleration error (labels).
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cmath>
#include <cstdint>

#include "../common.h"

using namespace otoo;

namespace {

constexpr int NI = OTOO_MLP_IN;
constexpr int NH = OTOO_MLP_H;
constexpr int NP = OTOO_MLP_NPARAM;
// parameter offsets
constexpr int OW1 = 0;
constexpr int OB1 = OW1 + NH * NI;
constexpr int OW2 = OB1 + NH;
constexpr int OB2 = OW2 + NH * NH;
constexpr int OW3 = OB2 + NH;
constexpr int OB3 = OW3 + NH;
static_assert(OB3 + 1 == NP, "parameter layout");

constexpr int kRowsPerCta = 128;
__device__ __forceinline__ float bf16_to_f(uint16_t b) { return __uint_as_float((uint32_t)b << 16); }

__device__ __forceinline__ void load_weights(const uint16_t* __restrict__ wbf16, float* s_w)
{
    for (int k = threadIdx.x; k < NP; k += blockDim.x) s_w[k] = bf16_to_f(wbf16[k]);
    __syncthreads();
}

// Forward pass of one row; keeps the activations.
__device__ __forceinline__ float forward_row(const float* __restrict__ w, const float x[NI], float h1[NH], float h2[NH])
{
#pragma unroll
    for (int i = 0; i < NH; ++i) {
        float z = w[OB1 + i];
#pragma unroll
        for (int k = 0; k < NI; ++k) z = fmaf(w[OW1 + i * NI + k], x[k], z);
        h1[i] = tanhf(z);
    }
#pragma unroll 4
    for (int i = 0; i < NH; ++i) {
        float z = w[OB2 + i];
#pragma unroll
        for (int j = 0; j < NH; ++j) z = fmaf(w[OW2 + i * NH + j], h1[j], z);
        h2[i] = tanhf(z);
    }
    float y = w[OB3];
#pragma unroll
    for (int j = 0; j < NH; ++j) y = fmaf(w[OW3 + j], h2[j], y);
    return y;
}

__global__ void k_mlp_forward(const uint16_t* __restrict__ wbf16, const float* __restrict__ x, float* __restrict__ y,
                              int64_t n)
{
    __shared__ float s_w[NP];
    load_weights(wbf16, s_w);
    const int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= n) return;
    float xr[NI], h1[NH], h2[NH];
#pragma unroll
    for (int k = 0; k < NI; ++k) xr[k] = x[r * NI + k];
    y[r] = forward_row(s_w, xr, h1, h2);
}

// Loss L = (1/n) sum_r (y_r - t_r)^2 and its gradient, per-CTA partials:
// part[cta][0..NP) = gradient sum over the CTA's rows, part[cta][NP] = sum of
// squared residuals / n.
//
// Four threads per row: each computes eight hidden units of each layer and
// eight deltas of the first, exchanging them through shared memory; every sum
// of a row is in forward_row's order.  Then the outer products over the rows:
// the second layer's 32 x 32 as 4 x 4 tiles per thread (two 16-byte loads for
// 16 products) with the rows in eight slices, the rest likewise with more
// slices, the slices added in order.  A batch of 8192 rows gives 64 CTAs, one
// per SM on less than half the GPU, so a CTA's own time counts, and in the form
// before (a thread per row, then a thread per parameter over all rows) that was
// shared-memory loads, two for each product: 12.4 us against 22.8 us.
constexpr int kBackThreads = 4 * kRowsPerCta;
constexpr int kU = NH / 4;   // hidden units per thread
constexpr int kSt = NH + 4;  // floats per row of a unit array (16-byte aligned rows, spread over the banks)

struct BackShared {
    float h1[kRowsPerCta][kSt], h2[kRowsPerCta][kSt], d1[kRowsPerCta][kSt], d2[kRowsPerCta][kSt];
    float x[kRowsPerCta][8];  // the row's inputs, 1 (past the last row 0), 0
    float dy[kRowsPerCta];
    float w2t[NH][NH];        // second layer's weights, transposed
    float w[NP + 3];
    float red[8 * NH * NH];   // slice sums
};

__device__ __forceinline__ float4 ld4(const float* p) { return *reinterpret_cast<const float4*>(p); }

// g[4][4] += a (column) b (row)
__device__ __forceinline__ void outer4(float g[16], float4 a, float4 b)
{
    const float av[4] = {a.x, a.y, a.z, a.w}, bv[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) g[4 * i + j] = fmaf(av[i], bv[j], g[4 * i + j]);
}

__global__ void __launch_bounds__(kBackThreads) k_mlp_backward(const uint16_t* __restrict__ wbf16,
                                                               const float* __restrict__ x,
                                                               const float* __restrict__ tgt, int64_t n,
                                                               float* __restrict__ part)
{
    extern __shared__ __align__(16) unsigned char back_smem[];
    BackShared& sh = *reinterpret_cast<BackShared*>(back_smem);
    const int64_t r0 = (int64_t)blockIdx.x * kRowsPerCta;
    const int tid = threadIdx.x;
    const int row = tid >> 2, u0 = (tid & 3) * kU;
    const int64_t r = r0 + row;
    const bool on = r < n;
    const float inv_n = 1.0f / (float)n;
    const float* __restrict__ xp = on ? x + r * NI : x;
    float xr[NI], target = 0.f;
#pragma unroll
    for (int k = 0; k < NI; ++k) xr[k] = xp[k];
    if (on) target = tgt[r];
    for (int k = tid; k < NP; k += kBackThreads) {
        const float w = bf16_to_f(wbf16[k]);
        sh.w[k] = w;
        if (k >= OW2 && k < OB2) sh.w2t[(k - OW2) % NH][(k - OW2) / NH] = w;
    }
    if (u0 == 0) {
#pragma unroll
        for (int k = 0; k < NI; ++k) sh.x[row][k] = xr[k];
        sh.x[row][NI] = on ? 1.f : 0.f;
        sh.x[row][NI + 1] = 0.f;
    }
    __syncthreads();
    float h1[kU], h2[kU];
#pragma unroll
    for (int u = 0; u < kU; ++u) {
        const int i = u0 + u;
        float z = sh.w[OB1 + i];
#pragma unroll
        for (int k = 0; k < NI; ++k) z = fmaf(sh.w[OW1 + i * NI + k], xr[k], z);
        h1[u] = tanhf(z);
    }
#pragma unroll
    for (int u = 0; u < kU; u += 4)
        *reinterpret_cast<float4*>(&sh.h1[row][u0 + u]) = make_float4(h1[u], h1[u + 1], h1[u + 2], h1[u + 3]);
    __syncwarp();
    {
        float z[kU];
#pragma unroll
        for (int u = 0; u < kU; ++u) z[u] = sh.w[OB2 + u0 + u];
#pragma unroll 4
        for (int j = 0; j < NH; ++j) {
            const float h = sh.h1[row][j];
            const float4 wa = ld4(&sh.w2t[j][u0]), wb = ld4(&sh.w2t[j][u0 + 4]);
            z[0] = fmaf(wa.x, h, z[0]), z[1] = fmaf(wa.y, h, z[1]), z[2] = fmaf(wa.z, h, z[2]), z[3] = fmaf(wa.w, h, z[3]);
            z[4] = fmaf(wb.x, h, z[4]), z[5] = fmaf(wb.y, h, z[5]), z[6] = fmaf(wb.z, h, z[6]), z[7] = fmaf(wb.w, h, z[7]);
        }
#pragma unroll
        for (int u = 0; u < kU; ++u) h2[u] = tanhf(z[u]);
#pragma unroll
        for (int u = 0; u < kU; u += 4)
            *reinterpret_cast<float4*>(&sh.h2[row][u0 + u]) = make_float4(h2[u], h2[u + 1], h2[u + 2], h2[u + 3]);
    }
    __syncwarp();
    {
        float yv = sh.w[OB3];
#pragma unroll
        for (int j = 0; j < NH; j += 4) {
            const float4 h = ld4(&sh.h2[row][j]);
            yv = fmaf(sh.w[OW3 + j], h.x, yv), yv = fmaf(sh.w[OW3 + j + 1], h.y, yv);
            yv = fmaf(sh.w[OW3 + j + 2], h.z, yv), yv = fmaf(sh.w[OW3 + j + 3], h.w, yv);
        }
        // places past the last row repeat the first without a residual: every delta is zero
        // (with zero inputs an infinite weight would make their hidden values NaN)
        const float dy = on ? 2.0f * (yv - target) * inv_n : 0.f;
        float d[kU];
#pragma unroll
        for (int u = 0; u < kU; ++u) d[u] = dy * sh.w[OW3 + u0 + u] * (1.0f - h2[u] * h2[u]);
#pragma unroll
        for (int u = 0; u < kU; u += 4)
            *reinterpret_cast<float4*>(&sh.d2[row][u0 + u]) = make_float4(d[u], d[u + 1], d[u + 2], d[u + 3]);
        if (u0 == 0) sh.dy[row] = dy;
    }
    __syncwarp();
    {
        float sd[kU];
#pragma unroll
        for (int u = 0; u < kU; ++u) sd[u] = 0.f;
#pragma unroll 4
        for (int i = 0; i < NH; ++i) {
            const float d = sh.d2[row][i];
            const float4 wa = ld4(&sh.w[OW2 + i * NH + u0]), wb = ld4(&sh.w[OW2 + i * NH + u0 + 4]);
            sd[0] = fmaf(wa.x, d, sd[0]), sd[1] = fmaf(wa.y, d, sd[1]), sd[2] = fmaf(wa.z, d, sd[2]), sd[3] = fmaf(wa.w, d, sd[3]);
            sd[4] = fmaf(wb.x, d, sd[4]), sd[5] = fmaf(wb.y, d, sd[5]), sd[6] = fmaf(wb.z, d, sd[6]), sd[7] = fmaf(wb.w, d, sd[7]);
        }
#pragma unroll
        for (int u = 0; u < kU; ++u) sd[u] *= 1.0f - h1[u] * h1[u];
#pragma unroll
        for (int u = 0; u < kU; u += 4)
            *reinterpret_cast<float4*>(&sh.d1[row][u0 + u]) = make_float4(sd[u], sd[u + 1], sd[u + 2], sd[u + 3]);
    }
    __syncthreads();
    float* out = part + (int64_t)blockIdx.x * (NP + 1);
    // W2: slice tid / 64 of 16 rows, tile (tid % 64)
    {
        const int s0 = (tid >> 6) * 16, ti = ((tid >> 3) & 7) * 4, tj = (tid & 7) * 4;
        float g[16];
#pragma unroll
        for (int k = 0; k < 16; ++k) g[k] = 0.f;
#pragma unroll 4
        for (int q = s0; q < s0 + 16; ++q) outer4(g, ld4(&sh.d2[q][ti]), ld4(&sh.h1[q][tj]));
        float* red = sh.red + (tid >> 6) * NH * NH;
#pragma unroll
        for (int k = 0; k < 4; ++k)
            *reinterpret_cast<float4*>(red + (ti + k) * NH + tj) = make_float4(g[4 * k], g[4 * k + 1], g[4 * k + 2], g[4 * k + 3]);
    }
    __syncthreads();
    for (int p = tid; p < NH * NH; p += kBackThreads) {
        float g = sh.red[p];
#pragma unroll
        for (int k = 1; k < 8; ++k) g += sh.red[k * NH * NH + p];
        out[OW2 + p] = g;
    }
    __syncthreads();
    // W1 and b1: d1 (x, 1): slice tid / 16 of 4 rows, tile tid % 16 (8 x 2 tiles); then b2 and w3:
    // column tid % 64 of (d2, dy h2), slice tid / 64 of 16 rows
    {
        const int s0 = (tid >> 4) * 4, ti = ((tid >> 1) & 7) * 4, tj = (tid & 1) * 4;
        float g[16];
#pragma unroll
        for (int k = 0; k < 16; ++k) g[k] = 0.f;
#pragma unroll
        for (int q = s0; q < s0 + 4; ++q) outer4(g, ld4(&sh.d1[q][ti]), ld4(&sh.x[q][tj]));
        float* red = sh.red + (tid >> 4) * 8 * NH;
#pragma unroll
        for (int k = 0; k < 4; ++k)
            *reinterpret_cast<float4*>(red + (ti + k) * 8 + tj) = make_float4(g[4 * k], g[4 * k + 1], g[4 * k + 2], g[4 * k + 3]);
    }
    float v = 0.f;
    {
        const int c = tid & 63, s0 = (tid >> 6) * 16;
#pragma unroll 8
        for (int q = s0; q < s0 + 16; ++q) v = c < NH ? v + sh.d2[q][c] : fmaf(sh.dy[q], sh.h2[q][c - NH], v);
    }
    __syncthreads();
    if (tid < 8 * NH) {
        float g = sh.red[tid];
#pragma unroll 8
        for (int k = 1; k < 32; ++k) g += sh.red[k * 8 * NH + tid];
        const int i = tid >> 3, k = tid & 7;
        if (k < NI)
            out[OW1 + i * NI + k] = g;
        else if (k == NI)
            out[OB1 + i] = g;
    } else if (tid < 8 * NH + 32) {
        // b3 and the loss (residual = dy n / 2): lane l sums rows 4 l .. 4 l + 3
        const int l = tid & 31;
        float gb = 0.f, gl = 0.f;
#pragma unroll
        for (int q = 4 * l; q < 4 * l + 4; ++q) {
            const float dy = sh.dy[q], res = dy * (0.5f * (float)n);
            gb += dy;
            gl = fmaf(res, res, gl);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            gb += __shfl_xor_sync(0xffffffffu, gb, o);
            gl += __shfl_xor_sync(0xffffffffu, gl, o);
        }
        if (l == 0) out[OB3] = gb, out[NP] = gl * inv_n;
    }
    __syncthreads();
    sh.red[(tid >> 6) * 64 + (tid & 63)] = v;
    __syncthreads();
    if (tid < 64) {
        float g = sh.red[tid];
#pragma unroll
        for (int k = 1; k < 8; ++k) g += sh.red[64 * k + tid];
        out[tid < NH ? OB2 + tid : OW3 + tid - NH] = g;
    }
}

// The sum of the CTA partials of parameter p (p = NP: the loss), by the eight
// threads of a block that hold slices threadIdx.y of it: slice y sums the
// partials y, y + 8, ... in order, then slice 0 adds the slices in order.  The
// result is in slice 0's thread.
constexpr int kSumX = 32, kSumY = 8;

__device__ __forceinline__ float sum_partials(const float* __restrict__ part, int nblk, int p)
{
    __shared__ float s[kSumY][kSumX];
    float g = 0.f;
    if (p <= NP) {
#pragma unroll 4
        for (int b = threadIdx.y; b < nblk; b += kSumY) g += part[(int64_t)b * (NP + 1) + p];
    }
    s[threadIdx.y][threadIdx.x] = g;
    __syncthreads();
    if (threadIdx.y == 0) {
#pragma unroll
        for (int k = 1; k < kSumY; ++k) g += s[k][threadIdx.x];
    }
    return g;
}

// Sum the CTA partials into grad and loss.
__global__ void k_mlp_reduce(const float* __restrict__ part, int nblk, float* __restrict__ grad, float* __restrict__ loss)
{
    const int p = blockIdx.x * kSumX + threadIdx.x;
    const float g = sum_partials(part, nblk, p);
    if (threadIdx.y != 0 || p > NP) return;
    if (p < NP)
        grad[p] = g;
    else if (loss)
        loss[0] = g;
}

// Adam (Kingma & Ba 2015) on the FP32 master weights, bias-corrected, then
// the bf16 copy is refreshed.
__global__ void k_mlp_adam(float* __restrict__ w, uint16_t* __restrict__ wbf16, float* __restrict__ m,
                           float* __restrict__ v, const float* __restrict__ part, int nblk, float lr, float b1,
                           float b2, float eps, float c1, float c2, float* __restrict__ loss)
{
    const int p = blockIdx.x * kSumX + threadIdx.x;
    const float g = sum_partials(part, nblk, p);
    if (threadIdx.y != 0 || p > NP) return;
    if (p == NP) {
        if (loss) loss[0] = g;
        return;
    }
    const float mm = b1 * m[p] + (1.f - b1) * g;
    const float vv = b2 * v[p] + (1.f - b2) * g * g;
    m[p] = mm;
    v[p] = vv;
    const float mh = mm / c1, vh = vv / c2;
    const float nw = w[p] - lr * mh / (sqrtf(vh) + eps);
    w[p] = nw;
    wbf16[p] = __bfloat16_as_ushort(__float2bfloat16_rn(nw));
}

__global__ void k_to_bf16(const float* __restrict__ w, uint16_t* __restrict__ o, int n)
{
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p < n) o[p] = __bfloat16_as_ushort(__float2bfloat16_rn(w[p]));
}

__global__ void k_select_theta(const uint16_t* __restrict__ wbf16, const float* __restrict__ x,
                               const float* __restrict__ grid, int nth, int64_t ng, float target,
                               const float* __restrict__ target_g, float fallback, float* __restrict__ out)
{
    __shared__ float s_w[NP];
    load_weights(wbf16, s_w);
    const int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (g >= ng) return;
    if (target_g) target = target_g[g];
    float best = grid[0];
    bool bad = false;
    for (int k = 0; k < nth; ++k) {
        float xr[NI], h1[NH], h2[NH];
        const float* xs = x + (g * nth + k) * NI;
#pragma unroll
        for (int c = 0; c < NI; ++c) xr[c] = xs[c];
        const float y = forward_row(s_w, xr, h1, h2);
        if (!isfinite(y)) bad = true;
        if (y <= target) best = fmaxf(best, grid[k]);
    }
    out[g] = bad ? fallback : best;
}

// ---- learned angle from raw list statistics ---------------------------------

constexpr int kThetaBlock = 128;

struct ThetaArgs {
    const uint16_t* wbf16;
    const float* mean;
    const float* std;
    const float* lo;
    const float* hi;
    const float* feat;     // [n][NI - 1]
    const int32_t* count;  // [n]
    int64_t n;
    float theta0, alpha, beta;
};

// Standardised row of group g's statistics with angle th.
__device__ __forceinline__ void theta_row(const ThetaArgs& a, int64_t g, float th, float x[NI])
{
#pragma unroll
    for (int k = 0; k < NI - 1; ++k) x[k] = __fdiv_rn(__fsub_rn(a.feat[g * (NI - 1) + k], a.mean[k]), a.std[k]);
    x[NI - 1] = __fdiv_rn(__fsub_rn(th, a.mean[NI - 1]), a.std[NI - 1]);
}

// Budget weight of every group (0 outside the training range or for a
// non-finite prediction): w = 10^(alpha y0 + beta log10 L), y0 the predicted
// log10 error at theta0, L = 2^feat[0] the list length at theta0; and the
// block's sums of count * w^2 and count over the groups that have a weight,
// in a fixed order (FP64).
__global__ void __launch_bounds__(kThetaBlock) k_theta_weights(const ThetaArgs a, float* __restrict__ wg,
                                                               double* __restrict__ part)
{
    __shared__ float s_w[NP];
    __shared__ double s_a[kThetaBlock], s_b[kThetaBlock];
    load_weights(a.wbf16, s_w);
    const int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    double nw2 = 0.0, nn = 0.0;
    if (g < a.n) {
        bool ok = true;
#pragma unroll
        for (int k = 0; k < NI - 1; ++k) {
            const float f = a.feat[g * (NI - 1) + k];
            ok = ok && isfinite(f);
            if (a.lo) ok = ok && f >= a.lo[k] && f <= a.hi[k];
        }
        float w = 0.f;
        if (ok) {
            float x[NI], h1[NH], h2[NH];
            theta_row(a, g, a.theta0, x);
            const float y0 = forward_row(s_w, x, h1, h2);
            // log10 L = feat[0] log10(2)
            const float e = fmaf(a.alpha, y0, a.beta * a.feat[g * (NI - 1)] * 0.30102999566398120f);
            w = isfinite(e) ? exp10f(e) : 0.f;
            if (!(w > 0.f) || !isfinite(w)) w = 0.f;
        }
        wg[g] = w;
        if (w > 0.f) {
            const double c = (double)a.count[g];
            nw2 = c * (double)w * (double)w;
            nn = c;
        }
    }
    s_a[threadIdx.x] = nw2;
    s_b[threadIdx.x] = nn;
    __syncthreads();
    for (int h = kThetaBlock / 2; h > 0; h >>= 1) {
        if (threadIdx.x < h) {
            s_a[threadIdx.x] += s_a[threadIdx.x + h];
            s_b[threadIdx.x] += s_b[threadIdx.x + h];
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        part[2 * blockIdx.x] = s_a[0];
        part[2 * blockIdx.x + 1] = s_b[0];
    }
}

// lambda = target / sqrt(sum count w^2 / sum count): the common factor that
// makes the particle-weighted RMS of the group targets equal to target.  One
// block sums the block partials: thread t those of t, t + 256, ..., then a
// fixed tree (one thread alone took 72 us for the 782 partials of 100003
// groups).
__global__ void __launch_bounds__(256) k_theta_lambda(const double* __restrict__ part, int nblk, double target,
                                                      double* __restrict__ lambda)
{
    __shared__ double s_a[256], s_b[256];
    double a = 0.0, b = 0.0;
    for (int k = threadIdx.x; k < nblk; k += 256) {
        a += part[2 * k];
        b += part[2 * k + 1];
    }
    s_a[threadIdx.x] = a;
    s_b[threadIdx.x] = b;
    __syncthreads();
    for (int h = 128; h > 0; h >>= 1) {
        if (threadIdx.x < h) {
            s_a[threadIdx.x] += s_a[threadIdx.x + h];
            s_b[threadIdx.x] += s_b[threadIdx.x + h];
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) lambda[0] = (s_a[0] > 0.0 && s_b[0] > 0.0) ? target / sqrt(s_a[0] / s_b[0]) : target;
}

// The choice: groups with a weight aim at log10(lambda w), the largest grid
// angle whose prediction is at most that (grid[0] when none); the others,
// and groups with a non-finite prediction, take the fallback angle.
//
// S threads per group, two angles each at a time from the end of the grid; the
// predictions are forward_row's, operation for operation (the angle is the
// last input, so the first layer's sums over the statistics are shared by all
// angles).  Where no prediction of the group can overflow (finite weights and
// inputs far inside the FP32 range: hidden values are within [-1, 1]) a group
// is done at the first angle that passes when the grid increases, and a warp
// at its last group's; otherwise every angle is evaluated.  A weight read from
// shared memory (four per load) serves both angles.  Bound by issue, half of
// it in tanhf.  100003 groups, 53 angles: 554 us against 770 us for one angle
// at a time over the whole grid.
constexpr int kChooseBlock = 64;

// Predictions of one group at two angles (x0, x1: the standardised angles):
// forward_row's operations, with the first layer's sums over the statistics
// from zs[i * zstride] and the second layer's weights as w2.
__device__ __forceinline__ void forward_two(const float* __restrict__ w, const float* __restrict__ w2,
                                            const float* __restrict__ zs, int zstride, float x0, float x1, float& y0,
                                            float& y1)
{
    float a[NH], b[NH];
#pragma unroll
    for (int i = 0; i < NH; ++i) {
        const float z = zs[i * zstride], wi = w[OW1 + i * NI + NI - 1];
        a[i] = tanhf(fmaf(wi, x0, z));
        b[i] = tanhf(fmaf(wi, x1, z));
    }
    y0 = y1 = w[OB3];
#pragma unroll 2
    for (int i = 0; i < NH; ++i) {
        float z0 = w[OB2 + i], z1 = z0;
        const float4* r = reinterpret_cast<const float4*>(w2 + NH * i);
#pragma unroll
        for (int q = 0; q < NH / 4; ++q) {
            const float4 v = r[q];
            z0 = fmaf(v.x, a[4 * q], z0), z1 = fmaf(v.x, b[4 * q], z1);
            z0 = fmaf(v.y, a[4 * q + 1], z0), z1 = fmaf(v.y, b[4 * q + 1], z1);
            z0 = fmaf(v.z, a[4 * q + 2], z0), z1 = fmaf(v.z, b[4 * q + 2], z1);
            z0 = fmaf(v.w, a[4 * q + 3], z0), z1 = fmaf(v.w, b[4 * q + 3], z1);
        }
        y0 = fmaf(w[OW3 + i], tanhf(z0), y0);
        y1 = fmaf(w[OW3 + i], tanhf(z1), y1);
    }
}

template <int S>
__global__ void __launch_bounds__(kChooseBlock) k_theta_choose(const ThetaArgs a, const float* __restrict__ wg,
                                                               const double* __restrict__ lambda,
                                                               const float* __restrict__ grid, int nth,
                                                               float fallback, float* __restrict__ tgt_out,
                                                               float* __restrict__ out)
{
    constexpr float kSafe = 1.0e6f;  // weights and inputs up to this leave every sum far below the FP32 range
    __shared__ __align__(16) float s_w2[NH * NH];
    __shared__ float s_w[NP];
    constexpr int G = kChooseBlock / S;  // groups per block
    __shared__ float s_z[NH * G];
    load_weights(a.wbf16, s_w);
    const float mean_t = a.mean[NI - 1], std_t = a.std[NI - 1];
    bool ok = true;
    for (int k = threadIdx.x; k < NP; k += kChooseBlock) ok = ok && fabsf(s_w[k]) <= kSafe;
    for (int k = threadIdx.x; k < NH * NH; k += kChooseBlock) s_w2[k] = s_w[OW2 + k];
    for (int k = threadIdx.x; k < nth; k += kChooseBlock)
        ok = ok && fabsf(__fdiv_rn(__fsub_rn(grid[k], mean_t), std_t)) <= kSafe && (k + 1 == nth || grid[k] < grid[k + 1]);
    const int gl = threadIdx.x / S, sub = threadIdx.x % S;
    const int64_t g = (int64_t)blockIdx.x * G + gl;
    const float w = g < a.n ? wg[g] : 0.f;
    const bool live = w > 0.f;
    float target = 0.f;
    if (live) {
        target = (float)log10(lambda[0] * (double)w);
        if (tgt_out && sub == 0) tgt_out[g] = target;
        float x[NI];
        theta_row(a, g, a.theta0, x);
#pragma unroll
        for (int k = 0; k < NI - 1; ++k) ok = ok && fabsf(x[k]) <= kSafe;
        for (int i = sub; i < NH; i += S) {
            float z = s_w[OB1 + i];
#pragma unroll
            for (int k = 0; k < NI - 1; ++k) z = fmaf(s_w[OW1 + i * NI + k], x[k], z);
            s_z[i * G + gl] = z;
        }
    }
    // (the barrier also publishes s_w2)
    const bool safe = __syncthreads_and(ok);
    const float th0 = grid[0];
    float best = th0;
    bool bad = false, done = !live;
    for (int k0 = nth - 1; k0 >= 0; k0 -= 2 * S) {
        if (!__any_sync(0xffffffffu, !done)) break;
        const int k = k0 - 2 * sub, k2 = k > 0 ? k - 1 : 0;
        bool pass = false;
        if (!done && k >= 0) {
            const float ta = grid[k], tb = grid[k2];
            float ya, yb;
            forward_two(s_w, s_w2, s_z + gl, G, __fdiv_rn(__fsub_rn(ta, mean_t), std_t),
                        __fdiv_rn(__fsub_rn(tb, mean_t), std_t), ya, yb);
            bad = bad || !isfinite(ya) || !isfinite(yb);
            pass = ya <= target || yb <= target;
            if (ya <= target) best = fmaxf(best, ta);
            if (yb <= target) best = fmaxf(best, tb);
        }
        // the group's threads stop together, after the round with its first passing angle
        const unsigned m = __ballot_sync(0xffffffffu, pass) >> (threadIdx.x & 31 & ~(S - 1));
        done = done || (safe && (m & ((1u << S) - 1u)) != 0u);
    }
#pragma unroll
    for (int o = S / 2; o > 0; o >>= 1) {
        best = fmaxf(best, __shfl_xor_sync(0xffffffffu, best, o));
        bad = __shfl_xor_sync(0xffffffffu, (int)bad, o) != 0 || bad;
    }
    if (sub != 0) return;
    if (g >= a.n) return;
    if (live) {
        out[g] = bad ? fallback : best;
    } else {
        if (tgt_out) tgt_out[g] = __int_as_float(0x7fc00000);  // no target: NaN
        out[g] = fallback;
    }
}

// Rows standardised with the training set's statistics: (x - mean) / std.
__global__ void k_standardise(const float* __restrict__ x, int64_t n, const float* __restrict__ mean,
                              const float* __restrict__ std, float* __restrict__ out)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n * NI) return;
    const int k = (int)(i % NI);
    out[i] = __fdiv_rn(__fsub_rn(x[i], mean[k]), std[k]);
}

// Per-group RMS of the relative acceleration error |a - ref| / |ref| over the
// targets [off[g], off[g + 1]) (one warp per group, lanes in a fixed order):
// out[g] = log10(max(rms, floor)).
__global__ void k_group_rms(const double* __restrict__ acc, const double* __restrict__ ref,
                            const int64_t* __restrict__ off, int64_t ng, float floor_v, float* __restrict__ out,
                            uint32_t* __restrict__ status)
{
    const int64_t g = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (g >= ng) return;
    const int64_t b = off[g], e = off[g + 1];
    if (b < 0 || e <= b) {
        if (lane == 0) {
            atomicOr(status, 1u);
            out[g] = __int_as_float(0x7fc00000);
        }
        return;
    }
    double s = 0.0;
    for (int64_t t = b + lane; t < e; t += 32) {
        double d2 = 0.0, r2 = 0.0;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const double d = acc[3 * t + c] - ref[3 * t + c];
            d2 = fma(d, d, d2);
            r2 = fma(ref[3 * t + c], ref[3 * t + c], r2);
        }
        s += d2 / r2;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) out[g] = (float)log10(fmax(sqrt(s / (double)(e - b)), (double)floor_v));
}

#define CUDA_TRY(expr)                                                                                 \
    do {                                                                                               \
        cudaError_t e_ = (expr);                                                                       \
        if (e_ != cudaSuccess) return set_error(OTOO_ECUDA, "%s: %s", #expr, cudaGetErrorString(e_));  \
    } while (0)

int backward(const uint16_t* wbf16, const float* x, const float* t, int64_t n, float* scratch, cudaStream_t s,
             int* nblk_out)
{
    const int64_t nb = (n + kRowsPerCta - 1) / kRowsPerCta;
    OTOO_REQUIRE(nb <= (1 << 20), OTOO_EINVAL, "too many rows");
    const size_t sm = sizeof(BackShared);
    CUDA_TRY(cudaFuncSetAttribute(k_mlp_backward, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm));
    k_mlp_backward<<<(unsigned)nb, kBackThreads, sm, s>>>(wbf16, x, t, n, scratch);
    CUDA_TRY(cudaGetLastError());
    *nblk_out = (int)nb;
    return OTOO_OK;
}

}  // namespace

extern "C" {

int64_t otoo_mlp_scratch_floats(int64_t n_rows)
{
    if (n_rows < 1) return 0;
    return ((n_rows + kRowsPerCta - 1) / kRowsPerCta) * (NP + 1);
}

int otoo_mlp_predict(const uint16_t* wbf16, const float* x, float* y, int64_t n_rows, void* stream)
{
    OTOO_REQUIRE(wbf16 && x && y, OTOO_EINVAL, "otoo_mlp_predict: NULL pointer");
    OTOO_REQUIRE(n_rows >= 0, OTOO_EINVAL, "otoo_mlp_predict: n_rows < 0");
    if (n_rows == 0) return OTOO_OK;
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    k_mlp_forward<<<(unsigned)((n_rows + 127) / 128), 128, 0, s>>>(wbf16, x, y, n_rows);
    CUDA_TRY(cudaGetLastError());
    return OTOO_OK;
}

int otoo_mlp_grad(const uint16_t* wbf16, const float* x, const float* target, int64_t n_rows, float* scratch,
                  float* grad, float* loss, void* stream)
{
    OTOO_REQUIRE(wbf16 && x && target && scratch && grad, OTOO_EINVAL, "otoo_mlp_grad: NULL pointer");
    OTOO_REQUIRE(n_rows >= 1, OTOO_EINVAL, "otoo_mlp_grad: n_rows < 1");
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    int nb = 0;
    int rc = backward(wbf16, x, target, n_rows, scratch, s, &nb);
    if (rc) return rc;
    k_mlp_reduce<<<(NP + 1 + kSumX - 1) / kSumX, dim3(kSumX, kSumY), 0, s>>>(scratch, nb, grad, loss);
    CUDA_TRY(cudaGetLastError());
    return OTOO_OK;
}

int otoo_mlp_train_step(float* w, uint16_t* wbf16, float* m, float* v, float* scratch, const float* x,
                        const float* target, int64_t n_rows, float lr, float beta1, float beta2, float eps_adam,
                        int32_t t, float* loss, void* stream)
{
    otoo::Range range_("otoo_mlp_train_step");
    OTOO_REQUIRE(w && wbf16 && m && v && scratch && x && target, OTOO_EINVAL, "otoo_mlp_train_step: NULL pointer");
    OTOO_REQUIRE(n_rows >= 1 && t >= 1, OTOO_EINVAL, "otoo_mlp_train_step: n_rows and t must be >= 1");
    OTOO_REQUIRE(lr > 0 && beta1 >= 0 && beta1 < 1 && beta2 >= 0 && beta2 < 1 && eps_adam > 0, OTOO_EINVAL,
                 "otoo_mlp_train_step: bad Adam hyper-parameters");
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    int nb = 0;
    int rc = backward(wbf16, x, target, n_rows, scratch, s, &nb);
    if (rc) return rc;
    const float c1 = 1.0f - powf(beta1, (float)t), c2 = 1.0f - powf(beta2, (float)t);
    k_mlp_adam<<<(NP + 1 + kSumX - 1) / kSumX, dim3(kSumX, kSumY), 0, s>>>(w, wbf16, m, v, scratch, nb, lr, beta1, beta2, eps_adam, c1, c2,
                                                     loss);
    CUDA_TRY(cudaGetLastError());
    return OTOO_OK;
}

int otoo_mlp_to_bf16(const float* w, uint16_t* wbf16, int32_t n, void* stream)
{
    OTOO_REQUIRE(w && wbf16 && n >= 0, OTOO_EINVAL, "otoo_mlp_to_bf16: bad argument");
    if (n == 0) return OTOO_OK;
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    k_to_bf16<<<(n + 255) / 256, 256, 0, s>>>(w, wbf16, n);
    CUDA_TRY(cudaGetLastError());
    return OTOO_OK;
}

int otoo_select_theta(const uint16_t* wbf16, const float* x, const float* theta_grid, int32_t n_theta,
                      int64_t n_groups, float log10_target, const float* log10_target_per_group, float fallback,
                      float* theta_out, void* stream)
{
    otoo::Range range_("otoo_select_theta");
    OTOO_REQUIRE(wbf16 && x && theta_grid && theta_out, OTOO_EINVAL, "otoo_select_theta: NULL pointer");
    OTOO_REQUIRE(n_theta >= 1 && n_groups >= 0, OTOO_EINVAL, "otoo_select_theta: bad sizes");
    if (n_groups == 0) return OTOO_OK;
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    k_select_theta<<<(unsigned)((n_groups + 127) / 128), 128, 0, s>>>(wbf16, x, theta_grid, n_theta, n_groups,
                                                                      log10_target, log10_target_per_group, fallback,
                                                                      theta_out);
    CUDA_TRY(cudaGetLastError());
    return OTOO_OK;
}

int otoo_mlp_standardise(const float* x, int64_t n_rows, const float* mean, const float* std, float* out,
                         void* stream)
{
    OTOO_REQUIRE(x && mean && std && out && n_rows >= 0, OTOO_EINVAL, "otoo_mlp_standardise: bad argument");
    if (n_rows == 0) return OTOO_OK;
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    const int64_t n = n_rows * NI;
    k_standardise<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(x, n_rows, mean, std, out);
    CUDA_TRY(cudaGetLastError());
    return OTOO_OK;
}

int64_t otoo_learned_theta_scratch_floats(int64_t n_groups)
{
    if (n_groups < 1) return 0;
    const int64_t nblk = (n_groups + kThetaBlock - 1) / kThetaBlock;
    // weights, then (aligned to 8 bytes) 2 doubles per block and lambda
    return ((n_groups + 1) & ~(int64_t)1) + 4 * nblk + 2;
}

int otoo_learned_theta(const otoo_theta_net* net, const otoo_theta_rule* rule, const float* feat,
                       const int32_t* count, int64_t n_groups, const float* grid, int32_t n_theta, float* scratch,
                       float* log10_target, float* theta_out, void* stream)
{
    otoo::Range range_("otoo_learned_theta");
    OTOO_REQUIRE(net && rule && feat && count && grid && scratch && theta_out, OTOO_EINVAL,
                 "otoo_learned_theta: NULL pointer");
    OTOO_REQUIRE(net->wbf16 && net->mean && net->std && ((net->lo == nullptr) == (net->hi == nullptr)), OTOO_EINVAL,
                 "otoo_learned_theta: network arrays missing (lo and hi are both set or both NULL)");
    OTOO_REQUIRE(n_theta >= 1 && n_groups >= 0 && n_groups < ((int64_t)1 << 31), OTOO_EINVAL,
                 "otoo_learned_theta: bad sizes");
    OTOO_REQUIRE(rule->target_rms > 0.f && rule->calib > 0.f && rule->theta0 > 0.f && std::isfinite(rule->alpha) &&
                     std::isfinite(rule->beta) && std::isfinite(rule->target_rms * rule->calib),
                 OTOO_EINVAL, "otoo_learned_theta: bad rule");
    OTOO_REQUIRE((reinterpret_cast<uintptr_t>(scratch) & 7) == 0, OTOO_EINVAL,
                 "otoo_learned_theta: scratch must be 8-byte aligned");
    if (n_groups == 0) return OTOO_OK;
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    ThetaArgs a;
    a.wbf16 = net->wbf16;
    a.mean = net->mean;
    a.std = net->std;
    a.lo = net->lo;
    a.hi = net->hi;
    a.feat = feat;
    a.count = count;
    a.n = n_groups;
    a.theta0 = rule->theta0;
    a.alpha = rule->alpha;
    a.beta = rule->beta;
    const int nblk = (int)((n_groups + kThetaBlock - 1) / kThetaBlock);
    float* wg = scratch;
    double* part = reinterpret_cast<double*>(scratch + ((n_groups + 1) & ~(int64_t)1));
    double* lambda = part + 2 * nblk;
    k_theta_weights<<<nblk, kThetaBlock, 0, s>>>(a, wg, part);
    CUDA_TRY(cudaGetLastError());
    k_theta_lambda<<<1, 256, 0, s>>>(part, nblk, (double)rule->target_rms * (double)rule->calib, lambda);
    CUDA_TRY(cudaGetLastError());
    // threads per group: as many as keep the launch within the threads that are
    // resident at once (about 500 per SM), where more would only wait
    int dev = 0, sms = 0;
    CUDA_TRY(cudaGetDevice(&dev));
    CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    const int64_t resident = (int64_t)sms * 500;
    if (8 * n_groups <= resident)
        k_theta_choose<8><<<(unsigned)((n_groups + kChooseBlock / 8 - 1) / (kChooseBlock / 8)), kChooseBlock, 0, s>>>(
            a, wg, lambda, grid, n_theta, rule->fallback, log10_target, theta_out);
    else if (2 * n_groups <= resident)
        k_theta_choose<2><<<(unsigned)((n_groups + kChooseBlock / 2 - 1) / (kChooseBlock / 2)), kChooseBlock, 0, s>>>(
            a, wg, lambda, grid, n_theta, rule->fallback, log10_target, theta_out);
    else
        k_theta_choose<1><<<(unsigned)((n_groups + kChooseBlock - 1) / kChooseBlock), kChooseBlock, 0, s>>>(
            a, wg, lambda, grid, n_theta, rule->fallback, log10_target, theta_out);
    CUDA_TRY(cudaGetLastError());
    return OTOO_OK;
}

int otoo_group_rms_error(const double* acc, const double* ref, const int64_t* group_off, int64_t n_groups,
                         float floor_value, float* log10_rms, uint32_t* status, void* stream)
{
    otoo::Range range_("otoo_group_rms_error");
    OTOO_REQUIRE(acc && ref && group_off && log10_rms && status, OTOO_EINVAL, "otoo_group_rms_error: NULL pointer");
    OTOO_REQUIRE(n_groups >= 0 && floor_value > 0.f, OTOO_EINVAL, "otoo_group_rms_error: bad argument");
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    CUDA_TRY(cudaMemsetAsync(status, 0, sizeof(uint32_t), s));
    if (n_groups == 0) return OTOO_OK;
    const int64_t threads = 32 * n_groups;
    k_group_rms<<<(unsigned)((threads + 127) / 128), 128, 0, s>>>(acc, ref, group_off, n_groups, floor_value,
                                                                  log10_rms, status);
    CUDA_TRY(cudaGetLastError());
    return OTOO_OK;
}

}  // extern "C"
