// The tree walk on the device and the device work plan.
//
// Paper: Section III-D (the walk runs on the GPU; a group of particles
// shares one traversal and the acceptance test uses the group-to-cell
// minimum distance, after Barnes 1990) and Section II-A (the traversal rules:
// accept a cell, open a cell into its children, take a leaf's particles).
// The paper walks with one work-item per group along next/more links; here
// one warp walks a set of neighbouring groups over a shared-memory stack, 64
// cells at a time, and writes each group's list for the force kernels (the host walk's lists,
// entry for entry, as sets per group).
//
// Kernels
//   k_walk_set<0>   pass 1: the groups' boxes (warp min/max over their particles),
//                   the walk, entry counts into the group records.
//   k_scan_*        exclusive prefix sums in group order (list offsets, plan
//                   slots): block sums, one-CTA scan of the block sums,
//                   block-level scans with the block offsets.
//   k_walk_set<1>   pass 2: the same walk, entries written at the offsets.
//   k_walk_set<2>   both in one pass, entries written into fixed slots.
//   k_plan_count    per group: particle and list chunks (the cost model of the
//                   host plan), cost class histogram, sums per block.
//   k_plan_scan     prefixes of the block sums; start of each cost class, most
//                   expensive class first.
//   k_plan_fill     work items and split records.
#include <cuda_runtime.h>

#include <cstdint>
#include <mutex>

#include "../common.h"
#include "../plan_chunks.h"

using namespace otoo;

namespace {

constexpr int kWalkWarps = 8;       // warps per CTA
#ifndef OTOO_WALK_HALVES
#define OTOO_WALK_HALVES 2
#endif
constexpr int kWalkHalves = OTOO_WALK_HALVES;  // cells per lane per walk step
#ifndef OTOO_WALK_MIN_BLOCKS
#define OTOO_WALK_MIN_BLOCKS 3  // resident CTAs per SM asked of the register allocator (85 registers)
#endif
constexpr int kWide = 32 * kWalkHalves;         // cells per walk step at most
constexpr int kStack = 512;         // stack entries (runs of sibling cells) per warp
constexpr int kMaxLevels = 22;      // tree levels (root level 0 to the 2^21 grid level)
constexpr int kScanThreads = 1024;  // scan kernels: threads per CTA
constexpr int kScanBlock = 2048;    // elements per scan block
constexpr int kClasses = 128;       // cost classes of the plan's launch order
constexpr int kTotals = 6;          // walk totals: entries, interactions, cell interactions,
                                    // largest n_cell, largest n_part, groups beyond their slots

#include "pair.cuh"

constexpr double kCubeAngle = 0.57;  // below 1/sqrt(3) = 0.5774 the test needs no cube overlap part

// status bits (counter[1])
constexpr uint32_t kWalkBadRecord = 1u;   // a cell record failed its bounds check
constexpr uint32_t kWalkOverflow = 2u;    // a group's stack or node budget ran out
constexpr uint32_t kWalkMismatch = 4u;    // pass 2 counted other entries than pass 1
constexpr uint32_t kWalkNoRoom = 8u;      // the output array is too small
constexpr uint32_t kWalkBadGroup = 16u;   // a group range failed its check

struct WalkArgs {
    int64_t n_part, n_cell;
    int32_t n_groups, exact, mac, pad;
    double theta, eps2;
    const otoo_src* src;
    const otoo_wcell* cell;
    const otoo_wcell64* cell64;
    const int32_t* gfirst;
    const int32_t* gcount;
    const float* tpg;
    uint32_t* counter;
    int64_t* totals;
};

// Per-group FP32 data of the filter: the group centre c as a float pair and
// the box relative to c.
struct BoxF {
    float c32[3], cl32[3], bl[3], bh[3];
    float B;    // sum over axes of max(|bl|, |bh|)
    float A;    // sum of |c32|: scale of the float-pair truncation error
};

// The acceptance test of the host walk, operation for operation in FP64
// (no contraction: every operation is an explicitly rounded intrinsic).
// Called for the few tests the FP32 filter cannot decide, so kept out of line
// (a smaller walk loop for the instruction cache).
__device__ __noinline__ bool mac_exact(const otoo_wcell64* __restrict__ c64, int k, const double blo[3],
                                       const double bhi[3], double theta)
{
    if (!(theta > 0.0)) return false;
    const otoo_wcell64 c = c64[k];
    bool overlap = true;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const double chi = __dadd_rn(c.lo[a], c.side);
        if (!(c.lo[a] <= bhi[a] && blo[a] <= chi)) overlap = false;
    }
    if (overlap) return false;
    double d2 = 0.0, s2 = 0.0;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        double d = 0.0;
        const double t0 = __dsub_rn(blo[a], c.com[a]);
        if (t0 > d) d = t0;
        const double t1 = __dsub_rn(c.com[a], bhi[a]);
        if (t1 > d) d = t1;
        d2 = __dadd_rn(d2, __dmul_rn(d, d));
        const double e = __dsub_rn(c.com[a], c.gc[a]);
        s2 = __dadd_rn(s2, __dmul_rn(e, e));
    }
    return __dsqrt_rn(d2) > __dadd_rn(__ddiv_rn(c.side, theta), __dsqrt_rn(s2));
}

// FP32 filter of the acceptance test: 1 = accept, 0 = reject, -1 = too close
// to call.  Without kOverlap (opening angles below 1/sqrt(3)) the cube
// overlap part is left out: a cube that overlaps the box puts its centre of
// mass within sqrt(3) l of the box, below l / theta + s, so the distance part
// alone already rejects it.  u = com - c from the float pairs; every rounded quantity is
// within 2^-20 K of its exact value (K: sum of the magnitudes the test
// combines, plus 2^-24 of the absolute coordinates for the truncated low
// words), so a comparison decided by more than 2^-18 K (box overlap) or
// 2^-16 K^2 (squared distances) is decided the same way by the exact
// arithmetic and by the host's FP64.
template <bool kOverlap>
__device__ __forceinline__ int mac_filter(const otoo_wcell& w, const BoxF& g, float invth)
{
    float u[3], au = 0.f, A = g.A;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        u[a] = __fadd_rn(__fsub_rn(w.com_hi[a], g.c32[a]), __fsub_rn(w.com_lo[a], g.cl32[a]));
        au += fabsf(u[a]);
        A += fabsf(w.com_hi[a]);
    }
    const float thr = __fadd_rn(__fmul_rn(w.side, invth), w.s);
    const float K = au + g.B + thr + w.side + A * 0x1p-24f;
    if (kOverlap) {
        const float del = K * 0x1p-18f;
        bool sep = false, ovl = true;
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const float lo = __fsub_rn(u[a], w.e[a]);
            const float hi = __fadd_rn(lo, w.side);
            sep = sep || (lo > g.bh[a] + del) || (g.bl[a] > hi + del);
            ovl = ovl && (lo < g.bh[a] - del) && (g.bl[a] < hi - del);
        }
        if (ovl) return 0;
        if (!sep) return -1;
    }
    float d2 = 0.f;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const float d = fmaxf(0.f, fmaxf(g.bl[a] - u[a], u[a] - g.bh[a]));
        d2 = fmaf(d, d, d2);
    }
    const float thr2 = thr * thr, m = K * K * 0x1p-16f;
    if (d2 > thr2 + m) return 1;
    if (d2 < thr2 - m) return 0;
    return -1;
}

// One 32-byte sector per load (256-bit vector loads, sm_100 and later): the
// 64-byte record in two requests instead of four.
__device__ __forceinline__ void ld256(const void* p, float v[8])
{
    asm("ld.global.nc.v8.f32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
        : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]), "=f"(v[6]), "=f"(v[7])
        : "l"(p));
}

// The absolute MAC of the host walk (Eq. SW_MAC): d_min > r_b, FP64,
// operation for operation (out of line, as mac_exact).
__device__ __noinline__ bool sw_exact(const otoo_wcell64* __restrict__ c64, int k, const double blo[3],
                                      const double bhi[3])
{
    const otoo_wcell64 c = c64[k];
    double d2 = 0.0;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        double d = 0.0;
        const double t0 = __dsub_rn(blo[a], c.com[a]);
        if (t0 > d) d = t0;
        const double t1 = __dsub_rn(c.com[a], bhi[a]);
        if (t1 > d) d = t1;
        d2 = __dadd_rn(d2, __dmul_rn(d, d));
    }
    return __dsqrt_rn(d2) > c.rb;
}

// FP32 filter of the absolute MAC with the same bound as mac_filter: the
// squared distance against r_b^2 decides when they differ by more than
// 2^-16 K^2 (K now includes r_b, rounded once from the host's FP64 value).
__device__ __forceinline__ int mac_filter_sw(const otoo_wcell& w, const BoxF& g)
{
    const float rb = w.rb;
    if (!(rb <= 3.0e38f)) return 0;  // infinite r_b (delta = 0): nothing is accepted
    float u[3], au = 0.f, A = g.A;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        u[a] = __fadd_rn(__fsub_rn(w.com_hi[a], g.c32[a]), __fsub_rn(w.com_lo[a], g.cl32[a]));
        au += fabsf(u[a]);
        A += fabsf(w.com_hi[a]);
    }
    const float K = au + g.B + rb + A * 0x1p-24f;
    float d2 = 0.f;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const float d = fmaxf(0.f, fmaxf(g.bl[a] - u[a], u[a] - g.bh[a]));
        d2 = fmaf(d, d, d2);
    }
    const float rb2 = rb * rb, m = K * K * 0x1p-16f;
    if (d2 > rb2 + m) return 1;
    if (d2 < rb2 - m) return 0;
    return -1;
}

__device__ __forceinline__ otoo_wcell load_wcell(const otoo_wcell* __restrict__ cell, int k)
{
    float v[16];
    ld256(cell + k, v);
    ld256(reinterpret_cast<const char*>(cell + k) + 32, v + 8);
    otoo_wcell w;
    w.com_hi[0] = v[0], w.com_hi[1] = v[1], w.com_hi[2] = v[2];
    w.com_lo[0] = v[3], w.com_lo[1] = v[4], w.com_lo[2] = v[5];
    w.e[0] = v[6], w.e[1] = v[7], w.e[2] = v[8];
    w.side = v[9];
    w.s = v[10];
    w.child0 = __float_as_int(v[11]);
    w.nchild = __float_as_int(v[12]);
    w.begin = __float_as_int(v[13]);
    w.end = __float_as_int(v[14]);
    w.rb = v[15];
    return w;
}

__device__ __forceinline__ int warp_incl_scan(int v, int lane)
{
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(kFull, v, o);
        if (lane >= o) v += t;
    }
    return v;
}

// Order-preserving integer key of a double (for non-NaN values): min/max on
// the keys is min/max on the values, on the integer pipe.
__device__ __forceinline__ long long dkey(double x)
{
    const long long b = __double_as_longlong(x);
    return b ^ ((b >> 63) & 0x7fffffffffffffffLL);
}
__device__ __forceinline__ double dval(long long k) { return __longlong_as_double(k ^ ((k >> 63) & 0x7fffffffffffffffLL)); }

// Of signed 64-bit keys: the high words, then the low words of the lanes that
// hold that high word (two reductions instead of five rounds of shuffles).
__device__ __forceinline__ long long warp_min(long long v)
{
    const int h = (int)(v >> 32), m = __reduce_min_sync(kFull, h);
    const unsigned l = __reduce_min_sync(kFull, h == m ? (unsigned)v : 0xffffffffu);
    return ((long long)m << 32) | l;
}
__device__ __forceinline__ long long warp_max(long long v)
{
    const int h = (int)(v >> 32), m = __reduce_max_sync(kFull, h);
    const unsigned l = __reduce_max_sync(kFull, h == m ? (unsigned)v : 0u);
    return ((long long)m << 32) | l;
}

// A stack entry is a run of consecutive cells (the children of one cell):
// first cell in the low 28 bits, run length - 1 (0..7) above.
constexpr uint32_t kRunShift = 28;
constexpr uint32_t kRunMask = (1u << kRunShift) - 1u;
__device__ __forceinline__ uint32_t run(int first, int n) { return (uint32_t)first | ((uint32_t)(n - 1) << kRunShift); }

// Geometry and acceptance rule of one group's walk.
struct GroupWalk {
    double blo[3], bhi[3], c[3];  // the particles' box (exact) and its centre
    BoxF bf;
    double theta;                 // opening angle of this group (0 for the absolute MAC / SPH)
    float invth;                  // 1 / theta rounded to FP32
    bool sw;                      // absolute MAC or SPH radius: accept when d_min > r_b
    bool drop;                    // SPH: accepted cells enter no list
    bool open_all;                // opening angle 0: nothing is accepted
    bool small_angle;             // theta < 1/sqrt(3): the filter skips the cube-overlap part
};

// The box of particles [first, first + count) (min/max on order-preserving
// integer keys, exact).
__device__ __forceinline__ void group_box(const WalkArgs& a, int32_t first, int32_t count, int lane, double lo[3],
                                          double hi[3])
{
    long long klo[3], khi[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) klo[k] = 0x7fffffffffffffffLL, khi[k] = -klo[k] - 1;
    for (int i = lane; i < count; i += 32) {
        const double2* ps = reinterpret_cast<const double2*>(a.src + first + i);
        const double2 xy = __ldg(ps), zm = __ldg(ps + 1);
        const long long kx = dkey(xy.x), ky = dkey(xy.y), kz = dkey(zm.x);
        klo[0] = kx < klo[0] ? kx : klo[0], khi[0] = kx > khi[0] ? kx : khi[0];
        klo[1] = ky < klo[1] ? ky : klo[1], khi[1] = ky > khi[1] ? ky : khi[1];
        klo[2] = kz < klo[2] ? kz : klo[2], khi[2] = kz > khi[2] ? kz : khi[2];
    }
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        lo[k] = dval(warp_min(klo[k]));
        hi[k] = dval(warp_max(khi[k]));
    }
}

// A group's box, its FP32 form for the filter, and the group's rule.
__device__ __forceinline__ void group_walk_setup(const WalkArgs& a, int g, int32_t first, int32_t count, int lane,
                                                 GroupWalk& w)
{
    group_box(a, first, count, lane, w.blo, w.bhi);
    w.bf.B = 0.f;
    w.bf.A = 0.f;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        w.c[k] = __dmul_rn(__dadd_rn(w.blo[k], w.bhi[k]), 0.5);
        w.bf.c32[k] = __double2float_rn(w.c[k]);
        w.bf.cl32[k] = __double2float_rn(__dsub_rn(w.c[k], (double)w.bf.c32[k]));
        w.bf.bl[k] = __double2float_rn(__dsub_rn(w.blo[k], w.c[k]));
        w.bf.bh[k] = __double2float_rn(__dsub_rn(w.bhi[k], w.c[k]));
        w.bf.B += fmaxf(fabsf(w.bf.bl[k]), fabsf(w.bf.bh[k]));
        w.bf.A += fabsf(w.bf.c32[k]);
    }
    // the absolute MAC and the SPH radius share the test d_min > r_b; an
    // SPH walk drops the cells that pass it (no neighbour inside)
    w.sw = a.mac == OTOO_MAC_SW || a.mac == OTOO_MAC_SPH;
    w.drop = a.mac == OTOO_MAC_SPH;
    w.theta = w.sw ? 0.0 : a.tpg ? (double)a.tpg[g] : a.theta;
    // the per-group choices as bits of an integer, taken through an opaque
    // move: the compiler must not re-derive them from theta inside the
    // walk loop, where FP64 compares would occupy GB300's narrow FP64 pipe
    int fl = (!w.sw && !(w.theta > 0.0) ? 1 : 0) | (w.theta < kCubeAngle ? 2 : 0);
    asm volatile("mov.b32 %0, %0;" : "+r"(fl));
    w.open_all = (fl & 1) != 0;
    w.small_angle = (fl & 2) != 0;
    // 1/theta within 2^-23 (the filter's margins allow 2^-21)
    w.invth = w.open_all ? 0.f : __frcp_rn(__double2float_rn(w.theta));
}

// The cells one walk step took and their decisions: lane j holds positions
// j + 32 h of the taken runs; kind 1 accept, 2 rejected leaf, 3 open, 0 none.
struct StepCells {
    int node[kWalkHalves], kind[kWalkHalves], c0[kWalkHalves], nch[kWalkHalves], pb[kWalkHalves],
        pe[kWalkHalves];
};

// Takes up to kWide cells from the top runs of the stack (the last run may be
// split, its rest goes back) and tests them.  False when the stack or the
// cell budget ran out (the walk stops).
__device__ __forceinline__ bool walk_take(const WalkArgs& a, const GroupWalk& w, uint32_t* stk, int& sp,
                                          int64_t& budget, int lane, StepCells& sc, uint32_t* status)
{
    if (sp + 2 > kStack) return false;
    const int wcap = sp + kWide + 1 + kMaxLevels <= kStack ? kWide : 1;
    // the top runs: lane l reads the l-th entry from the top
    const int nr = sp < 32 ? sp : 32;
    uint32_t e = 0;
    int rn = 0;
    if (lane < nr) {
        e = stk[sp - 1 - lane];
        rn = (int)(e >> kRunShift) + 1;
    }
    const int rinc = warp_incl_scan(rn, lane);
    const int rstart = rinc - rn;
    // runs wholly taken, and a run cut at wcap
    const bool whole = lane < nr && rinc <= wcap;
    const bool cut = lane < nr && rstart < wcap && rinc > wcap;
    const int nwhole = __popc(__ballot_sync(kFull, whole));
    const unsigned cutm = __ballot_sync(kFull, cut);
    const int in_whole = __shfl_sync(kFull, rinc, nwhole > 0 ? nwhole - 1 : 0);
    const int W = cutm ? wcap : (nwhole > 0 ? in_whole : 0);
    // start positions of the taken runs, 32 positions per mask word
    unsigned starts[kWalkHalves];
#pragma unroll
    for (int h = 0; h < kWalkHalves; ++h)
        starts[h] = __reduce_or_sync(kFull, (whole || cut) && rstart >= 32 * h && rstart < 32 * h + 32
                                                ? (1u << (rstart - 32 * h))
                                                : 0u);
    // the run that continues after the cut goes back on the stack first
    sp -= nwhole + (cutm ? 1 : 0);
    if (cut) {
        const int taken = wcap - rstart;
        stk[sp] = run((int)(e & kRunMask) + taken, rn - taken);
    }
    sp += cutm ? 1 : 0;
    budget -= W;
    if (budget < 0) return false;
    // lane j takes the cells at positions j, j + 32, ... of the taken
    // runs; position q lies in the run whose start is the last one <= q
#pragma unroll
    for (int h = 0; h < kWalkHalves; ++h) {
        int r = -1;
#pragma unroll
        for (int k = 0; k <= h; ++k) r += __popc(starts[k] & (k < h ? 0xffffffffu : (2u << lane) - 1u));
        const uint32_t er = __shfl_sync(kFull, e, r < 0 ? 0 : r);
        const int sr = __shfl_sync(kFull, rstart, r < 0 ? 0 : r);
        const int q = lane + 32 * h;
        sc.node[h] = q < W ? (int)(er & kRunMask) + (q - sr) : -1;
        sc.kind[h] = 0;
        sc.c0[h] = sc.nch[h] = sc.pb[h] = sc.pe[h] = 0;
    }
    __syncwarp();
#pragma unroll
    for (int h = 0; h < kWalkHalves; ++h) {
        if (lane + 32 * h >= W) continue;
        const int nd = sc.node[h];
        bool ok = nd >= 0 && nd < a.n_cell;
        if (ok) {
            const otoo_wcell c = load_wcell(a.cell, nd);
            sc.nch[h] = c.nchild;
            sc.c0[h] = c.child0;
            sc.pb[h] = c.begin;
            sc.pe[h] = c.end;
            ok = sc.nch[h] >= 0 && sc.nch[h] <= 8 &&
                 (sc.nch[h] == 0 || (sc.c0[h] > nd && (int64_t)sc.c0[h] + sc.nch[h] <= a.n_cell)) &&
                 sc.pb[h] >= 0 && sc.pb[h] <= sc.pe[h] && (int64_t)sc.pe[h] <= a.n_part;
            if (ok) {
                int dec = 0;
                if (w.sw) {
                    dec = a.exact ? -1 : mac_filter_sw(c, w.bf);
                    if (dec < 0) dec = sw_exact(a.cell64, nd, w.blo, w.bhi) ? 1 : 0;
                } else if (!w.open_all) {
                    dec = a.exact ? -1
                          : w.small_angle ? mac_filter<false>(c, w.bf, w.invth)
                                          : mac_filter<true>(c, w.bf, w.invth);
                    if (dec < 0) dec = mac_exact(a.cell64, nd, w.blo, w.bhi, w.theta) ? 1 : 0;
                }
                sc.kind[h] = dec ? 1 : (sc.nch[h] == 0 ? 2 : 3);
            }
        }
        if (!ok) atomicOr(status, kWalkBadRecord);
    }
    return true;
}

// One run per rejected inner cell of the step, the lowest position's on top:
// the last positions are pushed first.
__device__ __forceinline__ void walk_push(uint32_t* stk, int& sp, const StepCells& sc, unsigned lt)
{
#pragma unroll
    for (int h = kWalkHalves - 1; h >= 0; --h) {
        const unsigned om = __ballot_sync(kFull, sc.kind[h] == 3);
        const int no = __popc(om);
        if (sc.kind[h] == 3) stk[sp + no - 1 - __popc(om & lt)] = run(sc.c0[h], sc.nch[h]);
        sp += no;
    }
    __syncwarp();
}

// ---- the walk over lists -------------------------------------------------------
//
// Groups that are neighbours in tree order lie close together, and their walks
// test mostly the same cells: for the sets of groups under one parent cell of
// a Hernquist halo (7.6 groups per set at n_crit 128) the per-group walks
// visit 5.9 times as many cells as one walk over the union of their visited
// cells.  k_walk_set walks up to kSet consecutive groups with one warp: every
// stack run carries the mask of the set's groups for which the run's cells
// are still open (all their ancestors rejected), a taken cell's record is
// loaded once and tested against each group of its mask, and each group keeps
// its own counts and list slots.  A cell a group accepts is emitted for that
// group, a rejected leaf's particles go to every group that rejected it, and
// an inner cell rejected by any group is opened with the mask of the groups
// that rejected it.  Restricted to one group, the walk visits exactly the
// cells the group's own walk visits and takes the same decisions (those of the
// FP64 test), so each group's entries are the same set whatever the sets are;
// their order is the union walk's.
//
// The stack holds runs of sibling cells; each step takes up to kWide = 32
// kWalkHalves cells from the top runs (set_take; lane j tests the cells at
// positions j, j + 32, ...) and pushes one run per rejected inner cell
// (set_push).  A kWide-cell step adds at most kWide entries and runs only with
// kWide + 1 + kMaxLevels entries free; otherwise the step takes one cell,
// which adds at most one entry, and only when it descends a level (a tree has
// at most kMaxLevels levels below any cell), so the stack never overflows.
//
// Bound by instruction issue.  Everything of the test that the cell alone
// decides (its centre of mass relative to the set's common centre, the squared
// distances beyond which it is accepted and below which it is rejected) is
// computed once per cell, with the rounding margin of the set's largest
// group, and the groups are taken in a loop that the whole warp runs in step:
// a test is 12 operations and two comparisons, its accepted cells are written
// in the same turn.  Before, every lane went through its own cell's groups with
// their own margins (5.8 tests of 18 lanes a step where four of 27 do, N = 2^20
// taken two groups at a time; 977 instructions a step in all) and a second
// loop wrote the entries.  Plummer N = 2^20, n_crit 128: 1.24 -> 0.81 ms (980
// -> 642 million instructions) in sets of two, 0.68 ms in the sets taken now;
// Hernquist N = 2^23 6.37 -> 3.81 ms; absolute MAC, N = 2^23 1.90 -> 1.42 ms.

constexpr int kSet = 8;  // groups per set at most (one bit each in a run's mask)

// One group of a set: its box relative to the set's centre, its rule, and where
// its entries go.
struct SetGroup {
    float bl[3], bh[3];
    float invth;           // 1 / theta rounded to FP32
    int32_t flags;         // 1: opening angle 0 (nothing accepted), 2: theta < 1/sqrt(3)
    double blo[3], bhi[3]; // the particles' box
    double theta;          // opening angle (0 for the absolute MAC / SPH)
    int64_t off_c, off_p;  // where cell r and particle k go (cells backwards in the single pass)
    int32_t want_c, want_p;
};

// What the set's groups have in common.
struct SetRule {
    float4 c;   // centre of the set rounded to FP32; 1 / theta (if it is one for all)
    float4 cl;  // the centre's low words; sum over axes of |c| 2^-24 + the largest group's sum of max(|bl|, |bh|)
};

// One cell of a step in the filter: the centre of mass relative to the set's
// centre, the distance test's two limits, and what the cube test needs.
struct SetCell {
    float u[3], tu, tl;
    float e[3], side, s, K, del;
};

// The limits for threshold thr (a length): the squared distance decides when it
// differs from thr^2 by more than 2^-16 K^2.  Every rounded quantity is within
// 2^-20 K of its exact value (K: sum of the magnitudes the test combines, plus
// 2^-24 of the absolute coordinates for the truncated low words), so what the
// limits decide the exact arithmetic and the host's FP64 decide the same way.
__device__ __forceinline__ void set_limits(SetCell& c, float thr)
{
    const float K = c.K + thr, thr2 = thr * thr, m = K * K * 0x1p-16f;
    c.tu = thr2 + m;
    c.tl = thr2 - m;
    c.del = K * 0x1p-18f;
}

__device__ __forceinline__ SetCell set_cell(const otoo_wcell& w, const SetRule& r, bool sw, bool none, bool exact)
{
    SetCell c;
    const float4 h = r.c, l = r.cl;
    c.u[0] = __fadd_rn(__fsub_rn(w.com_hi[0], h.x), __fsub_rn(w.com_lo[0], l.x));
    c.u[1] = __fadd_rn(__fsub_rn(w.com_hi[1], h.y), __fsub_rn(w.com_lo[1], l.y));
    c.u[2] = __fadd_rn(__fsub_rn(w.com_hi[2], h.z), __fsub_rn(w.com_lo[2], l.z));
    float au = 0.f, ac = 0.f;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        au += fabsf(c.u[a]);
        ac += fabsf(w.com_hi[a]);
        c.e[a] = w.e[a];
    }
    c.side = w.side;
    c.s = w.s;
    c.K = au + l.w + ac * 0x1p-24f + (sw ? 0.f : w.side);
    set_limits(c, sw ? w.rb : __fadd_rn(__fmul_rn(w.side, h.w), w.s));
    if (exact) c.tu = __int_as_float(0x7f800000), c.tl = -c.tu;
    // angle 0, or an infinite r_b (delta = 0): nothing is accepted
    if (none || (sw && !(w.rb <= 3.0e38f))) c.tu = c.tl = __int_as_float(0x7f800000);
    return c;
}

// Takes up to kWide cells from the top runs of the stack (the last run may be
// split, its rest goes back): the cell at position lane + 32 h and the mask of
// its groups (0: no cell there).  False when the stack or the cell budget ran
// out (the walk stops).
__device__ __forceinline__ bool set_take(uint32_t* stk, uint8_t* msk, int& sp, int& budget, int lane,
                                         int node[kWalkHalves], unsigned cm[kWalkHalves])
{
    if (sp + 2 > kStack) return false;
    const int wcap = sp + kWide + 1 + kMaxLevels <= kStack ? kWide : 1;
    // the top runs: lane l reads the l-th entry from the top
    const int nr = sp < 32 ? sp : 32;
    uint32_t e = 0;
    unsigned em = 0;
    int rn = 0;
    if (lane < nr) {
        e = stk[sp - 1 - lane];
        em = msk[sp - 1 - lane];
        rn = (int)(e >> kRunShift) + 1;
    }
    const int rinc = warp_incl_scan(rn, lane);
    const int rstart = rinc - rn;
    // runs wholly taken, and a run cut at wcap
    const bool whole = lane < nr && rinc <= wcap;
    const bool cut = lane < nr && rstart < wcap && rinc > wcap;
    const int nwhole = __popc(__ballot_sync(kFull, whole));
    const unsigned cutm = __ballot_sync(kFull, cut);
    const int in_whole = __shfl_sync(kFull, rinc, nwhole > 0 ? nwhole - 1 : 0);
    const int W = cutm ? wcap : (nwhole > 0 ? in_whole : 0);
    // start positions of the taken runs, 32 positions per mask word
    unsigned starts[kWalkHalves];
#pragma unroll
    for (int h = 0; h < kWalkHalves; ++h)
        starts[h] = __reduce_or_sync(kFull, (whole || cut) && rstart >= 32 * h && rstart < 32 * h + 32
                                                ? (1u << (rstart - 32 * h))
                                                : 0u);
    // the run that continues after the cut goes back on the stack first
    sp -= nwhole + (cutm ? 1 : 0);
    if (cut) {
        const int taken = wcap - rstart;
        stk[sp] = run((int)(e & kRunMask) + taken, rn - taken);
        msk[sp] = (uint8_t)em;
    }
    sp += cutm ? 1 : 0;
    budget -= W;
    if (budget < 0) return false;
    // position q lies in the run whose start is the last one <= q
#pragma unroll
    for (int h = 0; h < kWalkHalves; ++h) {
        int r = -1;
#pragma unroll
        for (int k = 0; k <= h; ++k) r += __popc(starts[k] & (k < h ? 0xffffffffu : (2u << lane) - 1u));
        r = r < 0 ? 0 : r;
        const uint32_t er = __shfl_sync(kFull, e, r);
        const int sr = __shfl_sync(kFull, rstart, r);
        const unsigned mr = __shfl_sync(kFull, em, r);
        const int q = lane + 32 * h;
        node[h] = (int)(er & kRunMask) + (q - sr);
        cm[h] = q < W ? mr : 0u;
    }
    __syncwarp();
    return true;
}

// Rejected leaves of a walk with the masks of the groups that rejected them, in
// the order their particles are listed: a ring per warp.  A step finds one to
// six of them among its 64 cells; their particles are counted, scanned and
// written for 32 leaves at once (set_flush).  A step adds at most kWide with
// fewer than 32 held, so the ring is never full.
constexpr int kLeafRing = 128;
static_assert(kLeafRing >= kWide + 32 && (kLeafRing & (kLeafRing - 1)) == 0, "leaf ring");
struct LeafRing {
    int2 range[kLeafRing];  // first particle, one past the last
    uint8_t mask[kLeafRing];
};

// Lists the particles of the ring's n <= 32 oldest leaves for the groups that
// rejected them (lane j holds group j's count).
template <bool kWrite>
__device__ __forceinline__ void set_flush(const LeafRing& q, int head, int n, int lane, const SetGroup* sg,
                                          int32_t* __restrict__ list, int& my_np)
{
    __syncwarp();
    int2 r = make_int2(0, 0);
    unsigned m = 0u;
    if (lane < n) {
        r = q.range[(head + lane) & (kLeafRing - 1)];
        m = q.mask[(head + lane) & (kLeafRing - 1)];
    }
    // (not unrolled: the walk loop must stay small for the instruction cache)
#pragma unroll 1
    for (unsigned gm = __reduce_or_sync(kFull, m); gm; gm &= gm - 1u) {
        const int j = __ffs(gm) - 1;
        const int np = (m >> j) & 1u ? r.y - r.x : 0;
        const int pin = warp_incl_scan(np, lane);
        const int had = __shfl_sync(kFull, my_np, j);
        if (kWrite) {
            const int32_t base = had + pin - np;
            const int c = min(np, sg[j].want_p - base);
            int32_t* o = list + sg[j].off_p + base;
            for (int k = 0; k < c; ++k) o[k] = r.x + k;
        }
        const int sum = __shfl_sync(kFull, pin, 31);
        if (lane == j) my_np = had + sum;
    }
}

// One warp per set of gs <= kSet consecutive groups (atomic ticket over sets).
// kMode 0: count (group records, totals); 1: fill the list at the offsets
// of pass 0; 2: single pass -- count as pass 0 and write each group's entries
// into its fixed slot of list (capacity cells + pcap particles per slot):
// cells backwards from slot position capacity - 1, particles forwards from
// capacity, so that they end up contiguous, cells first, and the slots serve
// as the list (list_off set here; groups that outgrow their slot get -1).
// kGen: opening angles per group, or 1/sqrt(3) and more (plain_rule says which
// form a walk needs); without it the loop over the groups holds five values of
// a cell instead of twelve.
template <int kMode, bool kGen>
__global__ void __launch_bounds__(kWalkWarps * 32, OTOO_WALK_MIN_BLOCKS)
    k_walk_set(WalkArgs a, int32_t n_sets, int32_t gs, otoo_group* __restrict__ groups, int32_t* __restrict__ list,
               int64_t capacity, int64_t pcap)
{
    constexpr bool kFill = kMode == 1;
    constexpr bool kCount = kMode != 1;
    constexpr bool kWrite = kMode != 0;
    __shared__ uint32_t stack_s[kWalkWarps][kStack];
    __shared__ uint8_t mask_s[kWalkWarps][kStack];
    __shared__ SetGroup sg_s[kWalkWarps][kSet];
    __shared__ LeafRing ring_s[kWalkWarps];
    const int lane = threadIdx.x & 31;
    const int wid = threadIdx.x >> 5;
    uint32_t* stk = stack_s[wid];
    uint8_t* msk = mask_s[wid];
    SetGroup* sg = sg_s[wid];
    LeafRing& ring = ring_s[wid];
    const unsigned lt = (1u << lane) - 1u;
    uint32_t* status = a.counter + 1;
    // the absolute MAC and the SPH radius share the test d_min > r_b; an
    // SPH walk drops the cells that pass it (no neighbour inside)
    const bool sw = a.mac == OTOO_MAC_SW || a.mac == OTOO_MAC_SPH;
    const bool drop = a.mac == OTOO_MAC_SPH;
    if (kFill && a.totals[0] > capacity) {
        if (threadIdx.x == 0) atomicOr(status, kWalkNoRoom);
        return;
    }
    for (;;) {
        int set = 0;
        if (lane == 0) set = (int)atomicAdd(a.counter, 1u);
        set = __shfl_sync(kFull, set, 0);
        if (set >= n_sets) break;
        const int g0 = set * gs;
        const int ng = min(gs, a.n_groups - g0);
        unsigned valid = 0u;  // groups with a record to write (pass 0 / single pass) or check (pass 1)
        for (int j = 0; j < ng; ++j) {
            const int g = g0 + j;
            const int32_t first = a.gfirst[g], count = a.gcount[g];
            if (first < 0 || count < 1 || count > kMaxGroup || (int64_t)first + count > a.n_part) {
                if (lane == 0) {
                    atomicOr(status, kWalkBadGroup);
                    if (kCount) {
                        otoo_group z = {};
                        z.first = first;
                        z.eps2 = a.eps2;
                        z.theta = -1.f;
                        groups[g] = z;
                    }
                }
                continue;
            }
            double lo[3], hi[3];
            group_box(a, first, count, lane, lo, hi);
            if (lane == 0)
#pragma unroll
                for (int k = 0; k < 3; ++k) sg[j].blo[k] = lo[k], sg[j].bhi[k] = hi[k];
            valid |= 1u << j;
        }
        // lane j: group j's rule and offsets
        bool mine = lane < ng && ((valid >> lane) & 1u);
        bool walks = false;
        float my_inv = 0.f;
        int my_fl = 0;
        if (mine) {
            SetGroup& q = sg[lane];
            const double theta = sw ? 0.0 : a.tpg ? (double)a.tpg[g0 + lane] : a.theta;
            int64_t off_c = 0, off_p = 0;
            int32_t want_c = 0, want_p = 0;
            if (kMode == 2) {
                // cell r at off_c - r, particle k at off_p + k
                off_p = (int64_t)(g0 + lane) * (capacity + pcap) + capacity;
                off_c = off_p - 1;
                want_c = (int32_t)capacity;
                want_p = (int32_t)pcap;
            }
            if (kFill) {
                const otoo_group gr = groups[g0 + lane];
                off_c = gr.list_off;
                want_c = gr.n_cell;
                want_p = gr.n_part;
                off_p = off_c + want_c;
                if (off_c < 0 || want_c < 0 || want_p < 0 || off_p + want_p > capacity) {
                    atomicOr(status, kWalkNoRoom);
                    mine = false;
                }
            }
            my_fl = (!sw && !(theta > 0.0) ? 1 : 0) | (theta < kCubeAngle ? 2 : 0);
            // 1/theta within 2^-23 (the filter's margins allow 2^-21)
            my_inv = sw || (my_fl & 1) ? 0.f : __frcp_rn(__double2float_rn(theta));
            q.theta = theta;
            q.invth = my_inv;
            q.flags = my_fl;
            q.off_c = off_c;
            q.off_p = off_p;
            q.want_c = want_c;
            q.want_p = want_p;
            walks = mine && theta >= 0.0;
        }
        const unsigned live = __ballot_sync(kFull, walks);  // groups that walk
        __syncwarp();
        // the set's centre: that of the box of its walking groups
        SetRule rule = {};
        bool uni = true, none = false, overlap = false;  // one angle; nothing accepted; the test needs the cubes
        if (live) {
            double lo[3], hi[3];
            const int j0 = __ffs(live) - 1;
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                lo[k] = dval(warp_min(dkey(sg[walks ? lane : j0].blo[k])));
                hi[k] = dval(warp_max(dkey(sg[walks ? lane : j0].bhi[k])));
            }
            float B = 0.f, A = 0.f, ch[3], cl[3];
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                const double c = __dmul_rn(__dadd_rn(lo[k], hi[k]), 0.5);
                ch[k] = __double2float_rn(c);
                cl[k] = __double2float_rn(__dsub_rn(c, (double)ch[k]));
                A += fabsf(ch[k]);
                if (walks) {
                    SetGroup& q = sg[lane];
                    q.bl[k] = __double2float_rn(__dsub_rn(q.blo[k], c));
                    q.bh[k] = __double2float_rn(__dsub_rn(q.bhi[k], c));
                    B += fmaxf(fabsf(q.bl[k]), fabsf(q.bh[k]));
                }
            }
            // (B >= 0: its bits are ordered as the value)
            B = __uint_as_float(__reduce_max_sync(kFull, __float_as_uint(B)));
            const float inv0 = __shfl_sync(kFull, my_inv, j0);
            const int fl0 = __shfl_sync(kFull, my_fl, j0);
            uni = __all_sync(kFull, !walks || (my_inv == inv0 && my_fl == fl0));
            none = (fl0 & 1) != 0;
            overlap = !sw && __any_sync(kFull, walks && !(my_fl & 2));
            rule.c = make_float4(ch[0], ch[1], ch[2], inv0);
            rule.cl = make_float4(cl[0], cl[1], cl[2], B + A * 0x1p-24f);
            __syncwarp();
        }
        int my_nc = 0, my_np = 0;  // lane j: counts of group j
        int sp = 0;
        if (live) {
            if (lane == 0) {
                stk[0] = run(0, 1);
                msk[0] = (uint8_t)live;
            }
            sp = 1;
        }
        __syncwarp();
        int budget = (int)a.n_cell;  // the union of the walks visits each cell at most once
        bool failed = false;
        int head = 0, held = 0;  // the ring's leaves
        while (sp > 0) {
            // at, num: an inner cell's first child and -(number of children), a leaf's
            // first particle and one past its last
            int node[kWalkHalves], at[kWalkHalves], num[kWalkHalves];
            unsigned cm[kWalkHalves], acc[kWalkHalves];
            SetCell sc[kWalkHalves];
            if (!set_take(stk, msk, sp, budget, lane, node, cm)) {
                failed = true;
                break;
            }
#pragma unroll
            for (int h = 0; h < kWalkHalves; ++h) {
                const int nd = node[h];
                otoo_wcell c = {};
                bool ok = nd >= 0 && nd < a.n_cell;
                if (cm[h] && ok) c = load_wcell(a.cell, nd);
                ok = ok && c.nchild >= 0 && c.nchild <= 8 &&
                     (c.nchild == 0 || (c.child0 > nd && (int64_t)c.child0 + c.nchild <= a.n_cell)) && c.begin >= 0 &&
                     c.begin <= c.end && (int64_t)c.end <= a.n_part;
                at[h] = c.nchild ? c.child0 : c.begin;
                num[h] = c.nchild ? -c.nchild : c.end;
                if (cm[h] && !ok) {
                    atomicOr(status, kWalkBadRecord);
                    cm[h] = 0u;
                }
                acc[h] = 0u;
                sc[h] = set_cell(c, rule, sw, none, a.exact != 0);
            }
            // group by group: the decisions, and its accepted cells in position order
            // (not unrolled: the walk loop must stay small for the instruction cache)
            unsigned any = 0u;
#pragma unroll
            for (int h = 0; h < kWalkHalves; ++h) any |= cm[h];
#pragma unroll 1
            for (unsigned gm = __reduce_or_sync(kFull, any); gm; gm &= gm - 1u) {
                const int j = __ffs(gm) - 1;
                const SetGroup& q = sg[j];
                float bl[3], bh[3];
#pragma unroll
                for (int k = 0; k < 3; ++k) bl[k] = q.bl[k], bh[k] = q.bh[k];
                if (kGen && !uni) {
#pragma unroll
                    for (int h = 0; h < kWalkHalves; ++h) {
                        set_limits(sc[h], __fadd_rn(__fmul_rn(sc[h].side, q.invth), sc[h].s));
                        if (a.exact) sc[h].tu = __int_as_float(0x7f800000), sc[h].tl = -sc[h].tu;
                        if (q.flags & 1) sc[h].tu = sc[h].tl = __int_as_float(0x7f800000);
                    }
                }
                bool in[kWalkHalves], tc[kWalkHalves];
#pragma unroll
                for (int h = 0; h < kWalkHalves; ++h) {
                    const SetCell& c = sc[h];
                    float d2 = 0.f;
#pragma unroll
                    for (int k = 0; k < 3; ++k) {
                        const float d = fmaxf(0.f, fmaxf(bl[k] - c.u[k], c.u[k] - bh[k]));
                        d2 = fmaf(d, d, d2);
                    }
                    in[h] = d2 > c.tu;
                    tc[h] = !in[h] && !(d2 < c.tl);
                }
                // Opening angles of 1/sqrt(3) and more: a cell whose cube
                // overlaps the box is rejected.  (Below, a cube that overlaps
                // the box puts its centre of mass within sqrt(3) l of the box,
                // below l / theta + s, so the distance alone rejects it.)
                if (kGen && overlap) {
#pragma unroll
                    for (int h = 0; h < kWalkHalves; ++h) {
                        const SetCell& c = sc[h];
                        bool sep = false, ovl = true;
#pragma unroll
                        for (int k = 0; k < 3; ++k) {
                            const float lo = __fsub_rn(c.u[k], c.e[k]);
                            const float hi = __fadd_rn(lo, c.side);
                            sep = sep || (lo > bh[k] + c.del) || (bl[k] > hi + c.del);
                            ovl = ovl && (lo < bh[k] - c.del) && (bl[k] < hi - c.del);
                        }
                        tc[h] = a.exact ? tc[h] : !ovl && (!sep || tc[h]);
                        in[h] = in[h] && sep;
                    }
                }
#pragma unroll
                for (int h = 0; h < kWalkHalves; ++h) {
                    const bool m = (cm[h] >> j) & 1u;
                    if (m && tc[h])  // too close to call
                        in[h] = sw ? sw_exact(a.cell64, node[h], q.blo, q.bhi)
                                        : mac_exact(a.cell64, node[h], q.blo, q.bhi, q.theta);
                    in[h] = in[h] && m;
                    acc[h] |= in[h] ? 1u << j : 0u;
                }
                if (drop) continue;
                int n = __shfl_sync(kFull, my_nc, j);
                int32_t* o = nullptr;
                if (kWrite) o = list + q.off_c;
#pragma unroll
                for (int h = 0; h < kWalkHalves; ++h) {
                    const unsigned am = __ballot_sync(kFull, in[h]);
                    if (kWrite) {
                        const int32_t r = n + __popc(am & lt);
                        if (in[h] && r < q.want_c) o[kMode == 2 ? -r : r] = (int32_t)(a.n_part + node[h]);
                    }
                    n += __popc(am);
                }
                if (lane == j) my_nc = n;
            }
            // rejected leaves, in position order; one run per inner cell some
            // group rejected, with the mask of the groups that rejected it, the
            // lowest position's run on top (the last positions are pushed first)
#pragma unroll
            for (int h = 0; h < kWalkHalves; ++h) {
                cm[h] &= ~acc[h];
                const bool leaf = num[h] >= 0 && cm[h] != 0u;
                const unsigned lm = __ballot_sync(kFull, leaf);
                if (leaf) {
                    const int i = (head + held + __popc(lm & lt)) & (kLeafRing - 1);
                    ring.range[i] = make_int2(at[h], num[h]);
                    ring.mask[i] = (uint8_t)cm[h];
                }
                held += __popc(lm);
            }
#pragma unroll
            for (int h = kWalkHalves - 1; h >= 0; --h) {
                const bool op = num[h] < 0 && cm[h] != 0u;
                const unsigned om = __ballot_sync(kFull, op);
                const int no = __popc(om);
                if (op) {
                    const int i = sp + no - 1 - __popc(om & lt);
                    stk[i] = run(at[h], -num[h]);
                    msk[i] = (uint8_t)cm[h];
                }
                sp += no;
            }
            for (; held >= 32; held -= 32, head += 32) set_flush<kWrite>(ring, head, 32, lane, sg, list, my_np);
            __syncwarp();
        }
        set_flush<kWrite>(ring, head, held, lane, sg, list, my_np);
        if (failed && lane == 0) atomicOr(status, kWalkOverflow);
        // the groups' records (lane j writes group j's)
        if (mine) {
            const SetGroup& q = sg[lane];
            const int nc = my_nc, npt = my_np;
            if (kCount) {
                otoo_group r;
                r.first = a.gfirst[g0 + lane];
                r.count = a.gcount[g0 + lane];
                r.n_cell = nc;
                r.n_part = npt;
                // pass 0: the offsets come from the scan that follows
                r.list_off = kMode == 2 ? (nc <= q.want_c && npt <= q.want_p ? q.off_p - nc : -1) : 0;
                r.eps2 = a.eps2;
                r.cx = __dmul_rn(__dadd_rn(q.blo[0], q.bhi[0]), 0.5);
                r.cy = __dmul_rn(__dadd_rn(q.blo[1], q.bhi[1]), 0.5);
                r.cz = __dmul_rn(__dadd_rn(q.blo[2], q.bhi[2]), 0.5);
                r.theta = (float)q.theta;
                r.sys = 0;
                groups[g0 + lane] = r;
                const int64_t len = (int64_t)nc + npt;
                atomicAdd(reinterpret_cast<unsigned long long*>(a.totals), (unsigned long long)len);
                atomicAdd(reinterpret_cast<unsigned long long*>(a.totals + 1), (unsigned long long)(len * r.count));
                atomicAdd(reinterpret_cast<unsigned long long*>(a.totals + 2),
                          (unsigned long long)((int64_t)nc * r.count));
                atomicMax(reinterpret_cast<unsigned long long*>(a.totals + 3), (unsigned long long)nc);
                atomicMax(reinterpret_cast<unsigned long long*>(a.totals + 4), (unsigned long long)npt);
                if (kMode == 2 && (nc > q.want_c || npt > q.want_p))
                    atomicAdd(reinterpret_cast<unsigned long long*>(a.totals + 5), 1ull);
            } else if (nc != q.want_c || npt != q.want_p) {
                atomicOr(status, kWalkMismatch);
            }
        }
        __syncwarp();
    }
}

// ---- the walk fused with the force (the paper's GPU design) ------------------
// One warp per group walks the tree as k_walk_set does one group, but the entries do not go
// to a list in device memory: accepted cells and the particles of rejected
// leaves collect in two shared-memory index buffers, and whenever one holds a
// tile of entries the warp stages the tile as pair records (the layout of
// k_force_warp2) and evaluates it against the group's particles, IB per lane
// in lane subsets, with packed FP32 pairs and per-tile Kahan sums.  No list,
// no plan, no work items: the group is the work item.
constexpr int kFuseWarps = 4;                 // warps per CTA
constexpr int kFuseTP = 128;                  // pair records per tile at most
constexpr int kFusePPL = kFuseTP / 32;        // pair records staged per lane
constexpr int kFuseBuf = 2 * kFuseTP + kWide; // index buffer: a tile plus one step's cells

struct FuseArgs {
    const float4* split;    // [2 n_src] float pairs of the sources
    const otoo_quad* quad;  // [n_cell] or NULL (monopole cells)
    const int64_t* perm;    // [n_part] tree order -> caller order, or NULL
    double* accel;          // [n_part][3]
    double* pot;            // [n_part]
};

// Stages cnt entries buf[0..cnt) (cells: source n_part + k, else particles)
// as pair records relative to the group centre c and evaluates them for the
// lane's IB targets; the tile sums go into the Kahan sums acc.
template <int IB>
__device__ __forceinline__ void fuse_tile(const WalkArgs& a, const FuseArgs& f, const int32_t* buf, int cnt, bool cell,
                                          float4* rec, int lane, int nsub, int js, bool active, float cx, float cy,
                                          float cz, const f2 nx[IB], const f2 ny[IB], const f2 nz[IB], f2 e2,
                                          float eps2, Acc<float> acc[IB], uint32_t* status)
{
    const bool cq = cell && f.quad != nullptr;
    const int npair = (cnt + 1) / 2;
    const int npair_pad = (npair + nsub - 1) / nsub * nsub;
    const float4 zero4 = make_float4(0.f, 0.f, 0.f, 0.f);
    const int64_t n_src = a.n_part + a.n_cell;
#pragma unroll
    for (int pp = 0; pp < kFusePPL; ++pp) {
        const int m = lane + 32 * pp;
        if (m >= npair_pad) continue;
        float4 hh[2], ll[2], qa[2], qb[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int k = 2 * m + h;
            hh[h] = ll[h] = qa[h] = qb[h] = zero4;
            if (k < cnt) {
                const int idx = buf[k];
                const bool good = cell ? (idx >= a.n_part && idx < n_src) : (idx >= 0 && idx < a.n_part);
                if (good) {
                    hh[h] = __ldg(f.split + 2 * (int64_t)idx);
                    ll[h] = __ldg(f.split + 2 * (int64_t)idx + 1);
                    if (cq) {
                        const float4* qp = reinterpret_cast<const float4*>(f.quad + (idx - a.n_part));
                        qa[h] = __ldg(qp);
                        qb[h] = __ldg(qp + 1);
                    }
                } else {
                    atomicOr(status, kWalkBadRecord);
                }
            }
        }
        // padding and rejected entries were loaded as zeros: mass (and
        // quadrupole) 0, so they add exactly nothing
        float x[2], y[2], z[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            x[h] = rel32(hh[h].x, ll[h].x, cx);
            y[h] = rel32(hh[h].y, ll[h].y, cy);
            z[h] = rel32(hh[h].z, ll[h].z, cz);
        }
        const float w[2] = {hh[0].w, hh[1].w};
        put_rec2(rec, m, cq, x, y, z, w, qa, qb, eps2);
    }
    __syncwarp();
    if (active) {
        const f2 zero2 = f2pack(0.f, 0.f);
        Acc2 P2[IB];
#pragma unroll
        for (int k = 0; k < IB; ++k) P2[k].v[0] = P2[k].v[1] = P2[k].v[2] = P2[k].v[3] = zero2;
        const int niter = npair_pad / nsub;
        // loops not unrolled: the walk and the evaluation alternate in one
        // warp and must fit the instruction cache together
        if (cq)
            eval_cells2<IB, 1>(rec, js, nsub, niter, nx, ny, nz, e2, P2);
        else
            eval_parts2<IB, 1>(rec, js, nsub, niter, nx, ny, nz, e2, P2);
#pragma unroll
        for (int k = 0; k < IB; ++k) {
            float t4[4];
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                float lo, hi;
                f2unpack(P2[k].v[c], lo, hi);
                t4[c] = lo + hi;
            }
            acc[k].add(t4);
        }
    }
    __syncwarp();
}

// Drops the first `used` entries of buf (n in total; n - used < used).
__device__ __forceinline__ void fuse_shift(int32_t* buf, int n, int used, int lane)
{
    for (int k = lane; k < n - used; k += 32) buf[k] = buf[used + k];
    __syncwarp();
}

template <int IB>
#ifndef OTOO_FUSE_MIN_BLOCKS
#define OTOO_FUSE_MIN_BLOCKS 3  // resident CTAs per SM asked of the register allocator (168 registers)
#endif
__global__ void __launch_bounds__(kFuseWarps * 32, OTOO_FUSE_MIN_BLOCKS) k_walk_force(WalkArgs a, FuseArgs f)
{
    __shared__ uint32_t stack_s[kFuseWarps][kStack];
    __shared__ int32_t cbuf_s[kFuseWarps][kFuseBuf];
    __shared__ int32_t pbuf_s[kFuseWarps][kFuseBuf];
    __shared__ float4 rec_s[kFuseWarps][kCellRecF4 * kFuseTP];
    const int lane = threadIdx.x & 31;
    const int wid = threadIdx.x >> 5;
    uint32_t* stk = stack_s[wid];
    int32_t* cbuf = cbuf_s[wid];
    int32_t* pbuf = pbuf_s[wid];
    float4* rec = rec_s[wid];
    const unsigned lt = (1u << lane) - 1u;
    uint32_t* status = a.counter + 1;
    for (;;) {
        int g = 0;
        if (lane == 0) g = (int)atomicAdd(a.counter, 1u);
        g = __shfl_sync(kFull, g, 0);
        if (g >= a.n_groups) break;
        const int32_t first = a.gfirst[g], count = a.gcount[g];
        if (first < 0 || count < 1 || count > 32 * IB || (int64_t)first + count > a.n_part) {
            if (lane == 0) atomicOr(status, kWalkBadGroup);
            continue;
        }
        GroupWalk w;
        group_walk_setup(a, g, first, count, lane, w);
        if (!(w.theta >= 0.0)) continue;  // a negative per-group angle skips the group

        // the group's particles, IB per lane in nsub lane subsets
        const int P = (count + IB - 1) / IB;
        const int nsub = 32 / P;
        const int islot = lane % P, js = lane / P;
        const bool active = js < nsub;
        // entries per evaluated tile: a multiple of 2 nsub
        const int TE = 2 * ((kFuseTP / nsub) * nsub);
        const float eps2 = (float)a.eps2;
        const f2 e2 = f2pack(eps2, eps2);
        const float cx = __double2float_rn(w.c[0]), cy = __double2float_rn(w.c[1]), cz = __double2float_rn(w.c[2]);
        f2 nx[IB], ny[IB], nz[IB];
        Acc<float> acc[IB];
#pragma unroll
        for (int k = 0; k < IB; ++k) {
            const int i = islot + k * P;
            float x = 0.f, y = 0.f, z = 0.f;
            if (active && i < count) {
                const int64_t t = (int64_t)first + i;
                const float4 h = __ldg(f.split + 2 * t);
                const float4 l = __ldg(f.split + 2 * t + 1);
                x = rel32(h.x, l.x, cx);
                y = rel32(h.y, l.y, cy);
                z = rel32(h.z, l.z, cz);
            }
            nx[k] = f2pack(-x, -x);
            ny[k] = f2pack(-y, -y);
            nz[k] = f2pack(-z, -z);
            acc[k].zero();
        }

        int32_t ncell = 0, npart = 0;  // entries of the group's (virtual) list
        int nc = 0, npb = 0;           // entries waiting in the two buffers
        int sp = 1;
        if (lane == 0) stk[0] = run(0, 1);
        __syncwarp();
        int64_t budget = a.n_cell;
        bool failed = false;
        while (sp > 0) {
            StepCells sc;
            if (!walk_take(a, w, stk, sp, budget, lane, sc, status)) {
                failed = true;
                break;
            }
            // accepted cells into the cell buffer, in position order
#pragma unroll
            for (int h = 0; h < kWalkHalves; ++h) {
                const unsigned am = __ballot_sync(kFull, sc.kind[h] == 1);
                if (sc.kind[h] == 1) cbuf[nc + __popc(am & lt)] = (int32_t)(a.n_part + sc.node[h]);
                nc += __popc(am);
                ncell += __popc(am);
            }
            __syncwarp();
            // particles of rejected leaves into the particle buffer, in
            // position order, a buffer's worth at a time
#pragma unroll
            for (int h = 0; h < kWalkHalves; ++h) {
                if (!__any_sync(kFull, sc.kind[h] == 2)) continue;
                const int np = sc.kind[h] == 2 ? sc.pe[h] - sc.pb[h] : 0;
                const int pin = warp_incl_scan(np, lane);
                const int total = __shfl_sync(kFull, pin, 31);
                npart += total;
                for (int done = 0; done < total;) {
                    const int take = min(kFuseBuf - npb, total - done);
                    const int lo = max(pin - np, done), hi = min(pin, done + take);
                    for (int o = lo; o < hi; ++o) pbuf[npb + o - done] = sc.pb[h] + (o - (pin - np));
                    __syncwarp();
                    npb += take;
                    done += take;
                    while (npb >= TE) {
                        fuse_tile<IB>(a, f, pbuf, TE, false, rec, lane, nsub, js, active, cx, cy, cz, nx, ny, nz, e2,
                                      eps2, acc, status);
                        fuse_shift(pbuf, npb, TE, lane);
                        npb -= TE;
                    }
                }
            }
            walk_push(stk, sp, sc, lt);
            while (nc >= TE) {
                fuse_tile<IB>(a, f, cbuf, TE, true, rec, lane, nsub, js, active, cx, cy, cz, nx, ny, nz, e2, eps2, acc,
                              status);
                fuse_shift(cbuf, nc, TE, lane);
                nc -= TE;
            }
        }
        if (failed) {
            if (lane == 0) atomicOr(status, kWalkOverflow);
            continue;
        }
        if (nc > 0)
            fuse_tile<IB>(a, f, cbuf, nc, true, rec, lane, nsub, js, active, cx, cy, cz, nx, ny, nz, e2, eps2, acc, status);
        if (npb > 0)
            fuse_tile<IB>(a, f, pbuf, npb, false, rec, lane, nsub, js, active, cx, cy, cz, nx, ny, nz, e2, eps2, acc,
                          status);

        // merge the lane subsets, FP64 outputs in caller order; the self pair
        // (always in the list: a group never accepts a cell overlapping its
        // box) added exactly -m_i rsqrt(eps^2) in FP32
#pragma unroll
        for (int k = 0; k < IB; ++k) {
            double r[4];
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                float S = acc[k].s[c], C = acc[k].c[c];
                merge_subsets(S, C, js, nsub, P);
                r[c] = (double)S - (double)C;
            }
            r[3] = -r[3];
            const int i = islot + k * P;
            if (js == 0 && i < count) {
                const int64_t t = (int64_t)first + i;
                const float4 h = __ldg(f.split + 2 * t);
                r[3] += (double)(h.w * rsqrt_r(eps2));
                const int64_t o = f.perm ? f.perm[t] : t;
                f.accel[3 * o] = r[0];
                f.accel[3 * o + 1] = r[1];
                f.accel[3 * o + 2] = r[2];
                f.pot[o] = r[3];
            }
        }
        if (lane == 0) {
            const int64_t len = (int64_t)ncell + npart;
            atomicAdd(reinterpret_cast<unsigned long long*>(a.totals), (unsigned long long)len);
            atomicAdd(reinterpret_cast<unsigned long long*>(a.totals + 1), (unsigned long long)(len * count));
            atomicAdd(reinterpret_cast<unsigned long long*>(a.totals + 2), (unsigned long long)((int64_t)ncell * count));
            atomicMax(reinterpret_cast<unsigned long long*>(a.totals + 3), (unsigned long long)ncell);
            atomicMax(reinterpret_cast<unsigned long long*>(a.totals + 4), (unsigned long long)npart);
        }
    }
}

// One warp per group: the group's slot (filled by the single pass) copied to
// its place in the dense list (list_off, already rewritten by the scan),
// cells back in walk order, then particles.  Nothing is copied when a group
// did not fit its slot (totals[5] > 0: the caller walks again in two passes)
// or when the list is too small.
__global__ void k_compact(const otoo_group* __restrict__ groups, int32_t G, const int32_t* __restrict__ slots,
                          int64_t ccap, int64_t pcap, int32_t* __restrict__ list, int64_t capacity,
                          const int64_t* __restrict__ totals, uint32_t* __restrict__ status)
{
    const int64_t g = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (g >= G) return;
    if (totals[5] > 0 || totals[0] > capacity) {
        if (g == 0 && lane == 0) atomicOr(status, kWalkNoRoom);
        return;
    }
    const otoo_group gr = groups[g];
    if (gr.n_cell < 0 || gr.n_part < 0 || gr.n_cell > ccap || gr.n_part > pcap || gr.list_off < 0 ||
        gr.list_off + gr.n_cell + gr.n_part > capacity) {
        if (lane == 0) atomicOr(status, kWalkNoRoom);
        return;
    }
    const int32_t* ps = slots + g * (ccap + pcap) + ccap;  // particle 0; cell k at ps[-1 - k]
    int32_t* d = list + gr.list_off;
    for (int k = lane; k < gr.n_cell; k += 32) d[k] = ps[-1 - k];
    d += gr.n_cell;
    for (int k = lane; k < gr.n_part; k += 32) d[k] = ps[k];
}

// ---- exclusive prefix sums in index order ---------------------------------
// In: functor int64 operator()(int64 i); Out: functor void operator()(int64 i,
// int64 prefix).  Three launches: sums of blocks of kScanBlock elements, a
// one-CTA exclusive scan of those sums (total to *total), block-level scans.

struct GroupLen {
    const otoo_group* g;
    __device__ int64_t operator()(int64_t i) const { return (int64_t)g[i].n_cell + g[i].n_part; }
};
struct GroupOff {
    otoo_group* g;
    __device__ void operator()(int64_t i, int64_t v) const { g[i].list_off = v; }
};
__device__ int64_t block_excl_scan(int64_t v, int64_t* warp_s, int64_t* total)
{
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    int64_t inc = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int64_t t = __shfl_up_sync(kFull, inc, o);
        if (lane >= o) inc += t;
    }
    if (lane == 31) warp_s[wid] = inc;
    __syncthreads();
    if (wid == 0) {
        int64_t w = lane < (int)(blockDim.x >> 5) ? warp_s[lane] : 0;
        int64_t wi = w;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int64_t t = __shfl_up_sync(kFull, wi, o);
            if (lane >= o) wi += t;
        }
        warp_s[lane] = wi - w;
        if (lane == 31) warp_s[32] = wi;
    }
    __syncthreads();
    const int64_t r = warp_s[wid] + inc - v;
    *total = warp_s[32];
    __syncthreads();
    return r;
}

template <class In>
__global__ void __launch_bounds__(kScanThreads) k_scan_sums(In in, int64_t n, int64_t* __restrict__ bsum)
{
    __shared__ int64_t ws[33];
    const int64_t b0 = (int64_t)blockIdx.x * kScanBlock;
    int64_t v = 0;
    for (int k = 0; k < kScanBlock / kScanThreads; ++k) {
        const int64_t i = b0 + (int64_t)k * kScanThreads + threadIdx.x;
        if (i < n) v += in(i);
    }
    int64_t tot;
    block_excl_scan(v, ws, &tot);
    if (threadIdx.x == 0) bsum[blockIdx.x] = tot;
}

__global__ void __launch_bounds__(kScanThreads) k_scan_top(int64_t* __restrict__ bsum, int64_t nblk,
                                                            int64_t* __restrict__ total)
{
    __shared__ int64_t ws[33];
    int64_t carry = 0;
    for (int64_t b0 = 0; b0 < nblk; b0 += kScanThreads) {
        const int64_t i = b0 + threadIdx.x;
        const int64_t v = i < nblk ? bsum[i] : 0;
        int64_t tot;
        const int64_t e = block_excl_scan(v, ws, &tot);
        if (i < nblk) bsum[i] = carry + e;
        carry += tot;
    }
    if (threadIdx.x == 0 && total) *total = carry;
}

template <class In, class Out>
__global__ void __launch_bounds__(kScanThreads) k_scan_apply(In in, Out out, int64_t n,
                                                              const int64_t* __restrict__ bsum)
{
    __shared__ int64_t ws[33];
    constexpr int kPer = kScanBlock / kScanThreads;
    const int64_t b0 = (int64_t)blockIdx.x * kScanBlock + (int64_t)threadIdx.x * kPer;
    int64_t v[kPer], s = 0;
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
        v[k] = b0 + k < n ? in(b0 + k) : 0;
        s += v[k];
    }
    int64_t tot;
    int64_t e = block_excl_scan(s, ws, &tot) + bsum[blockIdx.x];
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
        if (b0 + k < n) out(b0 + k, e);
        e += v[k];
    }
}

template <class In, class Out>
cudaError_t excl_scan(In in, Out out, int64_t n, int64_t* bsum, int64_t* total, cudaStream_t s)
{
    const int64_t nblk = (n + kScanBlock - 1) / kScanBlock;
    if (nblk == 0) return cudaSuccess;
    k_scan_sums<In><<<(unsigned)nblk, kScanThreads, 0, s>>>(in, n, bsum);
    k_scan_top<<<1, kScanThreads, 0, s>>>(bsum, nblk, total);
    k_scan_apply<In, Out><<<(unsigned)nblk, kScanThreads, 0, s>>>(in, out, n, bsum);
    return cudaGetLastError();
}

int64_t scan_blocks(int64_t n) { return (n + kScanBlock - 1) / kScanBlock; }

// ---- device plan ------------------------------------------------------------

struct PlanScratch {
    int64_t* slots;   // [blocks] partial slots of each block's groups, then their exclusive prefix
    int64_t* splits;  // [blocks] split lists of each block's groups, then their exclusive prefix
    int32_t* hist;    // [kClasses] items per cost class
    int32_t* cursor;  // [kClasses] next free item position of each class
    int32_t* split;   // the list chunk length the counts were made with
};

// The plan kernels run 256 threads per block, one group each.  The chunk
// table (a kernel parameter) is copied to shared memory first: threads index
// it by their own group sizes, which the parameter bank would serialise.
// Counts and totals are summed per warp and block, so each block makes one
// global atomic per class and per total.  Three launches: k_plan_count also
// leaves each block's sums of slots and split lists, k_plan_scan turns them and
// the class counts into prefixes, k_plan_fill adds the prefix inside the block.
// With 64-bit shared-memory atomics per group, two three-launch scans over all
// groups and a one-thread prefix of the classes, ten launches took 49 us for
// 260 groups and 84 us for 221169; these take 16 and 40 us.
constexpr int kPlanThreads = 256;
constexpr int kPlanWarps = kPlanThreads / 32;

PlanScratch plan_layout(int32_t* base, int64_t G)
{
    const int64_t nb = (G + kPlanThreads - 1) / kPlanThreads;
    PlanScratch p;
    p.slots = reinterpret_cast<int64_t*>(base);
    p.splits = p.slots + nb;
    p.hist = reinterpret_cast<int32_t*>(p.splits + nb);
    p.cursor = p.hist + kClasses;
    p.split = p.cursor + kClasses;
    return p;
}

__device__ void plan_table_to_shared(const ChunkTable& tab, ChunkTable& st)
{
    for (int k = threadIdx.x; k <= kMaxGroup; k += blockDim.x) st.last[k] = tab.last[k];
    if (threadIdx.x == 0) st.ib = tab.ib;
}

// A group's particle chunks (plan_chunks.h), list chunks and cost class, the
// host plan's: class = quarter octaves of the largest item's ni * (j1 - j0).
// nic = nch = 0 for an empty list or a group size out of range.
__device__ __forceinline__ void plan_group(const otoo_group& gr, const ChunkTable& st, int32_t split, int32_t& nic,
                                           int32_t& nch, int32_t& cls)
{
    nic = nch = cls = 0;
    const int64_t len = (int64_t)gr.n_cell + gr.n_part;
    if (len <= 0 || gr.count <= 0 || gr.count > kMaxGroup) return;
    int32_t big = 0;
    nic = chunk_count(st, gr.count, &big);
    nch = (int32_t)((len + split - 1) / split);
    const int64_t c0 = (int64_t)big * ((len + nch - 1) / nch);
    const int msb = 63 - __clzll((long long)c0);
    const int frac = msb >= 2 ? (int)((c0 >> (msb - 2)) & 3) : (int)((c0 << (2 - msb)) & 3);
    cls = 4 * msb + frac;
    if (cls >= kClasses) cls = kClasses - 1;
}

__device__ __forceinline__ int64_t warp_sum64(int64_t v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
    return v;
}

__global__ void __launch_bounds__(kPlanThreads) k_plan_count(const otoo_group* __restrict__ groups, int32_t G,
                                                             const ChunkTable tab, int32_t split, PlanScratch p,
                                                             int64_t* __restrict__ totals)
{
    __shared__ ChunkTable st;
    __shared__ int32_t shist[kClasses];
    __shared__ int64_t s_sum[3][kPlanWarps];  // items, split lists, slots
    __shared__ int32_t s_max[kPlanWarps];
    plan_table_to_shared(tab, st);
    for (int c = threadIdx.x; c < kClasses; c += blockDim.x) shist[c] = 0;
    __syncthreads();
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int32_t g = blockIdx.x * blockDim.x + threadIdx.x;
    int32_t nic = 0, nch = 0, cls = 0, cnt = 1;
    if (g < G) {
        const otoo_group gr = groups[g];
        cnt = gr.count > 1 ? gr.count : 1;
        plan_group(gr, st, split, nic, nch, cls);
        if (nic > 0) atomicAdd(shist + cls, nic * nch);
    }
    __syncwarp();
    const int64_t items = warp_sum64((int64_t)nic * nch), slots = warp_sum64(nch > 1 ? nch : 0);
    const int32_t splits = __reduce_add_sync(kFull, nch > 1 ? 1 : 0), mx = __reduce_max_sync(kFull, cnt);
    if (lane == 0) s_sum[0][w] = items, s_sum[1][w] = splits, s_sum[2][w] = slots, s_max[w] = mx;
    __syncthreads();
    for (int c = threadIdx.x; c < kClasses; c += blockDim.x)
        if (shist[c]) atomicAdd(p.hist + c, shist[c]);
    if (threadIdx.x == 0) {
        int64_t a[3] = {0, 0, 0};
        int32_t m = 1;
        for (int k = 0; k < kPlanWarps; ++k) {
            for (int q = 0; q < 3; ++q) a[q] += s_sum[q][k];
            m = s_max[k] > m ? s_max[k] : m;
        }
        unsigned long long* t = reinterpret_cast<unsigned long long*>(totals);
        if (a[0]) atomicAdd(t, (unsigned long long)a[0]);
        if (a[1]) {
            atomicAdd(t + 1, (unsigned long long)a[1]);
            atomicAdd(t + 2, (unsigned long long)a[2]);
        }
        atomicMax(t + 3, (unsigned long long)m);
        p.splits[blockIdx.x] = a[1];
        p.slots[blockIdx.x] = a[2];
        if (blockIdx.x == 0) *p.split = split;
    }
}

// One block: exclusive prefixes of the blocks' slots and split lists, and the
// start of each cost class, most expensive class first.
__global__ void __launch_bounds__(kScanThreads) k_plan_scan(PlanScratch p, int32_t nblk,
                                                             const int64_t* __restrict__ totals)
{
    __shared__ int64_t ws[33];
    const int c = kClasses - 1 - (int)threadIdx.x;
    int64_t tot;
    const int64_t pos = block_excl_scan(c >= 0 ? p.hist[c] : 0, ws, &tot);
    if (c >= 0) p.cursor[c] = (int32_t)pos;
    if (totals[1] == 0) return;  // no list is split: no slots
    for (int a = 0; a < 2; ++a) {
        int64_t* v = a ? p.splits : p.slots;
        int64_t carry = 0;
        for (int32_t b0 = 0; b0 < nblk; b0 += kScanThreads) {
            const int32_t i = b0 + threadIdx.x;
            const int64_t e = block_excl_scan(i < nblk ? v[i] : 0, ws, &tot);
            if (i < nblk) v[i] = carry + e;
            carry += tot;
        }
    }
}

__global__ void __launch_bounds__(kPlanThreads) k_plan_fill(const otoo_group* __restrict__ groups, int32_t G,
                                                            const ChunkTable tab, PlanScratch p,
                                                            const int64_t* __restrict__ totals,
                                                            otoo_item* __restrict__ items, int64_t items_cap,
                                                            otoo_split* __restrict__ splits, int64_t splits_cap,
                                                            uint32_t* __restrict__ status)
{
    __shared__ ChunkTable st;
    __shared__ int32_t scount[kClasses], sbase[kClasses];
    __shared__ int64_t ws[33];
    plan_table_to_shared(tab, st);
    for (int c = threadIdx.x; c < kClasses; c += blockDim.x) scount[c] = 0;
    __syncthreads();
    // the block's items of each class take one run of that class's items
    const int32_t g = blockIdx.x * blockDim.x + threadIdx.x;
    otoo_group gr = {};
    int32_t nic = 0, nch = 0, cls = 0;
    if (g < G) {
        gr = groups[g];
        plan_group(gr, st, *p.split, nic, nch, cls);
    }
    const bool on = nic > 0 && nch > 0;
    const int32_t local = on ? atomicAdd(scount + cls, nic * nch) : 0;
    // first slot and split record of the group, in group order
    int64_t slot0 = 0, si = 0;
    if (totals[1] != 0) {  // (uniform)
        int64_t tot;
        slot0 = p.slots[blockIdx.x] + block_excl_scan(nch > 1 ? nch : 0, ws, &tot);
        si = p.splits[blockIdx.x] + block_excl_scan(nch > 1 ? 1 : 0, ws, &tot);
    }
    __syncthreads();
    for (int c = threadIdx.x; c < kClasses; c += blockDim.x)
        if (scount[c]) sbase[c] = atomicAdd(p.cursor + c, scount[c]);
    __syncthreads();
    if (!on) return;
    const int64_t len = (int64_t)gr.n_cell + gr.n_part;
    const int32_t pos = sbase[cls] + local;
    if ((int64_t)pos + nic * nch > items_cap) {
        atomicOr(status, kWalkNoRoom);
        return;
    }
    if (nch > 1) {
        if (si >= splits_cap) {
            atomicOr(status, kWalkNoRoom);
            return;
        }
        otoo_split s;
        s.g = g;
        s.slot0 = (int32_t)slot0;
        s.n_chunks = nch;
        s.pad = 0;
        splits[si] = s;
    }
    int32_t k = pos, i0 = 0;
    for (int32_t rest = gr.count; rest > 0;) {
        const int32_t ni = st.last[rest];
        for (int32_t q = 0; q < nch; ++q) {
            otoo_item it;
            it.g = g;
            it.i0 = i0;
            it.ni = ni;
            it.j0 = (int32_t)(len * q / nch);
            it.j1 = (int32_t)(len * (q + 1) / nch);
            it.slot = nch > 1 ? (int32_t)slot0 + q : -1;
            it.pad0 = it.pad1 = 0;
            items[k++] = it;
        }
        i0 += ni;
        rest -= ni;
    }
}

#define CUDA_TRY(expr)                                                                                 \
    do {                                                                                               \
        cudaError_t e_ = (expr);                                                                       \
        if (e_ != cudaSuccess) return set_error(OTOO_ECUDA, "%s: %s", #expr, cudaGetErrorString(e_));  \
    } while (0)

// The particle-chunk table of the plan for ib targets per lane, built once
// per process for each ib in {1, 2, 4} (others each call).
const ChunkTable& chunk_table(int32_t ib)
{
    static ChunkTable tabs[3];
    static std::once_flag once[3];
    const int k = ib == 1 ? 0 : ib == 2 ? 1 : ib == 4 ? 2 : -1;
    if (k < 0) {
        thread_local ChunkTable t;
        chunk_table_build(ib, t);
        return t;
    }
    std::call_once(once[k], [&] { chunk_table_build(ib, tabs[k]); });
    return tabs[k];
}

int check_walk(const otoo_dev_walk* w)
{
    OTOO_REQUIRE(w, OTOO_EINVAL, "walk is NULL");
    OTOO_REQUIRE(w->src && w->cell && w->cell64 && w->group_first && w->group_count && w->counter && w->totals,
                 OTOO_EINVAL, "walk: NULL device pointer");
    OTOO_REQUIRE(w->n_part >= 1 && w->n_cell >= 1 && w->n_part + w->n_cell <= INT32_MAX, OTOO_EINVAL,
                 "walk: n_part/n_cell out of range");
    OTOO_REQUIRE(w->n_cell <= (int64_t)kRunMask + 1, OTOO_EINVAL, "walk: more than 2^28 cells");
    OTOO_REQUIRE(w->n_groups >= 1, OTOO_EINVAL, "walk: n_groups < 1");
    OTOO_REQUIRE(w->eps2 > 0.0, OTOO_EINVAL, "walk: eps2 must be > 0");
    OTOO_REQUIRE(w->theta >= 0.0 && w->theta < 1e300, OTOO_EINVAL, "walk: theta must be finite and >= 0");
    OTOO_REQUIRE(w->set >= 0 && w->set <= kSet, OTOO_EINVAL, "walk: set must be in [0, %d]", kSet);
    OTOO_REQUIRE(w->mac == OTOO_MAC_THETA || w->mac == OTOO_MAC_SW || w->mac == OTOO_MAC_SPH, OTOO_EINVAL,
                 "walk: unknown mac %d", w->mac);
    return OTOO_OK;
}

WalkArgs walk_args(const otoo_dev_walk* w)
{
    WalkArgs a;
    a.n_part = w->n_part;
    a.n_cell = w->n_cell;
    a.n_groups = w->n_groups;
    a.exact = w->exact ? 1 : 0;
    a.mac = w->mac;
    a.pad = 0;
    a.theta = w->theta;
    a.eps2 = w->eps2;
    a.src = w->src;
    a.cell = w->cell;
    a.cell64 = w->cell64;
    a.gfirst = w->group_first;
    a.gcount = w->group_count;
    a.tpg = w->theta_per_group;
    a.counter = w->counter;
    a.totals = w->totals;
    return a;
}

// One threshold rule for every group and no cube test: the absolute MAC, the SPH
// radius, or one opening angle below the limit of group flag 2.
bool plain_rule(const otoo_dev_walk* w)
{
    return w->mac == OTOO_MAC_SW || w->mac == OTOO_MAC_SPH || (!w->theta_per_group && w->theta < kCubeAngle);
}

template <int kMode, bool kGen>
int launch_walk_form(const otoo_dev_walk* w, otoo_group* groups, int32_t* list, int64_t capacity, cudaStream_t s,
                     int64_t pcap)
{
    int dev = 0, sms = 0, occ = 0;
    CUDA_TRY(cudaGetDevice(&dev));
    CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_walk_set<kMode, kGen>, kWalkWarps * 32, 0));
    if (occ < 1) occ = 1;
    // groups per warp: as asked, or (0) about as many as give every resident
    // warp one set (a quarter more goes to a second round rather than to larger
    // sets), kSet at most: a larger set shares more of its cells, fewer sets
    // than warps leave warps idle.  Microseconds with 1 / 2 / 3 / 4 / 6 / 8 groups on
    // 3648 warps: 5353 groups (King 100003, theta 0.75) 126 / 115 / 126 / 142 /
    // 169 / 205; 11162 groups (Plummer 200000) 407 / 321 / 260 / 298 / 339 / 399;
    // 21230 groups (Hernquist 400000) 765 / 534 / 476 / 482 / 432 / 517; 27005 groups
    // (Plummer 2^20) 1113 / 793 / 724 / 664 / 726 / 686.
    int gs = w->set;
    if (gs == 0) {
        const int64_t warps = (int64_t)sms * occ * kWalkWarps;
        const int64_t fit = ((int64_t)w->n_groups - warps / 4 + warps - 1) / warps;
        gs = fit < 1 ? 1 : fit > kSet ? kSet : (int)fit;
    }
    // one set per warp, spread over all SMs, while there are fewer sets than warps
    const int64_t units = ((int64_t)w->n_groups + gs - 1) / gs;
    const int64_t blocks = units < (int64_t)sms * occ ? units : (int64_t)sms * occ;
    const int64_t need = (units + blocks - 1) / blocks;
    const int nw = need < kWalkWarps ? (int)need : kWalkWarps;
    if (kMode == 1) CUDA_TRY(cudaMemsetAsync(w->counter, 0, sizeof(uint32_t), s));  // (the others start with clear_walk)
    k_walk_set<kMode, kGen><<<(unsigned)blocks, nw * 32, 0, s>>>(walk_args(w), (int32_t)units, gs, groups, list, capacity,
                                                                 pcap);
    CUDA_TRY(cudaGetLastError());
    return OTOO_OK;
}

template <int kMode>
int launch_walk(const otoo_dev_walk* w, otoo_group* groups, int32_t* list, int64_t capacity, cudaStream_t s,
                int64_t pcap = 0)
{
    return plain_rule(w) ? launch_walk_form<kMode, false>(w, groups, list, capacity, s, pcap)
                         : launch_walk_form<kMode, true>(w, groups, list, capacity, s, pcap);
}

}  // namespace

extern "C" {

int64_t otoo_walk_totals_len(int64_t n_groups) { return kTotals + scan_blocks(n_groups < 0 ? 0 : n_groups) + 1; }

// Clears the ticket, the status and the totals before a walk: one operation
// when the caller keeps the totals right behind the four counter words.
static int clear_walk(const otoo_dev_walk* w, cudaStream_t s)
{
    const size_t nc = 4 * sizeof(uint32_t), nt = kTotals * sizeof(int64_t);
    if (reinterpret_cast<char*>(w->counter) + nc == reinterpret_cast<char*>(w->totals)) {
        CUDA_TRY(cudaMemsetAsync(w->counter, 0, nc + nt, s));
    } else {
        CUDA_TRY(cudaMemsetAsync(w->counter, 0, nc, s));
        CUDA_TRY(cudaMemsetAsync(w->totals, 0, nt, s));
    }
    return OTOO_OK;
}

int otoo_walk_count(const otoo_dev_walk* w, otoo_group* groups, void* stream)
{
    otoo::Range range_("otoo_walk_count");
    const int rc = check_walk(w);
    if (rc) return rc;
    OTOO_REQUIRE(groups, OTOO_EINVAL, "otoo_walk_count: groups is NULL");
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    const int r1 = clear_walk(w, s);
    if (r1) return r1;
    const int r2 = launch_walk<0>(w, groups, nullptr, 0, s);
    if (r2) return r2;
    CUDA_TRY(excl_scan(GroupLen{groups}, GroupOff{groups}, w->n_groups, w->totals + kTotals, nullptr, s));
    return OTOO_OK;
}

int otoo_walk_single(const otoo_dev_walk* w, otoo_group* groups, int32_t* slots, int64_t cell_cap, int64_t part_cap,
                     void* stream)
{
    otoo::Range range_("otoo_walk_single");
    const int rc = check_walk(w);
    if (rc) return rc;
    OTOO_REQUIRE(groups && slots, OTOO_EINVAL, "otoo_walk_single: NULL pointer");
    OTOO_REQUIRE(cell_cap >= 1 && part_cap >= 1 && cell_cap + part_cap <= INT32_MAX, OTOO_EINVAL,
                 "otoo_walk_single: slot sizes out of range");
    OTOO_REQUIRE(w->n_groups <= INT64_MAX / (cell_cap + part_cap), OTOO_EINVAL, "otoo_walk_single: slots too large");
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    const int r1 = clear_walk(w, s);
    if (r1) return r1;
    return launch_walk<2>(w, groups, slots, cell_cap, s, part_cap);
}

int otoo_walk_compact(const otoo_dev_walk* w, otoo_group* groups, const int32_t* slots, int64_t cell_cap,
                      int64_t part_cap, int32_t* list, int64_t capacity, void* stream)
{
    otoo::Range range_("otoo_walk_compact");
    const int rc = check_walk(w);
    if (rc) return rc;
    OTOO_REQUIRE(groups && slots && list, OTOO_EINVAL, "otoo_walk_compact: NULL pointer");
    OTOO_REQUIRE(cell_cap >= 1 && part_cap >= 1 && cell_cap + part_cap <= INT32_MAX, OTOO_EINVAL,
                 "otoo_walk_compact: slot sizes out of range");
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    CUDA_TRY(excl_scan(GroupLen{groups}, GroupOff{groups}, w->n_groups, w->totals + kTotals, nullptr, s));
    const int64_t warps = w->n_groups;
    k_compact<<<(unsigned)((warps * 32 + 255) / 256), 256, 0, s>>>(groups, w->n_groups, slots, cell_cap, part_cap,
                                                                   list, capacity, w->totals, w->counter + 1);
    CUDA_TRY(cudaGetLastError());
    return OTOO_OK;
}

int otoo_walk_fill(const otoo_dev_walk* w, const otoo_group* groups, int32_t* list, int64_t capacity, void* stream)
{
    otoo::Range range_("otoo_walk_fill");
    const int rc = check_walk(w);
    if (rc) return rc;
    OTOO_REQUIRE(groups && list, OTOO_EINVAL, "otoo_walk_fill: NULL pointer");
    OTOO_REQUIRE(capacity >= 0, OTOO_EINVAL, "otoo_walk_fill: negative capacity");
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    return launch_walk<1>(w, const_cast<otoo_group*>(groups), list, capacity, s);
}

int otoo_walk_force(const otoo_dev_walk* w, const otoo_quad* quad, const int64_t* perm, float* split, int32_t iblock,
                    double* accel, double* pot, void* stream)
{
    otoo::Range range_("otoo_walk_force");
    const int rc = check_walk(w);
    if (rc) return rc;
    OTOO_REQUIRE(split && accel && pot, OTOO_EINVAL, "otoo_walk_force: NULL pointer");
    OTOO_REQUIRE(w->mac != OTOO_MAC_SPH, OTOO_EINVAL, "otoo_walk_force: the SPH walk has no force");
    OTOO_REQUIRE(iblock == 1 || iblock == 2 || iblock == 4, OTOO_EINVAL, "otoo_walk_force: iblock must be 1, 2 or 4");
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    CUDA_TRY(cudaMemsetAsync(w->counter, 0, 4 * sizeof(uint32_t), s));
    CUDA_TRY(cudaMemsetAsync(w->totals, 0, kTotals * sizeof(int64_t), s));
    const int r1 = enqueue_split(w->src, split, w->n_part + w->n_cell, stream);
    if (r1) return r1;
    FuseArgs f;
    f.split = reinterpret_cast<const float4*>(split);
    f.quad = quad;
    f.perm = perm;
    f.accel = accel;
    f.pot = pot;
    void (*fn)(WalkArgs, FuseArgs) = iblock == 1 ? k_walk_force<1> : iblock == 2 ? k_walk_force<2> : k_walk_force<4>;
    int dev = 0, sms = 0, occ = 0;
    CUDA_TRY(cudaGetDevice(&dev));
    CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, fn, kFuseWarps * 32, 0));
    if (occ < 1) return set_error(OTOO_EINVAL, "otoo_walk_force: kernel does not fit on an SM");
    int64_t blocks = (int64_t)sms * occ;
    const int64_t need = ((int64_t)w->n_groups + kFuseWarps - 1) / kFuseWarps;
    if (blocks > need) blocks = need;
    fn<<<(unsigned)blocks, kFuseWarps * 32, 0, s>>>(walk_args(w), f);
    CUDA_TRY(cudaGetLastError());
    return OTOO_OK;
}

int otoo_walk_check_status(const otoo_dev_walk* w, void* stream)
{
    OTOO_REQUIRE(w && w->counter, OTOO_EINVAL, "walk/counter is NULL");
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    uint32_t h[2] = {0, 0};
    CUDA_TRY(cudaMemcpyAsync(h, w->counter, sizeof(h), cudaMemcpyDeviceToHost, s));
    CUDA_TRY(cudaStreamSynchronize(s));
    if (h[1] & kWalkBadGroup) return set_error(OTOO_EDEVICE, "walk: a group range failed its bounds check");
    if (h[1] & kWalkBadRecord) return set_error(OTOO_EDEVICE, "walk: a cell record failed its bounds check");
    if (h[1] & kWalkOverflow) return set_error(OTOO_EDEVICE, "walk: a group's stack or node budget ran out");
    if (h[1] & kWalkMismatch) return set_error(OTOO_EDEVICE, "walk: the two passes counted different entries");
    if (h[1] & kWalkNoRoom) return set_error(OTOO_EDEVICE, "walk/plan: output array too small");
    return OTOO_OK;
}

int64_t otoo_plan_scratch_ints(int64_t n_groups)
{
    if (n_groups < 0) n_groups = 0;
    return 4 * ((n_groups + kPlanThreads - 1) / kPlanThreads + 1) + 2 * kClasses + 2;
}

int otoo_plan_count(const otoo_group* groups, int32_t n_groups, const otoo_tune* tune, int32_t* plan_scratch,
                    int64_t* plan_totals, void* stream)
{
    otoo::Range range_("otoo_plan_count");
    OTOO_REQUIRE(groups && tune && plan_scratch && plan_totals, OTOO_EINVAL, "otoo_plan_count: NULL pointer");
    OTOO_REQUIRE(n_groups >= 1, OTOO_EINVAL, "otoo_plan_count: n_groups < 1");
    OTOO_REQUIRE(tune->split >= 1, OTOO_EINVAL, "split must be >= 1");
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    const int32_t ib = tune->iblock > 1 ? tune->iblock : 1;
    PlanScratch p = plan_layout(plan_scratch, n_groups);
    CUDA_TRY(cudaMemsetAsync(plan_totals, 0, 4 * sizeof(int64_t), s));
    CUDA_TRY(cudaMemsetAsync(p.hist, 0, kClasses * sizeof(int32_t), s));
    k_plan_count<<<(n_groups + kPlanThreads - 1) / kPlanThreads, kPlanThreads, 0, s>>>(
        groups, n_groups, chunk_table(ib), tune->split, p, plan_totals);
    k_plan_scan<<<1, kScanThreads, 0, s>>>(p, (n_groups + kPlanThreads - 1) / kPlanThreads, plan_totals);
    CUDA_TRY(cudaGetLastError());
    return OTOO_OK;
}

int otoo_plan_fill(const otoo_group* groups, int32_t n_groups, const otoo_tune* tune, int32_t* plan_scratch,
                   const int64_t* plan_totals, otoo_item* items, int64_t items_capacity, otoo_split* splits,
                   int64_t splits_capacity, uint32_t* counter, void* stream)
{
    otoo::Range range_("otoo_plan_fill");
    OTOO_REQUIRE(groups && tune && plan_scratch && plan_totals && counter, OTOO_EINVAL,
                 "otoo_plan_fill: NULL pointer");
    OTOO_REQUIRE(items || items_capacity == 0, OTOO_EINVAL, "otoo_plan_fill: items is NULL");
    OTOO_REQUIRE(splits || splits_capacity == 0, OTOO_EINVAL, "otoo_plan_fill: splits is NULL");
    OTOO_REQUIRE(n_groups >= 1, OTOO_EINVAL, "otoo_plan_fill: n_groups < 1");
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    const int32_t ib = tune->iblock > 1 ? tune->iblock : 1;
    PlanScratch p = plan_layout(plan_scratch, n_groups);
    k_plan_fill<<<(n_groups + kPlanThreads - 1) / kPlanThreads, kPlanThreads, 0, s>>>(
        groups, n_groups, chunk_table(ib), p, plan_totals, items, items_capacity, splits, splits_capacity,
        counter + 1);
    CUDA_TRY(cudaGetLastError());
    return OTOO_OK;
}

}  // extern "C"
