// The octree built on the device (Section III-B: root cube, keys, sort,
// cells; Section III-C: cell properties), producing the inputs of the device
// walk and the force step directly in device memory.
//
// The root cube, the grid coordinates, the Hilbert keys and the cube of every
// cell are computed with the host build's operations (treegeom.h), and the
// sort is stable on (key, caller index), so the particle order, the cells (as
// (level, first particle, last particle) ranges), their cubes and the groups
// are the host build's.  Cells are numbered level by level (the host numbers
// them in expansion order); children stay consecutive.  Moments are summed
// bottom-up (children combined by the parallel-axis rule), so they equal the
// host's direct sums to rounding.
//
// Kernels
//   k_bbox                  min/max of the positions (order-preserving integer
//                           keys: exact); its last block sets the root cube.
//   k_keys                  grid coordinates and Hilbert key per particle.
//   k_sort_pass / k_sort_tile  stable LSD radix sort of (key, index), 8 bits
//                           per pass: one launch per pass with a decoupled
//                           look-back between tiles, or all passes in one
//                           block for at most one tile.
//   k_permute               particles in tree order (sources, permutation).
//   k_levels / k_cells      every cell of every level at once, from the
//                           number of key digits that neighbouring particles
//                           share.
//   k_leaves / k_parents    the cells' links and the leaves' moments, then the
//                           parents combine their children, deepest level
//                           first, in one cooperative launch.
//   k_bmax                  largest distance of a cell's particles from its
//                           centre of mass (FP64, on the particles an FP32
//                           bound leaves), or the SPH radius bound (FP32);
//                           chunks of particles, atomic max.
//   k_records               sources, quadrupoles and walk records of the cells,
//                           first particle of every group (maximal cells with
//                           at most n_crit particles; larger leaves in chunks).
//   k_group_sums / k_group_write  the groups in tree order.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>
#include <cstring>

#include "../common.h"
#include "../treegeom.h"

using namespace otoo;

namespace {

constexpr unsigned kFull = 0xffffffffu;
constexpr int kLvThreads = 256;  // cells: threads per block
constexpr int kLvWarps = kLvThreads / 32;
constexpr int kLvTile = 2048;    // particles per block, in contiguous runs per warp
constexpr int kLv = kLevels + 1;  // levels 0 .. 21
constexpr int kBmaxChunk = 2048;                // particles per b_max work item

// status bits
constexpr uint32_t kTreeBadInput = 1u;   // a non-finite position or a mass <= 0
constexpr uint32_t kTreeBadSort = 2u;    // the sorted order indexed outside the particles
constexpr uint32_t kTreeStuck = 4u;      // a wait between blocks ran into its limit

struct Geom {
    double lo[3], S, h, scale;
};

// What one build keeps in one place on the device: zeroed before the first
// kernel, copied to the host once after the last (kernels read the counts of
// the cells and groups here, so that nothing waits for the host in between).
struct Head {
    Geom g;
    int64_t cells, groups;        // totals (cells: also when they exceed the capacity)
    int32_t lev[kLevels + 4];     // first cell of each level; lev[22]: the number of cells
    int32_t pcount[kLevels + 1];  // parents per level
    uint32_t status, stop;        // error bits; more cells than the capacity
    uint32_t bar, done;           // arrivals: grid barrier of k_parents, blocks of k_bbox
    uint32_t extra;               // k_bmax's work items of the larger cells
};

__device__ __forceinline__ long long dkey(double x)
{
    const long long b = __double_as_longlong(x);
    return b ^ ((b >> 63) & 0x7fffffffffffffffLL);
}
__device__ __forceinline__ double dval(long long k) { return __longlong_as_double(k ^ ((k >> 63) & 0x7fffffffffffffffLL)); }

// ---- bounding box ------------------------------------------------------------

__global__ void __launch_bounds__(256) k_bbox(const double* __restrict__ pos, const float* __restrict__ mass, int64_t n,
                                              long long* __restrict__ part, Head* __restrict__ head)
{
    long long lo[3], hi[3];
    for (int a = 0; a < 3; ++a) lo[a] = 0x7fffffffffffffffLL, hi[a] = -lo[a] - 1;
    bool bad = false;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        for (int a = 0; a < 3; ++a) {
            const double x = pos[3 * i + a];
            bad |= !isfinite(x);
            const long long k = dkey(x);
            lo[a] = k < lo[a] ? k : lo[a];
            hi[a] = k > hi[a] ? k : hi[a];
        }
        const float m = mass[i];
        bad |= !(m > 0.0f) || !isfinite(m);
    }
    if (bad) atomicOr(&head->status, kTreeBadInput);
    __shared__ long long s[6][8];
    __shared__ bool last;
    for (int a = 0; a < 3; ++a) {
        for (int o = 16; o > 0; o >>= 1) {
            const long long t0 = __shfl_xor_sync(kFull, lo[a], o), t1 = __shfl_xor_sync(kFull, hi[a], o);
            lo[a] = t0 < lo[a] ? t0 : lo[a];
            hi[a] = t1 > hi[a] ? t1 : hi[a];
        }
    }
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (lane == 0)
        for (int a = 0; a < 3; ++a) s[a][w] = lo[a], s[3 + a][w] = hi[a];
    __syncthreads();
    if (threadIdx.x < 6) {
        long long v = s[threadIdx.x][0];
        for (int k = 1; k < (int)(blockDim.x >> 5); ++k) {
            const long long t = s[threadIdx.x][k];
            v = threadIdx.x < 3 ? (t < v ? t : v) : (t > v ? t : v);
        }
        part[6 * blockIdx.x + threadIdx.x] = v;
        __threadfence();
    }
    __syncthreads();
    // the block that finishes last folds the partials and sets the root cube
    if (threadIdx.x == 0) last = atomicAdd(&head->done, 1u) == gridDim.x - 1;
    __syncthreads();
    if (!last) return;
    __threadfence();
    for (int a = 0; a < 3; ++a) lo[a] = 0x7fffffffffffffffLL, hi[a] = -lo[a] - 1;
    for (int b = threadIdx.x; b < (int)gridDim.x; b += blockDim.x)
        for (int a = 0; a < 3; ++a) {
            const long long l = __ldcg(part + 6 * b + a), h = __ldcg(part + 6 * b + 3 + a);
            lo[a] = l < lo[a] ? l : lo[a];
            hi[a] = h > hi[a] ? h : hi[a];
        }
    for (int a = 0; a < 3; ++a)
        for (int o = 16; o > 0; o >>= 1) {
            const long long t0 = __shfl_xor_sync(kFull, lo[a], o), t1 = __shfl_xor_sync(kFull, hi[a], o);
            lo[a] = t0 < lo[a] ? t0 : lo[a];
            hi[a] = t1 > hi[a] ? t1 : hi[a];
        }
    if (lane == 0)
        for (int a = 0; a < 3; ++a) s[a][w] = lo[a], s[3 + a][w] = hi[a];
    __syncthreads();
    if (threadIdx.x != 0) return;
    for (int a = 0; a < 3; ++a) {
        lo[a] = s[a][0], hi[a] = s[3 + a][0];
        for (int k = 1; k < (int)(blockDim.x >> 5); ++k) {
            lo[a] = s[a][k] < lo[a] ? s[a][k] : lo[a];
            hi[a] = s[3 + a][k] > hi[a] ? s[3 + a][k] : hi[a];
        }
    }
    Geom* g = &head->g;
    double mn[3], mx[3];
    for (int a = 0; a < 3; ++a) mn[a] = dval(lo[a]), mx[a] = dval(hi[a]);
    root_cube(mn, mx, g->lo, &g->S, &g->h);
    g->scale = ddiv(kGrid, g->S);
}

// ---- keys ---------------------------------------------------------------------

// Bound by the FP64 pipe while floor, clamp and conversion ran there (seven FP64
// operations per axis); two are left: N = 2^23 294 -> 224 us, 2^20 41 -> 33 us, now
// by the key's integer operations.
// One key per particle, and the counts of all eight digits of all keys
// (ghist[pass][digit], zero before the launch) that the sort's passes start
// from: shared-memory counts per block (increments of one address by a whole
// warp count as one), one global atomic per block and digit present.
__global__ void __launch_bounds__(256) k_keys(const double* __restrict__ pos, int64_t n, const Geom* __restrict__ g,
                                              uint64_t* __restrict__ keys, int32_t* __restrict__ ghist)
{
    __shared__ int32_t h[8 * 256];
    for (int j = threadIdx.x; j < 8 * 256; j += 256) h[j] = 0;
    __syncthreads();
    for (int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x; i < n; i += (int64_t)gridDim.x * 256) {
        const uint32_t x = quantize(pos[3 * i], g->lo[0], g->scale);
        const uint32_t y = quantize(pos[3 * i + 1], g->lo[1], g->scale);
        const uint32_t z = quantize(pos[3 * i + 2], g->lo[2], g->scale);
        const uint64_t k = hilbert_key(x, y, z);
        keys[i] = k;
#pragma unroll
        for (int p = 0; p < 8; ++p) atomicAdd(&h[256 * p + (int)((k >> (8 * p)) & 255u)], 1);
    }
    __syncthreads();
    for (int j = threadIdx.x; j < 8 * 256; j += 256)
        if (h[j]) atomicAdd(ghist + j, h[j]);
}

// ---- stable LSD radix sort ----------------------------------------------------
// Eight passes of eight bits over (key, index), one launch each (Adinets and
// Merrill, "Onesweep", 2022, after Merrill and Garland's decoupled look-back,
// 2016).  A tile of 4096 keys ranks its keys by digit in input order (warp
// ballots of the digit's bits and per-warp running counts: stable), publishes its count of every
// digit, and finds how many keys of each digit precede it by walking back over
// the earlier tiles' published words (an aggregate, or a whole prefix that
// ends the walk), one digit per thread.  Tiles take their number from a
// ticket, so a tile only waits for tiles that already run.  The tile is staged
// in digit order in shared memory and each digit's run goes to consecutive
// addresses.  A pass reads and writes every pair once (24 bytes per key) and
// is bound by its barriers and ranking at large n (2.6 TB/s; the warp match
// instruction in place of the ballots made it a third slower), by latency at small n.
// Sums of launches under ncu, against the form before (counts, a scan and a
// scatter per pass over tiles of 2048 keys, 40 launches): N = 4096 33 against
// 150 us (one tile, one launch), 100003 83 against 212, 2^20 138 against 293,
// 2^23 0.63 against 1.23 ms.
// Every wait is bounded; a tile that gives up sets the status bit (the others
// then stop waiting too) and its writes stay inside the arrays.

constexpr int kSortThreads = 512;
constexpr int kSortItems = 8;
constexpr int kSortWarps = kSortThreads / 32;
constexpr int kSortTile = kSortThreads * kSortItems;
constexpr uint32_t kSortAgg = 1u << 30, kSortPre = 2u << 30, kSortVal = kSortAgg - 1u;  // counts below 2^30

struct SortShared {
    uint64_t key[kSortTile];
    uint32_t val[kSortTile];
    int32_t wcount[kSortWarps][256];
    int32_t dstart[256], gstart[256];
    int32_t wsum[2][8];
    int32_t tile;
};

// Ranks the tile's keys (warp w owns a contiguous run) and fills dstart; each
// thread gets the tile position of its keys and thread d < 256 the tile's
// count of digit d.
__device__ __forceinline__ int32_t sort_rank(SortShared& sh, const uint64_t key[kSortItems], int64_t left, int shift,
                                             int32_t lp[kSortItems])
{
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const unsigned lt = (1u << lane) - 1u;
    for (int d = lane; d < 256; d += 32) sh.wcount[w][d] = 0;
    __syncwarp();
#pragma unroll
    for (int r = 0; r < kSortItems; ++r) {
        const bool ok = w * 32 * kSortItems + r * 32 + lane < left;
        const int d = ok ? (int)((key[r] >> shift) & 255u) : 256;
        unsigned peers = __ballot_sync(kFull, ok);
        if (!ok) peers = ~peers;
#pragma unroll
        for (int b = 0; b < 8; ++b) {
            const bool one = (d >> b) & 1;
            const unsigned m = __ballot_sync(kFull, one);
            peers &= one ? m : ~m;
        }
        const int lead = __ffs(peers) - 1;
        int32_t before = 0;
        if (ok && lane == lead) {
            before = sh.wcount[w][d];
            sh.wcount[w][d] = before + __popc(peers);
        }
        __syncwarp();
        lp[r] = __shfl_sync(kFull, before, lead) + __popc(peers & lt);
    }
    __syncthreads();
    int32_t cnt = 0, incl = 0;
    if (threadIdx.x < 256) {
        for (int k = 0; k < kSortWarps; ++k) {
            const int32_t c = sh.wcount[k][threadIdx.x];
            sh.wcount[k][threadIdx.x] = cnt;
            cnt += c;
        }
        incl = cnt;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int32_t t = __shfl_up_sync(kFull, incl, o);
            if (lane >= o) incl += t;
        }
        if (lane == 31) sh.wsum[0][w] = incl;
    }
    __syncthreads();
    if (threadIdx.x < 256) {
        int32_t e = incl - cnt;
        for (int k = 0; k < w; ++k) e += sh.wsum[0][k];
        sh.dstart[threadIdx.x] = e;
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < kSortItems; ++r) {
        const bool ok = w * 32 * kSortItems + r * 32 + lane < left;
        if (ok) {
            const int d = (int)((key[r] >> shift) & 255u);
            lp[r] += sh.wcount[w][d] + sh.dstart[d];
        }
    }
    return cnt;
}

// ghist: this pass's digit counts; ticket: this pass's tile counter (zero);
// look: this pass's published words (zero), look_next: the next pass's, zeroed
// here (the pass before this one is done with them).  vin NULL: the index
// itself (first pass).
__global__ void __launch_bounds__(kSortThreads, 3) k_sort_pass(const uint64_t* __restrict__ kin,
                                                             const uint32_t* __restrict__ vin, int64_t n, int shift,
                                                             const int32_t* __restrict__ ghist,
                                                             uint32_t* __restrict__ ticket,
                                                             uint32_t* __restrict__ look,
                                                             uint32_t* __restrict__ look_next,
                                                             uint64_t* __restrict__ kout,
                                                             uint32_t* __restrict__ vout,
                                                             uint32_t* __restrict__ status)
{
    extern __shared__ __align__(16) unsigned char sort_smem[];
    SortShared& sh = *reinterpret_cast<SortShared*>(sort_smem);
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    if (threadIdx.x == 0) sh.tile = (int32_t)atomicAdd(ticket, 1u);
    __syncthreads();
    const int32_t tile = sh.tile;
    const int64_t b0 = (int64_t)tile * kSortTile;
    const int64_t left = n - b0;
    uint64_t key[kSortItems];
    int32_t lp[kSortItems];
#pragma unroll
    for (int r = 0; r < kSortItems; ++r) {
        const int q = w * 32 * kSortItems + r * 32 + lane;
        key[r] = q < left ? kin[b0 + q] : 0;
    }
    const int32_t cnt = sort_rank(sh, key, left, shift, lp);
    const int d = threadIdx.x;
    volatile uint32_t* my = look + (int64_t)tile * 256;
    if (d < 256) {
        my[d] = (tile == 0 ? kSortPre : kSortAgg) | (uint32_t)cnt;
        look_next[(int64_t)tile * 256 + d] = 0u;
    }
    // the tile in digit order, while the look-back's words arrive
#pragma unroll
    for (int r = 0; r < kSortItems; ++r) {
        const int q = w * 32 * kSortItems + r * 32 + lane;
        if (q < left) {
            sh.key[lp[r]] = key[r];
            sh.val[lp[r]] = vin ? vin[b0 + q] : (uint32_t)(b0 + q);
        }
    }
    if (d < 256) {
        // keys of smaller digits, then keys of this digit in earlier tiles
        const int32_t gh = ghist[d];
        int32_t incl = gh;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int32_t t = __shfl_up_sync(kFull, incl, o);
            if (lane >= o) incl += t;
        }
        if (lane == 31) sh.wsum[1][w] = incl;
        uint32_t before = 0;
        bool done = tile == 0;
        // eight earlier tiles' words at a time, so that the walk does not wait
        // for one load after another
        for (int32_t t = tile - 1; !done;) {
            uint32_t v[8];
#pragma unroll
            for (int k = 0; k < 8; ++k)
                v[k] = t - k >= 0 ? *(const volatile uint32_t*)(look + (int64_t)(t - k) * 256 + d) : kSortPre;
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                if (done) continue;
                for (int spin = 0; v[k] < kSortAgg; ++spin) {
                    if (spin >= (1 << 20) || ((spin & 255) == 255 && (*(volatile uint32_t*)status & kTreeStuck))) {
                        atomicOr(status, kTreeStuck);
                        v[k] = kSortPre;
                        break;
                    }
                    v[k] = *(const volatile uint32_t*)(look + (int64_t)(t - k) * 256 + d);
                }
                before += v[k] & kSortVal;
                done = v[k] >= kSortPre;
            }
            t -= 8;
        }
        if (tile > 0) my[d] = kSortPre | ((before + (uint32_t)cnt) & kSortVal);
        sh.gstart[d] = incl - gh + (int32_t)before;
    }
    __syncthreads();
    if (d < 256) {
        int32_t e = 0;
        for (int k = 0; k < w; ++k) e += sh.wsum[1][k];
        sh.gstart[d] += e - sh.dstart[d];
    }
    __syncthreads();
    const int nvalid = (int)(left < kSortTile ? left : kSortTile);
    for (int j = threadIdx.x; j < nvalid; j += kSortThreads) {
        const uint64_t k = sh.key[j];
        const int64_t gp = (int64_t)sh.gstart[(int)((k >> shift) & 255u)] + j;
        if (gp >= 0 && gp < n) {  // (always, unless a wait gave up)
            kout[gp] = k;
            vout[gp] = sh.val[j];
        }
    }
}

// The whole sort of at most one tile: all passes in one block.
__global__ void __launch_bounds__(kSortThreads) k_sort_tile(const uint64_t* __restrict__ kin, int64_t n,
                                                             uint64_t* __restrict__ kout, uint32_t* __restrict__ vout)
{
    extern __shared__ __align__(16) unsigned char sort_smem[];
    SortShared& sh = *reinterpret_cast<SortShared*>(sort_smem);
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    uint64_t key[kSortItems];
    uint32_t val[kSortItems];
    int32_t lp[kSortItems];
#pragma unroll
    for (int r = 0; r < kSortItems; ++r) {
        const int q = w * 32 * kSortItems + r * 32 + lane;
        key[r] = q < n ? kin[q] : 0;
        val[r] = (uint32_t)q;
    }
    for (int shift = 0;; shift += 8) {
        sort_rank(sh, key, n, shift, lp);
        if (shift == 56) break;
        // (every thread has read its digits' starts: dstart and wcount are
        // rewritten only after the barriers below)
#pragma unroll
        for (int r = 0; r < kSortItems; ++r)
            if (w * 32 * kSortItems + r * 32 + lane < n) sh.key[lp[r]] = key[r], sh.val[lp[r]] = val[r];
        __syncthreads();
#pragma unroll
        for (int r = 0; r < kSortItems; ++r) {
            const int q = w * 32 * kSortItems + r * 32 + lane;
            if (q < n) key[r] = sh.key[q], val[r] = sh.val[q];
        }
        __syncthreads();
    }
#pragma unroll
    for (int r = 0; r < kSortItems; ++r)
        if (w * 32 * kSortItems + r * 32 + lane < n) kout[lp[r]] = key[r], vout[lp[r]] = val[r];
}

// ---- tree order ------------------------------------------------------------------

// (The grid coordinates of a cell's first particle, which the records need, are
// worked out there; one triple per particle here cost 282 us for 250 at N = 2^23.)
__global__ void k_permute(const double* __restrict__ pos, const float* __restrict__ mass,
                          const uint32_t* __restrict__ order, int64_t n, otoo_src* __restrict__ src, int64_t* __restrict__ perm, uint32_t* __restrict__ status)
{
    const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n) return;
    const int64_t i = order[k];
    if (i >= n) {  // the sort is a permutation; this only guards the reads
        atomicOr(status, kTreeBadSort);
        return;
    }
    otoo_src s;
    s.x = pos[3 * i];
    s.y = pos[3 * i + 1];
    s.z = pos[3 * i + 2];
    s.m = mass[i];
    s.pad = 0;
    src[k] = s;
    perm[k] = i;
}

// ---- cells, one level at a time ---------------------------------------------------

struct Cells {
    int32_t* begin;
    int32_t* end;
    int32_t* level;
    int32_t* parent;
    int32_t* child0;
    int32_t* nchild;
};

// All cells at once from the sorted keys, with no loop over levels.  With
// cd(i, j) the number of leading key digits (levels) that particles i and j
// share, the cell at level L that holds particle b has more than leaf_size
// particles exactly when some window of leaf_size + 1 consecutive particles
// that contains b shares L digits.  So the deepest cell that holds b, its
// leaf, is at level
//   D(b) = min(21, 1 + max over i in [b - leaf_size, b] of cd(i, i + leaf_size))
// (0 when there is no such window), and the cells whose first particle is b
// are those of levels cd(b - 1, b) + 1 .. D(b) (from level 0 for b = 0).
// Cells are numbered by (level, first particle), which keeps a cell's
// children consecutive: a cell's index is the start of its level plus the
// number of cells of that level that start before it.
//
//   k_levels   both levels of every particle and, per tile, how many cells of
//              each level start in it
//   (scan)     counts in (level, tile) order: where each tile's cells of each
//              level go; the last sum is the number of cells
//   k_cells    the cells of a tile, ranked per level by warp ballots
//   k_leaves   children and end of every cell (and the leaves' moments)
//
// Four to six launches, bound by their latency at small N and by the keys and
// cell arrays they read and write at large N; expanding one level after
// another took five launches per level for 22 possible levels, most of them
// over few cells.  Device time of the two forms (Plummer, Hernquist at 2^23;
// sums of launches under ncu): N = 4096 0.031 against 0.372 ms, 2^20 0.049
// against 0.501 ms, 2^23 0.19 against 0.73 ms.

constexpr int kLvRounds = kLvTile / kLvThreads;
constexpr int kLvLeaf = 64;           // leaf sizes up to this take the window maximum in shared memory

// Leading digits two keys share (21 for equal keys; bit 63 of a key is 0).
__device__ __forceinline__ int common_digits(uint64_t a, uint64_t b)
{
    const uint64_t x = a ^ b;
    return x ? (__clzll((long long)x) - 1) / 3 : kLevels;
}

// Windows for leaf sizes above kLvLeaf, in global memory, padded in front by
// leaf_size zeros: win[j] = 1 + cd(i, i + leaf) for i = j - leaf in [0, n -
// leaf), else 0; then maxima over runs of 2, 4, ... windows by doubling.
__global__ void k_win_init(const uint64_t* __restrict__ keys, int64_t n, int64_t leaf, uint8_t* __restrict__ win)
{
    const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= n + leaf) return;
    const int64_t i = j - leaf;
    win[j] = i >= 0 && i + leaf < n ? (uint8_t)(1 + common_digits(keys[i], keys[i + leaf])) : (uint8_t)0;
}

__global__ void k_win_double(const uint8_t* __restrict__ in, int64_t len, int64_t step, uint8_t* __restrict__ out)
{
    const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= len) return;
    const uint8_t a = in[j], b = j + step < len ? in[j + step] : (uint8_t)0;
    out[j] = a > b ? a : b;
}

// lv[b] = lo | D << 8, lo the level of the first cell that starts at b (above
// D when none does); hist[L * gridDim.x + blk]: cells of level L that start in
// the tile.  win: NULL for leaf <= kLvLeaf, else the maxima over runs of span
// windows (span the largest power of two <= leaf + 1).
__global__ void __launch_bounds__(kLvThreads) k_levels(const uint64_t* __restrict__ keys, int64_t n, int64_t leaf,
                                                        const uint8_t* __restrict__ win, int64_t span,
                                                        uint16_t* __restrict__ lv, int32_t* __restrict__ hist)
{
    __shared__ uint64_t sk[kLvTile + 2 * kLvLeaf];
    __shared__ uint8_t sw[kLvTile + kLvLeaf];
    __shared__ int32_t wcnt[kLvWarps][kLv];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int64_t t0 = (int64_t)blockIdx.x * kLvTile;
    const int halo = win ? 1 : (int)leaf;  // keys staged before and after the tile
    for (int j = threadIdx.x; j < kLvTile + 2 * halo; j += kLvThreads) {
        const int64_t i = t0 - halo + j;
        sk[j] = i >= 0 && i < n ? keys[i] : 0;
    }
    __syncthreads();
    if (!win) {
        for (int j = threadIdx.x; j < kLvTile + halo; j += kLvThreads) {
            const int64_t i = t0 - halo + j;  // window [i, i + leaf]
            sw[j] = i >= 0 && i + halo < n ? (uint8_t)(1 + common_digits(sk[j], sk[j + halo])) : (uint8_t)0;
        }
        __syncthreads();
    }
    int32_t mine = 0;  // lane L: cells of level L that start in the warp's run
    for (int r = 0; r < kLvRounds; ++r) {
        const int q = w * 32 * kLvRounds + r * 32 + lane;
        const int64_t b = t0 + q;
        int lo = kLv, dp = 0;
        if (b < n) {
            lo = b == 0 ? 0 : common_digits(sk[q + halo - 1], sk[q + halo]) + 1;
            int m = 0;
            if (win) {
                const int m0 = win[b], m1 = win[b + leaf + 1 - span];
                m = m0 > m1 ? m0 : m1;
            } else {
                for (int k = 0; k <= halo; ++k) m = sw[q + k] > m ? sw[q + k] : m;
            }
            dp = m < kLevels ? m : kLevels;
            lv[b] = (uint16_t)(lo | (dp << 8));
        }
        const bool any = lo <= dp && b < n;
        const int l0 = __reduce_min_sync(kFull, any ? lo : kLv), l1 = __reduce_max_sync(kFull, any ? dp : -1);
        for (int L = l0; L <= l1; ++L) {
            const int c = __popc(__ballot_sync(kFull, any && lo <= L && L <= dp));
            if (lane == L) mine += c;
        }
    }
    if (lane < kLv) wcnt[w][lane] = mine;
    __syncthreads();
    if (threadIdx.x < kLv) {
        int32_t c = 0;
        for (int k = 0; k < kLvWarps; ++k) c += wcnt[k][threadIdx.x];
        hist[(int64_t)threadIdx.x * gridDim.x + blockIdx.x] = c;
    }
}

// Writes the cells that start in the tile.  offs: the exclusive scan of
// k_levels' counts, *total their sum; block 0 writes the levels' first cells
// lev[0 .. 22].  More than cap cells, or an error found before (status: a position
// that is not finite would put every particle into one leaf, which one thread sums
// for a second at N = 2^23): nothing is written, so that every later kernel finds no
// cells, and stop is set.
__global__ void __launch_bounds__(kLvThreads) k_cells(int64_t n, const uint16_t* __restrict__ lv,
                                                       const int32_t* __restrict__ offs,
                                                       const int64_t* __restrict__ total, int64_t cap, Cells c,
                                                       int32_t* __restrict__ lev,
                                                       const uint32_t* __restrict__ status,
                                                       uint32_t* __restrict__ stop)
{
    __shared__ int32_t wcnt[kLvWarps][kLv];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const unsigned lt = (1u << lane) - 1u;
    if (*total > cap || *status != 0u) {
        if (blockIdx.x == 0 && threadIdx.x == 0) *stop = 1u;
        return;
    }
    if (blockIdx.x == 0 && threadIdx.x <= kLv)
        lev[threadIdx.x] = threadIdx.x < kLv ? offs[(int64_t)threadIdx.x * gridDim.x] : (int32_t)*total;
    const int64_t t0 = (int64_t)blockIdx.x * kLvTile + (int64_t)w * 32 * kLvRounds;
    uint16_t v[kLvRounds];
    int32_t mine = 0;
#pragma unroll
    for (int r = 0; r < kLvRounds; ++r) {
        const int64_t b = t0 + r * 32 + lane;
        v[r] = b < n ? lv[b] : (uint16_t)kLv;
        const int lo = v[r] & 255, dp = v[r] >> 8;
        const bool any = lo <= dp;
        const int l0 = __reduce_min_sync(kFull, any ? lo : kLv), l1 = __reduce_max_sync(kFull, any ? dp : -1);
        for (int L = l0; L <= l1; ++L) {
            const int k = __popc(__ballot_sync(kFull, any && lo <= L && L <= dp));
            if (lane == L) mine += k;
        }
    }
    if (lane < kLv) wcnt[w][lane] = mine;
    __syncthreads();
    // lane L: index of the next cell of level L
    int32_t next = 0;
    if (lane < kLv) {
        next = offs[(int64_t)lane * gridDim.x + blockIdx.x];
        for (int k = 0; k < w; ++k) next += wcnt[k][lane];
    }
#pragma unroll
    for (int r = 0; r < kLvRounds; ++r) {
        const int64_t b = t0 + r * 32 + lane;
        const int lo = v[r] & 255, dp = v[r] >> 8;
        const bool any = lo <= dp;
        const int l0 = __reduce_min_sync(kFull, any ? lo : kLv), l1 = __reduce_max_sync(kFull, any ? dp : -1);
        int32_t up = 0;    // the last cell of level L - 1 that starts at or before b
        int32_t mine_up = -1;  // the cell of level L - 1 that starts at b
        for (int L = l0 > 0 ? l0 - 1 : 0; L <= l1; ++L) {
            const bool on = any && lo <= L && L <= dp;
            const unsigned m = __ballot_sync(kFull, on);
            const int32_t base = __shfl_sync(kFull, next, L);
            const int32_t id = base + __popc(m & lt);
            if (on) {
                c.begin[id] = (int32_t)b;
                c.level[id] = L;
                c.parent[id] = L == 0 ? -1 : up;
                if (L == dp) c.child0[id] = 0;
                if (mine_up >= 0) c.child0[mine_up] = id;
                mine_up = id;
            }
            up = base + __popc(m & lt) - (on ? 0 : 1);
            if (lane == L) next += __popc(m);
        }
    }
}

// ---- moments ------------------------------------------------------------------------

struct Moments {
    double* m;      // [cap]
    double* com;    // [cap][3]
    double* q;      // [cap][6] central second moment Cxx Cyy Czz Cxy Cxz Cyz
    double* b2;     // [cap]
    unsigned long long* dmax2;  // [cap] bits of the largest squared distance (FP64), or of
                                //   the SPH radius (FP32, zero-extended)
};

// A positive float widened to double by integer operations on its bits (the
// FP64 pipe, which the conversion instruction would occupy, is what bounds
// these kernels); subnormal, infinite and NaN values take the conversion.
__device__ __forceinline__ double widen(float f)
{
    const uint32_t u = __float_as_uint(f);
    if (u - 0x00800000u < 0x7f000000u) return __hiloint2double((int)((u >> 3) + 0x38000000u), (int)(u << 29));
    return (double)f;
}

// Moments of every cell, in one pass over its members (its particles for a
// leaf, its children for a parent): with x0 a member's position (a leaf's
// first particle, a parent's heaviest child's centre of mass) and d = x - x0,
// M = sum m, S1 = sum m d, S2 = sum m d d^T (+ the child's own central second
// moment C_c), then com = x0 + S1 / M and the central second moment C = S2 -
// S1 S1^T / M (the parallel-axis shift to the centre of mass).  S1 S1^T / M =
// M g g^T with g = com - x0, while C holds at least m_0 M / (M - m_0) g g^T
// (the reference member, mass m_0, against the rest), so the subtraction
// loses about log2((M - m_0) / m_0) bits: under 3 for a parent (the heaviest
// of up to 8 children), about log2 of the leaf size for equal masses in a
// leaf.  Stored: m, com, C (Cxx Cyy Czz Cxy Cxz Cyz) and B_2 = tr C; the
// records take the quadrupole Q = 3 C - tr(C) I.  GB300's FP64 pipe (1/76 of
// the FP32 rate) bounds both kernels at large N, latency at small N.

// The end of a cell, and the moments of a leaf (nch = 0) of one particle; returns
// the number of particles of a leaf of several, else 0.
__device__ __forceinline__ int32_t close_cell(int32_t cell, int32_t b, int lvl, int32_t nch,
                                           const uint64_t* __restrict__ keys, int64_t n, int64_t leaf_size,
                                           const otoo_src* __restrict__ src, const Cells& c, const Moments& mo)
{
    const int sh = 3 * (kLevels - lvl);
    const uint64_t pre = keys[b] >> sh;
    int64_t l = nch > 0 ? b + leaf_size : b, hi, step = 1;
    for (hi = l + step; hi < n && (keys[hi] >> sh) == pre; hi = l + step) {
        l = hi;
        step *= 2;
    }
    if (hi > n) hi = n;
    while (hi - l > 1) {
        const int64_t mid = l + ((hi - l) >> 1);
        if ((keys[mid] >> sh) == pre)
            l = mid;
        else
            hi = mid;
    }
    const int32_t e = (int32_t)hi;
    c.end[cell] = e;
    mo.dmax2[cell] = 0ull;
    if (nch > 0) return 0;
    if (e - b == 1) {
        const otoo_src p0 = src[b];
        double* q = mo.q + 6 * (int64_t)cell;
        double* com = mo.com + 3 * (int64_t)cell;
        mo.m[cell] = widen(p0.m);
        com[0] = p0.x, com[1] = p0.y, com[2] = p0.z;
        q[0] = q[1] = q[2] = q[3] = q[4] = q[5] = 0.0;
        mo.b2[cell] = 0.0;
        return 0;
    }
    return e - b;
}

// The moments of a leaf of several particles [b, e).
__device__ __forceinline__ void leaf_moments(int32_t cell, int32_t b, int32_t e, const otoo_src* __restrict__ src,
                                             const Moments& mo)
{
    const otoo_src p0 = src[b];
    double m = widen(p0.m);
    double* q = mo.q + 6 * (int64_t)cell;
    double* com = mo.com + 3 * (int64_t)cell;
    double s1[3] = {0, 0, 0}, s2[6] = {0, 0, 0, 0, 0, 0};
#pragma unroll 1
    for (int32_t i = b + 1; i < e; ++i) {
        const otoo_src p = src[i];
        const double mi = widen(p.m);
        const double dx = p.x - p0.x, dy = p.y - p0.y, dz = p.z - p0.z;
        const double mx = mi * dx, my = mi * dy, mz = mi * dz;
        m += mi;
        s1[0] += mx, s1[1] += my, s1[2] += mz;
        s2[0] = fma(mx, dx, s2[0]), s2[1] = fma(my, dy, s2[1]), s2[2] = fma(mz, dz, s2[2]);
        s2[3] = fma(mx, dy, s2[3]), s2[4] = fma(mx, dz, s2[4]), s2[5] = fma(my, dz, s2[5]);
    }
    const double inv = 1.0 / m;
    const double gx = s1[0] * inv, gy = s1[1] * inv, gz = s1[2] * inv;  // com - x0
    mo.m[cell] = m;
    com[0] = p0.x + gx;
    com[1] = p0.y + gy;
    com[2] = p0.z + gz;
    const double cxx = fma(-s1[0], gx, s2[0]), cyy = fma(-s1[1], gy, s2[1]), czz = fma(-s1[2], gz, s2[2]);
    q[0] = cxx, q[1] = cyy, q[2] = czz;
    q[3] = fma(-s1[0], gy, s2[3]), q[4] = fma(-s1[0], gz, s2[4]), q[5] = fma(-s1[1], gz, s2[5]);
    mo.b2[cell] = cxx + cyy + czz;
}

// One thread per cell: the cell's links (children: the consecutive cells from
// child0 on that name it as their parent; end: the first particle past it, by
// a galloping search over the keys' leading digits; a cell that splits holds
// at least leaf_size + 1 particles), and for a leaf its moments.  The
// reference particle's own terms are zero and are left out (a leaf of leaf size
// 8 holds 2.7 particles on average).  An FP64 instruction costs its warp the
// same for one lane as for 32, so the block sorts its leaves of several
// particles by their number (counting sort in shared memory) and a warp takes
// leaves of about one size.  Bound by the FP64 pipe: N = 2^20 96 -> 64 us, 2^23
// with leaves of 16 635 -> 440 us against a thread per cell in cell order (16.6 of
// 32 lanes in an instruction, N = 2^22); 4096 17 -> 18 us, links included.
constexpr int kLeafThreads = 256;  // cells per block at most

__global__ void __launch_bounds__(kLeafThreads) k_leaves(const int32_t* __restrict__ lev,
                                                         const uint64_t* __restrict__ keys, int64_t n,
                                                         int64_t leaf_size, const otoo_src* __restrict__ src, Cells c,
                                                         Moments mo, int32_t* __restrict__ plist,
                                                         int32_t* __restrict__ pcount)
{
    constexpr int kBins = 64;  // leaves of 64 particles and more first, of 2 last
    __shared__ int32_t bins[kBins], total;
    __shared__ int32_t leaf[kLeafThreads][3];  // cell, first particle, one past the last
    const int32_t n_cell = lev[kLv];
    const int lane = threadIdx.x & 31;
    for (int64_t w0 = (int64_t)blockIdx.x * blockDim.x; w0 < n_cell; w0 += (int64_t)gridDim.x * blockDim.x) {
        for (int j = threadIdx.x; j < kBins; j += blockDim.x) bins[j] = 0;
        __syncthreads();
        const bool in = w0 + threadIdx.x < n_cell;
        const int32_t cell = (int32_t)(in ? w0 + threadIdx.x : w0);
        int32_t k = 0;
        const int32_t c0 = in ? c.child0[cell] : 0;
        if (c0 > 0)
            while (k < 8 && c0 + k < n_cell && c.parent[c0 + k] == cell) ++k;
        const int lvl = c.level[cell];
        __syncwarp();
        // parents into their level's list, one atomic per warp and level (a
        // warp's cells are nearly always of one level)
        const unsigned peers = __match_any_sync(kFull, k > 0 ? lvl : -1 - lane);
        const int lead = __ffs(peers) - 1;
        int32_t at = 0;
        if (k > 0 && lane == lead) at = atomicAdd(pcount + lvl, __popc(peers));
        at = __shfl_sync(kFull, at, lead);
        if (k > 0) plist[lev[lvl] + at + __popc(peers & ((1u << lane) - 1u))] = cell;
        int32_t np = 0, rank = 0, b = 0;
        if (in) {
            c.nchild[cell] = k;
            b = c.begin[cell];
            np = close_cell(cell, b, lvl, k, keys, n, leaf_size, src, c, mo);
        }
        const int bin = np < kBins ? kBins - np : 0;
        if (np > 0) rank = atomicAdd(bins + bin, 1);
        __syncthreads();
        if (threadIdx.x < 32) {
            const int32_t n0 = bins[2 * lane], n1 = bins[2 * lane + 1];
            int32_t incl = n0 + n1;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int32_t t = __shfl_up_sync(kFull, incl, o);
                if (lane >= o) incl += t;
            }
            bins[2 * lane] = incl - n0 - n1;
            bins[2 * lane + 1] = incl - n1;
            if (lane == 31) total = incl;
        }
        __syncthreads();
        if (np > 0) {
            int32_t* q = leaf[bins[bin] + rank];
            q[0] = cell, q[1] = b, q[2] = b + np;
        }
        __syncthreads();
        if ((int)threadIdx.x < total) {
            const int32_t* q = leaf[threadIdx.x];
            leaf_moments(q[0], q[1], q[2], src, mo);
        }
        __syncthreads();
    }
}

// A grid-wide barrier of a cooperative launch: bar counts arrivals (zero
// before the launch).  The wait is bounded (about a second); a block that
// gives up sets the status bit and the others see it, so that the kernel ends
// in any case.  False: leave the kernel.
__device__ __forceinline__ bool grid_wait(uint32_t* bar, uint32_t round, uint32_t* status)
{
    __shared__ int ok;
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        atomicAdd(bar, 1u);
        const uint32_t want = round * gridDim.x;
        int good = 0;
        for (int spin = 0; spin < (1 << 22); ++spin) {
            if (*(volatile uint32_t*)bar >= want) {
                good = 1;
                break;
            }
            if (spin > 64) __nanosleep(100);
            if ((spin & 1023) == 1023 && (*(volatile uint32_t*)status & kTreeStuck)) break;
        }
        if (!good) atomicOr(status, kTreeStuck);
        __threadfence();
        ok = good;
    }
    __syncthreads();
    return ok != 0;
}

// One parent per eight lanes (lane j of eight holds child j of ch0, ch0 + 1,
// ...; nch = 0: none, the lanes only take part in the shuffles).
__device__ __forceinline__ void combine_children(int32_t cell, int nch, int32_t ch0, int j, const Moments& mo)
{
    const bool on = j < nch;
    const int64_t ch = on ? ch0 + j : 0;
    double v[10], x[3] = {0, 0, 0};
#pragma unroll
    for (int q = 0; q < 10; ++q) v[q] = 0.0;
    if (on) {
        v[0] = __ldcg(mo.m + ch);
#pragma unroll
        for (int q = 0; q < 3; ++q) x[q] = __ldcg(mo.com + 3 * (int64_t)ch + q);
#pragma unroll
        for (int q = 0; q < 6; ++q) v[4 + q] = __ldcg(mo.q + 6 * (int64_t)ch + q);
    }
    // the heaviest child, the first of equals (positive doubles order
    // like their bits)
    unsigned long long mb = (unsigned long long)__double_as_longlong(v[0]);
    int jh = j;
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) {
        const unsigned long long mo_ = __shfl_xor_sync(kFull, mb, o, 8);
        const int jo = __shfl_xor_sync(kFull, jh, o, 8);
        if (mo_ > mb || (mo_ == mb && jo < jh)) mb = mo_, jh = jo;
    }
    double x0[3];
#pragma unroll
    for (int q = 0; q < 3; ++q) x0[q] = __shfl_sync(kFull, x[q], jh, 8);
    if (on) {
        const double dx = x[0] - x0[0], dy = x[1] - x0[1], dz = x[2] - x0[2];
        v[1] = v[0] * dx, v[2] = v[0] * dy, v[3] = v[0] * dz;
        v[4] = fma(v[1], dx, v[4]), v[5] = fma(v[2], dy, v[5]), v[6] = fma(v[3], dz, v[6]);
        v[7] = fma(v[1], dy, v[7]), v[8] = fma(v[1], dz, v[8]), v[9] = fma(v[2], dz, v[9]);
    }
    // lanes with bit 2 clear keep sums 0..4, the others 5..9; then of
    // those five the first three or the last two, then two or one
    double a[5];
    const bool b2 = j & 4, b1 = j & 2, b0 = j & 1;
#pragma unroll
    for (int q = 0; q < 5; ++q) {
        const double got = __shfl_xor_sync(kFull, b2 ? v[q] : v[5 + q], 4, 8);
        a[q] = (b2 ? v[5 + q] : v[q]) + got;
    }
    double d[3];
#pragma unroll
    for (int q = 0; q < 3; ++q) {
        const double hi3 = q < 2 ? a[3 + q] : 0.0;
        const double got = __shfl_xor_sync(kFull, b1 ? a[q] : hi3, 2, 8);
        d[q] = (b1 ? hi3 : a[q]) + got;
    }
    double s[2];
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        const double hi2 = q < 1 ? d[2] : 0.0;
        const double got = __shfl_xor_sync(kFull, b0 ? d[q] : hi2, 1, 8);
        s[q] = (b0 ? hi2 : d[q]) + got;
    }
    // sums now: lane 0: 0, 1; 1: 2; 2: 3, 4; 4: 5, 6; 5: 7; 6: 8, 9
    const double M = __shfl_sync(kFull, s[0], 0, 8);
    double s1[3], g[3], s2[6];
    s1[0] = __shfl_sync(kFull, s[1], 0, 8);
    s1[1] = __shfl_sync(kFull, s[0], 1, 8);
    s1[2] = __shfl_sync(kFull, s[0], 2, 8);
    s2[0] = __shfl_sync(kFull, s[1], 2, 8);
    s2[1] = __shfl_sync(kFull, s[0], 4, 8);
    s2[2] = __shfl_sync(kFull, s[1], 4, 8);
    s2[3] = __shfl_sync(kFull, s[0], 5, 8);
    s2[4] = __shfl_sync(kFull, s[0], 6, 8);
    s2[5] = __shfl_sync(kFull, s[1], 6, 8);
    const double inv = 1.0 / (nch > 0 ? M : 1.0);  // (a zero divisor takes the division's slow path)
#pragma unroll
    for (int q = 0; q < 3; ++q) g[q] = s1[q] * inv;  // com - x0
    // lane 0 .. 5: one entry of C = S2 - S1 g^T; lane 6: M; lanes 0 .. 2 also com
    const double ca = j == 0 || j == 3 || j == 4 ? s1[0] : j == 1 || j == 5 ? s1[1] : s1[2];
    const double cg = j == 0 ? g[0] : j == 1 || j == 3 ? g[1] : g[2];
    double sv = s2[0];
#pragma unroll
    for (int q = 1; q < 6; ++q) sv = j == q ? s2[q] : sv;
    const double cv = fma(-ca, cg, sv);
    const double c1 = __shfl_sync(kFull, cv, 1, 8), c2 = __shfl_sync(kFull, cv, 2, 8);
    if (nch == 0) return;
    if (j < 6) mo.q[6 * (int64_t)cell + j] = cv;
    if (j < 3) {
        const double xr = j == 0 ? x0[0] : j == 1 ? x0[1] : x0[2], gr = j == 0 ? g[0] : j == 1 ? g[1] : g[2];
        mo.com[3 * (int64_t)cell + j] = xr + gr;
    }
    if (j == 6) mo.m[cell] = M;
    if (j == 0) mo.b2[cell] = cv + c1 + c2;
}

// Parents, deepest level first, eight lanes per parent (lane j holds child j):
// the children's loads and products run side by side, then the ten sums are
// halved over the lanes (a lane ends with one or two of them), so four parents
// cost a warp about 40 FP64 instructions in a short chain; one thread per
// parent is a chain of 8 dependent loads and 200 FP64 instructions.  One
// cooperative launch walks the levels: a level of at most kSoloParents parents
// is block 0's alone (block barriers), the others take a grid barrier before
// and after, and each warp has its first parents' links in registers when the
// barrier opens.  40 us at N = 4096, 97 us at 2^20, 0.20 ms at 2^23 (Plummer);
// leaves and parents together 58, 190 and 770 us against 149, 382 and 1056 us
// with one thread per cell and one launch per level, the links not counted
// there.  The line at 64 parents: 16 warps of one SM take them in one round.
// plist: k_leaves' parents of each level, pcount of them from
// the level's first cell on.  mo's arrays are read past L1 (other blocks of
// this launch write them).
constexpr int kSoloParents = 64;

__global__ void __launch_bounds__(512) k_parents(const int32_t* __restrict__ lev, Cells c, Moments mo,
                                                  const int32_t* __restrict__ plist,
                                                  const int32_t* __restrict__ pcount, uint32_t* __restrict__ bar,
                                                  uint32_t* __restrict__ status)
{
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    uint32_t round = 0;
    bool wide_done = false;  // a level shared by all blocks has been summed since the last barrier
    for (int L = kLevels - 1; L >= 0; --L) {
        const int32_t np = pcount[L];
        if (np == 0) continue;
        const bool solo = np <= kSoloParents;
        // neighbouring parents go to different SMs (each has one narrow FP64 pipe)
        const int64_t nwarp = solo ? nw : (int64_t)gridDim.x * nw;
        const int64_t warp = solo ? wid : (int64_t)wid * gridDim.x + blockIdx.x;
        const int32_t* pl = plist + lev[L];
        int64_t k = 4 * warp + (lane >> 3);
        int32_t cell = 0, n = 0, c0 = 0;
        auto links = [&]() {
            cell = k < np ? pl[k] : 0;
            n = k < np ? c.nchild[cell] : 0;
            c0 = k < np ? c.child0[cell] : 0;
        };
        if (!solo || blockIdx.x == 0) links();
        if (wide_done || !solo) {
            if (!grid_wait(bar, ++round, status)) return;
        } else {
            __syncthreads();
        }
        wide_done = !solo;
        if (solo && blockIdx.x != 0) continue;
        for (int64_t w0 = 4 * warp; w0 < np; w0 += 4 * nwarp) {
            combine_children(cell, n, c0, lane & 7, mo);
            k += 4 * nwarp;
            if (w0 + 4 * nwarp < np) links();
        }
    }
}

// FP32 distance |c~ - x~_j| between a cell's rounded centre of mass c~ and a
// rounded particle x~_j (k_bmax), and the particle's rounding bound
// e_j = 2^-23 (|x~| + |y~| + |z~|).
__device__ __forceinline__ float bmax_dist(const float4 cc, const float4 p, float& ej)
{
    const float dx = cc.x - p.x, dy = cc.y - p.y, dz = cc.z - p.z;
    ej = 0x1p-23f * (fabsf(p.x) + fabsf(p.y) + fabsf(p.z));
    return sqrtf(fmaf(dx, dx, fmaf(dy, dy, dz * dz)));
}

// pk[j] = (x_j, y_j, z_j rounded to FP32, h_j or 0) in tree order,
// cf[cell] = (com rounded to FP32, e_c).  Rounding a value v to FP32 moves it
// by at most 2^-24 |v| per coordinate, so |com - x_j| lies within
// e_c + e_j (twice that bound, which also covers rounding in e itself) of
// |com~ - x~_j|, and the FP32 distance errs by a few 2^-24 relative, covered
// by a factor 1 -+ 2^-20.
//
// SPH (sph != 0): an upper bound on the cell's SPH radius, the largest
// |com - x_j| + h_j (Eq. SPH_RAD), in FP32 throughout; dmax2 holds the float
// bits, zero-extended.  The radius can only be larger than the exact one: a
// cell may keep particles that contribute W = 0 but never loses a neighbour.
//
// Absolute MAC: the largest squared distance in FP64, as the host computes
// it; dmax2 holds double bits.  A first FP32 pass finds a lower bound L on
// the largest distance of the lanes' particles; the FP64 distance is then
// taken only for the particles whose FP32 upper bound reaches L.  That set
// holds every particle whose FP64 value could be the largest (their exact
// distances lie within 2^-40 or so of the largest, far inside the bounds'
// margin), so the result is the same bits as the FP64 maximum over all
// particles.
//
// kW lanes (8 or 32) share the particles [i0, i1) of one cell; the lanes of a
// warp run the same number of rounds (trips, uniform).  SPH: returns, in each of
// the kW lanes, the largest of their particles' radius bounds.
template <int kW>
__device__ __forceinline__ float bmax_sph(int i0, int i1, int trips, int j, float4 cc, const float4* __restrict__ pk)
{
    float hi = 0.f;
#pragma unroll 4
    for (int t = 0; t < trips; ++t) {
        const int i = i0 + t * kW + j;
        if (i < i1) {
            const float4 p = pk[i];
            float ej;
            const float d = bmax_dist(cc, p, ej);
            hi = fmaxf(hi, d + (p.w + ej));
        }
    }
    __syncwarp();
#pragma unroll
    for (int o = kW / 2; o > 0; o >>= 1) hi = fmaxf(hi, __shfl_xor_sync(kFull, hi, o));
    return (hi + cc.w) * (1.0f + 0x1p-20f);
}

// A distance within 2^-22 (the margins allow 2^-20).
__device__ __forceinline__ float bmax_dist_approx(const float4 cc, const float4 p, float& ej)
{
    const float dx = cc.x - p.x, dy = cc.y - p.y, dz = cc.z - p.z;
    ej = 0x1p-23f * (fabsf(p.x) + fabsf(p.y) + fabsf(p.z));
    float d;
    asm("sqrt.approx.f32 %0, %1;" : "=f"(d) : "f"(fmaf(dx, dx, fmaf(dy, dy, dz * dz))));
    return d;
}

// Absolute MAC, first pass: the kW lanes' largest lower bound lo, and of the
// lane's own particles the largest upper bound u1 with its particle, and the
// second largest u2 (infinite when a bound is not finite).
struct BmaxLane {
    float lo, u1, u2;
    int i1;
};
template <int kW>
__device__ __forceinline__ BmaxLane bmax_scan(int i0, int i1, int trips, int j, float4 cc, const float4* __restrict__ pk)
{
    BmaxLane r = {0.f, -1.f, -1.f, i0};
#pragma unroll 4
    for (int t = 0; t < trips; ++t) {
        const int i = i0 + t * kW + j;
        if (i < i1) {
            float ej;
            const float d = bmax_dist_approx(cc, pk[i], ej);
            const float e2 = 2.0f * (ej + cc.w), u = (d + e2) * (1.0f + 0x1p-20f);
            r.lo = fmaxf(r.lo, d * (1.0f - 0x1p-20f) - e2);
            r.u2 = u <= 3.0e38f ? fmaxf(r.u2, fminf(r.u1, u)) : __int_as_float(0x7f800000);
            r.i1 = u > r.u1 ? i : r.i1;
            r.u1 = fmaxf(r.u1, u);
        }
    }
    __syncwarp();
#pragma unroll
    for (int o = kW / 2; o > 0; o >>= 1) r.lo = fmaxf(r.lo, __shfl_xor_sync(kFull, r.lo, o));
    return r;
}

// The (cell, particle) pairs whose FP64 distance is to be taken, a queue per
// warp: an FP64 instruction costs the warp the same for one pair as for 32, so
// the pairs of several cells are taken together.
struct BmaxQueue {
    int2 q[64];
};

__device__ __forceinline__ void bmax_flush(const BmaxQueue& s, int n, int lane, const double* __restrict__ com,
                                           const otoo_src* __restrict__ src, unsigned long long* __restrict__ dmax2)
{
    __syncwarp();
    if (lane < n) {
        const int2 c = s.q[lane];
        const otoo_src p = src[c.y];
        const double* x = com + 3 * (int64_t)c.x;
        const double dx = x[0] - p.x, dy = x[1] - p.y, dz = x[2] - p.z;
        atomicMax(dmax2 + c.x, (unsigned long long)__double_as_longlong(dx * dx + dy * dy + dz * dz));
    }
    __syncwarp();
}

__device__ __forceinline__ void bmax_push(BmaxQueue& s, int& held, bool near, int32_t cell, int i, int lane,
                                          const double* __restrict__ com, const otoo_src* __restrict__ src,
                                          unsigned long long* __restrict__ dmax2)
{
    const unsigned m = __ballot_sync(kFull, near);
    if (near) s.q[held + __popc(m & ((1u << lane) - 1u))] = make_int2(cell, i);
    held += __popc(m);
    if (held >= 32) {
        bmax_flush(s, 32, lane, com, src, dmax2);
        int2 rest = make_int2(0, 0);
        if (lane < held - 32) rest = s.q[32 + lane];
        __syncwarp();
        if (lane < held - 32) s.q[lane] = rest;
        held -= 32;
    }
}

// Absolute MAC, the candidates of a cell: nearly always a lane has at most one, the
// one that the first pass kept; if some lane may have a second, all particles
// are gone through again.
template <int kW>
__device__ __forceinline__ void bmax_candidates(BmaxQueue& s, int& held, int32_t cell, const BmaxLane& r, int i0, int i1,
                                                int trips, int j, int lane, float4 cc, const double* __restrict__ com,
                                                const otoo_src* __restrict__ src, const float4* __restrict__ pk,
                                                unsigned long long* __restrict__ dmax2)
{
    if (!__any_sync(kFull, r.u2 >= r.lo && trips > 0)) {
        bmax_push(s, held, r.u1 >= r.lo, cell, r.i1, lane, com, src, dmax2);
        return;
    }
    for (int t = 0; t < trips; ++t) {
        const int i = i0 + t * kW + j;
        bool near = false;
        if (i < i1) {
            float ej;
            const float d = bmax_dist_approx(cc, pk[i], ej);
            near = !((d + 2.0f * (ej + cc.w)) * (1.0f + 0x1p-20f) < r.lo);  // NaN bounds count as candidates
        }
        bmax_push(s, held, near, cell, i, lane, com, src, dmax2);
    }
}

// Cells of up to kBmaxSmall particles, four per warp (eight lanes each); larger
// cells as the work items items[0, head->extra) = (cell, chunk of kBmaxChunk
// particles), one warp each.  The results fold into dmax2 (zero before) by an
// atomic max on the bits (non-negative floating-point values order like their
// bit patterns).  Bound by the loads of the particles' FP32 records and the
// instructions around them: one pass over them instead of two, approximate square
// roots inside the bounds' margins and 32-bit indices took the absolute MAC's
// radii at N = 2^23 (leaves of 16) from 841 to 465 us and the SPH radii at 2^20 from
// 64 to 53 us; the FP64 distances, in rounds of 32, no longer count.
constexpr int kBmaxSmall = 64;

__global__ void __launch_bounds__(256) k_bmax(const Head* __restrict__ head, const int2* __restrict__ items,
                                              const otoo_src* __restrict__ src, const float4* __restrict__ pk,
                                              const float4* __restrict__ cf, Cells c, Moments mo, int sph)
{
    __shared__ BmaxQueue queue[8];
    BmaxQueue& s = queue[threadIdx.x >> 5];
    int held = 0;  // (uniform)
    const int lane = threadIdx.x & 31;
    const int64_t nwarp = ((int64_t)gridDim.x * blockDim.x) >> 5;
    const int32_t n_cell = head->lev[kLv];
    const int64_t nbig = head->extra, n_units = nbig + ((int64_t)n_cell + 3) / 4;
    for (int64_t w = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; w < n_units; w += nwarp) {
        if (w < nbig) {
            const int2 it = items[w];
            const int i0 = c.begin[it.x] + it.y * kBmaxChunk, e = c.end[it.x];
            const int i1 = min(i0 + kBmaxChunk, e), trips = (i1 - i0 + 31) / 32;
            const float4 cc = cf[it.x];
            if (sph) {
                const float h = bmax_sph<32>(i0, i1, trips, lane, cc, pk);
                if (lane == 0) atomicMax(mo.dmax2 + it.x, (unsigned long long)__float_as_uint(h));
            } else {
                const BmaxLane r = bmax_scan<32>(i0, i1, trips, lane, cc, pk);
                bmax_candidates<32>(s, held, it.x, r, i0, i1, trips, lane, lane, cc, mo.com, src, pk, mo.dmax2);
            }
        } else {
            const int64_t k = 4 * (w - nbig) + (lane >> 3);
            const int32_t cell = (int32_t)(k < n_cell ? k : n_cell - 1);
            const int32_t b = c.begin[cell], e = c.end[cell];
            // a single particle is its own centre of mass: distance 0
            const bool on = k < n_cell && e - b <= kBmaxSmall && (sph || e - b > 1);
            const int trips = __reduce_max_sync(kFull, on ? (e - b + 7) / 8 : 0);
            const int i1 = on ? e : b;
            const float4 cc = cf[cell];
            if (sph) {
                const float h = bmax_sph<8>(b, i1, trips, lane & 7, cc, pk);
                if (on && (lane & 7) == 0) mo.dmax2[cell] = (unsigned long long)__float_as_uint(h);
            } else {
                const BmaxLane r = bmax_scan<8>(b, i1, trips, lane & 7, cc, pk);
                bmax_candidates<8>(s, held, cell, r, b, i1, trips, lane & 7, lane, cc, mo.com, src, pk, mo.dmax2);
            }
        }
    }
    bmax_flush(s, held, lane, mo.com, src, mo.dmax2);
}

// The work items of the cells of more than kBmaxSmall particles (any order;
// one atomic per warp), and every cell's FP32 centre of mass with its rounding
// bound e_c.
__global__ void __launch_bounds__(128) k_chunks(Head* __restrict__ head, Cells c, const double* __restrict__ com,
                                                int2* __restrict__ items, float4* __restrict__ cf)
{
    const int32_t n_cell = head->lev[kLv];
    const int lane = threadIdx.x & 31;
    for (int64_t w0 = (int64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31); w0 < n_cell;
         w0 += (int64_t)gridDim.x * blockDim.x) {
        const int64_t cell = w0 + lane;
        const bool in = cell < n_cell;
        const int32_t cnt = in ? c.end[cell] - c.begin[cell] : 0;
        const int32_t more = cnt > kBmaxSmall ? (cnt + kBmaxChunk - 1) / kBmaxChunk : 0;
        int32_t incl = more;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int32_t t = __shfl_up_sync(kFull, incl, o);
            if (lane >= o) incl += t;
        }
        uint32_t at = 0;
        const int32_t all = __shfl_sync(kFull, incl, 31);
        if (lane == 0 && all > 0) at = atomicAdd(&head->extra, (uint32_t)all);
        at = __shfl_sync(kFull, at, 0) + (uint32_t)(incl - more);
        for (int32_t k = 0; k < more; ++k) items[at + k] = make_int2((int)cell, k);
        if (in) {
            const float x = (float)com[3 * cell], y = (float)com[3 * cell + 1], z = (float)com[3 * cell + 2];
            cf[cell] = make_float4(x, y, z, 0x1p-23f * (fabsf(x) + fabsf(y) + fabsf(z)));
        }
        __syncwarp();
    }
}

// Tree-order FP32 positions with each particle's SPH radius, or 0 without h
// (k_bmax).
__global__ void k_bpack(int64_t n, const otoo_src* __restrict__ src, const float* __restrict__ h,
                        const int64_t* __restrict__ perm, float4* __restrict__ pk)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const otoo_src p = src[i];
    pk[i] = make_float4((float)p.x, (float)p.y, (float)p.z, h ? h[perm[i]] : 0.0f);
}

// ---- records and groups ----------------------------------------------------------

struct RecArgs {
    int64_t n_part;
    int32_t use_quad, mac, n_crit;
    double delta, m_limit;
};

// Stores a record in 16-byte words (wide: its array starts on a 16-byte boundary).
// Field by field a cell's 224 bytes were some forty stores of 4 and 8 bytes that
// throttled the load/store path: N = 2^20 83 -> 56 us, SPH 76 -> 44 us, 2^23 with the
// absolute MAC's radii 378 -> 363 us.
template <typename T> __device__ __forceinline__ void put_record(T* __restrict__ p, const T& v, bool wide)
{
    static_assert(sizeof(T) % 16 == 0, "record size");
    if (wide) {
        float4 t[sizeof(T) / 16];
        memcpy(t, &v, sizeof(T));
#pragma unroll
        for (int k = 0; k < (int)(sizeof(T) / 16); ++k) reinterpret_cast<float4*>(p)[k] = t[k];
    } else {
        *p = v;
    }
}

// The records of one cell, and the groups that start in it: a group starts at
// the first particle of each maximal cell with at most n_crit particles, and
// every n_crit particles inside a leaf that holds more (one bit per particle
// in bits).
__device__ __forceinline__ void cell_records(const RecArgs& ra, int32_t cell, const Geom* __restrict__ g,
                                             const Cells& c, const Moments& mo,
                                             otoo_src* __restrict__ src, otoo_quad* __restrict__ quad,
                                             otoo_wcell* __restrict__ wc, otoo_wcell64* __restrict__ wc64,
                                             int32_t* __restrict__ level_out, uint32_t* __restrict__ bits, bool wide)
{
    const int L = c.level[cell];
    const int32_t b = c.begin[cell], e = c.end[cell], par = c.parent[cell];
    if (par < 0 || c.end[par] - c.begin[par] > ra.n_crit) {
        if (e - b <= ra.n_crit)
            atomicOr(bits + (b >> 5), 1u << (b & 31));
        else if (c.nchild[cell] == 0)
            for (int64_t k = b; k < e; k += ra.n_crit) atomicOr(bits + (k >> 5), 1u << (k & 31));
    }
    const int sh = kLevels - L;
    const double side = cube_side(g->h, L);
    const otoo_src p0 = src[b];
    const double first[3] = {p0.x, p0.y, p0.z};
    double lo[3], gc[3], com[3];
    for (int a = 0; a < 3; ++a) {
        // (sh = 21: the root)
        const uint32_t org = quantize(first[a], g->lo[a], g->scale) >> sh << sh;
        lo[a] = cube_lo(g->lo[a], org, g->h);
        gc[a] = cube_centre(lo[a], side);
        com[a] = mo.com[3 * (int64_t)cell + a];
    }
    const double m = mo.m[cell];
    otoo_src s;
    s.x = com[0];
    s.y = com[1];
    s.z = com[2];
    s.m = narrow(m);
    s.pad = 0;
    put_record(src + ra.n_part + cell, s, wide);
    otoo_quad qd;
    const bool u = ra.use_quad != 0;
    // Q = 3 C - tr(C) I from the central second moment C
    const double* cm = mo.q + 6 * (int64_t)cell;
    const double tr = mo.b2[cell];
    qd.xx = u ? narrow(3.0 * cm[0] - tr) : 0.f;
    qd.yy = u ? narrow(3.0 * cm[1] - tr) : 0.f;
    qd.zz = u ? narrow(3.0 * cm[2] - tr) : 0.f;
    qd.xy = u ? narrow(3.0 * cm[3]) : 0.f;
    qd.xz = u ? narrow(3.0 * cm[4]) : 0.f;
    qd.yz = u ? narrow(3.0 * cm[5]) : 0.f;
    qd.b2 = u ? narrow(tr) : 0.f;
    qd.pad = 0.f;
    put_record(quad + cell, qd, wide);
    const double dm = __longlong_as_double((long long)mo.dmax2[cell]);
    const double rb = ra.mac == OTOO_MAC_SW    ? sw_radius(mo.b2[cell], __dsqrt_rn(dm), m, ra.delta, ra.m_limit, g->S)
                      : ra.mac == OTOO_MAC_SPH ? (double)__uint_as_float((unsigned)mo.dmax2[cell])
                                               : 0.0;
    otoo_wcell w;
    wcell_geometry(com, lo, gc, side, &w);
    w.nchild = c.nchild[cell];
    w.child0 = w.nchild > 0 ? c.child0[cell] : 0;
    w.begin = b;
    w.end = e;
    w.rb = narrow(rb);
    put_record(wc + cell, w, wide);
    otoo_wcell64 w64;
    for (int a = 0; a < 3; ++a) w64.lo[a] = lo[a], w64.com[a] = com[a], w64.gc[a] = gc[a];
    w64.side = side;
    w64.rb = rb;
    w64.pad = 0.0;
    put_record(wc64 + cell, w64, wide);
    level_out[cell] = L;
}

__global__ void __launch_bounds__(128) k_records(RecArgs ra, const Head* __restrict__ head, Cells c, Moments mo,
                                                 otoo_src* __restrict__ src, otoo_quad* __restrict__ quad, otoo_wcell* __restrict__ wc,
                                                 otoo_wcell64* __restrict__ wc64, int32_t* __restrict__ level_out,
                                                 uint32_t* __restrict__ bits)
{
    const int32_t n_cell = head->lev[kLv];
    const bool wide = ((reinterpret_cast<uintptr_t>(src) | reinterpret_cast<uintptr_t>(quad) |
                        reinterpret_cast<uintptr_t>(wc) | reinterpret_cast<uintptr_t>(wc64)) & 15) == 0;
    for (int32_t cell = blockIdx.x * blockDim.x + threadIdx.x; cell < n_cell; cell += gridDim.x * blockDim.x)
        cell_records(ra, cell, &head->g, c, mo, src, quad, wc, wc64, level_out, bits, wide);
}

// Groups in tree order from their first particles' bits: words of 32 particles,
// kGroupWords words per block.  k_group_sums counts a block's bits, k_group_write
// adds up the blocks before its own and writes its groups; a group ends where
// the next bit is set.  Two launches and n / 8 bytes, against a flag per
// particle, a copy, a three-launch scan, a compaction and a pass for the counts
// (seven launches).
constexpr int kGroupWords = 1024;

__global__ void __launch_bounds__(256) k_group_sums(const uint32_t* __restrict__ bits, int64_t nw,
                                                     int32_t* __restrict__ bsum)
{
    __shared__ int32_t s[8];
    int32_t v = 0;
    for (int k = 0; k < kGroupWords / 256; ++k) {
        const int64_t i = (int64_t)blockIdx.x * kGroupWords + k * 256 + threadIdx.x;
        if (i < nw) v += __popc(bits[i]);
    }
    v = __reduce_add_sync(kFull, v);
    if ((threadIdx.x & 31) == 0) s[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int k = 1; k < 8; ++k) v += s[k];
        bsum[blockIdx.x] = v;
    }
}

__global__ void __launch_bounds__(256) k_group_write(const uint32_t* __restrict__ bits, int64_t nw, int64_t n,
                                                      const int32_t* __restrict__ bsum, int32_t* __restrict__ first,
                                                      int32_t* __restrict__ count, Head* __restrict__ head,
                                                      uint32_t* __restrict__ status_out)
{
    __shared__ int32_t s[2][8];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    // groups of the blocks before this one
    int32_t v = 0;
    for (int b = threadIdx.x; b < (int)blockIdx.x; b += 256) v += bsum[b];
    v = __reduce_add_sync(kFull, v);
    // this block's words, four consecutive ones per thread
    const int64_t i0 = (int64_t)blockIdx.x * kGroupWords + 4 * threadIdx.x;
    uint32_t m[4];
    int32_t mine = 0;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        m[k] = i0 + k < nw ? bits[i0 + k] : 0u;
        mine += __popc(m[k]);
    }
    int32_t incl = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int32_t t = __shfl_up_sync(kFull, incl, o);
        if (lane >= o) incl += t;
    }
    if (lane == 31) s[0][w] = incl;
    if (lane == 0) s[1][w] = v;
    __syncthreads();
    int32_t g = incl - mine;
    for (int k = 0; k < 8; ++k) g += s[1][k] + (k < w ? s[0][k] : 0);
    if (blockIdx.x == gridDim.x - 1 && threadIdx.x == 255) {
        head->groups = g + mine;
        status_out[0] = head->status;
    }
#pragma unroll 1
    for (int k = 0; k < 4; ++k)
        for (uint32_t x = m[k]; x; x &= x - 1u, ++g) {
            const int64_t p = 32 * (i0 + k) + (__ffs(x) - 1);
            // the next bit: in this word, or in the first word after it that has one
            uint32_t up = x & (x - 1u);
            int64_t j = i0 + k;
            while (!up && ++j < nw) up = bits[j];
            first[g] = (int32_t)p;
            count[g] = (int32_t)((up ? 32 * j + (__ffs(up) - 1) : n) - p);
        }
}

// ---- scans (exclusive, in place, int32) --------------------------------------------

constexpr int kScanThreads = 1024;

__device__ int64_t block_excl_scan64(int64_t v, int64_t* ws, int64_t* total)
{
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    int64_t inc = v;
    for (int o = 1; o < 32; o <<= 1) {
        const int64_t t = __shfl_up_sync(kFull, inc, o);
        if (lane >= o) inc += t;
    }
    if (lane == 31) ws[wid] = inc;
    __syncthreads();
    if (wid == 0) {
        const int64_t w = lane < (int)(blockDim.x >> 5) ? ws[lane] : 0;
        int64_t wi = w;
        for (int o = 1; o < 32; o <<= 1) {
            const int64_t t = __shfl_up_sync(kFull, wi, o);
            if (lane >= o) wi += t;
        }
        ws[lane] = wi - w;
        if (lane == 31) ws[32] = wi;
    }
    __syncthreads();
    const int64_t r = ws[wid] + inc - v;
    *total = ws[32];
    __syncthreads();
    return r;
}

__global__ void __launch_bounds__(kScanThreads) k_scan_sums(const int32_t* __restrict__ a, int64_t n,
                                                             int64_t* __restrict__ bsum)
{
    __shared__ int64_t ws[33];
    const int64_t i = (int64_t)blockIdx.x * kScanThreads + threadIdx.x;
    int64_t tot;
    block_excl_scan64(i < n ? a[i] : 0, ws, &tot);
    if (threadIdx.x == 0) bsum[blockIdx.x] = tot;
}

__global__ void __launch_bounds__(kScanThreads) k_scan_top(int64_t* __restrict__ bsum, int64_t nblk,
                                                            int64_t* __restrict__ total)
{
    __shared__ int64_t ws[33];
    int64_t carry = 0;
    for (int64_t b0 = 0; b0 < nblk; b0 += kScanThreads) {
        const int64_t i = b0 + threadIdx.x;
        int64_t tot;
        const int64_t e = block_excl_scan64(i < nblk ? bsum[i] : 0, ws, &tot);
        if (i < nblk) bsum[i] = carry + e;
        carry += tot;
    }
    if (threadIdx.x == 0) *total = carry;
}

__global__ void __launch_bounds__(kScanThreads) k_scan_apply(int32_t* __restrict__ a, int64_t n,
                                                              const int64_t* __restrict__ bsum)
{
    __shared__ int64_t ws[33];
    const int64_t i = (int64_t)blockIdx.x * kScanThreads + threadIdx.x;
    int64_t tot;
    const int64_t e = block_excl_scan64(i < n ? a[i] : 0, ws, &tot) + bsum[blockIdx.x];
    if (i < n) a[i] = (int32_t)e;
}

#define CUDA_TRY(expr)                                                                                 \
    do {                                                                                               \
        cudaError_t e_ = (expr);                                                                       \
        if (e_ != cudaSuccess) return set_error(OTOO_ECUDA, "%s: %s", #expr, cudaGetErrorString(e_));  \
    } while (0)

// One block: an exclusive scan of a[0, n) in place, four elements per thread
// and round, the total to *total.  For arrays of up to 16 * kScanThreads
// elements, where the three launches below (2.8 us each at least) cost more
// than the serial rounds (3.4 us at n = 512, 7.8 us at 11264).
__global__ void __launch_bounds__(kScanThreads) k_scan_one(int32_t* __restrict__ a, int64_t n,
                                                            int64_t* __restrict__ total)
{
    __shared__ int64_t ws[33];
    int64_t carry = 0;
    for (int64_t b0 = 0; b0 < n; b0 += 4 * kScanThreads) {
        const int64_t i = b0 + 4 * (int64_t)threadIdx.x;
        int32_t v[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) v[k] = i + k < n ? a[i + k] : 0;
        int64_t tot;
        int64_t e = carry + block_excl_scan64((int64_t)v[0] + v[1] + v[2] + v[3], ws, &tot);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            if (i + k < n) a[i + k] = (int32_t)e;
            e += v[k];
        }
        carry += tot;
    }
    if (threadIdx.x == 0) *total = carry;
}

// exclusive scan of a[0, n) in place; the total to *total (device)
int scan32(int32_t* a, int64_t n, int64_t* bsum, int64_t* total, cudaStream_t s)
{
    const int64_t nblk = (n + kScanThreads - 1) / kScanThreads;
    if (nblk == 0) {
        CUDA_TRY(cudaMemsetAsync(total, 0, sizeof(int64_t), s));
        return OTOO_OK;
    }
    if (n <= 16 * kScanThreads) {
        k_scan_one<<<1, kScanThreads, 0, s>>>(a, n, total);
        CUDA_TRY(cudaGetLastError());
        return OTOO_OK;
    }
    k_scan_sums<<<(unsigned)nblk, kScanThreads, 0, s>>>(a, n, bsum);
    k_scan_top<<<1, kScanThreads, 0, s>>>(bsum, nblk, total);
    k_scan_apply<<<(unsigned)nblk, kScanThreads, 0, s>>>(a, n, bsum);
    CUDA_TRY(cudaGetLastError());
    return OTOO_OK;
}

// Scratch layout (byte offsets, each part 256-byte aligned).
struct Layout {
    size_t keys0, keys1, vals0, vals1, head, bits, hist, bsum, part, cells[6], mom_m, mom_com, mom_q, mom_b2,
        mom_dmax, dig, total;
};

size_t up(size_t x) { return (x + 255) & ~(size_t)255; }

Layout layout(int64_t n, int64_t cap)
{
    Layout l;
    size_t o = 0;
    auto take = [&](size_t bytes) {
        const size_t at = o;
        o += up(bytes);
        return at;
    };
    const int64_t nblk = (n + kLvTile - 1) / kLvTile;
    l.keys0 = take(8 * n);
    l.keys1 = take(8 * n);
    l.vals0 = take(4 * n);
    l.vals1 = take(4 * n);
    // zeroed together before the first kernel: the head, a bit per particle,
    // the sort's counts and first words
    l.head = take(sizeof(Head));
    l.bits = take(4 * ((n + 31) / 32));
    // the sort's counts, tickets and two sets of published words; later the
    // cells' counts (kLv per tile of kLvTile)
    const int64_t ntile = (n + kSortTile - 1) / kSortTile;
    l.hist = take(4 * std::max<int64_t>(256 * (9 + 2 * ntile), kLv * nblk));
    // block sums of the cells' scan, later the groups' per block
    l.bsum = take(8 * ((256 * nblk + n) / kScanThreads + 8));
    l.part = take(8 * 6 * 1024);
    for (int k = 0; k < 6; ++k) l.cells[k] = take(4 * cap);
    l.mom_m = take(8 * cap);
    l.mom_com = take(24 * cap);
    l.mom_q = take(48 * cap);
    l.mom_b2 = take(8 * cap);
    l.mom_dmax = take(8 * cap);
    l.dig = take(32 * cap);
    l.total = o;
    return l;
}

}  // namespace

extern "C" {

int64_t otoo_devtree_scratch_bytes(int64_t n_part, int64_t cap_cell)
{
    if (n_part < 1 || cap_cell < 1) return 0;
    return (int64_t)layout(n_part, cap_cell).total;
}

int otoo_devtree_build(const double* pos, const float* mass, otoo_devtree* t, void* scratch, int64_t scratch_bytes,
                       void* stream)
{
    otoo::Range range_("otoo_devtree_build");
    OTOO_REQUIRE(pos && mass && t && scratch, OTOO_EINVAL, "otoo_devtree_build: NULL pointer");
    const int64_t n = t->n_part, cap = t->cap_cell;
    OTOO_REQUIRE(n >= 1 && n <= INT32_MAX / 2 && cap >= 1 && n + cap <= INT32_MAX, OTOO_EINVAL,
                 "otoo_devtree_build: n_part / cap_cell out of range");
    OTOO_REQUIRE(t->leaf_size >= 1 && t->n_crit >= 1 && t->n_crit <= kMaxGroup, OTOO_EINVAL,
                 "otoo_devtree_build: leaf_size < 1 or n_crit outside [1, %d]", kMaxGroup);
    OTOO_REQUIRE(t->mac == OTOO_MAC_THETA || t->mac == OTOO_MAC_SW || t->mac == OTOO_MAC_SPH, OTOO_EINVAL,
                 "unknown mac %d", t->mac);
    OTOO_REQUIRE(t->mac != OTOO_MAC_SPH || t->h_sph, OTOO_EINVAL, "OTOO_MAC_SPH needs h_sph");
    OTOO_REQUIRE(t->mac != OTOO_MAC_SW || (t->delta >= 0.0 && std::isfinite(t->delta) && std::isfinite(t->m_limit)),
                 OTOO_EINVAL, "delta must be finite and >= 0, m_limit finite");
    OTOO_REQUIRE(t->src && t->quad && t->cell && t->cell64 && t->group_first && t->group_count && t->perm &&
                     t->cell_level && t->status,
                 OTOO_EINVAL, "otoo_devtree_build: NULL output array");
    const Layout ly = layout(n, cap);
    OTOO_REQUIRE(scratch_bytes >= (int64_t)ly.total, OTOO_EINVAL, "otoo_devtree_build: scratch too small (%lld < %lld)",
                 (long long)scratch_bytes, (long long)ly.total);
    OTOO_REQUIRE((reinterpret_cast<uintptr_t>(scratch) & 15) == 0, OTOO_EINVAL,
                 "otoo_devtree_build: scratch not 16-byte aligned");
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    char* base = static_cast<char*>(scratch);
    uint64_t* keys[2] = {reinterpret_cast<uint64_t*>(base + ly.keys0), reinterpret_cast<uint64_t*>(base + ly.keys1)};
    uint32_t* vals[2] = {reinterpret_cast<uint32_t*>(base + ly.vals0), reinterpret_cast<uint32_t*>(base + ly.vals1)};
    int32_t* hist = reinterpret_cast<int32_t*>(base + ly.hist);
    int64_t* bsum = reinterpret_cast<int64_t*>(base + ly.bsum);
    long long* part = reinterpret_cast<long long*>(base + ly.part);
    Head* head = reinterpret_cast<Head*>(base + ly.head);
    Geom* geom = &head->g;
    uint32_t* bits = reinterpret_cast<uint32_t*>(base + ly.bits);
    const int64_t nw = (n + 31) / 32;
    Cells c;
    c.begin = reinterpret_cast<int32_t*>(base + ly.cells[0]);
    c.end = reinterpret_cast<int32_t*>(base + ly.cells[1]);
    c.level = reinterpret_cast<int32_t*>(base + ly.cells[2]);
    c.parent = reinterpret_cast<int32_t*>(base + ly.cells[3]);
    c.child0 = reinterpret_cast<int32_t*>(base + ly.cells[4]);
    c.nchild = reinterpret_cast<int32_t*>(base + ly.cells[5]);
    Moments mo;
    mo.m = reinterpret_cast<double*>(base + ly.mom_m);
    mo.com = reinterpret_cast<double*>(base + ly.mom_com);
    mo.q = reinterpret_cast<double*>(base + ly.mom_q);
    mo.b2 = reinterpret_cast<double*>(base + ly.mom_b2);
    mo.dmax2 = reinterpret_cast<unsigned long long*>(base + ly.mom_dmax);
    int32_t* dig = reinterpret_cast<int32_t*>(base + ly.dig);
    uint32_t* status = &head->status;
    int dev = 0, sms = 0;
    CUDA_TRY(cudaGetDevice(&dev));
    CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));

    // root cube, keys, sort
    const int nblk = (int)((n + kLvTile - 1) / kLvTile);
    const int ntile = (int)((n + kSortTile - 1) / kSortTile);
    // digit counts and tickets of the eight passes, then the first pass's words
    int32_t* ghist = hist;
    uint32_t* ticket = reinterpret_cast<uint32_t*>(ghist + 8 * 256);
    uint32_t* look[2] = {ticket + 256, ticket + 256 + (size_t)256 * ntile};
    CUDA_TRY(cudaMemsetAsync(head, 0, ly.hist - ly.head + 4 * (8 * 256 + 256 + (size_t)256 * ntile), s));
    const int nbb = (int)std::min<int64_t>(1024, (n + 255) / 256);
    k_bbox<<<nbb, 256, 0, s>>>(pos, mass, n, part, head);
    k_keys<<<(unsigned)std::min<int64_t>((n + 255) / 256, (int64_t)sms * 8), 256, 0, s>>>(pos, n, geom, keys[0], ghist);
    CUDA_TRY(cudaGetLastError());
    CUDA_TRY(cudaFuncSetAttribute(k_sort_pass, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(SortShared)));
    CUDA_TRY(cudaFuncSetAttribute(k_sort_tile, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(SortShared)));
    int cur = 0;
    if (ntile == 1) {
        k_sort_tile<<<1, kSortThreads, sizeof(SortShared), s>>>(keys[0], n, keys[1], vals[1]);
        cur = 1;
    } else {
        for (int p = 0; p < 8; ++p, cur ^= 1)
            k_sort_pass<<<ntile, kSortThreads, sizeof(SortShared), s>>>(
                keys[cur], p ? vals[cur] : nullptr, n, 8 * p, ghist + 256 * p, ticket + p, look[p & 1],
                look[(p & 1) ^ 1], keys[cur ^ 1], vals[cur ^ 1], status);
    }
    CUDA_TRY(cudaGetLastError());
    k_permute<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(pos, mass, vals[cur], n, t->src, t->perm,
                                                          status);
    CUDA_TRY(cudaGetLastError());
    const uint64_t* skeys = keys[cur];

    // cells; the unsorted copy of the keys is dead, its memory holds the
    // particles' levels (2 n bytes) and the windows of large leaf sizes
    // (2 (n + leaf_size) bytes, leaf_size < n)
    int32_t* lev = head->lev;
    uint16_t* lv = reinterpret_cast<uint16_t*>(keys[cur ^ 1]);
    const uint8_t* win = nullptr;
    int64_t span = 1;
    const int64_t leaf = std::min<int64_t>(t->leaf_size, n);
    if (leaf > kLvLeaf) {
        const int64_t len = n + leaf;
        uint8_t* wb[2] = {reinterpret_cast<uint8_t*>(lv + n), reinterpret_cast<uint8_t*>(lv + n) + len};
        const unsigned g = (unsigned)((len + 255) / 256);
        k_win_init<<<g, 256, 0, s>>>(skeys, n, leaf, wb[0]);
        int k = 0;
        for (; 2 * span <= leaf + 1; span *= 2, k ^= 1) k_win_double<<<g, 256, 0, s>>>(wb[k], len, span, wb[k ^ 1]);
        win = wb[k];
    }
    k_levels<<<nblk, kLvThreads, 0, s>>>(skeys, n, leaf, win, span, lv, hist);
    CUDA_TRY(cudaGetLastError());
    {
        const int r = scan32(hist, (int64_t)kLv * nblk, bsum, &head->cells, s);
        if (r) return r;
    }
    k_cells<<<nblk, kLvThreads, 0, s>>>(n, lv, hist, &head->cells, cap, c, lev, status, &head->stop);
    CUDA_TRY(cudaGetLastError());

    // links, leaves, then the parents level by level (grid-stride over the
    // cells: their number is on the device)
    const unsigned cg = (unsigned)std::min<int64_t>((cap + 127) / 128, (int64_t)sms * 16);
    int32_t* pcount = head->pcount;
    // (small trees: smaller blocks use more SMs)
    const int lt = n < 32768 ? 64 : n < 262144 ? 128 : kLeafThreads;
    k_leaves<<<(unsigned)std::min<int64_t>((cap + lt - 1) / lt, (int64_t)sms * 8 * kLeafThreads / lt), lt, 0, s>>>(
        lev, skeys, n, leaf, t->src, c, mo, dig, pcount);
    if (n > leaf) {
        uint32_t* bar = &head->bar;
        void* args[] = {&lev, &c, &mo, &dig, &pcount, &bar, &status};
        const unsigned pg = (unsigned)std::min<int64_t>(sms, (cap + 63) / 64);  // at most one block per SM
        CUDA_TRY(cudaLaunchCooperativeKernel((const void*)k_parents, dim3(pg), dim3(512), args, 0, s));
    }
    CUDA_TRY(cudaGetLastError());
    const bool sph = t->mac == OTOO_MAC_SPH;
    if (t->mac == OTOO_MAC_SW || sph) {
        // The sorted keys, the sort's values and the parents' lists are dead
        // once the moments exist: keys0..keys1 (two adjacent 256-byte-aligned
        // parts of 8 n bytes) hold the FP32 particles, vals0..vals1 the larger
        // cells' work items (8 bytes each; a level has at most n / 64 cells of
        // more than 64 particles and n / 2048 further chunks, 22 levels: below
        // 3 n bytes of 8 n), dig (32 cap bytes) the FP32 centres.
        float4* pk = reinterpret_cast<float4*>(base + ly.keys0);
        float4* cf = reinterpret_cast<float4*>(dig);
        int2* extra = reinterpret_cast<int2*>(base + ly.vals0);
        k_chunks<<<cg, 128, 0, s>>>(head, c, mo.com, extra, cf);
        k_bpack<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(n, t->src, sph ? t->h_sph : nullptr, t->perm, pk);
        k_bmax<<<(unsigned)std::min<int64_t>((cap + 31) / 32, (int64_t)sms * 8), 256, 0, s>>>(
            head, extra, t->src, pk, cf, c, mo, sph ? 1 : 0);
        CUDA_TRY(cudaGetLastError());
    }
    RecArgs ra;
    ra.n_part = n;
    ra.use_quad = t->use_quad ? 1 : 0;
    ra.mac = t->mac;
    ra.n_crit = t->n_crit;
    ra.delta = t->delta;
    ra.m_limit = t->m_limit;
    k_records<<<cg, 128, 0, s>>>(ra, head, c, mo, t->src, t->quad, t->cell, t->cell64, t->cell_level, bits);
    // groups
    int32_t* gsum = reinterpret_cast<int32_t*>(bsum);
    const unsigned gg = (unsigned)((nw + kGroupWords - 1) / kGroupWords);
    k_group_sums<<<gg, 256, 0, s>>>(bits, nw, gsum);
    k_group_write<<<gg, 256, 0, s>>>(bits, nw, n, gsum, t->group_first, t->group_count, head, t->status);
    CUDA_TRY(cudaGetLastError());
    Head h;
    CUDA_TRY(cudaMemcpyAsync(&h, head, sizeof(h), cudaMemcpyDeviceToHost, s));
    CUDA_TRY(cudaStreamSynchronize(s));
    if (h.status & kTreeBadInput) return set_error(OTOO_EINVAL, "otoo_devtree_build: non-finite position or mass <= 0");
    if (h.status & kTreeStuck) return set_error(OTOO_EDEVICE, "otoo_devtree_build: a wait between blocks ran into its limit");
    if (h.status & kTreeBadSort) return set_error(OTOO_EDEVICE, "otoo_devtree_build: sort produced an invalid order");
    if (h.stop) {
        t->n_cell = -1;
        return set_error(OTOO_ENOMEM, "otoo_devtree_build: more than cap_cell = %lld cells", (long long)cap);
    }
    // level L holds [lev[L], lev[L + 1]); the last non-empty level is the depth
    int depth = 0;
    for (int L = 0; L <= kLevels; ++L)
        if (h.lev[L + 1] > h.lev[L]) depth = L;
    const Geom& hg = h.g;
    const int32_t n_cell = h.lev[kLv];
    const int64_t G = h.groups;
    t->n_cell = n_cell;
    t->n_groups = G;
    t->depth = depth;
    for (int a = 0; a < 3; ++a) t->root_lo[a] = hg.lo[a];
    t->root_side = hg.S;
    return OTOO_OK;
}

}  // extern "C"
