// Leaf decomposition on the GPU: chaining mesh or recursive coordinate bisection
// (Sec. 3.1 names the RCB tree; Sec. 5.3 runs the kernels over leaf pairs),
// then the periodic leaf-pair image lists used by every pair kernel.
//
// RCB without per-node sorts: every particle is ranked once per axis by a
// stable radix sort of (coordinate, index).  Each level keeps three lists,
// each sorted along its axis inside every node, whose entries carry the
// particle's ranks along the two other axes.  A node's tight box is read off
// the ends of its three segments; the split takes the first floor(n/2) of the
// chosen axis' segment, which is a threshold on the rank along that axis, so
// the two other lists are stably partitioned by comparing the ranks they
// carry (a prefix sum of the left flags orders the output).  The shape of the
// tree depends on n alone, so the host precomputes every level's segments.
#include <cooperative_groups.h>

#include <algorithm>
#include <chrono>
#include <cmath>
#include <cstdio>
#include <cstring>

#include "crk_internal.cuh"

namespace {

constexpr int kMaxLeafCap = 1024;

// Positions in [0, L_box), gas h > 0 and finite; largest gas h per box.
// Each block takes `items` rows of 256 consecutive particles and combines
// its counts (and, when its range lies in one box, its h maximum) in shared
// memory, so the global atomics are a few per block: same-address atomics
// from every warp of a 33M-particle launch serialise at L2 (about 1.7 ms).
// 16 rows where that leaves blocks for every SM, else 4 (2x64^3: 20 -> 7.5 us).

__global__ void __launch_bounds__(256) validate_kernel(const float *__restrict__ x, const float *__restrict__ y,
                                                       const float *__restrict__ z, const uint8_t *__restrict__ sp,
                                                       const float *__restrict__ h, int64_t n, int items,
                                                       const int32_t *__restrict__ box_of,
                                                       const float *__restrict__ box_L,
                                                       int32_t *__restrict__ flags /* [0] bad pos, [1] bad h, [2] n_gas */,
                                                       unsigned *__restrict__ hmax_bits /* per box */) {
    __shared__ unsigned part[4][8];
    const int64_t tile = 256 * (int64_t)items, base = (int64_t)blockIdx.x * tile;
    const int64_t last = (base + tile < n ? base + tile : n) - 1;
    const int bfirst = box_of ? box_of[base] : 0;
    const bool one_box = !box_of || box_of[last] == bfirst;  // boxes are contiguous ranges
    unsigned nbad = 0, nbadh = 0, ngas = 0, hb_blk = 0;
    for (int k = 0; k < items; ++k) {
        const int64_t i = base + (int64_t)k * 256 + threadIdx.x;
        if (i >= n) break;
        const int b = box_of ? box_of[i] : 0;
        const float L = box_L[b];
        const float c[3] = {x[i], y[i], z[i]};
        bool bad = false;
        for (int a = 0; a < 3; ++a) bad |= !(c[a] >= 0.0f && c[a] < L);
        nbad += bad;
        if (sp[i] == 0) {
            ++ngas;
            const float hi = h[i];
            if (!(hi > 0.0f) || !isfinite(hi)) {
                ++nbadh;
            } else {
                const unsigned hb = __float_as_uint(hi);  // positive floats order like their bits
                if (one_box) hb_blk = hb > hb_blk ? hb : hb_blk;
                else atomicMax(&hmax_bits[b], hb);
            }
        }
    }
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    nbad = __reduce_add_sync(CRK_FULL_MASK, nbad);
    nbadh = __reduce_add_sync(CRK_FULL_MASK, nbadh);
    ngas = __reduce_add_sync(CRK_FULL_MASK, ngas);
    hb_blk = __reduce_max_sync(CRK_FULL_MASK, hb_blk);
    if (lane == 0) {
        part[0][w] = nbad;
        part[1][w] = nbadh;
        part[2][w] = ngas;
        part[3][w] = hb_blk;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int v = 1; v < 8; ++v) {
            for (int q = 0; q < 3; ++q) part[q][0] += part[q][v];
            part[3][0] = part[3][v] > part[3][0] ? part[3][v] : part[3][0];
        }
        for (int q = 0; q < 3; ++q)
            if (part[q][0]) atomicAdd(&flags[q], (int)part[q][0]);
        if (part[3][0]) atomicMax(&hmax_bits[bfirst], part[3][0]);
    }
}

// box of each particle from the box starts (binary search)
__global__ void box_of_kernel(int64_t n, const int64_t *__restrict__ box_start, int nbox, int32_t *__restrict__ box_of) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    int lo = 0, hi = nbox - 1;
    while (lo < hi) {
        int mid = (lo + hi + 1) >> 1;
        if (box_start[mid] <= i) lo = mid;
        else hi = mid - 1;
    }
    box_of[i] = lo;
}

// chaining mesh cell: c = min(nc-1, floor(x nc / L)) per axis in FP64, id = (cx nc + cy) nc + cz
__global__ void mesh_keys_kernel(const float *__restrict__ x, const float *__restrict__ y, const float *__restrict__ z,
                                 int64_t n, int nc, double L, uint32_t *__restrict__ keys, int32_t *__restrict__ vals,
                                 int32_t *__restrict__ counts) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    float c3[3] = {x[i], y[i], z[i]};
    int c[3];
    for (int a = 0; a < 3; ++a) {
        double f = floor(__ddiv_rn(__dmul_rn((double)c3[a], (double)nc), L));
        int ci = (int)f;
        c[a] = ci > nc - 1 ? nc - 1 : (ci < 0 ? 0 : ci);
    }
    uint32_t id = (uint32_t)((c[0] * nc + c[1]) * nc + c[2]);
    keys[i] = id;
    vals[i] = (int32_t)i;
    atomicAdd(&counts[id], 1);
}

// --- RCB level kernels ------------------------------------------------------
struct LevelDev {
    const int32_t *lo, *hi, *k, *child, *node;
    int32_t *axis;
    const int32_t *leftbase;  // sum of k over the earlier segments of the level
};

// everything the partition needs about one segment, in one 32-byte record
struct __align__(16) SegRec {
    int32_t lo, hi, k, child;
    int32_t axis, leftbase, thr, pad;  // thr: rank along the split axis of the first right-going particle
};

// The three axis lists carry ranks, not particle ids.  S[t] is the stable
// (coordinate, index) order along axis t (box-major for batches) and R[t] its
// inverse (the rank of each particle along t).  Entry p of list a holds the
// ranks of its particle along the two other axes:
// A[a][c][p] = rank along axis (a + 1 + c) % 3.  Inside a node, list a is
// sorted by rank along a, so the node's split is a rank threshold: an entry of
// another list goes left iff its rank along the split axis is below the rank
// of the first right-going entry of the split axis' own list.  A level is then
// pure streaming (no per-particle side flag is scattered or gathered).
struct RankLists {
    const int32_t *A[3][2];
};
struct RankListsOut {
    int32_t *A[3][2];
};
struct AxisOrder {
    const int32_t *S[3];
    const int32_t *R[3];
};
struct RankOut {
    int32_t *r[3];
};

__device__ __forceinline__ unsigned lanemask_lt_u() {
    unsigned m;
    asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
    return m;
}

__device__ __forceinline__ int rank_comp(int a, int t) { return (t - a + 2) % 3; }  // component of list a holding t

// particle id of entry p of list a
__device__ __forceinline__ int32_t rank_entry_id(const RankLists &L, const AxisOrder &o, int a, int64_t p) {
    const int32_t r = L.A[a][0][p];
    return a == 0 ? o.S[1][r] : (a == 1 ? o.S[2][r] : o.S[0][r]);
}

// R[S[p]] = p: the inverse of each axis order (blocks run in launch order, axis by axis, so the
// randomly written array, n ints, stays about the size of L2)
__global__ void rank_of_kernel(int64_t n, AxisOrder o, RankOut R) {
    int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int t = blockIdx.y;
    if (p < n) (t == 0 ? R.r[0] : (t == 1 ? R.r[1] : R.r[2]))[(t == 0 ? o.S[0] : (t == 1 ? o.S[1] : o.S[2]))[p]] = (int32_t)p;
}

// the six rank columns: list a, column c holds R[S_a[p]] of axis t = (a + 1 + c) % 3; columns in
// the order of t, two per randomly read source array
__global__ void rank_column_kernel(int64_t n, AxisOrder o, RankListsOut A) {
    int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= n) return;
    auto col = [&](int a, int c, int t) { A.A[a][c][p] = __ldg(o.R[t] + o.S[a][p]); };
    switch (blockIdx.y) {
        case 0: col(2, 0, 0); break;
        case 1: col(1, 1, 0); break;
        case 2: col(0, 0, 1); break;
        case 3: col(2, 1, 1); break;
        case 4: col(1, 0, 2); break;
        default: col(0, 1, 2); break;
    }
}

// final member order (list 0) as particle ids
__global__ void rank_members_kernel(int64_t n, RankLists L, AxisOrder o, int32_t *__restrict__ members) {
    int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p < n) members[p] = rank_entry_id(L, o, 0, p);
}

// Record of segment s of a level; for a split node the tight box from the ends of its three list
// segments, the split axis (longest extent, ties to the lower axis) and the rank threshold, with
// the box and the axis stored when `store`.
__device__ __forceinline__ SegRec rcb_segment(int s, const LevelDev &lv, const RankLists &L, const AxisOrder &o,
                                              const float *__restrict__ x, const float *__restrict__ y,
                                              const float *__restrict__ z, float *__restrict__ node_box, bool store) {
    int k = lv.k[s];
    int lo = lv.lo[s], hi = lv.hi[s];
    SegRec r{lo, hi, k, lv.child[s], 0, lv.leftbase[s], 0, 0};
    if (k <= 0) return r;
    const float *cs[3] = {x, y, z};
    float blo[3], bhi[3];
    double ext[3];
    for (int a = 0; a < 3; ++a) {
        blo[a] = cs[a][rank_entry_id(L, o, a, lo)];
        bhi[a] = cs[a][rank_entry_id(L, o, a, hi - 1)];
        ext[a] = __dsub_rn((double)bhi[a], (double)blo[a]);
    }
    int axis = 0;
    if (ext[1] > ext[axis]) axis = 1;
    if (ext[2] > ext[axis]) axis = 2;
    r.axis = axis;
    r.thr = o.R[axis][rank_entry_id(L, o, axis, lo + k)];
    if (store) {
        lv.axis[s] = axis;
        float *nb = node_box + 6 * (int64_t)lv.node[s];
        for (int a = 0; a < 3; ++a) {
            nb[a] = blo[a];
            nb[3 + a] = bhi[a];
        }
    }
    return r;
}

__global__ void rcb_axis_kernel(int nseg, LevelDev lv, RankLists L, AxisOrder o, const float *__restrict__ x,
                                const float *__restrict__ y, const float *__restrict__ z, float *__restrict__ node_box,
                                SegRec *__restrict__ seg) {
    int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s < nseg) seg[s] = rcb_segment(s, lv, L, o, x, y, z, node_box, true);
}

// Stable partition of the three lists, one level at a time.  The prefix count
// of left-going entries at a segment's start equals the sum of k over the
// earlier split segments (every split segment sends exactly k entries left in
// every list), so the prefix is never materialised: tiles count, a 3-column
// scan orders the tiles, and the scatter re-derives the tile-local prefixes.
constexpr int kPartThreads = 256;
constexpr int kPartItems = 8;
constexpr int kPartTile = kPartThreads * kPartItems;

// left flags of entry p (bit b: list b), or 0 for entries of unsplit segments
__device__ __forceinline__ unsigned rcb_left3(const SegRec &sr, const RankLists &L, int64_t p) {
    const int ks = sr.k;
    if (ks <= 0) return 0u;
    const int ax = sr.axis, lo = sr.lo;
    const int32_t th = sr.thr;
    unsigned f = 0;
#pragma unroll
    for (int b = 0; b < 3; ++b) {
        bool left;
        if (b == ax) {
            left = (int)p - lo < ks;
        } else {
            const int32_t *col = rank_comp(b, ax) == 0 ? L.A[b][0] : L.A[b][1];  // no dynamic index into the parameter
            left = col[p] < th;
        }
        f |= (unsigned)left << b;
    }
    return f;
}

// Exclusive scan of the three columns of tile sums in place, by one block (nb entries each).
__device__ void rcb_scan_columns(int32_t *bsum, int64_t nb, int32_t *wt) {
    constexpr int kItems = 8;
    for (int b = 0; b < 3; ++b) {
        int32_t carry = 0;
        int32_t *col = bsum + (int64_t)b * nb;
        for (int64_t s0 = 0; s0 < nb; s0 += (int64_t)blockDim.x * kItems) {
            const int64_t i0 = s0 + (int64_t)threadIdx.x * kItems;
            int32_t v[kItems], s = 0;
#pragma unroll
            for (int k = 0; k < kItems; ++k) {
                v[k] = i0 + k < nb ? __ldcg(col + i0 + k) : 0;
                s += v[k];
            }
            int32_t tot;
            int32_t e = carry + crk_block_scan(s, wt, tot);
#pragma unroll
            for (int k = 0; k < kItems; ++k) {
                if (i0 + k < nb) col[i0 + k] = e;
                e += v[k];
            }
            carry += tot;
        }
    }
}

// kAxis (one box: a streamed level's segments hold over 1024 entries, so a tile of 2048 meets at
// most kTileSegs): the blocks make the segment records they need themselves instead of a launch of
// their own.  ctr != NULL: the last block to finish scans the tile sums (no block waits on another).
constexpr int kTileSegs = 4;
constexpr int64_t kFusedTiles = 1024;  // up to here (2M particles) launches cost more than the repeated work

template <bool kAxis>
__global__ void __launch_bounds__(kPartThreads) rcb_count3_kernel(int64_t n, SegRec *__restrict__ segs,
                                                                   const int32_t *__restrict__ node_of, RankLists L,
                                                                   int32_t *bsum, int64_t nb, unsigned *ctr, LevelDev lv,
                                                                   AxisOrder o, const float *__restrict__ x,
                                                                   const float *__restrict__ y,
                                                                   const float *__restrict__ z,
                                                                   float *__restrict__ node_box, int32_t *__restrict__ err) {
    __shared__ int32_t wt[32];
    __shared__ SegRec own[kTileSegs];
    __shared__ bool last;
    const int64_t base = (int64_t)blockIdx.x * kPartTile;
    int s0 = 0;
    if constexpr (kAxis) {
        s0 = node_of[base];
        const int ns = node_of[(base + kPartTile < n ? base + kPartTile : n) - 1] - s0 + 1;
        const int t = threadIdx.x >> 5;  // one warp's first lane per segment
        if ((threadIdx.x & 31) == 0 && t < kTileSegs) {
            if (t < ns) {
                const int lo = lv.lo[s0 + t];
                const bool mine = lo >= base && lo < base + kPartTile;
                own[t] = rcb_segment(s0 + t, lv, L, o, x, y, z, node_box, mine);
                if (mine) segs[s0 + t] = own[t];
            }
            if (t == 0 && ns > kTileSegs) atomicAdd(err, 1);  // excluded by the host's choice of levels
        }
        __syncthreads();
    }
    int32_t seg[kPartItems];
#pragma unroll
    for (int k = 0; k < kPartItems; ++k) {
        int64_t p = base + (int64_t)k * kPartThreads + threadIdx.x;
        seg[k] = p < n ? node_of[p] : -1;
    }
    int32_t c[3] = {0, 0, 0};
#pragma unroll
    for (int k = 0; k < kPartItems; ++k) {
        int64_t p = base + (int64_t)k * kPartThreads + threadIdx.x;
        unsigned f = 0u;
        if (seg[k] >= 0) {
            const SegRec sr = kAxis ? own[min(seg[k] - s0, kTileSegs - 1)] : segs[seg[k]];
            f = rcb_left3(sr, L, p);
        }
        c[0] += f & 1u;
        c[1] += (f >> 1) & 1u;
        c[2] += (f >> 2) & 1u;
    }
    for (int b = 0; b < 3; ++b) {
        int32_t tot;
        crk_block_scan(c[b], wt, tot);
        if (threadIdx.x == 0) bsum[(int64_t)b * nb + blockIdx.x] = tot;
    }
    if (!ctr) return;
    if (threadIdx.x == 0) {
        __threadfence();
        last = atomicInc(ctr, gridDim.x - 1) == gridDim.x - 1;  // wraps to 0 for the next level
        __threadfence();
    }
    __syncthreads();
    if (last) rcb_scan_columns(bsum, nb, wt);
}

// single block: exclusive scan of the three columns of tile sums, in place
__global__ void __launch_bounds__(1024) rcb_scan3_kernel(int32_t *__restrict__ bsum, int64_t nb) {
    __shared__ int32_t wt[32];
    rcb_scan_columns(bsum, nb, wt);
}

// Entries are taken in rows of kPartThreads consecutive positions (entry k of
// thread t is position base + k kPartThreads + t), so the left-going (and the
// right-going) entries of one warp row land in consecutive output positions:
// coalesced stores.  The tile-local prefix of an entry is the count over
// earlier (row, warp) pairs plus the ballot rank inside its warp.  The kernel
// waits on its loads (segment record, rank columns): compiled for six
// resident blocks per SM (40 registers) it ran the 14 streamed levels of the
// 33.5M-particle build 2.0 ms faster than at four.
constexpr int kPartWarps = kPartThreads / 32;

__global__ void __launch_bounds__(kPartThreads, 6) rcb_scatter3_kernel(int64_t n, const SegRec *__restrict__ segs,
                                                                      const int32_t *__restrict__ node_of, RankLists L,
                                                                      const int32_t *__restrict__ bsum, int64_t nb,
                                                                      RankListsOut O, int32_t *__restrict__ node_of_next,
                                                                      int32_t *__restrict__ err) {
    static_assert(kPartItems * kPartWarps == 64, "prefix table: two entries per lane of one warp");
    __shared__ int32_t wc[3][kPartItems * kPartWarps];  // left count per (list, row, warp), then its prefix
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const unsigned below = lanemask_lt_u();
    const int64_t base = (int64_t)blockIdx.x * kPartTile;
    int32_t seg[kPartItems];
    unsigned f[kPartItems];
#pragma unroll
    for (int k = 0; k < kPartItems; ++k) {
        int64_t p = base + (int64_t)k * kPartThreads + threadIdx.x;
        seg[k] = p < n ? node_of[p] : -1;
    }
#pragma unroll
    for (int k = 0; k < kPartItems; ++k) {
        int64_t p = base + (int64_t)k * kPartThreads + threadIdx.x;
        f[k] = 0u;
        if (seg[k] >= 0) {
            const SegRec sr = segs[seg[k]];
            f[k] = rcb_left3(sr, L, p);
        }
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            const unsigned m = __ballot_sync(0xffffffffu, (f[k] >> b) & 1u);
            if (lane == 0) wc[b][k * kPartWarps + warp] = __popc(m);
        }
    }
    __syncthreads();
    if (warp == 0) {
        for (int b = 0; b < 3; ++b) {
            const int32_t e0 = wc[b][2 * lane], e1 = wc[b][2 * lane + 1];
            int32_t v = e0 + e1;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                int32_t t = __shfl_up_sync(0xffffffffu, v, o);
                if (lane >= o) v += t;
            }
            const int32_t ex = v - e0 - e1;
            wc[b][2 * lane] = ex;
            wc[b][2 * lane + 1] = ex + e0;
        }
    }
    __syncthreads();
    int32_t tile0[3];
#pragma unroll
    for (int b = 0; b < 3; ++b) tile0[b] = bsum[(int64_t)b * nb + blockIdx.x];
#pragma unroll
    for (int k = 0; k < kPartItems; ++k) {
        const int64_t p = base + (int64_t)k * kPartThreads + threadIdx.x;
        const bool valid = seg[k] >= 0;
        SegRec sr{0, 0, 0, 0, 0, 0, 0, 0};
        if (valid) sr = segs[seg[k]];
        const int ks = sr.k, lo = sr.lo;
        if (valid) node_of_next[p] = sr.child + ((ks > 0 && (int)p - lo >= ks) ? 1 : 0);
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            const bool left = (f[k] >> b) & 1u;
            const unsigned m = __ballot_sync(0xffffffffu, left);
            if (!valid) continue;
            const int32_t r0 = L.A[b][0][p], r1 = L.A[b][1][p];
            int64_t np = p;
            if (ks > 0) {
                // left-going entries before p in this segment
                const int lb = tile0[b] + wc[b][k * kPartWarps + warp] + __popc(m & below) - sr.leftbase;
                np = left ? lo + lb : lo + ks + ((int)p - lo - lb);
                if (!(np >= lo && np < sr.hi)) {
                    atomicAdd(err, 1);  // inconsistent partition: reported, never written out of the segment
                    continue;
                }
            }
            O.A[b][0][np] = r0;
            O.A[b][1][np] = r1;
        }
    }
}

// --- RCB bottom levels in shared memory --------------------------------------
// Once every segment of a level holds at most kLocalCap entries, one block
// takes one segment and runs all the remaining levels on it in shared memory:
// the same boxes, axes, rank thresholds and stable partitions as the level
// kernels above (so the same tree, bit for bit), but a level costs a few
// shared-memory passes instead of three DRAM passes over the six rank
// columns.  The block ends by writing the final member order of its range.
// The three levels before that run in clusters of up to eight such blocks per segment (at most 16384
// entries): a streamed level is two launches that wait on chains of dependent loads, 25 us at any size
// below 2M particles.  Three levels take 12 us more in this kernel instead of 75 on 30,011 particles and
// 40 us instead of 80 on 2x64^3.  Only while the clusters fit in one wave of resident blocks: beyond that
// the remote stores are slower than the streamed levels (2x256^3 5.5 ms against 4.5, 24 boxes 537 us
// against 380).
constexpr int kLocalCap = 2048;
constexpr int kLocalThreads = 512;
constexpr int kLocalBlocks = 2;                         // resident blocks per SM (shared memory: ~113 KB each)
constexpr int kLocalItems = kLocalCap / kLocalThreads;  // consecutive positions per thread
constexpr int kLocalLevels = 7;                         // levels one block may run
constexpr int kLocalSegs = 1 << kLocalLevels;           // segments per block at its deepest level
constexpr int kClusterLevels = 3;                       // levels a cluster of blocks runs before
constexpr int kClusterBlocks = 1 << kClusterLevels;
constexpr size_t kLocalSmem = sizeof(int32_t) * 2 * 6 * kLocalCap + sizeof(int16_t) * 2 * kLocalCap;
static_assert(kLocalItems == 4, "positions are moved as int4");

// the level tables a block walks: tab[l] = 7 columns of m[l] segments (lo, hi, k, child, node, axis, leftbase)
struct LocalShape {
    int32_t *tab[kClusterLevels + kLocalLevels];
    int32_t m[kClusterLevels + kLocalLevels];
    int pre, nlev;  // levels run by clusters of 2^pre blocks, all levels
};

struct __align__(16) LocalSeg {
    int32_t lo, hi, k, child;  // lo, hi relative to the block's range; child relative to the next level's first
    int32_t axis, thr, lb, pad;  // lb: left entries of the block's earlier segments (every list alike)
};

// three 21-bit counters in one word (at most kLocalCap per counter)
__device__ __forceinline__ uint64_t pack3(unsigned f) {
    return (uint64_t)(f & 1u) | ((uint64_t)((f >> 1) & 1u) << 21) | ((uint64_t)((f >> 2) & 1u) << 42);
}
__device__ __forceinline__ int field3(uint64_t v, int b) { return (int)((v >> (21 * b)) & 0x1fffffu); }

template <bool kClusters>
__global__ void __launch_bounds__(kLocalThreads, kLocalBlocks) rcb_local_kernel(int64_t n, LocalShape sh, RankLists L, AxisOrder o,
                                                                       const float *__restrict__ x,
                                                                       const float *__restrict__ y,
                                                                       const float *__restrict__ z,
                                                                       float *__restrict__ node_box,
                                                                       int32_t *__restrict__ members,
                                                                       int32_t *__restrict__ rank_y,
                                                                       int32_t *__restrict__ rank_z,
                                                                       int32_t *__restrict__ err) {
    extern __shared__ int4 local_smem[];
    int32_t *cur = reinterpret_cast<int32_t *>(local_smem);  // [6][kLocalCap]: column 2b + c of list b
    int32_t *nxt = cur + 6 * kLocalCap;
    int16_t *sc = reinterpret_cast<int16_t *>(nxt + 6 * kLocalCap);  // segment of each position
    int16_t *sn = sc + kLocalCap;
    __shared__ LocalSeg seg[kLocalSegs];
    __shared__ uint64_t wsum[kLocalThreads / 32];
    __shared__ uint64_t rows[64], totals[kClusterBlocks];  // cluster levels: left counts of the rows, of the blocks,
    __shared__ int own[kClusterBlocks + 1];                // and the positions that each block keeps
    __shared__ int bad;
    const int t = threadIdx.x, lane = t & 31, w = t >> 5;
    const unsigned below = lanemask_lt_u();
    // this block's segment at its first level of its own, and those of the blocks of its cluster (the
    // children of a level's neighbouring segments follow one another)
    const int pre = kClusters ? sh.pre : 0, top = blockIdx.x >> pre, rank = blockIdx.x - (top << pre);
    int f = top, e = f + 1;
    if constexpr (kClusters) {
        for (int lev = 0; lev < pre; ++lev) {
            const int32_t *tab = sh.tab[lev];
            const int m = sh.m[lev], fn = tab[3 * m + f];
            e = tab[3 * m + e - 1] + (tab[2 * m + e - 1] > 0 ? 2 : 1);
            f = fn;
        }
    }
    const int32_t *t0 = sh.tab[pre];
    const int m0 = sh.m[pre], nown = e - f, s0 = f + rank;
    const int lo = rank < nown ? t0[s0] : t0[m0 + e - 1], cnt = rank < nown ? t0[m0 + s0] - lo : 0;
    if (t == 0) bad = 0;
    bool over = nown > (1 << pre);
    for (int r = 0; r < nown; ++r) over |= t0[m0 + f + r] - t0[f + r] > kLocalCap;
    if (over) {  // excluded by the host's choice of levels; the whole cluster leaves
        if (t == 0) atomicAdd(err, 1);
        return;
    }
    for (int q = t; q < cnt; q += kLocalThreads) {
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            cur[(2 * b) * kLocalCap + q] = L.A[b][0][lo + q];
            cur[(2 * b + 1) * kLocalCap + q] = L.A[b][1][lo + q];
        }
        sc[q] = 0;
    }
    const float *cs[3] = {x, y, z};
    // a rank used as an index; a partition found inconsistent (reported through err) may leave
    // positions unwritten, whose values then never index out of the arrays
    auto rk = [n](int32_t r) -> int64_t { return (uint64_t)r < (uint64_t)n ? r : 0; };
    // The records of the ns segments from f on, positions relative to `base`: the tight box from the ends
    // of the three list segments (entry p of list a: rank along axis (a + 1) % 3 in column 2 a), the axis
    // and the threshold.
    auto records = [&](int32_t *tab, int m, int f, int ns, int base, bool store, auto entry) {
        for (int u = t; u < ns; u += kLocalThreads) {
            const int s = f + u;
            LocalSeg r{tab[s] - base, tab[m + s] - base, tab[2 * m + s], tab[3 * m + s] - tab[3 * m + f], 0, 0,
                       tab[6 * m + s] - tab[6 * m + f], 0};
            const int k = r.k;
            if (k > 0) {
                float blo[3], bhi[3];
                double ext[3];
                for (int a = 0; a < 3; ++a) {
                    const int32_t *S = o.S[(a + 1) % 3];
                    blo[a] = cs[a][S[rk(entry(2 * a, r.lo))]];
                    bhi[a] = cs[a][S[rk(entry(2 * a, r.hi - 1))]];
                    ext[a] = __dsub_rn((double)bhi[a], (double)blo[a]);
                }
                int axis = 0;
                if (ext[1] > ext[axis]) axis = 1;
                if (ext[2] > ext[axis]) axis = 2;
                r.axis = axis;
                r.thr = o.R[axis][o.S[(axis + 1) % 3][rk(entry(2 * axis, r.lo + k))]];
                if (store) {
                    tab[5 * m + s] = axis;
                    float *nb = node_box + 6 * (int64_t)tab[4 * m + s];
                    for (int a = 0; a < 3; ++a) {
                        nb[a] = blo[a];
                        nb[3 + a] = bhi[a];
                    }
                }
            }
            seg[u] = r;
        }
    };
    // is entry q (relative to the segments' base; the block's entry ql) of list b in the left part
    auto goes_left = [&](const LocalSeg &r, int b, int q, int ql) {
        if (b == r.axis) return q - r.lo < r.k;
        const int c = (r.axis - b + 2) % 3;  // column of list b holding ranks along the axis
        return cur[(2 * b + c) * kLocalCap + ql] < r.thr;
    };
    // ---- levels of the cluster: each block keeps the positions that are its segment's in the end; entries
    // move to their block's next columns through distributed shared memory
    if constexpr (kClusters) {
        const int LO = t0[f];
        const cooperative_groups::cluster_group cl = cooperative_groups::this_cluster();
        if (t <= kClusterBlocks) own[t] = (t < nown ? t0[f + t] : t0[m0 + e - 1]) - LO;
        __syncthreads();
        auto owner = [&](int q) {
            int r = 0;  // own[] of the missing blocks is the end
#pragma unroll
            for (int d = kClusterBlocks / 2; d; d >>= 1) r += q >= own[r + d] ? d : 0;
            return min(r, nown - 1);
        };
        const int to = lo - LO;
        int fp = top, ep = top + 1;
        for (int lev = 0; lev < pre; ++lev) {
            int32_t *tab = sh.tab[lev];
            const int m = sh.m[lev], ns = ep - fp;  // at most 2^lev
            cl.sync();  // every block's columns of this level are in place
            records(tab, m, fp, ns, LO, rank == 0, [&](int col, int q) {
                const int b = owner(q);
                return cl.map_shared_rank(cur, b)[col * kLocalCap + q - own[b]];
            });
            __syncthreads();
            // entries in rows of one per thread, so that a warp's left-going and right-going ones are two
            // runs of words in the other blocks' memory (remote stores cost by the packet)
            unsigned fl[kLocalItems];
            int sg[kLocalItems];
#pragma unroll
            for (int i = 0; i < kLocalItems; ++i) {
                const int ql = i * kLocalThreads + t, q = to + ql;
                fl[i] = 0u;
                sg[i] = 0;
                for (int s = 1; s < ns; ++s) sg[i] += q >= seg[s].lo;
                const LocalSeg &r = seg[sg[i]];
                if (ql < cnt && r.k > 0) {
#pragma unroll
                    for (int b = 0; b < 3; ++b) fl[i] |= (unsigned)goes_left(r, b, q, ql) << b;
                }
                uint64_t c3 = 0;
#pragma unroll
                for (int b = 0; b < 3; ++b)
                    c3 |= (uint64_t)__popc(__ballot_sync(CRK_FULL_MASK, (fl[i] >> b) & 1u)) << (21 * b);
                if (lane == 0) rows[i * (kLocalThreads / 32) + w] = c3;
            }
            __syncthreads();
            if (w == 0) {  // exclusive scan of the rows' counts, two per lane
                static_assert(kLocalItems * (kLocalThreads / 32) == 64, "two counts per lane");
                const uint64_t v0 = rows[2 * lane], v = v0 + rows[2 * lane + 1];
                uint64_t iv = v;
#pragma unroll
                for (int d = 1; d < 32; d <<= 1) {
                    const uint64_t u = __shfl_up_sync(CRK_FULL_MASK, iv, d);
                    if (lane >= d) iv += u;
                }
                rows[2 * lane] = iv - v;
                rows[2 * lane + 1] = iv - v + v0;
                const uint64_t total = __shfl_sync(CRK_FULL_MASK, iv, 31);
                if (lane < (1 << pre)) cl.map_shared_rank(totals, lane)[rank] = total;
            }
            cl.sync();
            uint64_t before = 0;
            for (int r = 0; r < rank; ++r) before += totals[r];
#pragma unroll
            for (int i = 0; i < kLocalItems; ++i) {
                const int ql = i * kLocalThreads + t, q = to + ql;
                const LocalSeg &r = seg[sg[i]];
                const uint64_t run = before + rows[i * (kLocalThreads / 32) + w];
#pragma unroll
                for (int b = 0; b < 3; ++b) {
                    const bool left = (fl[i] >> b) & 1u;
                    const unsigned mk = __ballot_sync(CRK_FULL_MASK, left);
                    if (ql >= cnt) continue;
                    int np = q;
                    if (r.k > 0) {
                        const int lb = field3(run, b) + __popc(mk & below) - r.lb;
                        np = left ? r.lo + lb : r.lo + r.k + (q - r.lo - lb);
                        if (!(np >= r.lo && np < r.hi)) {
                            bad = 1;  // as below
                            continue;
                        }
                    }
                    const int ob = owner(np);
                    int32_t *dst = cl.map_shared_rank(nxt, ob) + np - own[ob];
                    dst[(2 * b) * kLocalCap] = cur[(2 * b) * kLocalCap + ql];
                    dst[(2 * b + 1) * kLocalCap] = cur[(2 * b + 1) * kLocalCap + ql];
                }
            }
            int32_t *tp = cur;
            cur = nxt;
            nxt = tp;
            const int fn = tab[3 * m + fp];
            ep = tab[3 * m + ep - 1] + (tab[2 * m + ep - 1] > 0 ? 2 : 1);
            fp = fn;
        }
        cl.sync();  // no block touches another one's memory from here on
        if (rank >= nown) return;
    }
    f = s0;
    e = s0 + 1;  // this block's segments at the current level
    for (int lev = pre; lev < sh.nlev; ++lev) {
        int32_t *tab = sh.tab[lev];
        const int m = sh.m[lev];
        const int ns = e - f;
        __syncthreads();  // the previous level is done with seg[], cur and sc
        if (ns > kLocalSegs) {  // excluded by the host's choice of levels
            if (t == 0) atomicAdd(err, 1);
            return;
        }
        records(tab, m, f, ns, lo, true, [&](int col, int q) { return cur[col * kLocalCap + q]; });
        // the next level's range of this block's segments
        const int fn = tab[3 * m + f];
        const int en = tab[3 * m + e - 1] + (tab[2 * m + e - 1] > 0 ? 2 : 1);
        __syncthreads();
        // left flags of this thread's kLocalItems consecutive positions (bit b: list b)
        const int q0 = t * kLocalItems;
        unsigned fl[kLocalItems];
        int sg[kLocalItems];
        uint64_t mine = 0;
#pragma unroll
        for (int i = 0; i < kLocalItems; ++i) {
            const int q = q0 + i;
            fl[i] = 0u;
            sg[i] = 0;
            if (q < cnt) {
                sg[i] = sc[q];
                const LocalSeg &r = seg[sg[i]];
                if (r.k > 0) {
#pragma unroll
                    for (int b = 0; b < 3; ++b) fl[i] |= (unsigned)goes_left(r, b, q, q) << b;
                }
                mine += pack3(fl[i]);
            }
        }
        // block exclusive scan of the three counters
        uint64_t incl = mine;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const uint64_t v = __shfl_up_sync(CRK_FULL_MASK, incl, d);
            if (lane >= d) incl += v;
        }
        if (lane == 31) wsum[w] = incl;
        __syncthreads();
        if (w == 0) {
            constexpr int kW = kLocalThreads / 32;
            uint64_t v = lane < kW ? wsum[lane] : 0, iv = v;
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const uint64_t u = __shfl_up_sync(CRK_FULL_MASK, iv, d);
                if (lane >= d) iv += u;
            }
            if (lane < kW) wsum[lane] = iv - v;
        }
        __syncthreads();
        uint64_t run = wsum[w] + incl - mine;
        // stable partition into nxt; the segment of each new position
#pragma unroll
        for (int i = 0; i < kLocalItems; ++i) {
            const int q = q0 + i;
            if (q >= cnt) break;
            const LocalSeg &r = seg[sg[i]];
#pragma unroll
            for (int b = 0; b < 3; ++b) {
                int np = q;
                if (r.k > 0) {
                    const int lb = field3(run, b) - r.lb;  // left entries before q in its segment
                    np = (fl[i] >> b) & 1u ? r.lo + lb : r.lo + r.k + (q - r.lo - lb);
                    if (!(np >= r.lo && np < r.hi)) {
                        bad = 1;  // inconsistent partition: reported, never written out of the segment
                        continue;
                    }
                }
                nxt[(2 * b) * kLocalCap + np] = cur[(2 * b) * kLocalCap + q];
                nxt[(2 * b + 1) * kLocalCap + np] = cur[(2 * b + 1) * kLocalCap + q];
            }
            sn[q] = (int16_t)(r.child + ((r.k > 0 && q - r.lo >= r.k) ? 1 : 0));
            run += pack3(fl[i]);
        }
        int32_t *tp = cur;
        cur = nxt;
        nxt = tp;
        int16_t *ts = sc;
        sc = sn;
        sn = ts;
        f = fn;
        e = en;
    }
    __syncthreads();
    if (t == 0 && bad) atomicAdd(err, 1);
    for (int q = t; q < cnt; q += kLocalThreads) {  // list 0: its columns are the ranks along y and z
        const int32_t ry = cur[q];
        members[lo + q] = o.S[1][rk(ry)];
        rank_y[lo + q] = ry;
        rank_z[lo + q] = cur[kLocalCap + q];
    }
}

// --- per-leaf data ------------------------------------------------------------
__device__ __forceinline__ uint32_t spread10(uint32_t v) {
    v &= 1023u;
    v = (v | (v << 16)) & 0x030000FFu;
    v = (v | (v << 8)) & 0x0300F00Fu;
    v = (v | (v << 4)) & 0x030C30C3u;
    v = (v | (v << 2)) & 0x09249249u;
    return v;
}

// box of the 32 leaf-relative positions r of a warp into cell[0] (lo, largest h), cell[1] (hi): the
// coordinates and h are >= 0 (-0 + 0 = 0), so their bits order like the values
__device__ __forceinline__ void store_cell(float4 *cell, const float4 &r, int lane) {
    const unsigned bits[3] = {__float_as_uint(r.x + 0.0f), __float_as_uint(r.y + 0.0f), __float_as_uint(r.z + 0.0f)};
    float l[3], u[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        l[k] = __uint_as_float(__reduce_min_sync(CRK_FULL_MASK, bits[k]));
        u[k] = __uint_as_float(__reduce_max_sync(CRK_FULL_MASK, bits[k]));
    }
    const float hm = __uint_as_float(__reduce_max_sync(CRK_FULL_MASK, __float_as_uint(r.w)));
    if (lane == 0) {
        cell[0] = make_float4(l[0], l[1], l[2], hm);
        cell[1] = make_float4(u[0], u[1], u[2], 0.0f);
    }
}

// Shared state of bisect32 (one per block) for leaves of at most kCap members.
template <int kCap>
struct Bisect32 {
    static constexpr int kMaxSeg = kCap / 32;
    int16_t a[kCap], b[kCap];  // orders (member slots), double-buffered
    float cax[kCap];           // coordinate of the member at each position on its part's axis
    uint32_t cid[kCap];        // its particle index (ties)
    int lo[kMaxSeg], hi[kMaxSeg], ax[kMaxSeg];
    int nseg, more;
};

// Bisects positions [0, m) of the order bs.a (member slots; m <= kCap) into
// groups of 32: each part above 32 is ranked along the longest extent of its
// members in (coordinate, index) order and split with 32 ceil(g/2) of its g
// groups of 32 on the left, until every part holds at most 32; then every run
// of 32 positions starting at a multiple of 32 is an RCB cell.  At most
// ceil(m/32) <= 32 parts, one per lane of warp 0.  All threads call it; returns
// the array (bs.a or bs.b) holding the result in [0, m).
template <int kCap>
__device__ int16_t *bisect32(Bisect32<kCap> &bs, int m, const float4 *pm, const uint64_t *key) {
    constexpr int U = 32;
    static_assert(kCap / U <= Bisect32<kCap>::kMaxSeg && kCap / U <= 32, "parts per leaf");
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
    int16_t *src = bs.a, *dst = bs.b;
    if (threadIdx.x == 0) {
        bs.nseg = 1;
        bs.lo[0] = 0;
        bs.hi[0] = m;
        bs.more = m > U;
    }
    __syncthreads();
    while (bs.more) {
        // axis of the longest extent of every part above 32 (one warp per part)
        for (int sg = w; sg < bs.nseg; sg += nw) {
            const int l = bs.lo[sg], hh = bs.hi[sg];
            if (hh - l <= U) {
                if (lane == 0) bs.ax[sg] = -1;
                continue;
            }
            float mn[3] = {INFINITY, INFINITY, INFINITY}, mx[3] = {-INFINITY, -INFINITY, -INFINITY};
            for (int u = l + lane; u < hh; u += 32) {
                const float4 c = pm[src[u]];
                mn[0] = fminf(mn[0], c.x); mx[0] = fmaxf(mx[0], c.x);
                mn[1] = fminf(mn[1], c.y); mx[1] = fmaxf(mx[1], c.y);
                mn[2] = fminf(mn[2], c.z); mx[2] = fmaxf(mx[2], c.z);
            }
            for (int o = 16; o > 0; o >>= 1)
                for (int q = 0; q < 3; ++q) {
                    mn[q] = fminf(mn[q], __shfl_xor_sync(CRK_FULL_MASK, mn[q], o));
                    mx[q] = fmaxf(mx[q], __shfl_xor_sync(CRK_FULL_MASK, mx[q], o));
                }
            const float e0 = mx[0] - mn[0], e1 = mx[1] - mn[1], e2 = mx[2] - mn[2];
            if (lane == 0) bs.ax[sg] = (e0 >= e1 && e0 >= e2) ? 0 : (e1 >= e2 ? 1 : 2);
        }
        __syncthreads();
        // each position's key on its part's axis, so the ranking reads two flat arrays
        for (int q = threadIdx.x; q < m; q += blockDim.x) {
            int sg = 0;
            while (bs.hi[sg] <= q) ++sg;
            const int ax = bs.ax[sg], t = src[q];
            const float4 c = pm[t];
            bs.cax[q] = ax == 0 ? c.x : (ax == 1 ? c.y : c.z);
            bs.cid[q] = (uint32_t)key[t];
        }
        __syncthreads();
        for (int q = threadIdx.x; q < m; q += blockDim.x) {
            int sg = 0;
            while (bs.hi[sg] <= q) ++sg;
            if (bs.ax[sg] < 0) {
                dst[q] = src[q];
                continue;
            }
            const float cv = bs.cax[q];
            const uint32_t iv = bs.cid[q];
            const int l = bs.lo[sg], hh = bs.hi[sg];
            int r = 0;
            for (int u = l; u < hh; ++u) {
                const float cu = bs.cax[u];
                r += (cu < cv) || (cu == cv && bs.cid[u] < iv);
            }
            dst[l + r] = src[q];
        }
        __syncthreads();
        if (w == 0) {
            // the children of every part, in order (one part per lane)
            const bool have = lane < bs.nseg;
            const int l = have ? bs.lo[lane] : 0, hh = have ? bs.hi[lane] : 0;
            const bool split = have && bs.ax[lane] >= 0;
            const int nch = have ? (split ? 2 : 1) : 0;
            int off = nch;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int v = __shfl_up_sync(CRK_FULL_MASK, off, o);
                if (lane >= o) off += v;
            }
            const int total = __shfl_sync(CRK_FULL_MASK, off, 31);
            off -= nch;
            const int g = (hh - l + U - 1) / U;
            const int left = split ? U * ((g + 1) / 2) : hh - l;
            __syncwarp();
            if (have) {
                bs.lo[off] = l;
                bs.hi[off] = l + left;
                if (split) {
                    bs.lo[off + 1] = l + left;
                    bs.hi[off + 1] = hh;
                }
            }
            const bool open = have && (left > U || (split && hh - l - left > U));
            const bool any = __any_sync(CRK_FULL_MASK, open);
            if (lane == 0) {
                bs.nseg = total;
                bs.more = any;
            }
        }
        __syncthreads();
        int16_t *tmp = src;
        src = dst;
        dst = tmp;
    }
    return src;
}

// One block per leaf: tight box, gas count, largest gas h; the canonical
// order (gas first, then dark matter, each by index) for export; the gas
// kernel order (gas first, then dark matter, each along a Z-order curve of the
// leaf box, ties by index; the gas part bisected into groups of 32 as below; RCB
// leaves of at most 128 have the kernel below, which takes both in canonical
// order instead, so that a part of at most 32 gas particles stays in index
// order); the gravity kernel order (species mixed): the leaf bisected into groups of 32,
// each split along the longest extent of its part in (coordinate, index)
// order with a multiple of 32 particles on the left, so that every group of 32
// consecutive particles is an RCB cell (the gravity tiles sweep the
// candidates within r_c of a group's box: at r_c = 3 such cells cut the
// candidates per in-range pair from ~4.0 to ~3.3 against Z-order groups); and
// the leaf-relative positions in both kernel orders.
// kCap: the largest leaf the launch may meet.
template <int kCap>
__global__ void leaf_data_kernel(int64_t n_leaves, const int32_t *__restrict__ leaf_start,
                                 const int32_t *__restrict__ members, const float *__restrict__ x,
                                 const float *__restrict__ y, const float *__restrict__ z,
                                 const uint8_t *__restrict__ sp, const float *__restrict__ h,
                                 int32_t *__restrict__ perm, int32_t *__restrict__ kperm,
                                 int32_t *__restrict__ leaf_ngas, float *__restrict__ bbox,
                                 float *__restrict__ hmax, float4 *__restrict__ pos, int32_t *__restrict__ kperm_g,
                                 float4 *__restrict__ pos_g, int32_t *__restrict__ kinv, int32_t *__restrict__ kinv_g,
                                 float4 *__restrict__ gcell, float4 *__restrict__ hcell, int32_t *__restrict__ err) {
    __shared__ uint64_t key[kCap], zkey[kCap];
    __shared__ Bisect32<kCap> bs;
    __shared__ float4 pm[kCap];  // member position and h (0 for dark matter), gathered once
    __shared__ float red[6][32];
    __shared__ int ngs[32];
    __shared__ float hms[32];
    const int64_t a = blockIdx.x;
    if (a >= n_leaves) return;
    const int lo = leaf_start[a], hi = leaf_start[a + 1], cnt = hi - lo;
    if (cnt > kCap) {
        if (threadIdx.x == 0) atomicAdd(err, 1);
        return;
    }
    float mn[3] = {INFINITY, INFINITY, INFINITY}, mx[3] = {-INFINITY, -INFINITY, -INFINITY};
    int ng = 0;
    float hm = 0.0f;
    for (int t = threadIdx.x; t < cnt; t += blockDim.x) {
        int32_t id = members[lo + t];
        const bool gas = sp[id] == 0;
        key[t] = ((uint64_t)!gas << 32) | (uint32_t)id;
        float c[3] = {x[id], y[id], z[id]};
        const float hh = gas ? h[id] : 0.0f;
        pm[t] = make_float4(c[0], c[1], c[2], hh);
        for (int q = 0; q < 3; ++q) {
            mn[q] = fminf(mn[q], c[q]);
            mx[q] = fmaxf(mx[q], c[q]);
        }
        if (gas) {
            ++ng;
            hm = fmaxf(hm, hh);
        }
    }
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
    for (int o = 16; o > 0; o >>= 1) {
        for (int q = 0; q < 3; ++q) {
            mn[q] = fminf(mn[q], __shfl_xor_sync(CRK_FULL_MASK, mn[q], o));
            mx[q] = fmaxf(mx[q], __shfl_xor_sync(CRK_FULL_MASK, mx[q], o));
        }
        ng += __shfl_xor_sync(CRK_FULL_MASK, ng, o);
        hm = fmaxf(hm, __shfl_xor_sync(CRK_FULL_MASK, hm, o));
    }
    if (lane == 0) {
        for (int q = 0; q < 3; ++q) {
            red[q][w] = mn[q];
            red[3 + q][w] = mx[q];
        }
        ngs[w] = ng;
        hms[w] = hm;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int v = 1; v < nw; ++v) {
            for (int q = 0; q < 3; ++q) {
                red[q][0] = fminf(red[q][0], red[q][v]);
                red[3 + q][0] = fmaxf(red[3 + q][0], red[3 + q][v]);
            }
            ngs[0] += ngs[v];
            hms[0] = fmaxf(hms[0], hms[v]);
        }
        for (int q = 0; q < 6; ++q) bbox[6 * a + q] = red[q][0];
        leaf_ngas[a] = ngs[0];
        hmax[a] = hms[0];
    }
    __syncthreads();
    const float ox = red[0][0], oy = red[1][0], oz = red[2][0];
    const float ext = fmaxf(fmaxf(red[3][0] - ox, red[4][0] - oy), fmaxf(red[5][0] - oz, 1e-30f));
    const float sc = 1023.0f / ext;
    // canonical ranks, and the Z-order keys of each member: zkey with the
    // species on top (gas first), gkey without (gravity order)
    for (int t = threadIdx.x; t < cnt; t += blockDim.x) {
        uint64_t kt = key[t];
        int r = 0;
        for (int u = 0; u < cnt; ++u) r += key[u] < kt;
        int32_t id = (int32_t)(uint32_t)kt;
        perm[lo + r] = id;
        const float4 c = pm[t];
        uint32_t mx3 = spread10((uint32_t)fminf((c.x - ox) * sc, 1023.0f)) |
                       (spread10((uint32_t)fminf((c.y - oy) * sc, 1023.0f)) << 1) |
                       (spread10((uint32_t)fminf((c.z - oz) * sc, 1023.0f)) << 2);
        zkey[t] = ((kt >> 32) << 62) | ((uint64_t)mx3 << 32) | (uint32_t)id;
    }
    __syncthreads();
    // gas order: gas first, then dark matter, each along the Z curve; then the gas part
    // bisected into groups of 32 (dark matter keeps the Z order)
    for (int t = threadIdx.x; t < cnt; t += blockDim.x) {
        uint64_t kt = zkey[t];
        int r = 0;
        for (int u = 0; u < cnt; ++u) r += zkey[u] < kt;
        bs.a[r] = (int16_t)t;
        bs.b[r] = (int16_t)t;
    }
    const int16_t *gsrc = bisect32(bs, ngs[0], pm, key);
    for (int q = threadIdx.x; q < cnt; q += blockDim.x) {
        const int t = gsrc[q];
        const float4 c = pm[t];
        const int32_t id = (int32_t)(uint32_t)key[t];
        kperm[lo + q] = id;
        kinv[id] = lo + q;  // the inverse permutations, written here rather than by a pass of their own
        pos[lo + q] = make_float4(c.x - ox, c.y - oy, c.z - oz, c.w);
    }
    for (int q0 = w * 32; q0 < ngs[0]; q0 += nw * 32) {  // boxes of the gas cells of 32
        const float4 c = pm[gsrc[q0 + lane < ngs[0] ? q0 + lane : ngs[0] - 1]];
        store_cell(hcell + 2 * ((int64_t)(lo >> 5) + a + (q0 >> 5)), make_float4(c.x - ox, c.y - oy, c.z - oz, c.w), lane);
    }
    __syncthreads();
    // gravity order: the whole leaf bisected into groups of 32
    for (int t = threadIdx.x; t < cnt; t += blockDim.x) bs.a[t] = (int16_t)t;
    int16_t *src = bisect32(bs, cnt, pm, key);
    for (int q0 = w * 32; q0 < cnt; q0 += nw * 32) {  // one warp per cell of 32
        const int q = q0 + lane;
        const int t = src[q < cnt ? q : cnt - 1];
        const float4 c = pm[t];
        const float4 r = make_float4(c.x - ox, c.y - oy, c.z - oz, c.w);
        if (q < cnt) {
            const int32_t id = (int32_t)(uint32_t)key[t];
            kperm_g[lo + q] = id;
            kinv_g[id] = lo + q;
            pos_g[lo + q] = r;
        }
        store_cell(gcell + 2 * ((int64_t)(lo >> 5) + a + (q0 >> 5)), r, lane);
    }
}

// The same for RCB leaves of at most kRcbLeaf members, with the gravity order bisected down to
// cells of 8.  Members arrive in x order with their ranks along y and z (integers, all different,
// ordered like (coordinate, index)), so every order inside the leaf follows from one ranking per
// axis (7-bit local ranks) and no coordinate is compared again:
//   * the ranking counts smaller 32-bit keys, four to a shared-memory load;
//   * a part's extents are the coordinates of its lowest and highest ranks (warp min and max);
//   * the rank inside a part counts the smaller local ranks four to a word: with 7-bit values the
//     byte differences of (rank | 0x80) - w never borrow, and bit 7 says rank >= w.
// What bounds it is issue and the chain of levels.  33.5M particles: 8.4 ms for the general kernel
// above with cells of 8, 5.2 here; 2x64^3: 156 -> 72 us; 30,011 particles: 71 -> 12.5 us.
constexpr int kRcbLeaf = 128;
struct LeafParts {
    int lo[2][kRcbLeaf / 8], hi[2][kRcbLeaf / 8];  // bounds of the parts, double-buffered
    int ax[kRcbLeaf / 8], left[kRcbLeaf / 8];      // split axis (-1: none), members that go left
    unsigned split[2];                             // parts that split
    uint8_t part[2][kRcbLeaf];                     // part of each position
    __align__(8) uint8_t ab[kRcbLeaf];             // local rank of each position's member on its part's axis
    uint8_t rk[3][kRcbLeaf], ord[3][kRcbLeaf];     // local rank of a member, member of a local rank
};

// Bisects positions [0, m) of the order src: parts above 32 with a multiple of 32 on the left, then
// (cells8) parts above 8 with a multiple of 8; returns the buffer (src or dst) with the result.
__device__ uint8_t *bisect_ranks(LeafParts &lp, int m, const float4 *pm, uint8_t *src, uint8_t *dst, bool cells8) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
    __syncthreads();
    if (threadIdx.x == 0) {
        lp.lo[0][0] = 0;
        lp.hi[0][0] = m;
        lp.split[0] = 0u;
    }
    for (int q = threadIdx.x; q < kRcbLeaf; q += blockDim.x) {
        lp.part[0][q] = 0;
        if (q >= m) lp.ab[q] = 0;  // (a 7-bit value: the differences never borrow)
    }
    int np = 1, b = 0;
    for (;;) {
        __syncthreads();
        if (threadIdx.x == 0) lp.split[b ^ 1] = 0u;
        bool any = false;
        for (int p = w; p < np; p += nw) {
            const int l = lp.lo[b][p], h = lp.hi[b][p], len = h - l;
            const int U = len > 32 ? 32 : (cells8 && len > 8 ? 8 : 0);
            if (U == 0) {
                if (lane == 0) lp.ax[p] = -1;
                continue;
            }
            unsigned mn[3] = {255u, 255u, 255u}, mx[3] = {0u, 0u, 0u};
            for (int q = l + lane; q < h; q += 32) {
                const int t = src[q];
#pragma unroll
                for (int a = 0; a < 3; ++a) {
                    const unsigned v = lp.rk[a][t];
                    mn[a] = min(mn[a], v);
                    mx[a] = max(mx[a], v);
                }
            }
            float e[3];
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                const float4 c0 = pm[lp.ord[a][__reduce_min_sync(CRK_FULL_MASK, mn[a])]];
                const float4 c1 = pm[lp.ord[a][__reduce_max_sync(CRK_FULL_MASK, mx[a])]];
                e[a] = a == 0 ? c1.x - c0.x : (a == 1 ? c1.y - c0.y : c1.z - c0.z);
            }
            any = true;
            if (lane == 0) {
                lp.ax[p] = (e[0] >= e[1] && e[0] >= e[2]) ? 0 : (e[1] >= e[2] ? 1 : 2);
                lp.left[p] = U * (((len + U - 1) / U + 1) / 2);
                atomicOr(&lp.split[b], 1u << p);
            }
        }
        if (!__syncthreads_or(any)) return src;
        const unsigned split = lp.split[b];
        for (int q = threadIdx.x; q < m; q += blockDim.x) {
            const int ax = lp.ax[lp.part[b][q]];
            if (ax >= 0) lp.ab[q] = lp.rk[ax][src[q]];
        }
        if (threadIdx.x < np) {  // the children's bounds
            const int p = threadIdx.x, c = p + __popc(split & ((1u << p) - 1u));
            const int l = lp.lo[b][p], h = lp.hi[b][p];
            lp.lo[b ^ 1][c] = l;
            lp.hi[b ^ 1][c] = h;
            if (split >> p & 1u) {
                lp.hi[b ^ 1][c] = l + lp.left[p];
                lp.lo[b ^ 1][c + 1] = l + lp.left[p];
                lp.hi[b ^ 1][c + 1] = h;
            }
        }
        __syncthreads();
        for (int q = threadIdx.x; q < m; q += blockDim.x) {
            const int p = lp.part[b][q], c = p + __popc(split & ((1u << p) - 1u));
            int to = q, cp = c;
            if (split >> p & 1u) {
                const unsigned r = (unsigned)lp.ab[q] * 0x01010101u | 0x80808080u;
                const int l = lp.lo[b][p], h = lp.hi[b][p];
                unsigned n4 = 0u;  // four byte counters
                for (int u = l; u < h; u += 8) {  // parts start at multiples of 8; only the last may end inside a word
                    const uint2 v = *reinterpret_cast<const uint2 *>(lp.ab + u);
                    unsigned c0 = (r - v.x) >> 7 & 0x01010101u, c1 = (r - v.y) >> 7 & 0x01010101u;
                    if (u + 8 > h) {  // the bytes past the end do not count
                        c0 &= h - u >= 4 ? ~0u : (1u << (8 * (h - u))) - 1u;
                        c1 &= h - u <= 4 ? 0u : (1u << (8 * (h - u - 4))) - 1u;
                    }
                    n4 += c0 + c1;
                }
                const int rank = (int)((n4 * 0x01010101u) >> 24) - 1;  // (the member itself counted)
                to = l + rank;
                cp = c + (rank >= lp.left[p]);
            }
            dst[to] = src[q];
            lp.part[b ^ 1][to] = (uint8_t)cp;
        }
        np += __popc(split);
        b ^= 1;
        uint8_t *t = src;
        src = dst;
        dst = t;
    }
}

__global__ void __launch_bounds__(128) leaf_data_rcb_kernel(
    const int32_t *__restrict__ leaf_start, const int32_t *__restrict__ members, const int32_t *__restrict__ rank_y,
    const int32_t *__restrict__ rank_z, const float *__restrict__ x, const float *__restrict__ y,
    const float *__restrict__ z, const uint8_t *__restrict__ sp, const float *__restrict__ h, int32_t *__restrict__ perm,
    int32_t *__restrict__ kperm, int32_t *__restrict__ leaf_ngas, float *__restrict__ bbox, float *__restrict__ hmax,
    float4 *__restrict__ pos, int32_t *__restrict__ kperm_g, float4 *__restrict__ pos_g, int32_t *__restrict__ kinv,
    int32_t *__restrict__ kinv_g, float4 *__restrict__ gcell, float4 *__restrict__ hcell, int32_t *__restrict__ err) {
    __shared__ float4 pm[kRcbLeaf];                                  // member position and h (0 for dark matter)
    __shared__ uint4 key4[3][kRcbLeaf / 4];                          // dark matter << 31 | id; ranks along y, z
    __shared__ LeafParts lp;
    __shared__ uint8_t can[kRcbLeaf], oa[kRcbLeaf], ob[kRcbLeaf];    // canonical order; working orders
    __shared__ float red[6][4], hms[4];
    __shared__ int ngs[4];
    uint32_t *const key = reinterpret_cast<uint32_t *>(key4[0]), *const gy = reinterpret_cast<uint32_t *>(key4[1]),
                   *const gz = reinterpret_cast<uint32_t *>(key4[2]);
    const int64_t a = blockIdx.x;
    const int lo = leaf_start[a], m = leaf_start[a + 1] - lo;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
    if (m > kRcbLeaf) {  // excluded by the tree's shape
        if (threadIdx.x == 0) atomicAdd(err, 1);
        return;
    }
    float mn[3] = {INFINITY, INFINITY, INFINITY}, mx[3] = {-INFINITY, -INFINITY, -INFINITY};
    int ng = 0;
    float hm = 0.0f;
    for (int t = threadIdx.x; t < kRcbLeaf; t += blockDim.x) {
        if (t >= m) {
            key[t] = gy[t] = gz[t] = 0xffffffffu;
            continue;
        }
        // (every order starts as one of valid members: a partition found inconsistent, which is
        // reported through err, may leave ranks that are not all different)
        can[t] = oa[t] = ob[t] = lp.ord[0][t] = lp.ord[1][t] = lp.ord[2][t] = lp.rk[0][t] = (uint8_t)t;
        const int32_t id = members[lo + t];
        gy[t] = (uint32_t)rank_y[lo + t];
        gz[t] = (uint32_t)rank_z[lo + t];
        const bool gas = sp[id] == 0;
        key[t] = (gas ? 0u : 0x80000000u) | (uint32_t)id;  // ids are below 2^31
        const float c[3] = {x[id], y[id], z[id]};
        const float hh = gas ? h[id] : 0.0f;
        pm[t] = make_float4(c[0], c[1], c[2], hh);
        for (int q = 0; q < 3; ++q) {
            mn[q] = fminf(mn[q], c[q]);
            mx[q] = fmaxf(mx[q], c[q]);
        }
        if (gas) {
            ++ng;
            hm = fmaxf(hm, hh);
        }
    }
    for (int o = 16; o > 0; o >>= 1) {
        for (int q = 0; q < 3; ++q) {
            mn[q] = fminf(mn[q], __shfl_xor_sync(CRK_FULL_MASK, mn[q], o));
            mx[q] = fmaxf(mx[q], __shfl_xor_sync(CRK_FULL_MASK, mx[q], o));
        }
        hm = fmaxf(hm, __shfl_xor_sync(CRK_FULL_MASK, hm, o));
    }
    ng = __reduce_add_sync(CRK_FULL_MASK, ng);
    if (lane == 0) {
        for (int q = 0; q < 3; ++q) {
            red[q][w] = mn[q];
            red[3 + q][w] = mx[q];
        }
        ngs[w] = ng;
        hms[w] = hm;
    }
    __syncthreads();
    // the leaf's box, gas count and h_max, and its members' ranks: canonical, along y, along z
    float ox = red[0][0], oy = red[1][0], oz = red[2][0], ux = red[3][0], uy = red[4][0], uz = red[5][0];
    ng = ngs[0];
    hm = hms[0];
    for (int v = 1; v < nw; ++v) {
        ox = fminf(ox, red[0][v]); oy = fminf(oy, red[1][v]); oz = fminf(oz, red[2][v]);
        ux = fmaxf(ux, red[3][v]); uy = fmaxf(uy, red[4][v]); uz = fmaxf(uz, red[5][v]);
        ng += ngs[v];
        hm = fmaxf(hm, hms[v]);
    }
    if (threadIdx.x == 0) {
        bbox[6 * a] = ox; bbox[6 * a + 1] = oy; bbox[6 * a + 2] = oz;
        bbox[6 * a + 3] = ux; bbox[6 * a + 4] = uy; bbox[6 * a + 5] = uz;
        leaf_ngas[a] = ng;
        hmax[a] = hm;
    }
    const int m4 = (m + 3) >> 2;
    for (int t = threadIdx.x; t < m; t += blockDim.x) {
        const uint32_t k = key[t], ky = gy[t], kz = gz[t];
        int r = 0, ry = 0, rz = 0;
#pragma unroll 4
        for (int u = 0; u < m4; ++u) {
            const uint4 c = key4[0][u], cy = key4[1][u], cz = key4[2][u];
            r += (c.x < k) + (c.y < k) + (c.z < k) + (c.w < k);
            ry += (cy.x < ky) + (cy.y < ky) + (cy.z < ky) + (cy.w < ky);
            rz += (cz.x < kz) + (cz.y < kz) + (cz.z < kz) + (cz.w < kz);
        }
        can[r] = (uint8_t)t;
        oa[r] = ob[r] = (uint8_t)t;
        perm[lo + r] = (int32_t)(k & 0x7fffffffu);
        lp.rk[1][t] = (uint8_t)ry;
        lp.rk[2][t] = (uint8_t)rz;
        lp.ord[1][ry] = (uint8_t)t;
        lp.ord[2][rz] = (uint8_t)t;
    }
    // gas order: gas first, bisected into groups of 32, then dark matter in canonical order
    const uint8_t *gsrc = bisect_ranks(lp, ng, pm, oa, ob, false);
    for (int q = threadIdx.x; q < m; q += blockDim.x) {
        const int t = q < ng ? gsrc[q] : can[q];
        const float4 c = pm[t];
        const int32_t id = (int32_t)(key[t] & 0x7fffffffu);
        kperm[lo + q] = id;
        kinv[id] = lo + q;
        pos[lo + q] = make_float4(c.x - ox, c.y - oy, c.z - oz, c.w);
    }
    for (int q0 = w * 32; q0 < ng; q0 += nw * 32) {  // boxes of the gas cells of 32
        const float4 c = pm[gsrc[q0 + lane < ng ? q0 + lane : ng - 1]];
        store_cell(hcell + 2 * ((int64_t)(lo >> 5) + a + (q0 >> 5)), make_float4(c.x - ox, c.y - oy, c.z - oz, c.w), lane);
    }
    __syncthreads();
    // gravity order: every member, down to cells of 8
    for (int t = threadIdx.x; t < m; t += blockDim.x) oa[t] = (uint8_t)t;
    const uint8_t *src = bisect_ranks(lp, m, pm, oa, ob, true);
    for (int q0 = w * 32; q0 < m; q0 += nw * 32) {  // one warp per cell of 32
        const int q = q0 + lane;
        const int t = src[q < m ? q : m - 1];
        const float4 c = pm[t];
        const float4 r = make_float4(c.x - ox, c.y - oy, c.z - oz, c.w);
        if (q < m) {
            const int32_t id = (int32_t)(key[t] & 0x7fffffffu);
            kperm_g[lo + q] = id;
            kinv_g[id] = lo + q;
            pos_g[lo + q] = r;
        }
        store_cell(gcell + 2 * ((int64_t)(lo >> 5) + a + (q0 >> 5)), r, lane);
    }
}

// --- leaf-pair images ------------------------------------------------------------
struct TreeDev {
    const float *node_box;       // [nodes][6]
    const float *node_hmax;      // [nodes] largest gas h below the node
    const int32_t *node_left;    // child ids, -1 for leaves
    const int32_t *node_right;
    const int32_t *node_leaf;    // leaf id for leaves, -1 otherwise
    int32_t root;
};

// FP32 periodic box gap, used only to discard candidates that are clearly out
// of range (the caller adds a margin far above the FP32 rounding of the sums)
__device__ __forceinline__ float axis_gap32(float loa, float hia, float lob, float hib, float L) {
    float best = INFINITY;
#pragma unroll
    for (int k = -1; k <= 1; ++k) {
        float s = (float)k * L;
        float g = fmaxf(fmaxf((lob + s) - hia, (loa - hib) - s), 0.0f);
        best = fminf(best, g);
    }
    return best;
}

__device__ __forceinline__ bool clearly_apart(const float *A, const float *B, float L, float cut) {
    float gx = axis_gap32(A[0], A[3], B[0], B[3], L);
    float gy = axis_gap32(A[1], A[4], B[1], B[4], L);
    float gz = axis_gap32(A[2], A[5], B[2], B[5], L);
    float c = cut + 1e-5f * L + 1e-6f;
    return gx * gx + gy * gy + gz * gz > c * c;
}

__device__ __forceinline__ double axis_gap_shift(double loa, double hia, double lob, double hib, double s) {
    double t1 = __dsub_rn(__dadd_rn(lob, s), hia);
    double t2 = __dsub_rn(__dsub_rn(loa, hib), s);
    double g = t1 > t2 ? t1 : t2;
    return g < 0.0 ? 0.0 : g;
}

__device__ __forceinline__ double sum_sq(double gx, double gy, double gz) {
    return __dadd_rn(__dadd_rn(__dmul_rn(gx, gx), __dmul_rn(gy, gy)), __dmul_rn(gz, gz));
}

// The gaps of two leaves per axis and box shift (-L, 0, L), in FP32.
struct Gaps {
    float g[3][3];
};
__device__ __forceinline__ float pick3(const float g[3], int k) { return k == 0 ? g[0] : (k == 1 ? g[1] : g[2]); }

// The FP64 test of one image (A, B: the two leaf boxes).  A call of its own: inlined, its per-axis
// parts were hoisted out of the image loops and evaluated for every candidate.
__device__ __noinline__ bool image_inside(const float *A, const float *B, int ix, int iy, int iz, double L, double cut) {
    return sum_sq(axis_gap_shift(A[0], A[3], B[0], B[3], (double)(ix - 1) * L),
                  axis_gap_shift(A[1], A[4], B[1], B[4], (double)(iy - 1) * L),
                  axis_gap_shift(A[2], A[5], B[2], B[5], (double)(iz - 1) * L)) < __dmul_rn(cut, cut);
}

// The images of leaf B within cut of leaf A as bits 9 sx + 3 sy + sz (shift indices 0, 1, 2).  The
// decision is that of the FP64 gaps, squared and summed, against cut^2.  The FP32 gaps settle every
// image that is not within a margin far above their rounding of the cut: FP64 (1/64 of the FP32
// rate here) only sees those; square roots of cut^2 and two FP64 gap sums per candidate and list
// were the kernel's time before: 6.2 -> 1.5 ms on the 2x256^3 box.
__device__ __forceinline__ uint32_t image_mask(const float *A, const float *B, const Gaps &s, double L, double cut) {
    const float cf = (float)cut, m = 1e-5f * (float)L + 1e-6f, hi = cf + m, lo = cf - m;
    const float hi2 = hi * hi, lo2 = lo > 0.0f ? lo * lo : -1.0f;
    uint32_t keep[3];
#pragma unroll
    for (int q = 0; q < 3; ++q)
        keep[q] = (s.g[q][0] > hi ? 0u : 1u) | (s.g[q][1] > hi ? 0u : 2u) | (s.g[q][2] > hi ? 0u : 4u);
    uint32_t out = 0;
    for (uint32_t mx = keep[0]; mx; mx &= mx - 1) {
        const int ix = __ffs(mx) - 1;
        const float gx = pick3(s.g[0], ix);
        for (uint32_t my = keep[1]; my; my &= my - 1) {
            const int iy = __ffs(my) - 1;
            const float gy = pick3(s.g[1], iy);
            for (uint32_t mz = keep[2]; mz; mz &= mz - 1) {
                const int iz = __ffs(mz) - 1;
                const float gz = pick3(s.g[2], iz), d2 = gx * gx + gy * gy + gz * gz;
                bool in = d2 < lo2;
                if (!in && !(d2 > hi2)) in = image_inside(A, B, ix, iy, iz, L, cut);
                if (in) out |= 1u << (9 * ix + 3 * iy + iz);
            }
        }
    }
    return out;
}

// the float nearest b + (k - 1) L - a, each sum rounded to FP64 first; without a shift the FP32
// difference is that number (b - a is exact in FP64 or |b| < 2^-29 |a|).  A call of its own: inlined,
// the FP64 form was evaluated for every image and selected away.
__device__ __noinline__ float wrapped_shift(float b, float a, int k, double L) {
    return (float)__dsub_rn(__dadd_rn((double)b, (double)(k - 1) * L), (double)a);
}
__device__ __forceinline__ float image_shift(float b, float a, int k, double L) {
    return k == 1 ? __fsub_rn(__fadd_rn(b, 0.0f), a) : wrapped_shift(b, a, k, L);
}

// --- warp-cooperative leaf-pair finder ---------------------------------------------
// One warp per i-leaf.  The warp pops up to 32 tree nodes at a time from a
// shared-memory stack, tests them in parallel (FP32, with margin, against the
// larger of the gravity cut and the hydro cut bound), pushes the children of
// the survivors and collects surviving leaves.  The candidates are sorted,
// tested exactly (image_mask) for both lists, and
// the leaf's images are written with one atomic reservation per list, so each
// leaf's lists stay in ascending j-leaf order.
constexpr int kTravWarps = 4;
constexpr int kStackCap = 512;
constexpr int kCandCap = 1024;

struct PairOut {
    int32_t *start[4];  // gravity images, gravity pairs, hydro images, hydro pairs
    int32_t *count[4];
    crk_image *gimg, *himg;
    int32_t *gpair, *hpair;
    int64_t cap[4];
    unsigned long long *cursor;  // [4]
    int32_t *err;                // [0] traversal overflow, [1] output overflow
};

__device__ __forceinline__ int warp_excl_scan(int v, int lane, int &total) {
    int x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        int y = __shfl_up_sync(CRK_FULL_MASK, x, o);
        if (lane >= o) x += y;
    }
    total = __shfl_sync(CRK_FULL_MASK, x, 31);
    return x - v;
}

template <bool kBrute>
__global__ void __launch_bounds__(kTravWarps * 32) leaf_pairs_warp_kernel(
    int64_t n_leaves, const int32_t *__restrict__ leaf_start, const int32_t *__restrict__ leaf_ngas,
    const float *__restrict__ bbox, const float *__restrict__ hmax, TreeDev tree, double L0, double rc, PairOut o,
    const int32_t *__restrict__ leaf_box, const int32_t *__restrict__ box_root, const float *__restrict__ box_L) {
    // two per-warp buffers, each reused by a later phase (32 KB a block, five blocks per SM):
    // the traversal stack, then the sorted candidates; the candidates, then the image counts
    static_assert(kStackCap <= kCandCap, "stack inside the sorted-candidate buffer");
    __shared__ int32_t buf_a[kTravWarps][kCandCap];
    __shared__ int32_t buf_b[kTravWarps][kCandCap];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    int32_t *const stack = buf_a[warp], *const sorted = buf_a[warp];
    int32_t *const cand = buf_b[warp];
    // per sorted candidate: the number of its images, and above it the one image of a single
    uint16_t *const ng = reinterpret_cast<uint16_t *>(buf_b[warp]), *const nh = ng + kCandCap;
    const unsigned below = (1u << lane) - 1u;
    const int64_t a = (int64_t)blockIdx.x * kTravWarps + warp;
    if (a >= n_leaves) return;  // whole warp leaves together; no block barrier below
    const bool a_any = leaf_start[a + 1] > leaf_start[a];
    const bool a_gas = leaf_ngas[a] > 0;
    float A[6];
#pragma unroll
    for (int q = 0; q < 6; ++q) A[q] = bbox[6 * a + q];
    const float ha = hmax[a];
    const int bx = leaf_box ? leaf_box[a] : 0;
    const double L = leaf_box ? (double)box_L[bx] : L0;
    const int32_t root = leaf_box ? box_root[bx] : tree.root;
    const float Lf = (float)L;
    int nc = 0;
    bool bad = false;
    if (a_any) {
        if (kBrute) {
            for (int64_t b0 = 0; b0 < n_leaves; b0 += 32) {
                int64_t b = b0 + lane;
                bool keep = false;
                if (b < n_leaves && leaf_start[b + 1] > leaf_start[b]) {
                    float cut = fmaxf((float)rc, a_gas && leaf_ngas[b] > 0 ? 2.0f * fmaxf(ha, hmax[b]) : 0.0f);
                    keep = !clearly_apart(A, bbox + 6 * b, Lf, cut);
                }
                unsigned m = __ballot_sync(CRK_FULL_MASK, keep);
                int pos = nc + __popc(m & below);
                if (keep && pos < kCandCap) cand[pos] = (int32_t)b;
                nc += __popc(m);
            }
        } else {
            int top = 1;
            if (lane == 0) stack[0] = root;
            __syncwarp();
            while (top > 0) {
                const int take = top < 32 ? top : 32;
                const int32_t nd = lane < take ? stack[top - 1 - lane] : -1;
                top -= take;
                __syncwarp();
                bool pass = false;
                int32_t lf = -1;
                if (nd >= 0) {
                    float cut = fmaxf((float)rc, a_gas ? 2.0f * fmaxf(ha, tree.node_hmax[nd]) : 0.0f);
                    pass = !clearly_apart(A, tree.node_box + 6 * (int64_t)nd, Lf, cut);
                    lf = tree.node_leaf[nd];
                }
                const bool is_leaf = pass && lf >= 0, inner = pass && lf < 0;
                unsigned m = __ballot_sync(CRK_FULL_MASK, is_leaf);
                int pos = nc + __popc(m & below);
                if (is_leaf && pos < kCandCap) cand[pos] = lf;
                nc += __popc(m);
                unsigned m2 = __ballot_sync(CRK_FULL_MASK, inner);
                int sp = top + 2 * __popc(m2 & below);
                if (inner && sp + 1 < kStackCap) {
                    stack[sp] = tree.node_right[nd];
                    stack[sp + 1] = tree.node_left[nd];
                }
                top += 2 * __popc(m2);
                if (top > kStackCap || nc > kCandCap) {
                    bad = true;
                    break;
                }
                __syncwarp();
            }
        }
        if (nc > kCandCap) bad = true;
    }
    __syncwarp();
    // a leaf whose candidates or images do not fit is left without images: the gas lists of the
    // same build may read them before the host sees the error
    auto none = [&]() {
        if (lane < 4) {
            int32_t *const st = lane == 0 ? o.start[0] : (lane == 1 ? o.start[1] : (lane == 2 ? o.start[2] : o.start[3]));
            int32_t *const ct = lane == 0 ? o.count[0] : (lane == 1 ? o.count[1] : (lane == 2 ? o.count[2] : o.count[3]));
            st[a] = 0;
            ct[a] = 0;
        }
    };
    if (bad) {
        if (lane == 0) atomicAdd(&o.err[0], 1);
        none();
        return;
    }
    // ascending j-leaf order (rank sort; leaf ids are unique)
    for (int t = lane; t < nc; t += 32) {
        int32_t v = cand[t];
        int r = 0;
        for (int u = 0; u < nc; ++u) r += cand[u] < v;
        sorted[r] = v;
    }
    __syncwarp();
    // the images of both lists
    auto images = [&](int32_t b, uint32_t &mg, uint32_t &mh) {
        const float2 *Bp = reinterpret_cast<const float2 *>(bbox + 6 * (int64_t)b);
        const float2 b0 = Bp[0], b1 = Bp[1], b2 = Bp[2];
        const float B[6] = {b0.x, b0.y, b1.x, b1.y, b2.x, b2.y};
        Gaps s;
#pragma unroll
        for (int q = 0; q < 3; ++q)
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                const float sf = (float)(k - 1) * Lf;
                const float t1 = (B[q] + sf) - A[3 + q], t2 = (A[q] - B[3 + q]) - sf, g = t1 > t2 ? t1 : t2;
                s.g[q][k] = g < 0.0f ? 0.0f : g;  // a NaN stays, and gives no image
            }
        const float *pa = bbox + 6 * a, *pb = bbox + 6 * (int64_t)b;
        mg = image_mask(pa, pb, s, L, rc);
        mh = 0;
        if (a_gas && leaf_ngas[b] > 0) mh = image_mask(pa, pb, s, L, (double)(2.0f * fmaxf(ha, hmax[b])));
    };
    auto coded = [](uint32_t m) { return (uint16_t)(__popc(m) | ((31 - __clz(m | 1u)) << 8)); };
    // totals: images in the low half word, pairs in the high one (27 * kCandCap < 2^16)
    unsigned tg = 0, th = 0;
    for (int t0 = 0; t0 < nc; t0 += 32) {
        const int t = t0 + lane;
        uint32_t mg = 0, mh = 0;
        if (t < nc) {
            images(sorted[t], mg, mh);
            ng[t] = coded(mg);
            nh[t] = coded(mh);
        }
        tg += __reduce_add_sync(CRK_FULL_MASK, (unsigned)__popc(mg) | (mg ? 0x10000u : 0u));
        th += __reduce_add_sync(CRK_FULL_MASK, (unsigned)__popc(mh) | (mh ? 0x10000u : 0u));
    }
    __syncwarp();
    const int tot[4] = {(int)(tg & 0xffffu), (int)(tg >> 16), (int)(th & 0xffffu), (int)(th >> 16)};
    unsigned long long base[4] = {0, 0, 0, 0};
    if (lane == 0)
        for (int k = 0; k < 4; ++k) base[k] = tot[k] ? atomicAdd(&o.cursor[k], (unsigned long long)tot[k]) : 0ull;
    bool over = false;
    for (int k = 0; k < 4; ++k) {
        base[k] = __shfl_sync(CRK_FULL_MASK, base[k], 0);
        over |= base[k] + (unsigned long long)tot[k] > (unsigned long long)o.cap[k];
    }
    if (over) {
        if (lane == 0) atomicAdd(&o.err[1], 1);
        none();
        return;
    }
    if (lane == 0)
        for (int k = 0; k < 4; ++k) {
            o.start[k][a] = (int32_t)base[k];
            o.count[k][a] = tot[k];
        }
    unsigned rg = 0, rh = 0;
    for (int t0 = 0; t0 < nc; t0 += 32) {
        const int t = t0 + lane;
        const unsigned vg = t < nc ? ng[t] : 0u, vh = t < nc ? nh[t] : 0u;
        const unsigned cg = vg & 0xffu, ch = vh & 0xffu;
        int sg, sh;
        const unsigned og = rg + (unsigned)warp_excl_scan((int)(cg | (cg ? 0x10000u : 0u)), lane, sg);
        const unsigned oh = rh + (unsigned)warp_excl_scan((int)(ch | (ch ? 0x10000u : 0u)), lane, sh);
        rg += (unsigned)sg;
        rh += (unsigned)sh;
        if (cg | ch) {
            const int32_t b = sorted[t];
            uint32_t mg = cg ? 1u << (vg >> 8) : 0u, mh = ch ? 1u << (vh >> 8) : 0u;
            if (cg > 1 || ch > 1) images(b, mg, mh);
            if (cg) o.gpair[base[1] + (og >> 16)] = b;
            if (ch) o.hpair[base[3] + (oh >> 16)] = b;
            const float2 *Bp = reinterpret_cast<const float2 *>(bbox + 6 * (int64_t)b);
            const float2 b0 = Bp[0], b1 = Bp[1];
            float4 *gi = reinterpret_cast<float4 *>(o.gimg + base[0] + (og & 0xffffu));
            float4 *hi = reinterpret_cast<float4 *>(o.himg + base[2] + (oh & 0xffffu));
            for (uint32_t m = mg | mh; m; m &= m - 1) {
                const int k = __ffs(m) - 1;
                const float4 im = make_float4(__int_as_float(b), image_shift(b0.x, A[0], k / 9, L),
                                              image_shift(b0.y, A[1], k / 3 % 3, L), image_shift(b1.x, A[2], k % 3, L));
                if (mg >> k & 1u) *gi++ = im;
                if (mh >> k & 1u) *hi++ = im;
            }
        }
    }
}

__global__ void leaf_box_to_node_kernel(int64_t n_leaves, const float *__restrict__ bbox,
                                        const float *__restrict__ hmax, const int32_t *__restrict__ leaf_node,
                                        float *__restrict__ node_box, float *__restrict__ node_hmax) {
    int64_t a = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (a >= n_leaves) return;
    int64_t nd = leaf_node[a];
    for (int q = 0; q < 6; ++q) node_box[6 * nd + q] = bbox[6 * a + q];
    node_hmax[nd] = hmax[a];
}

// one level of split nodes, deepest level first: node h_max = max of the children
__global__ void node_hmax_kernel(int nseg, LevelDev lv, const int32_t *__restrict__ left,
                                 const int32_t *__restrict__ right, float *__restrict__ node_hmax) {
    int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= nseg || lv.k[s] <= 0) return;
    int nd = lv.node[s];
    node_hmax[nd] = fmaxf(node_hmax[left[nd]], node_hmax[right[nd]]);
}

// The small levels (at most kTreeLevel segments) of a tree, deepest first, in one block: the node
// h_max of split nodes, after the leaf boxes and h_max went into the nodes.
constexpr int kTreeLevel = 8192;
constexpr int kTreeLevels = 32;
struct TreeLevels {
    const int32_t *k[kTreeLevels], *node[kTreeLevels];
    int32_t m[kTreeLevels];
    int n;
};
__global__ void __launch_bounds__(1024) tree_hmax_kernel(TreeLevels t, const int32_t *__restrict__ left,
                                                         const int32_t *__restrict__ right, float *node_hmax) {
    for (int d = 0; d < t.n; ++d) {
        for (int s = threadIdx.x; s < t.m[d]; s += blockDim.x) {
            if (t.k[d][s] <= 0) continue;
            const int nd = t.node[d][s];
            node_hmax[nd] = fmaxf(node_hmax[left[nd]], node_hmax[right[nd]]);
        }
        __syncthreads();
    }
}

// The box tables of a build (layout: see build_leaves_impl) written by a kernel: a copy from
// pageable host memory waits for the stream's earlier work before it starts.
constexpr int kBoxTables = 64;
struct BoxTables {
    int64_t start[kBoxTables + 1];
    float side[kBoxTables];
    int32_t seg[kBoxTables];
};
__global__ void box_tables_kernel(BoxTables t, int nbox, int32_t *__restrict__ a, int32_t *__restrict__ b, int words,
                                  int start_at) {
    for (int w = threadIdx.x; w < words; w += blockDim.x) a[w] = b[w] = 0;
    __syncthreads();
    for (int k = threadIdx.x; k <= nbox; k += blockDim.x) {
        for (int c = 0; c < 2; ++c) {
            int32_t *d = c ? a : b;
            reinterpret_cast<int64_t *>(d + start_at)[k] = t.start[k];
            if (k == nbox) continue;
            reinterpret_cast<float *>(d)[16 + nbox + k] = t.side[k];
            d[start_at + 2 * (nbox + 1) + k] = t.seg[k];
        }
    }
}

struct HostSeg {
    int32_t lo, hi, k, child, node;
};

}  // namespace

// ---------------------------------------------------------------------------------
void crk_rcb_shape_free(crk_ctx *ctx) {
    if (!ctx || !ctx->rcb) return;
    crk_rcb_shape *r = ctx->rcb;
    cudaFree(r->dtab);
    cudaFree(r->leaf_start);
    cudaFree(r->left);
    cudaFree(r->right);
    cudaFree(r->leaf_of);
    cudaFree(r->leaf_node);
    cudaFree(r->d_leaf_box);
    cudaFree(r->d_box_root);
    delete r;
    ctx->rcb = nullptr;
}

// The RCB tree shape for the boxes [box_start[b], box_start[b+1]) and
// max_leaf: level segment tables, leaf starts, children (one root per box).
static int rcb_shape(crk_ctx *ctx, const std::vector<int64_t> &box_start, int ml, const crk_rcb_shape **out) {
    const int64_t n = box_start.back();
    if (ctx->rcb && ctx->rcb->box_start == box_start && ctx->rcb->max_leaf == ml) {
        *out = ctx->rcb;
        return CRK_OK;
    }
    CRK_CUDA(ctx, cudaStreamSynchronize(ctx->stream));  // the old shape may still be in use
    crk_rcb_shape_free(ctx);
    crk_rcb_shape *r = new crk_rcb_shape();
    r->n = n;
    r->max_leaf = ml;
    r->box_start = box_start;
    const int nbox = (int)box_start.size() - 1;
    std::vector<std::vector<HostSeg>> levels;
    std::vector<HostSeg> cur;
    std::vector<int32_t> left, right;
    int32_t next_node = 0;
    r->box_root.assign(nbox, -1);
    for (int b = 0; b < nbox; ++b)
        if (box_start[b + 1] > box_start[b]) {
            r->box_root[b] = next_node;
            cur.push_back({(int32_t)box_start[b], (int32_t)box_start[b + 1], 0, 0, next_node++});
        }
    left.assign(next_node > 0 ? next_node : 1, -1);
    right.assign(next_node > 0 ? next_node : 1, -1);
    while (!cur.empty()) {
        bool any = false;
        for (auto &sg : cur)
            if (sg.hi - sg.lo > ml) {
                sg.k = (sg.hi - sg.lo) / 2;
                any = true;
            }
        if (!any) break;
        std::vector<HostSeg> nxt;
        nxt.reserve(cur.size() * 2);
        for (auto &sg : cur) {
            sg.child = (int32_t)nxt.size();
            if (sg.k > 0) {
                int32_t l = next_node++, rr = next_node++;
                left.resize(next_node, -1);
                right.resize(next_node, -1);
                left[sg.node] = l;
                right[sg.node] = rr;
                nxt.push_back({sg.lo, sg.lo + sg.k, 0, 0, l});
                nxt.push_back({sg.lo + sg.k, sg.hi, 0, 0, rr});
            } else {
                nxt.push_back({sg.lo, sg.hi, 0, 0, sg.node});
            }
        }
        levels.push_back(cur);
        cur.swap(nxt);
    }
    const int64_t nl = (int64_t)cur.size();
    r->n_leaves = nl;
    r->n_nodes = next_node;
    std::vector<int32_t> leaf_start(nl + 1), leaf_of(next_node > 0 ? next_node : 1, -1), leaf_node(nl > 0 ? nl : 1);
    r->leaf_box.assign(nl > 0 ? nl : 1, 0);
    for (int64_t a = 0, b = 0; a < nl; ++a) {
        leaf_start[a] = cur[a].lo;
        leaf_of[cur[a].node] = (int32_t)a;
        leaf_node[a] = cur[a].node;
        while (b + 1 < nbox && box_start[b + 1] <= cur[a].lo) ++b;
        r->leaf_box[a] = (int32_t)b;
        r->max_leaf_size = std::max(r->max_leaf_size, cur[a].hi - cur[a].lo);
    }
    leaf_start[nl] = (int32_t)n;
    size_t tot = 0;
    for (auto &L : levels) {
        r->level_off.push_back(tot);
        r->level_size.push_back(L.size());
        int32_t mx = 0;
        for (auto &sg : L) mx = std::max(mx, sg.hi - sg.lo);
        r->level_max.push_back(mx);
        tot += 7 * L.size();
    }
    std::vector<int32_t> packed(tot > 0 ? tot : 1);
    for (size_t d = 0; d < levels.size(); ++d) {
        const auto &L = levels[d];
        size_t m = L.size(), off = r->level_off[d];
        int64_t leftbase = 0;
        for (size_t q = 0; q < m; ++q) {
            packed[off + q] = L[q].lo;
            packed[off + m + q] = L[q].hi;
            packed[off + 2 * m + q] = L[q].k;
            packed[off + 3 * m + q] = L[q].child;
            packed[off + 4 * m + q] = L[q].node;
            packed[off + 5 * m + q] = 0;
            packed[off + 6 * m + q] = (int32_t)leftbase;
            leftbase += L[q].k;
        }
    }
    auto dev = [&](int32_t **p, const std::vector<int32_t> &v) -> int {
        if (cudaMalloc(p, sizeof(int32_t) * (v.size() > 0 ? v.size() : 1)) != cudaSuccess) {
            cudaGetLastError();
            return CRK_ENOMEM;
        }
        return cudaMemcpy(*p, v.data(), sizeof(int32_t) * v.size(), cudaMemcpyHostToDevice) == cudaSuccess
                   ? CRK_OK
                   : CRK_ECUDA;
    };
    int rc = CRK_OK;
    if (!rc) rc = dev(&r->dtab, packed);
    if (!rc) rc = dev(&r->leaf_start, leaf_start);
    if (!rc) rc = dev(&r->left, left);
    if (!rc) rc = dev(&r->right, right);
    if (!rc) rc = dev(&r->leaf_of, leaf_of);
    if (!rc) rc = dev(&r->leaf_node, leaf_node);
    if (!rc) rc = dev(&r->d_leaf_box, r->leaf_box);
    if (!rc) rc = dev(&r->d_box_root, r->box_root);
    ctx->rcb = r;
    if (rc) {
        crk_rcb_shape_free(ctx);
        return crk_fail(ctx, rc, "RCB shape tables");
    }
    *out = r;
    return CRK_OK;
}

namespace {
struct Tracer {
    crk_ctx *ctx;
    bool on;  // never during a rebuild (it may be captured)
    std::chrono::steady_clock::time_point t;
    Tracer(crk_ctx *c, bool allowed) : ctx(c), on(allowed && c->trace), t(std::chrono::steady_clock::now()) {}
    void mark(const char *what) {
        if (!on) return;
        cudaStreamSynchronize(ctx->stream);
        auto now = std::chrono::steady_clock::now();
        fprintf(stderr, "[crk] %-18s %8.3f ms\n", what, std::chrono::duration<double, std::milli>(now - t).count());
        t = now;
    }
};
}  // namespace

__global__ void init_node_of_kernel(int64_t n, const int32_t *__restrict__ box_of, const int32_t *__restrict__ seg_of_box,
                                    int32_t *__restrict__ node_of) {
    int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p < n) node_of[p] = seg_of_box[box_of[p]];
}

// The host checks of a build as bits of the leaves' status word (rebuilds, which do not synchronise).
__global__ void leaf_status_kernel(const int32_t *__restrict__ flags, const unsigned *__restrict__ hbits,
                                   const float *__restrict__ box_L, int nbox, int32_t n_gas, int32_t *__restrict__ status) {
    int32_t s = 0;
    if (threadIdx.x == 0) {
        if (flags[0] > 0) s |= CRK_LEAVES_BAD_POSITION;
        if (flags[1] > 0) s |= CRK_LEAVES_BAD_H;
        if (flags[2] != n_gas) s |= CRK_LEAVES_GAS_COUNT;
        if (flags[4] > 0) s |= CRK_LEAVES_LEAF_SIZE;
        if (flags[5] > 0) s |= CRK_LEAVES_INTERNAL;
    }
    for (int b = threadIdx.x; b < nbox; b += blockDim.x) {
        const float hm = __uint_as_float(hbits[b]);
        if (!(2.0 * (double)hm < 0.5 * (double)box_L[b])) s |= CRK_LEAVES_HMAX;
    }
    if (s) atomicOr(status, s);
}

__global__ void pairs_status_kernel(const int32_t *__restrict__ err, int32_t *__restrict__ status) {
    int32_t s = 0;
    if (err[0] > 0) s |= CRK_LEAVES_CANDIDATES;
    if (err[1] > 0) s |= CRK_LEAVES_IMAGE_CAP;
    if (s) atomicOr(status, s);
}

// Leaves of one box (nbox = 1) or of several independent periodic boxes whose
// particles are the consecutive ranges box_start[b] .. box_start[b+1].
// re != NULL: rebuild those leaves in place (crk_leaves_rebuild): no host synchronisation and no
// allocation; the host checks become bits of the leaves' device status word.
static int build_leaves_impl(crk_ctx *ctx, const crk_particles *p, const float *h, const crk_leaf_params *lp,
                             const std::vector<int64_t> &box_start, const std::vector<float> &box_side,
                             crk_leaves **out, crk_leaves *re = nullptr) {
    if (!p || !lp || !out) return crk_fail(ctx, CRK_EINVAL, "null argument");
    if (!re) *out = nullptr;
    const int64_t n = p->n;
    const int nbox = (int)box_side.size();
    if (n < 0 || n > 2000000000LL) return crk_fail(ctx, CRK_EINVAL, "particle count out of range");
    if (n > 0 && (!p->x || !p->y || !p->z || !p->species || !h)) return crk_fail(ctx, CRK_EINVAL, "null array");
    if (lp->mode != 0 && lp->mode != 1) return crk_fail(ctx, CRK_EINVAL, "leaf mode must be 0 or 1");
    if (lp->mode == 0 && nbox != 1) return crk_fail(ctx, CRK_EINVAL, "chaining-mesh leaves take one box");
    if (lp->mode == 0 && (lp->cells_per_side < 1 || lp->cells_per_side > 40))
        return crk_fail(ctx, CRK_EINVAL, "cells_per_side must be in [1, 40]");
    if (lp->mode == 1 && (lp->max_leaf < 1 || lp->max_leaf > kMaxLeafCap))
        return crk_fail(ctx, CRK_EINVAL, "max_leaf must be in [1, 1024]");
    float box_max = 0.0f;
    for (int b = 0; b < nbox; ++b) {
        if (!(box_side[b] > 0.0f)) return crk_fail(ctx, CRK_EINVAL, "box %d: side must be positive", b);
        if (box_start[b + 1] < box_start[b]) return crk_fail(ctx, CRK_EINVAL, "box starts must not decrease");
        if (box_start[b + 1] > box_start[b] && (!(lp->r_cut_grav > 0.0f) ||
                                                !((double)lp->r_cut_grav < 0.5 * (double)box_side[b])))
            return crk_fail(ctx, CRK_EBOX, "box %d: r_cut_grav must be positive and below box/2", b);
        box_max = std::max(box_max, box_side[b]);
    }
    if (box_start[0] != 0 || box_start[nbox] != n) return crk_fail(ctx, CRK_EINVAL, "box starts must span [0, n]");
    if (re) {
        if (re->n != n || re->box_start != box_start || re->box_side != box_side || re->mode != lp->mode ||
            re->max_leaf != lp->max_leaf || re->cells != lp->cells_per_side || re->r_cut_grav != lp->r_cut_grav)
            return crk_fail(ctx, CRK_ESTATE, "rebuild: particles, boxes or leaf parameters differ from the leaves'");
        if (re->grav_lists.list) return crk_fail(ctx, CRK_ESTATE, "rebuild: leaves with gravity lists");
        if (re->gas_lists.list && !re->gas_lists.onepass)
            return crk_fail(ctx, CRK_ESTATE, "rebuild: gas lists of the exact two-pass build");
        if (!re->dev || !re->boxtab) return crk_fail(ctx, CRK_ESTATE, "rebuild: leaves without rebuild state");
        if (n > 0 && lp->mode == 1 && !(ctx->rcb && ctx->rcb->box_start == box_start && ctx->rcb->max_leaf == lp->max_leaf)) {
            cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
            cudaStreamIsCapturing(ctx->stream, &cs);
            if (cs != cudaStreamCaptureStatusNone)
                return crk_fail(ctx, CRK_ESTATE, "rebuild under capture: the context holds another RCB shape");
        }
    }

    Tracer tr(ctx, re == nullptr);
    crk_leaves *lv = re ? re : new crk_leaves();
    lv->n = n;
    lv->box = box_max;
    lv->nbox = nbox;
    lv->mode = lp->mode;
    lv->r_cut_grav = lp->r_cut_grav;
    lv->max_leaf = lp->max_leaf;
    lv->cells = lp->cells_per_side;
    lv->box_start = box_start;
    lv->box_side = box_side;
    cudaStream_t st = ctx->stream;
    int rc = CRK_OK;
#define TRY(expr)                          \
    do {                                   \
        rc = (expr);                       \
        if (rc != CRK_OK) goto fail;       \
    } while (0)
#define ALLOC(ptr, type, count)                                                                          \
    do {                                                                                                 \
        if (!re) { /* a rebuild keeps the buffers of the first build */                                \
            ptr = (type *)crk_leaves_alloc(ctx, lv, sizeof(type) * (size_t)((count) > 0 ? (count) : 1)); \
            if (!ptr) {                                                                                  \
                rc = crk_fail(ctx, CRK_ENOMEM, "leaf allocation");                                       \
                goto fail;                                                                               \
            }                                                                                            \
        }                                                                                                \
    } while (0)
#define KCHECK(what)                                       \
    do {                                                   \
        cudaError_t e_ = cudaGetLastError();               \
        if (e_ != cudaSuccess) {                           \
            rc = crk_check_cuda(ctx, e_, what);            \
            goto fail;                                     \
        }                                                  \
    } while (0)
    {
        // the box tables: flags[0..15] and per box hmax bits (zero), side, start (int64), segment index;
        // then the leaves' device words (zero)
        const size_t tbytes = (64 + 4 * (size_t)nbox + 4 * (size_t)nbox + 8 * (size_t)(nbox + 2) + 4 * (size_t)nbox + 127) &
                              ~(size_t)127;
        const size_t fbytes = tbytes + 256;
        int32_t *flags = (int32_t *)crk_scratch(ctx, 0, fbytes);
        if (!flags) { rc = crk_fail(ctx, CRK_ENOMEM, "scratch"); goto fail; }
        const size_t o_start = (64 + 8 * (size_t)nbox + 7) & ~(size_t)7;
        unsigned *hbits = (unsigned *)(flags + 16);
        float *box_L = (float *)(flags + 16 + nbox);
        int64_t *d_box_start = (int64_t *)((char *)flags + o_start);
        int32_t *seg_of_box = (int32_t *)(d_box_start + nbox + 1);
        if (!re) {
            // the rebuild state: a device copy of the box tables; status word, group counts and cursors
            lv->boxtab_bytes = fbytes;
            lv->boxtab = (unsigned char *)crk_leaves_alloc(ctx, lv, lv->boxtab_bytes);
            if (!lv->boxtab) { rc = crk_fail(ctx, CRK_ENOMEM, "leaf allocation"); goto fail; }
            lv->dev = (int32_t *)(lv->boxtab + tbytes);
            BoxTables bt{};
            for (int b = 0, q = 0; b < nbox && nbox <= kBoxTables; ++b) {
                bt.start[b] = box_start[b];
                bt.side[b] = box_side[b];
                bt.seg[b] = q;
                if (box_start[b + 1] > box_start[b]) ++q;
            }
            if (nbox <= kBoxTables) {
                bt.start[nbox] = n;
                box_tables_kernel<<<1, 256, 0, st>>>(bt, nbox, (int32_t *)lv->boxtab, flags, (int)(fbytes / 4),
                                                     (int)(o_start / 4));
                ++ctx->launches;
                KCHECK("box tables");
            } else {
                std::vector<char> tab(fbytes, 0);
                std::memcpy(tab.data() + 64 + 4 * (size_t)nbox, box_side.data(), 4 * (size_t)nbox);
                std::memcpy(tab.data() + o_start, box_start.data(), 8 * (size_t)(nbox + 1));
                int32_t *hs = (int32_t *)(tab.data() + o_start + 8 * (size_t)(nbox + 1));
                for (int b = 0, q = 0; b < nbox; ++b) {
                    hs[b] = q;
                    if (box_start[b + 1] > box_start[b]) ++q;
                }
                if (cudaMemcpyAsync(flags, tab.data(), fbytes, cudaMemcpyHostToDevice, st) != cudaSuccess ||
                    cudaMemcpyAsync(lv->boxtab, flags, fbytes, cudaMemcpyDeviceToDevice, st) != cudaSuccess) {
                    rc = crk_fail(ctx, CRK_ECUDA, "leaf build set-up copies");
                    goto fail;
                }
            }
        } else if (cudaMemsetAsync(lv->dev, 0, 256, st) != cudaSuccess ||
                   cudaMemcpyAsync(flags, lv->boxtab, lv->boxtab_bytes, cudaMemcpyDeviceToDevice, st) != cudaSuccess) {
            // (the table's flags and hmax bits are zero: the build works on the scratch copy)
            rc = crk_fail(ctx, CRK_ECUDA, "leaf build set-up copies");
            goto fail;
        }
        int32_t *box_of = nullptr;
        if (nbox > 1 && n > 0) {
            box_of = (int32_t *)crk_scratch(ctx, 16, sizeof(int32_t) * (size_t)n);
            if (!box_of) { rc = crk_fail(ctx, CRK_ENOMEM, "scratch"); goto fail; }
            box_of_kernel<<<crk_grid(n, 256), 256, 0, st>>>(n, d_box_start, nbox, box_of);
            ++ctx->launches;
        }
        if (n > 0) {
            const int items = n >= (int64_t)4096 * 8 * ctx->num_sms ? 16 : 4;
            validate_kernel<<<(unsigned)((n + 256 * items - 1) / (256 * items)), 256, 0, st>>>(
                p->x, p->y, p->z, p->species, h, n, items, box_of, box_L, flags, hbits);
            ++ctx->launches;
        }
        int32_t *members = nullptr;  // particle ids grouped by leaf
        int32_t *rank_yz[2] = {nullptr, nullptr};  // RCB: the members' ranks along y and z (members are in x order)
        int64_t nl = 0;
        const crk_rcb_shape *shape = nullptr;
        float *node_box = nullptr, *node_hmax = nullptr;

        if (lp->mode == 0) {
            int nc = lp->cells_per_side;
            nl = (int64_t)nc * nc * nc;
            uint32_t *keys = (uint32_t *)crk_scratch(ctx, 1, sizeof(uint32_t) * (size_t)(n > 0 ? n : 1));
            int32_t *vals = (int32_t *)crk_scratch(ctx, 2, sizeof(int32_t) * (size_t)(n > 0 ? n : 1));
            int32_t *cnts = (int32_t *)crk_scratch(ctx, 3, sizeof(int32_t) * (size_t)(nl + 1));
            if (!keys || !vals || !cnts) { rc = crk_fail(ctx, CRK_ENOMEM, "scratch"); goto fail; }
            ALLOC(lv->leaf_start, int32_t, nl + 1);
            if (cudaMemsetAsync(cnts, 0, sizeof(int32_t) * (size_t)(nl + 1), st) != cudaSuccess) {
                rc = crk_fail(ctx, CRK_ECUDA, "memset");
                goto fail;
            }
            if (n > 0) {
                mesh_keys_kernel<<<crk_grid(n, 256), 256, 0, st>>>(p->x, p->y, p->z, n, nc, (double)box_side[0], keys,
                                                                   vals, cnts);
                ++ctx->launches;
            }
            int bits = 1;
            while ((1LL << bits) < nl) ++bits;
            TRY(crk_radix_sort_u32(ctx, keys, vals, n, bits));
            TRY(crk_exclusive_scan_i32(ctx, cnts, lv->leaf_start, nl + 1, nullptr));
            members = vals;
        } else {
            TRY(rcb_shape(ctx, box_start, lp->max_leaf, &shape));
            nl = shape->n_leaves;
            ALLOC(lv->leaf_start, int32_t, nl + 1);
            if (cudaMemcpyAsync(lv->leaf_start, shape->leaf_start, sizeof(int32_t) * (size_t)(nl + 1),
                                cudaMemcpyDeviceToDevice, st) != cudaSuccess) {
                rc = crk_fail(ctx, CRK_ECUDA, "leaf starts");
                goto fail;
            }
            ALLOC(lv->node_box, float, 6 * shape->n_nodes);
            ALLOC(lv->node_hmax, float, shape->n_nodes);
            node_box = lv->node_box;
            node_hmax = lv->node_hmax;
            tr.mark("shape");
            int32_t *Lc[3];
            size_t nb = sizeof(int32_t) * (size_t)(n > 0 ? n : 1);
            int32_t *R[3], *Ac[3][2], *An[3][2];
            for (int a = 0; a < 3; ++a) {
                Lc[a] = nullptr;
                R[a] = (int32_t *)crk_scratch(ctx, 5 + a, nb);
                Ac[a][0] = (int32_t *)crk_scratch(ctx, 19 + a, nb);
            }
            int32_t *node_of = (int32_t *)crk_scratch(ctx, 8, nb);
            int32_t *node_nx = (int32_t *)crk_scratch(ctx, 9, nb);
            int32_t *mem = (int32_t *)crk_scratch(ctx, 10, nb);
            int32_t *flag = (int32_t *)crk_scratch(ctx, 11, nb + 3 * sizeof(int32_t) * (size_t)(n / 2048 + 2));
            size_t max_seg = 1;
            for (size_t m : shape->level_size) max_seg = std::max(max_seg, m);
            SegRec *segs = (SegRec *)crk_scratch(ctx, 31, sizeof(SegRec) * max_seg);
            bool ok = node_of && node_nx && mem && flag && segs;
            for (int a = 0; a < 3; ++a) ok = ok && R[a] && Ac[a][0];
            if (!ok) {
                rc = crk_fail(ctx, CRK_ENOMEM, "scratch");
                goto fail;
            }
            int32_t *spare[9] = {};  // the other nine rank columns live where the sort's keys and values were
            TRY(crk_sort_axes(ctx, p->x, p->y, p->z, n, box_of, nbox, Lc, spare));
            for (int a = 0; a < 3; ++a) {
                Ac[a][1] = spare[a];
                An[a][0] = spare[3 + a];
                An[a][1] = spare[6 + a];
            }
            tr.mark("axis sorts");
            const AxisOrder ord{{Lc[0], Lc[1], Lc[2]}, {R[0], R[1], R[2]}};
            if (n > 0) {
                const dim3 g3((unsigned)crk_grid(n, 256), 3), g6((unsigned)crk_grid(n, 256), 6);
                rank_of_kernel<<<g3, 256, 0, st>>>(n, ord, RankOut{{R[0], R[1], R[2]}});
                rank_column_kernel<<<g6, 256, 0, st>>>(
                    n, ord, RankListsOut{{{Ac[0][0], Ac[0][1]}, {Ac[1][0], Ac[1][1]}, {Ac[2][0], Ac[2][1]}}});
                ctx->launches += 2;
                if (box_of) {
                    init_node_of_kernel<<<crk_grid(n, 256), 256, 0, st>>>(n, box_of, seg_of_box, node_of);
                    ++ctx->launches;
                } else if (cudaMemsetAsync(node_of, 0, sizeof(int32_t) * (size_t)n, st) != cudaSuccess) {
                    rc = crk_fail(ctx, CRK_ECUDA, "memset");
                    goto fail;
                }
            }
            // levels [0, d_local) stream through DRAM; the rest run in shared memory, one block per
            // segment of level d_local (every segment there holds at most kLocalCap entries)
            const int n_lev = (int)shape->level_size.size();
            int d_local = n_lev;
            for (int d = 0; d < n_lev; ++d)
                if (shape->level_max[d] <= kLocalCap) {
                    d_local = d;
                    break;
                }
            if (n_lev - d_local > kLocalLevels) d_local = n_lev - kLocalLevels;
            // and a cluster of blocks per segment runs the last levels before d_local on the way
            int d_mid = d_local;
            if (d_local < n_lev) {
                const int d = d_local - std::min(d_local, kClusterLevels);
                if ((int64_t)shape->level_size[d] << (d_local - d) <= (int64_t)kLocalBlocks * ctx->num_sms) d_mid = d;
            }
            for (int d = 0; d < d_mid; ++d) {
                int m = (int)shape->level_size[d];
                int32_t *tab = shape->dtab + shape->level_off[d];
                LevelDev dv{tab, tab + m, tab + 2 * m, tab + 3 * m, tab + 4 * m, tab + 5 * m, tab + 6 * m};
                const RankLists Lr{{{Ac[0][0], Ac[0][1]}, {Ac[1][0], Ac[1][1]}, {Ac[2][0], Ac[2][1]}}};
                const RankListsOut Lo{{{An[0][0], An[0][1]}, {An[1][0], An[1][1]}, {An[2][0], An[2][1]}}};
                const int64_t nbt = (n + kPartTile - 1) / kPartTile;
                // small builds: one launch makes the records, counts and scans (in one box a level above
                // kLocalCap has no segment below kLocalCap / 2)
                const bool fused = nbt <= kFusedTiles, axis = fused && nbox == 1 && shape->level_max[d] > kLocalCap;
                unsigned *ctr = fused ? (unsigned *)(flags + 8) : nullptr;
                if (!axis) rcb_axis_kernel<<<crk_grid(m, 128), 128, 0, st>>>(m, dv, Lr, ord, p->x, p->y, p->z, node_box, segs);
                if (axis)
                    rcb_count3_kernel<true><<<(unsigned)nbt, kPartThreads, 0, st>>>(
                        n, segs, node_of, Lr, flag, nbt, ctr, dv, ord, p->x, p->y, p->z, node_box, flags + 5);
                else
                    rcb_count3_kernel<false><<<(unsigned)nbt, kPartThreads, 0, st>>>(
                        n, segs, node_of, Lr, flag, nbt, ctr, dv, ord, p->x, p->y, p->z, node_box, flags + 5);
                if (!fused) rcb_scan3_kernel<<<1, 1024, 0, st>>>(flag, nbt);
                ctx->launches += (axis ? 1 : 2) + (fused ? 0 : 1) + 1;
                rcb_scatter3_kernel<<<(unsigned)nbt, kPartThreads, 0, st>>>(n, segs, node_of, Lr, flag, nbt, Lo, node_nx,
                                                                            flags + 5);
                for (int a = 0; a < 3; ++a)
                    for (int c = 0; c < 2; ++c) std::swap(Ac[a][c], An[a][c]);
                std::swap(node_of, node_nx);
                KCHECK("rcb level");
            }
            const RankLists Lfin{{{Ac[0][0], Ac[0][1]}, {Ac[1][0], Ac[1][1]}, {Ac[2][0], Ac[2][1]}}};
            if (n > 0 && d_local < n_lev) {
                static bool smem_set = false;  // opt-in above 48 KB, once (never inside a capture: a
                if (!smem_set) {               // rebuild always follows a fresh build)
                    cudaFuncSetAttribute(rcb_local_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kLocalSmem);
                    cudaFuncSetAttribute(rcb_local_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kLocalSmem);
                    smem_set = true;
                }
                LocalShape ls{};
                ls.pre = d_local - d_mid;
                ls.nlev = n_lev - d_mid;
                for (int l = 0; l < ls.nlev; ++l) {
                    ls.tab[l] = shape->dtab + shape->level_off[d_mid + l];
                    ls.m[l] = (int32_t)shape->level_size[d_mid + l];
                }
                cudaLaunchConfig_t cfg{};
                cfg.gridDim = dim3((unsigned)shape->level_size[d_mid] << ls.pre);
                cfg.blockDim = dim3(kLocalThreads);
                cfg.dynamicSmemBytes = kLocalSmem;
                cfg.stream = st;
                cudaLaunchAttribute cluster{};
                cluster.id = cudaLaunchAttributeClusterDimension;
                cluster.val.clusterDim.x = 1u << ls.pre;
                cluster.val.clusterDim.y = cluster.val.clusterDim.z = 1;
                cfg.attrs = &cluster;
                cfg.numAttrs = ls.pre > 0 ? 1 : 0;
                cudaLaunchKernelEx(&cfg, ls.pre > 0 ? rcb_local_kernel<true> : rcb_local_kernel<false>, n, ls, Lfin, ord,
                                   p->x, p->y, p->z, node_box, mem, An[0][0], An[0][1], flags + 5);
                rank_yz[0] = An[0][0];
                rank_yz[1] = An[0][1];
                ++ctx->launches;
                KCHECK("rcb local levels");
            } else if (n > 0) {
                rank_members_kernel<<<crk_grid(n, 256), 256, 0, st>>>(n, Lfin, ord, mem);
                rank_yz[0] = Ac[0][0];
                rank_yz[1] = Ac[0][1];
                ++ctx->launches;
            }
            tr.mark("rcb levels");
            members = mem;
        }
        lv->n_leaves = nl;
        ALLOC(lv->perm, int32_t, n);
        ALLOC(lv->kperm, int32_t, n);
        ALLOC(lv->leaf_ngas, int32_t, nl);
        ALLOC(lv->bbox, float, 6 * nl);
        ALLOC(lv->hmax, float, nl);
        ALLOC(lv->pos, float4, n);
        ALLOC(lv->kperm_g, int32_t, n);
        ALLOC(lv->pos_g, float4, n);
        ALLOC(lv->kinv, int32_t, n);
        ALLOC(lv->kinv_g, int32_t, n);
        ALLOC(lv->gcell, float4, 2 * (n / 32 + nl + 1));
        ALLOC(lv->hcell, float4, 2 * (n / 32 + nl + 1));
        if (nl > 0) {
            if (lp->mode == 1 && shape && shape->max_leaf_size <= kRcbLeaf)
                // two warps a leaf; four where the leaves are too few to fill the GPU
                leaf_data_rcb_kernel<<<(unsigned)nl, nl < (int64_t)32 * ctx->num_sms ? 128 : 64, 0, st>>>(
                    lv->leaf_start, members, rank_yz[0], rank_yz[1], p->x, p->y, p->z, p->species, h, lv->perm,
                    lv->kperm, lv->leaf_ngas, lv->bbox, lv->hmax, lv->pos, lv->kperm_g, lv->pos_g, lv->kinv,
                    lv->kinv_g, lv->gcell, lv->hcell, flags + 4);
            else
                leaf_data_kernel<kMaxLeafCap><<<(unsigned)nl, 128, 0, st>>>(
                    nl, lv->leaf_start, members, p->x, p->y, p->z, p->species, h, lv->perm, lv->kperm, lv->leaf_ngas,
                    lv->bbox, lv->hmax, lv->pos, lv->kperm_g, lv->pos_g, lv->kinv, lv->kinv_g, lv->gcell,
                    lv->hcell, flags + 4);
            ++ctx->launches;
        }
        KCHECK("leaf data");
        if (re) {  // the checks below, on the device
            leaf_status_kernel<<<1, 256, 0, st>>>(flags, hbits, box_L, nbox, (int32_t)lv->n_gas, lv->dev);
            ++ctx->launches;
        }
        // the gas lists' groups are counted before the host looks, so that one read brings everything
        const bool gas_lists = re ? lv->gas_lists.list != nullptr : crk_wants_gas_lists(ctx);
        if (!re && gas_lists) TRY(crk_gas_groups(ctx, lv));
        // ---- host checks (first synchronisation)
        std::vector<int32_t> hflags(16 + nbox);
        const unsigned *hb = (const unsigned *)hflags.data() + 16;
        int32_t hdev[2] = {0, 0};
        std::vector<int32_t> ls(!re && lp->mode == 0 ? nl + 1 : 0);
        if (re) {
        } else if ((!ls.empty() && cudaMemcpyAsync(ls.data(), lv->leaf_start, sizeof(int32_t) * ls.size(),
                                                   cudaMemcpyDeviceToHost, st) != cudaSuccess) ||
            cudaMemcpyAsync(hflags.data(), flags, 64 + 4 * (size_t)nbox, cudaMemcpyDeviceToHost, st) != cudaSuccess ||
            cudaMemcpyAsync(hdev, lv->dev, sizeof(hdev), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
            cudaStreamSynchronize(st) != cudaSuccess) {
            rc = crk_fail(ctx, CRK_ECUDA, "leaf build: %s", cudaGetErrorString(cudaGetLastError()));
            goto fail;
        }
        tr.mark("leaf data");
        if (!re) {
        if (hflags[0] > 0) { rc = crk_fail(ctx, CRK_EBOX, "%d particle positions outside [0, box)", hflags[0]); goto fail; }
        if (hflags[1] > 0) { rc = crk_fail(ctx, CRK_EINVAL, "%d gas particles with h <= 0 or not finite", hflags[1]); goto fail; }
        if (hflags[4] > 0) { rc = crk_fail(ctx, CRK_EINVAL, "a leaf holds more than %d particles", kMaxLeafCap); goto fail; }
        if (hflags[5] > 0) { rc = crk_fail(ctx, CRK_ESTATE, "internal error: inconsistent RCB partition"); goto fail; }
        lv->n_gas = hflags[2];
        float hmax_all = 0.0f;
        for (int b = 0; b < nbox; ++b) {
            float hm;
            std::memcpy(&hm, &hb[b], sizeof(float));
            hmax_all = std::max(hmax_all, hm);
            if (!(2.0 * (double)hm < 0.5 * (double)box_side[b])) {
                rc = crk_fail(ctx, CRK_EBOX, "box %d: 2 h_max = %g is not below box/2", b, 2.0 * hm);
                goto fail;
            }
        }
        lv->hmax_all = hmax_all;
        if (lp->mode == 0) {
            int mx = 0;
            for (int64_t a = 0; a < nl; ++a) mx = std::max(mx, ls[a + 1] - ls[a]);
            lv->max_leaf_size = mx;
            if (mx > kMaxLeafCap) { rc = crk_fail(ctx, CRK_EINVAL, "a chaining-mesh cell holds more than %d particles", kMaxLeafCap); goto fail; }
        } else {
            lv->max_leaf_size = shape->max_leaf_size;
        }
        }
        // ---- tree for traversal (RCB): leaf boxes and h_max into the nodes, then bottom-up h_max
        TreeDev tree{};
        const int brute = lp->mode == 0 ? 1 : 0;
        if (!brute && nl > 0) {
            leaf_box_to_node_kernel<<<crk_grid(nl, 128), 128, 0, st>>>(nl, lv->bbox, lv->hmax, shape->leaf_node,
                                                                       node_box, node_hmax);
            ++ctx->launches;
            TreeLevels tl{};
            for (size_t d = shape->level_size.size(); d-- > 0;) {
                int m = (int)shape->level_size[d];
                int32_t *tab = shape->dtab + shape->level_off[d];
                LevelDev dv{tab, tab + m, tab + 2 * m, tab + 3 * m, tab + 4 * m, tab + 5 * m, tab + 6 * m};
                if (m > kTreeLevel) {  // (levels shrink towards the root)
                    node_hmax_kernel<<<crk_grid(m, 128), 128, 0, st>>>(m, dv, shape->left, shape->right, node_hmax);
                    ++ctx->launches;
                } else {
                    if (tl.n == kTreeLevels) {  // a full table runs before the levels that read its nodes
                        tree_hmax_kernel<<<1, 1024, 0, st>>>(tl, shape->left, shape->right, node_hmax);
                        ++ctx->launches;
                        tl.n = 0;
                    }
                    tl.k[tl.n] = dv.k;
                    tl.node[tl.n] = dv.node;
                    tl.m[tl.n++] = m;
                }
            }
            if (tl.n > 0) {
                tree_hmax_kernel<<<1, 1024, 0, st>>>(tl, shape->left, shape->right, node_hmax);
                ++ctx->launches;
            }
            KCHECK("node h_max");
            tree.node_box = node_box;
            tree.node_hmax = node_hmax;
            tree.node_left = shape->left;
            tree.node_right = shape->right;
            tree.node_leaf = shape->leaf_of;
            tree.root = 0;
        }
        bool lists_over = false;  // a gas list exceeded the one-pass capacities
        // ---- leaf-pair image lists, one warp per leaf; retried once with exact
        // capacities if the first estimate is too small
        {
            int32_t *se[8] = {lv->gimg_start, lv->gimg_cnt, lv->gpair_start, lv->gpair_cnt,
                              lv->himg_start, lv->himg_cnt, lv->hpair_start, lv->hpair_cnt};
            for (int q = 0; q < 8; ++q) ALLOC(se[q], int32_t, nl);
            // the list cursors live with the leaves (a rebuild refreshes the counts from them later); they
            // are zero at the start of a build and of a rebuild
            unsigned long long *cur = (unsigned long long *)(lv->dev + 16);
            // first capacities: 1.5 times the leaves of the mean size within the cut of one (clustered
            // boxes hold 34 images a leaf and list, cubes of 128 particles at r_c = 3 an estimated 38),
            // the hydro cut taken at the largest h but at most 128 a leaf; never below 48 images and 32
            // pairs a leaf, which rebuilds of particles that have since clustered may need
            double vol = 0.0;
            for (int b = 0; b < nbox; ++b)
                if (box_start[b + 1] > box_start[b]) vol += (double)box_side[b] * box_side[b] * box_side[b];
            const double ls = nl > 0 ? cbrt(vol / (double)nl) : 1.0;
            auto images = [&](double cut, double most) {
                const double w = 2.0 * ls;  // leaf boxes nearer than cut: Minkowski sum of two leaves and a ball
                const double v = w * w * w + 6.0 * w * w * cut + 9.42 * w * cut * cut + 4.19 * cut * cut * cut;
                return (int64_t)std::min(most, 1.5 * v / (ls * ls * ls) + 16.0);
            };
            const int64_t ig = images((double)lp->r_cut_grav, (double)kCandCap), ih = images(2.0 * lv->hmax_all, 128.0);
            int64_t cap[4] = {std::max<int64_t>(ig, 48), std::max<int64_t>(ig, 32), std::max<int64_t>(ih, 48),
                              std::max<int64_t>(ih, 32)};
            for (int64_t &c : cap) c = c * nl + 64;
            if (re)
                for (int k = 0; k < 4; ++k) cap[k] = lv->img_cap[k];
            crk_image *gimg = lv->gimg, *himg = lv->himg;
            int32_t *gpair = lv->gpair_list, *hpair = lv->hpair_list;
            unsigned long long hcur[6] = {(unsigned long long)lv->n_gimg, (unsigned long long)lv->n_gpairs,
                                          (unsigned long long)lv->n_himg, (unsigned long long)lv->n_hpairs, 0, 0};
            for (int attempt = 0; attempt < 2; ++attempt) {
                // capacity blocks come from the leaves' own allocations; a retry leaves the
                // first (too small) blocks unused until the leaves are freed
                ALLOC(gimg, crk_image, cap[0]);
                ALLOC(gpair, int32_t, cap[1]);
                ALLOC(himg, crk_image, cap[2]);
                ALLOC(hpair, int32_t, cap[3]);
                if (attempt > 0 && cudaMemsetAsync(lv->dev + 3, 0, 256 - 12, st) != cudaSuccess) {
                    rc = crk_fail(ctx, CRK_ECUDA, "memset");
                    goto fail;
                }
                PairOut po;
                for (int k = 0; k < 4; ++k) {
                    po.start[k] = se[2 * k];
                    po.count[k] = se[2 * k + 1];
                    po.cap[k] = cap[k];
                }
                po.gimg = gimg; po.gpair = gpair; po.himg = himg; po.hpair = hpair;
                po.cursor = cur;
                po.err = (int32_t *)(cur + 4);
                if (nl > 0) {
                    unsigned grid = (unsigned)((nl + kTravWarps - 1) / kTravWarps);
                    if (brute)
                        leaf_pairs_warp_kernel<true><<<grid, kTravWarps * 32, 0, st>>>(
                            nl, lv->leaf_start, lv->leaf_ngas, lv->bbox, lv->hmax, tree, (double)box_side[0],
                            (double)lp->r_cut_grav, po, nullptr, nullptr, nullptr);
                    else
                        leaf_pairs_warp_kernel<false><<<grid, kTravWarps * 32, 0, st>>>(
                            nl, lv->leaf_start, lv->leaf_ngas, lv->bbox, lv->hmax, tree, (double)box_side[0],
                            (double)lp->r_cut_grav, po, shape->d_leaf_box, shape->d_box_root, box_L);
                    ++ctx->launches;
                }
                KCHECK("pair lists");
                if (re) {  // one attempt at the first build's capacities; overflows go to the status word
                    pairs_status_kernel<<<1, 1, 0, st>>>(po.err, lv->dev);
                    ++ctx->launches;
                    break;
                }
                tr.mark("pair lists");
                if (gas_lists) {  // on these images; a leaf whose images did not fit has none (and the lists are redone)
                    lv->himg_start = se[4]; lv->himg_cnt = se[5]; lv->himg = himg;
                    TRY(crk_gas_lists_onepass(ctx, lv, hdev[1]));
                    tr.mark("gas lists");
                }
                // ---- second synchronisation: list sizes and overflows
                int32_t hall[64];
                if (cudaMemcpyAsync(hall, lv->dev, 256, cudaMemcpyDeviceToHost, st) != cudaSuccess ||
                    cudaStreamSynchronize(st) != cudaSuccess) {
                    rc = crk_fail(ctx, CRK_ECUDA, "pair lists: %s", cudaGetErrorString(cudaGetLastError()));
                    goto fail;
                }
                std::memcpy(hcur, hall + 16, 48);
                lists_over = hall[3] != 0;
                const int32_t *herr = (const int32_t *)(hcur + 4);
                if (herr[0] > 0) {
                    rc = crk_fail(ctx, CRK_EINVAL,
                                  "%d leaves have more than %d candidate leaves within the cut (leaves too small "
                                  "for r_cut or h)", herr[0], kCandCap);
                    goto fail;
                }
                if (herr[1] == 0) break;
                // exact counts plus an eighth (room for the rebuilds of moved particles)
                for (int k = 0; k < 4; ++k) cap[k] = (int64_t)hcur[k] + (int64_t)(hcur[k] / 8) + 64;
                if (attempt == 1) { rc = crk_fail(ctx, CRK_ESTATE, "pair list capacity"); goto fail; }
            }
            lv->gimg_start = se[0]; lv->gimg_cnt = se[1]; lv->gimg = gimg; lv->n_gimg = (int64_t)hcur[0];
            lv->gpair_start = se[2]; lv->gpair_cnt = se[3]; lv->gpair_list = gpair; lv->n_gpairs = (int64_t)hcur[1];
            lv->himg_start = se[4]; lv->himg_cnt = se[5]; lv->himg = himg; lv->n_himg = (int64_t)hcur[2];
            lv->hpair_start = se[6]; lv->hpair_cnt = se[7]; lv->hpair_list = hpair; lv->n_hpairs = (int64_t)hcur[3];
            for (int k = 0; k < 4; ++k) lv->img_cap[k] = cap[k];
        }
        if (re && gas_lists) TRY(crk_build_lists(ctx, lv, true, true));
        if (!re && gas_lists && lists_over) TRY(crk_build_lists(ctx, lv, true, false));  // the exact two-pass build
        if (!re && (ctx->variant[CRK_K_GRAVITY] == CRK_VARIANT_LISTS ||
                    ctx->variant[CRK_K_GRAVITY_ADJOINT] == CRK_VARIANT_LISTS))
            TRY(crk_build_lists(ctx, lv, false, false));
        tr.mark("gravity lists");
    }
#undef TRY
#undef ALLOC
#undef KCHECK
    *out = lv;
    return CRK_OK;
fail:
    if (!re) crk_leaves_free(ctx, lv);
    return rc;
}

int crk_build_leaves(crk_ctx *ctx, const crk_particles *p, const float *h, const crk_leaf_params *lp,
                     crk_leaves **out) {
    if (!ctx) return CRK_EINVAL;
    if (!p) return crk_fail(ctx, CRK_EINVAL, "null argument");
    if (p->n < 0) return crk_fail(ctx, CRK_EINVAL, "particle count out of range");
    std::vector<int64_t> bs = {0, p->n};
    std::vector<float> side = {p->box};
    return build_leaves_impl(ctx, p, h, lp, bs, side, out);
}

int crk_build_leaves_batch(crk_ctx *ctx, const crk_batch *bt, const float *h, const crk_leaf_params *lp,
                           crk_leaves **out) {
    if (!ctx) return CRK_EINVAL;
    if (!bt || !bt->box_start || !bt->box_side || bt->nbox < 1) return crk_fail(ctx, CRK_EINVAL, "bad batch");
    std::vector<int64_t> bs(bt->box_start, bt->box_start + bt->nbox + 1);
    std::vector<float> side(bt->box_side, bt->box_side + bt->nbox);
    crk_particles p{bt->x, bt->y, bt->z, bt->species, bt->n, 0.0f};
    for (float s : side) p.box = std::max(p.box, s);
    return build_leaves_impl(ctx, &p, h, lp, bs, side, out);
}

int crk_leaves_rebuild(crk_ctx *ctx, crk_leaves *lv, const crk_particles *p, const float *h) {
    if (!ctx) return CRK_EINVAL;
    if (!lv || !p) return crk_fail(ctx, CRK_EINVAL, "null argument");
    if (lv->nbox != 1) return crk_fail(ctx, CRK_ESTATE, "rebuild: the leaves hold several boxes");
    std::vector<int64_t> bs = {0, p->n};
    std::vector<float> side = {p->box};
    crk_leaf_params lp{lv->mode, lv->cells, lv->max_leaf, lv->r_cut_grav};
    crk_leaves *out = lv;
    return build_leaves_impl(ctx, p, h, &lp, bs, side, &out, lv);
}

int crk_leaves_rebuild_batch(crk_ctx *ctx, crk_leaves *lv, const crk_batch *bt, const float *h) {
    if (!ctx) return CRK_EINVAL;
    if (!lv || !bt || !bt->box_start || !bt->box_side || bt->nbox < 1) return crk_fail(ctx, CRK_EINVAL, "bad batch");
    std::vector<int64_t> bs(bt->box_start, bt->box_start + bt->nbox + 1);
    std::vector<float> side(bt->box_side, bt->box_side + bt->nbox);
    crk_particles p{bt->x, bt->y, bt->z, bt->species, bt->n, 0.0f};
    for (float s : side) p.box = std::max(p.box, s);
    crk_leaf_params lp{lv->mode, lv->cells, lv->max_leaf, lv->r_cut_grav};
    crk_leaves *out = lv;
    return build_leaves_impl(ctx, &p, h, &lp, bs, side, &out, lv);
}

int crk_leaves_status(crk_ctx *ctx, crk_leaves *lv, int32_t *status) {
    if (!ctx) return CRK_EINVAL;
    if (!lv || !status) return crk_fail(ctx, CRK_EINVAL, "null argument");
    *status = 0;
    if (!lv->dev) return CRK_OK;  // an empty box
    int32_t head[4];
    unsigned long long cur[6];
    CRK_CUDA(ctx, cudaMemcpyAsync(head, lv->dev, sizeof(head), cudaMemcpyDeviceToHost, ctx->stream));
    CRK_CUDA(ctx, cudaMemcpyAsync(cur, lv->dev + 16, sizeof(cur), cudaMemcpyDeviceToHost, ctx->stream));
    CRK_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
    *status = head[0];
    lv->n_gimg = (int64_t)cur[0];
    lv->n_gpairs = (int64_t)cur[1];
    lv->n_himg = (int64_t)cur[2];
    lv->n_hpairs = (int64_t)cur[3];
    return CRK_OK;
}

int crk_leaves_info(const crk_leaves *lv, int64_t info[6]) {
    if (!lv || !info) return CRK_EINVAL;
    info[0] = lv->n;
    info[1] = lv->n_leaves;
    info[2] = lv->n_gpairs;
    info[3] = lv->n_hpairs;
    info[4] = lv->n_gimg;
    info[5] = lv->n_himg;
    return CRK_OK;
}

int crk_leaves_export(crk_ctx *ctx, const crk_leaves *lv, int32_t *perm, int32_t *leaf_start, int32_t *grav_ptr,
                      int32_t *grav_list, int32_t *hydro_ptr, int32_t *hydro_list) {
    if (!ctx) return CRK_EINVAL;
    if (!lv) return crk_fail(ctx, CRK_EINVAL, "null leaves");
    CRK_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
    const int64_t n = lv->n, nl = lv->n_leaves;
    if (perm && n) CRK_CUDA(ctx, cudaMemcpy(perm, lv->perm, sizeof(int32_t) * n, cudaMemcpyDeviceToHost));
    if (leaf_start) CRK_CUDA(ctx, cudaMemcpy(leaf_start, lv->leaf_start, sizeof(int32_t) * (nl + 1), cudaMemcpyDeviceToHost));
    struct {
        int32_t *ptr, *list;
        const int32_t *start, *cnt, *data;
        int64_t total;
    } L[2] = {{grav_ptr, grav_list, lv->gpair_start, lv->gpair_cnt, lv->gpair_list, lv->n_gpairs},
              {hydro_ptr, hydro_list, lv->hpair_start, lv->hpair_cnt, lv->hpair_list, lv->n_hpairs}};
    for (auto &l : L) {
        if (!l.ptr && !l.list) continue;
        std::vector<int32_t> st(nl), ct(nl), data(l.total);
        if (nl) {
            CRK_CUDA(ctx, cudaMemcpy(st.data(), l.start, sizeof(int32_t) * nl, cudaMemcpyDeviceToHost));
            CRK_CUDA(ctx, cudaMemcpy(ct.data(), l.cnt, sizeof(int32_t) * nl, cudaMemcpyDeviceToHost));
        }
        if (l.total) CRK_CUDA(ctx, cudaMemcpy(data.data(), l.data, sizeof(int32_t) * l.total, cudaMemcpyDeviceToHost));
        int64_t k = 0;
        for (int64_t a = 0; a < nl; ++a) {
            if (l.ptr) l.ptr[a] = (int32_t)k;
            for (int32_t q = 0; q < ct[a]; ++q, ++k)
                if (l.list) l.list[k] = data[st[a] + q];
        }
        if (l.ptr) l.ptr[nl] = (int32_t)k;
    }
    return CRK_OK;
}

void crk_leaves_free(crk_ctx *ctx, crk_leaves *lv) {
    if (!lv) return;
    for (auto &b : lv->allocs) {
        if (ctx && ctx->block_cache.size() < 256) ctx->block_cache.push_back(b);
        else cudaFree(b.first);
    }
    delete lv;
}
