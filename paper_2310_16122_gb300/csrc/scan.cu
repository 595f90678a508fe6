// Device-wide exclusive scan and stable LSD radix sort used by the leaf build.
#include "crk_internal.cuh"

namespace {

constexpr int kScanThreads = 256;
constexpr int kScanItems = 8;
constexpr int kScanTile = kScanThreads * kScanItems;

// Block-wide exclusive scan of one int32 per thread; returns the block total.
__device__ __forceinline__ int32_t block_exclusive_scan(int32_t v, int32_t *warp_tot, int32_t &total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    int32_t x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        int32_t y = __shfl_up_sync(CRK_FULL_MASK, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) warp_tot[warp] = x;
    __syncthreads();
    if (warp == 0) {
        int32_t t = lane < nw ? warp_tot[lane] : 0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            int32_t y = __shfl_up_sync(CRK_FULL_MASK, t, o);
            if (lane >= o) t += y;
        }
        if (lane < nw) warp_tot[lane] = t;  // inclusive warp prefix
    }
    __syncthreads();
    total = warp_tot[nw - 1];
    int32_t base = warp > 0 ? warp_tot[warp - 1] : 0;
    int32_t r = base + x - v;
    __syncthreads();
    return r;
}

__global__ void scan_reduce_kernel(const int32_t *__restrict__ in, int64_t n, int32_t *__restrict__ sums) {
    __shared__ int32_t wt[32];
    int64_t base = (int64_t)blockIdx.x * kScanTile;
    int32_t s = 0;
#pragma unroll
    for (int k = 0; k < kScanItems; ++k) {
        int64_t i = base + (int64_t)k * kScanThreads + threadIdx.x;
        if (i < n) s += in[i];
    }
    int32_t tot;
    block_exclusive_scan(s, wt, tot);
    if (threadIdx.x == 0) sums[blockIdx.x] = tot;
}

// single block: exclusive scan of nb block sums in place; writes the grand total
__global__ void scan_sums_kernel(int32_t *sums, int64_t nb, int32_t *total) {
    __shared__ int32_t wt[32];
    int32_t carry = 0;
    for (int64_t s0 = 0; s0 < nb; s0 += blockDim.x) {
        int64_t i = s0 + threadIdx.x;
        int32_t v = i < nb ? sums[i] : 0;
        int32_t tot;
        int32_t e = block_exclusive_scan(v, wt, tot);
        if (i < nb) sums[i] = carry + e;
        carry += tot;
    }
    if (threadIdx.x == 0 && total) *total = carry;
}

__global__ void scan_tile_kernel(const int32_t *__restrict__ in, int32_t *__restrict__ out, int64_t n,
                                 const int32_t *__restrict__ sums) {
    __shared__ int32_t wt[32];
    int64_t base = (int64_t)blockIdx.x * kScanTile + (int64_t)threadIdx.x * kScanItems;  // blocked
    int32_t v[kScanItems];
    int32_t s = 0;
#pragma unroll
    for (int k = 0; k < kScanItems; ++k) {
        int64_t i = base + k;
        v[k] = i < n ? in[i] : 0;
        s += v[k];
    }
    int32_t tot;
    int32_t e = block_exclusive_scan(s, wt, tot) + sums[blockIdx.x];
#pragma unroll
    for (int k = 0; k < kScanItems; ++k) {
        int64_t i = base + k;
        if (i < n) out[i] = e;
        e += v[k];
    }
}

// one block, one pass: exclusive scan of n values (n at most kScanSmall, arrays 16-byte aligned)
// and the total; 32 consecutive values per thread
constexpr int64_t kScanSmall = 32768;
__global__ void __launch_bounds__(1024) scan_small_kernel(const int32_t *in, int32_t *out, int64_t n, int32_t *total) {
    __shared__ int32_t wt[32];
    const int64_t base = (int64_t)threadIdx.x * 32;
    int4 v[8];
    int32_t s = 0;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        const int64_t i = base + 4 * k;
        v[k] = make_int4(0, 0, 0, 0);
        if (i + 3 < n) {
            v[k] = *reinterpret_cast<const int4 *>(in + i);
        } else {
            if (i < n) v[k].x = in[i];
            if (i + 1 < n) v[k].y = in[i + 1];
            if (i + 2 < n) v[k].z = in[i + 2];
        }
        s += v[k].x + v[k].y + v[k].z + v[k].w;
    }
    int32_t tot;
    int32_t e = block_exclusive_scan(s, wt, tot);
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        const int64_t i = base + 4 * k;
        const int4 o = make_int4(e, e + v[k].x, e + v[k].x + v[k].y, e + v[k].x + v[k].y + v[k].z);
        e = o.w + v[k].w;
        if (i + 3 < n) {
            *reinterpret_cast<int4 *>(out + i) = o;
        } else {
            if (i < n) out[i] = o.x;
            if (i + 1 < n) out[i + 1] = o.y;
            if (i + 2 < n) out[i + 2] = o.z;
        }
    }
    if (threadIdx.x == 0 && total) *total = tot;
}

// ---------------------------------------------------------------- radix sort
// LSD radix sort with 8-bit digits: a histogram pass per tile, one exclusive
// scan of the digit-major counts, and a scatter pass that ranks each tile
// stably by digit and writes every digit's run to consecutive positions.
constexpr int kSortThreads = 256;
constexpr int kSortItems = 8;
constexpr int kSortTile = kSortThreads * kSortItems;
constexpr int kSortWarps = kSortThreads / 32;
constexpr int kRadix = 256;  // 8-bit digits
static_assert(kRadix == kSortThreads, "one digit per thread in the scatter's digit scan");

__device__ __forceinline__ unsigned lanemask_below() {
    unsigned m;
    asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
    return m;
}

// What a pass sorts: list l = blockIdx.y of the launch, n items each.
//   kRadixPairs   keys and values of the previous pass
//   kRadixCoords  the first pass of an axis sort: key = the coordinate's bits, value = the index
//   kRadixBoxes   the last pass of a batched axis sort: key = the box of the particle
enum : int { kRadixPairs = 0, kRadixCoords = 1, kRadixBoxes = 2 };
struct RadixIn {
    const uint32_t *key;
    const int32_t *val;
    const float *c[3];
    const int32_t *box_of;
    int64_t n;
    int shift;
};
template <int kMode>
__device__ __forceinline__ uint32_t radix_key(const RadixIn &in, int l, int64_t i, int32_t v) {
    if constexpr (kMode == kRadixCoords) {
        const float x = (l == 0 ? in.c[0] : (l == 1 ? in.c[1] : in.c[2]))[i];
        return crk_coord_key(x);
    } else if constexpr (kMode == kRadixBoxes) {
        return (uint32_t)__ldg(in.box_of + v);
    } else {
        return in.key[l * in.n + i];
    }
}

// per tile: the count of each digit (lanes with equal digits add once per warp step), at
// counts[(list, digit)][tile]
template <int kMode>
__global__ void __launch_bounds__(kSortThreads) radix_hist_kernel(RadixIn in, int32_t *__restrict__ counts, int64_t nb) {
    __shared__ int32_t h[kRadix];
    h[threadIdx.x] = 0;
    __syncthreads();
    const int64_t base = (int64_t)blockIdx.x * kSortTile;
    const int lane = threadIdx.x & 31, l = blockIdx.y;
    uint32_t key[kSortItems];  // every load in flight before the first count
#pragma unroll
    for (int k = 0; k < kSortItems; ++k) {
        const int64_t i = base + (int64_t)k * kSortThreads + threadIdx.x;
        key[k] = 0u;
        if (i < in.n) key[k] = radix_key<kMode>(in, l, i, kMode == kRadixBoxes ? in.val[l * in.n + i] : 0);
    }
#pragma unroll
    for (int k = 0; k < kSortItems; ++k) {
        const int64_t i = base + (int64_t)k * kSortThreads + threadIdx.x;
        const int d = i < in.n ? (int)((key[k] >> in.shift) & (kRadix - 1)) : kRadix;
        const unsigned peers = __match_any_sync(CRK_FULL_MASK, d);
        if (d < kRadix && lane == __ffs(peers) - 1) atomicAdd(&h[d], __popc(peers));
    }
    __syncthreads();
    counts[((int64_t)l * kRadix + threadIdx.x) * nb + blockIdx.x] = h[threadIdx.x];
}

// One LSD pass over a tile.  Warp w takes the tile's items w*256 .. w*256 + 255
// in 8 coalesced steps of 32 (8 items per thread keep the kernel at 48
// registers, five blocks per SM; 16 items took 80 registers and 0.4 ms more
// per 33.5M-particle leaf build); the lanes of a step with equal digits are found
// by __match_any_sync, so each item's rank among the earlier items of its warp
// with the same digit is a running per-warp count plus its rank among its
// peers.  The per-warp counts then give each warp's offset inside the digit,
// a scan over the 256 digits gives each digit's start in the tile, the tile is
// sorted in shared memory, and every digit's run is written to consecutive
// global positions (coalesced stores).  Stable: the tile order is item order.
// kKeys: the keys are written too (a later pass reads them).
template <int kMode, bool kKeys>
__global__ void __launch_bounds__(kSortThreads) radix_scatter_kernel(RadixIn in, uint32_t *__restrict__ kout,
                                                                     int32_t *__restrict__ vout,
                                                                     const int32_t *__restrict__ offsets, int64_t nb) {
    __shared__ int32_t whist[kSortWarps][kRadix];  // per-warp digit counts, then the warp's offset in the digit
    __shared__ int32_t dstart[kRadix];
    __shared__ int32_t goff[kRadix];
    __shared__ uint32_t skey[kSortTile];
    __shared__ int32_t sval[kSortTile];
    __shared__ int32_t wt[32];
    const int t = threadIdx.x, lane = t & 31, w = t >> 5;
    const int l = blockIdx.y;
    const int64_t n = in.n, first = l * n;
    const int shift = in.shift;
    // the scan runs over the lists one after the other: list l starts at l n (mod 2^32)
    goff[t] = (int32_t)((uint32_t)offsets[((int64_t)l * kRadix + t) * nb + blockIdx.x] - (uint32_t)first);
#pragma unroll
    for (int v = 0; v < kSortWarps; ++v) whist[v][t] = 0;
    __syncthreads();
    const int64_t tile0 = (int64_t)blockIdx.x * kSortTile;
    const unsigned below = lanemask_below();
    uint32_t key[kSortItems];
    int32_t val[kSortItems];
    int dig[kSortItems], rank[kSortItems];
#pragma unroll
    for (int r = 0; r < kSortItems; ++r) {
        const int64_t i = tile0 + (int64_t)w * (32 * kSortItems) + 32 * r + lane;
        const bool ok = i < n;
        val[r] = !ok ? 0 : (kMode == kRadixCoords ? (int32_t)i : in.val[first + i]);
        key[r] = ok ? radix_key<kMode>(in, l, i, val[r]) : 0u;
        const int d = ok ? (int)((key[r] >> shift) & (kRadix - 1)) : kRadix;
        dig[r] = d;
        const unsigned peers = __match_any_sync(CRK_FULL_MASK, d);
        const int leader = __ffs(peers) - 1;
        int before = 0;
        if (lane == leader && d < kRadix) {
            before = whist[w][d];
            whist[w][d] = before + __popc(peers);
        }
        before = __shfl_sync(CRK_FULL_MASK, before, leader);
        rank[r] = before + __popc(peers & below);
        __syncwarp();
    }
    __syncthreads();
    // thread t = digit t: the warps' offsets inside the digit, then the digits' starts in the tile
    int32_t tot = 0;
#pragma unroll
    for (int v = 0; v < kSortWarps; ++v) {
        const int32_t c = whist[v][t];
        whist[v][t] = tot;
        tot += c;
    }
    int32_t all;
    dstart[t] = block_exclusive_scan(tot, wt, all);
    __syncthreads();
#pragma unroll
    for (int r = 0; r < kSortItems; ++r) {
        const int d = dig[r];
        if (d < kRadix) {
            const int pos = dstart[d] + whist[w][d] + rank[r];
            skey[pos] = key[r];
            sval[pos] = val[r];
        }
    }
    __syncthreads();
    const int m = (int)(n - tile0 < kSortTile ? n - tile0 : kSortTile);
    for (int i = t; i < m; i += kSortThreads) {
        const uint32_t kk = skey[i];
        const int d = (int)((kk >> shift) & (kRadix - 1));
        const int64_t pos = (int64_t)goff[d] + (i - dstart[d]);
        if constexpr (kKeys) kout[first + pos] = kk;
        vout[first + pos] = sval[i];
    }
}

}  // namespace

int crk_exclusive_scan_i32(crk_ctx *ctx, const int32_t *in, int32_t *out, int64_t n, int32_t *total) {
    if (n <= 0) {
        if (total) CRK_CUDA(ctx, cudaMemsetAsync(total, 0, sizeof(int32_t), ctx->stream));
        return CRK_OK;
    }
    if (n <= kScanSmall && (((uintptr_t)in | (uintptr_t)out) & 15) == 0) {  // one launch instead of three
        scan_small_kernel<<<1, 1024, 0, ctx->stream>>>(in, out, n, total);
        ++ctx->launches;
        CRK_LAUNCH_CHECK(ctx, "exclusive scan");
        return CRK_OK;
    }
    int64_t nb = (n + kScanTile - 1) / kScanTile;
    int32_t *sums = (int32_t *)crk_scratch(ctx, 15, sizeof(int32_t) * (size_t)nb);
    if (!sums) return crk_fail(ctx, CRK_ENOMEM, "scan scratch");
    scan_reduce_kernel<<<(unsigned)nb, kScanThreads, 0, ctx->stream>>>(in, n, sums);
    scan_sums_kernel<<<1, 1024, 0, ctx->stream>>>(sums, nb, total);
    scan_tile_kernel<<<(unsigned)nb, kScanThreads, 0, ctx->stream>>>(in, out, n, sums);
    ctx->launches += 3;
    CRK_LAUNCH_CHECK(ctx, "exclusive scan");
    return CRK_OK;
}

namespace {
// one pass over `lists` lists: histogram, one scan of all the counts, scatter
template <int kMode, bool kKeys>
int radix_pass(crk_ctx *ctx, const RadixIn &in, int lists, uint32_t *kout, int32_t *vout, int32_t *counts, int64_t nb) {
    const dim3 grid((unsigned)nb, (unsigned)lists);
    radix_hist_kernel<kMode><<<grid, kSortThreads, 0, ctx->stream>>>(in, counts, nb);
    CRK_LAUNCH_CHECK(ctx, "radix hist");
    const int rc = crk_exclusive_scan_i32(ctx, counts, counts, lists * nb * kRadix, nullptr);
    if (rc) return rc;
    radix_scatter_kernel<kMode, kKeys><<<grid, kSortThreads, 0, ctx->stream>>>(in, kout, vout, counts, nb);
    ctx->launches += 2;
    CRK_LAUNCH_CHECK(ctx, "radix scatter");
    return CRK_OK;
}
}  // namespace

int crk_radix_sort_u32(crk_ctx *ctx, uint32_t *keys, int32_t *vals, int64_t n, int key_bits) {
    if (n <= 1) return CRK_OK;
    if (n > 2147483647LL) return crk_fail(ctx, CRK_EINVAL, "radix sort: n too large");
    int64_t nb = (n + kSortTile - 1) / kSortTile;
    int passes = (key_bits + 7) / 8;
    uint32_t *k2 = (uint32_t *)crk_scratch(ctx, 13, sizeof(uint32_t) * (size_t)n);
    int32_t *v2 = (int32_t *)crk_scratch(ctx, 14, sizeof(int32_t) * (size_t)n);
    int32_t *counts = (int32_t *)crk_scratch(ctx, 12, sizeof(int32_t) * (size_t)(nb * kRadix));
    if (!k2 || !v2 || !counts) return crk_fail(ctx, CRK_ENOMEM, "radix sort scratch");
    uint32_t *ka = keys, *kb = k2;
    int32_t *va = vals, *vb = v2;
    for (int p = 0; p < passes; ++p) {
        const RadixIn in{ka, va, {}, nullptr, n, 8 * p};
        const int rc = radix_pass<kRadixPairs, true>(ctx, in, 1, kb, vb, counts, nb);
        if (rc) return rc;
        uint32_t *tk = ka; ka = kb; kb = tk;
        int32_t *tv = va; va = vb; vb = tv;
    }
    if (ka != keys) {
        CRK_CUDA(ctx, cudaMemcpyAsync(keys, ka, sizeof(uint32_t) * (size_t)n, cudaMemcpyDeviceToDevice, ctx->stream));
        CRK_CUDA(ctx, cudaMemcpyAsync(vals, va, sizeof(int32_t) * (size_t)n, cudaMemcpyDeviceToDevice, ctx->stream));
    }
    return CRK_OK;
}

// The three axes are sorted by the same launches (a pass is one histogram, one
// scan and one scatter over all of them), the first pass reads the coordinates
// themselves, and the last writes no keys: 12 launches (20 on large boxes)
// instead of 63.  With the merged rank, level and tree launches of the leaf
// build and two host reads instead of four, leaf build + gravity on 30,011
// particles went from 810 to 490 us, the whole step on 2x64^3 from 3490 to 3152 us.
int crk_sort_axes(crk_ctx *ctx, const float *x, const float *y, const float *z, int64_t n, const int32_t *box_of,
                  int nbox, int32_t *order[3], int32_t *spare[9]) {
    if (n <= 0) return CRK_OK;
    if (n > 2147483647LL) return crk_fail(ctx, CRK_EINVAL, "radix sort: n too large");
    const int64_t nb = (n + kSortTile - 1) / kSortTile;
    const int64_t pitch = (n + 63) & ~(int64_t)63;  // of the spare columns: each starts on a 256-byte boundary
    uint32_t *k[2] = {(uint32_t *)crk_scratch(ctx, 1, sizeof(uint32_t) * 3 * (size_t)pitch),
                      (uint32_t *)crk_scratch(ctx, 13, sizeof(uint32_t) * 3 * (size_t)pitch)};
    int32_t *v[2] = {(int32_t *)crk_scratch(ctx, 2, sizeof(int32_t) * 3 * (size_t)pitch),
                     (int32_t *)crk_scratch(ctx, 14, sizeof(int32_t) * 3 * (size_t)pitch)};
    int32_t *counts = (int32_t *)crk_scratch(ctx, 12, sizeof(int32_t) * 3 * (size_t)(nb * kRadix));
    if (!k[0] || !k[1] || !v[0] || !v[1] || !counts) return crk_fail(ctx, CRK_ENOMEM, "radix sort scratch");
    int at = 0, rc;
    RadixIn in{nullptr, nullptr, {x, y, z}, box_of, n, 0};
    if ((rc = radix_pass<kRadixCoords, true>(ctx, in, 3, k[0], v[0], counts, nb))) return rc;
    for (int p = 1; p < 4; ++p, at ^= 1) {
        in.key = k[at];
        in.val = v[at];
        in.shift = 8 * p;
        rc = p < 3 ? radix_pass<kRadixPairs, true>(ctx, in, 3, k[at ^ 1], v[at ^ 1], counts, nb)
                   : radix_pass<kRadixPairs, false>(ctx, in, 3, nullptr, v[at ^ 1], counts, nb);
        if (rc) return rc;
    }
    // batches: stable by box, so the order is (box, coordinate, index); four digits at most (a shift by the
    // width of an int is undefined, and the loop did not end above 2^24 boxes)
    for (int shift = 0; box_of && (shift == 0 || (shift < 32 && (nbox - 1) >> shift)); shift += 8, at ^= 1) {
        in.val = v[at];
        in.shift = shift;
        if ((rc = radix_pass<kRadixBoxes, false>(ctx, in, 3, nullptr, v[at ^ 1], counts, nb))) return rc;
    }
    for (int a = 0; a < 3; ++a) {
        order[a] = v[at] + a * n;
        spare[a] = (int32_t *)k[0] + a * pitch;
        spare[3 + a] = (int32_t *)k[1] + a * pitch;
        spare[6 + a] = v[at ^ 1] + a * pitch;
    }
    return CRK_OK;
}
