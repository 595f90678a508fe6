// Short-range pair kernels of CRK-HACC (Sec. 5: Geometry, Corrections,
// Acceleration/Energy; Sec. 3.1: short-range gravity) and the two adjoints.
//
// Work decomposition (Sec. 5.3 runs the kernels over leaf pairs; the paper's
// "half-warp" lane split is prior art, not reused): one block per i-leaf, one
// warp per group of 32 consecutive i-particles of that leaf.  The warp walks
// the leaf's periodic images of j-leaves; every j-particle whose distance to
// the warp's i-box is below the cut is appended, already shifted into the
// i-leaf frame, to a per-warp buffer in shared memory (ballot compaction).
// Each full buffer is then swept by all 32 lanes, every lane accumulating the
// pair terms of its own i-particle (one-sided: no atomics, deterministic).
// Positions are FP32 relative to the i-leaf origin; sums are FP32 (Kahan-
// compensated for the moment sums); the CRK 3x3 inverse and the conservation
// reductions are FP64.
#include <cmath>
#include <mutex>

#include <type_traits>

#include "crk_internal.cuh"

namespace {

constexpr int kThreads = 128;
constexpr int kWarps = kThreads / 32;
constexpr int kCap = 64;                     // per-warp candidate buffer
constexpr int kCellPairs = 96;                // per-warp candidate pairs of the gravity cell sweeps
constexpr int kGroupImgCap = 128;            // image table of one i-leaf staged per warp in shared memory
// capacities of the one-pass gas lists (adaptive h keeps a gas particle near 58 neighbours;
// the largest lane list and group table seen in the clustered workloads are ~95 and ~360)
constexpr int kGasListCapRows = 128;
constexpr int kGasTableCap = 512;
constexpr float kSigmaW = 0.61548156588532f;  // 495 / (256 pi), Wendland C4 3-D normalisation

// Words of a stage record that are stored: all of it, or Rec::kWords leading ones.
template <class R, class = void>
struct rec_words {
    static constexpr int value = (int)(sizeof(R) / sizeof(float));
};
template <class R>
struct rec_words<R, std::void_t<decltype(R::kWords)>> {
    static constexpr int value = R::kWords;
};

// How the records of a stage are stored.  Planes (the rule): word quads
// 0..kQ-1 as float4 arrays, then a tail of one or two words.  Lanes that read
// different records of one 32-particle cell then touch the same few 128-byte
// lines per load (8 records a line and quad), where whole records cost a line
// per lane, and in shared memory the 16-byte stride spreads random records
// over all banks.  Whole (Rec::kWhole): records side by side, for one whose
// gather is bound by L1 misses rather than by lookups.  Single calls on the
// 2x64^3 clustered box, whole -> planes, us: Extras 275 -> 214, corrections 206
// -> 190, geometry adjoint 108 -> 87, hydro adjoint 687 -> 552, Energy 563 ->
// 355 (limited 471 -> 450).  Kept whole: hydro 319 -> 327, limited 387 -> 412,
// Acceleration 347 -> 354, limited 416 -> 430 (up to 15% on uniform boxes with
// less gas), corrections adjoint (its second kernel 300 -> 338).
template <class R, class = void>
struct rec_whole : std::false_type {};
template <class R>
struct rec_whole<R, std::void_t<decltype(R::kWhole)>> : std::bool_constant<R::kWhole> {};

template <class R>
struct Planes {
    static constexpr bool kWhole = rec_whole<R>::value;
    static constexpr int kW = kWhole ? (int)(sizeof(R) / sizeof(float)) : rec_words<R>::value;
    static constexpr int kQ = kW / 4 + (kW % 4 == 3 ? 1 : 0);
    static constexpr int kT = kW % 4 == 3 ? 0 : kW % 4;
    static constexpr size_t kBytes = 16 * kQ + 4 * kT;  // stored bytes of one record
    static_assert(kBytes <= sizeof(R) && !(kWhole && kT), "stored words lie inside the record");

    __device__ __forceinline__ static int64_t quad(int k, int64_t stride, int64_t i) {
        return kWhole ? i * kQ + k : k * stride + i;
    }
    template <bool kGlobal>
    __device__ __forceinline__ static R load(const void *base, int64_t stride, int64_t i) {
        const float4 *q = reinterpret_cast<const float4 *>(base);
        R r{};
        float *w = reinterpret_cast<float *>(&r);
#pragma unroll
        for (int k = 0; k < kQ; ++k) {
            float4 t;
            if constexpr (kGlobal) t = __ldg(q + quad(k, stride, i));
            else t = q[quad(k, stride, i)];
            w[4 * k] = t.x; w[4 * k + 1] = t.y; w[4 * k + 2] = t.z; w[4 * k + 3] = t.w;
        }
        const float4 *tail = q + kQ * stride;
        if constexpr (kT == 1) {
            const float *f = reinterpret_cast<const float *>(tail) + i;
            w[4 * kQ] = kGlobal ? __ldg(f) : *f;
        } else if constexpr (kT == 2) {
            const float2 *f = reinterpret_cast<const float2 *>(tail) + i;
            float2 t;
            if constexpr (kGlobal) t = __ldg(f);
            else t = *f;
            w[4 * kQ] = t.x; w[4 * kQ + 1] = t.y;
        }
        return r;
    }
    __device__ __forceinline__ static void store(void *base, int64_t stride, int64_t i, const R &r) {
        float4 *q = reinterpret_cast<float4 *>(base);
        const float *w = reinterpret_cast<const float *>(&r);
#pragma unroll
        for (int k = 0; k < kQ; ++k)
            q[quad(k, stride, i)] = make_float4(w[4 * k], w[4 * k + 1], w[4 * k + 2], w[4 * k + 3]);
        float4 *tail = q + kQ * stride;
        if constexpr (kT == 1) reinterpret_cast<float *>(tail)[i] = w[4 * kQ];
        if constexpr (kT == 2) reinterpret_cast<float2 *>(tail)[i] = make_float2(w[4 * kQ], w[4 * kQ + 1]);
    }
};

// The records of one stage in kernel order.
template <class R>
struct RecView {
    const void *base;
    int64_t n;
    __device__ __forceinline__ R operator[](int64_t i) const { return Planes<R>::template load<true>(base, n, i); }
};

struct LeafView {
    const int32_t *leaf_start;
    const int32_t *leaf_ngas;
    const float *bbox;
    const float *hmax;
    const float4 *pos;
    const int32_t *kperm;
    const int32_t *img_start;
    const int32_t *img_cnt;
    const crk_image *img;
    int64_t n_leaves;
    int32_t *queue;  // persistent mode: next leaf to take (zeroed before launch); NULL = one block per leaf
    int korder;      // 1: the stage's per-particle arrays are in kernel order (no permutation)
    int depth;       // gravity sweeps: candidates compacted before each sweep (32, 64 or 96)
    const float4 *gcell;  // boxes of the gravity order's cells of 32 (lo, hi), leaf-relative
};

// Next i-leaf of this block: the grid-stride successor, or (persistent mode)
// the next unclaimed leaf of the work queue.  Block-uniform; every thread calls it.
__device__ __forceinline__ int64_t next_leaf(const LeafView &lv, int64_t cur, int64_t *slot) {
    if (!lv.queue) return cur < 0 ? (int64_t)blockIdx.x : cur + gridDim.x;
    __syncthreads();
    if (threadIdx.x == 0) *slot = atomicAdd(lv.queue, 1);
    __syncthreads();
    return *slot;
}

// Next group of this warp (warp-granular work: one warp per group of 32
// consecutive kernel-order particles of one leaf): the grid-stride successor,
// or (persistent mode) the next unclaimed group of the work queue.  Warp-uniform.
__device__ __forceinline__ int64_t next_group(const LeafView &lv, int64_t cur, int lane) {
    if (!lv.queue) return cur < 0 ? (int64_t)blockIdx.x * kWarps + (threadIdx.x >> 5) : cur + (int64_t)gridDim.x * kWarps;
    int g = 0;
    if (lane == 0) g = atomicAdd(lv.queue, 1);
    return __shfl_sync(CRK_FULL_MASK, g, 0);
}

// index of kernel-order position q in the stage's per-particle arrays
__device__ __forceinline__ int32_t stage_index(const LeafView &lv, int q) { return lv.korder ? q : lv.kperm[q]; }

__device__ __forceinline__ unsigned lanemask_lt() {
    unsigned m;
    asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
    return m;
}

__device__ __forceinline__ void kahan_add(float &s, float &c, float v) {
    float y = v - c;
    float t = s + y;
    c = (t - s) - y;
    s = t;
}

// A value as the unevaluated sum h + l of two floats (h the rounded sum, 2^-47 relative): error-free
// transformations of Dekker (1971) and Knuth, products by FMA.  4-15 FP32 instructions an operation,
// each issued at 64 times the rate of an FP64 one.  Not for infinities or results near the subnormals.
struct Two {
    float h, l;
};
__device__ __forceinline__ Two quick_two(float a, float b) {  // |a| >= |b|, or a = 0
    const float s = __fadd_rn(a, b);
    return {s, __fsub_rn(b, __fsub_rn(s, a))};
}
__device__ __forceinline__ Two sum_two(float a, float b) {
    const float s = __fadd_rn(a, b), t = __fsub_rn(s, a);
    return {s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, t)), __fsub_rn(b, t))};
}
__device__ __forceinline__ Two prod_two(Two a, Two b) {  // not normalised
    const float p = __fmul_rn(a.h, b.h);
    return {p, __fmaf_rn(a.h, b.l, __fmaf_rn(a.l, b.h, __fmaf_rn(a.h, b.h, -p)))};
}
__device__ __forceinline__ Two prod_two(Two a, float b) {
    const float p = __fmul_rn(a.h, b);
    return {p, __fmaf_rn(a.l, b, __fmaf_rn(a.h, b, -p))};
}
__device__ __forceinline__ Two plus_two(Two a, Two b) {  // not normalised
    const Two s = sum_two(a.h, b.h);
    return {s.h, __fadd_rn(s.l, __fadd_rn(a.l, b.l))};
}
__device__ __forceinline__ Two norm_two(Two a) { return quick_two(a.h, a.l); }
__device__ __forceinline__ Two operator-(Two a) { return {-a.h, -a.l}; }
__device__ __forceinline__ Two operator+(Two a, Two b) { return norm_two(plus_two(a, b)); }
__device__ __forceinline__ Two operator+(Two a, float b) {
    const Two s = sum_two(a.h, b);
    return quick_two(s.h, __fadd_rn(s.l, a.l));
}
__device__ __forceinline__ Two operator*(Two a, Two b) { return norm_two(prod_two(a, b)); }
__device__ __forceinline__ Two operator*(Two a, float b) { return norm_two(prod_two(a, b)); }
// the same operations in FP64, so that code over either type reads alike
template <class B>
__device__ __forceinline__ Two mad(Two a, B b, Two c) { return norm_two(plus_two(c, prod_two(a, b))); }
__device__ __forceinline__ double mad(double a, double b, double c) { return fma(a, b, c); }
template <class B>
__device__ __forceinline__ Two dot3(Two a0, B b0, Two a1, B b1, Two a2, B b2) {
    return norm_two(plus_two(plus_two(prod_two(a0, b0), prod_two(a1, b1)), prod_two(a2, b2)));
}
__device__ __forceinline__ double dot3(double a0, double b0, double a1, double b1, double a2, double b2) {
    return fma(a2, b2, fma(a1, b1, a0 * b0));
}
__device__ __forceinline__ Two twice(Two a) { return {2.0f * a.h, 2.0f * a.l}; }
__device__ __forceinline__ double twice(double a) { return 2.0 * a; }
__device__ __forceinline__ Two inverse(Two a) {
    const float r = 1.0f / a.h;
    return quick_two(r, __fmul_rn(r, __fmaf_rn(-r, a.l, __fmaf_rn(-r, a.h, 1.0f))));
}
__device__ __forceinline__ double inverse(double a) { return 1.0 / a; }
__device__ __forceinline__ float rounded(Two a) { return a.h; }  // normalised values
__device__ __forceinline__ float rounded(double a) { return (float)a; }
// exact difference of two floats
__device__ __forceinline__ void difference(float a, float b, Two &d) { d = sum_two(a, -b); }
__device__ __forceinline__ void difference(double a, double b, double &d) { d = a - b; }
// what a float is read as beside a T
template <class T>
struct beside {
    using type = double;
};
template <>
struct beside<Two> {
    using type = float;
};

// 1/sqrt(x), 1/x and a/x by PTX's .approx.ftz instructions, which read a subnormal operand as zero; the
// arguments here are normal numbers.  Gravity's x = r^2 + eps^2 may be subnormal (eps = 0, r < 1e-19):
// x^-3/2 then overflows to infinity either way.  Against rsqrtf and __fdividef, gravity on the 2x128^3 box
// 3644 -> 3272 us, its adjoint 6324 -> 6006 us.
__device__ __forceinline__ float rsqrt_normal(float x) {
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float div_normal(float a, float x) {
    float y;
    asm("div.approx.ftz.f32 %0, %1, %2;" : "=f"(y) : "f"(a), "f"(x));
    return y;
}

// Wendland C4 with support 2h: W and (dW/dr)/r at distance^2 r2, h = hij.
__device__ __forceinline__ void wendland(float r2, float hij, float &W, float &dWr) {
    float r = r2 * rsqrt_normal(fmaxf(r2, 1e-30f));
    float ih = div_normal(1.0f, hij);
    float q = r * ih;
    float t = fmaxf(1.0f - 0.5f * q, 0.0f);
    float t2 = t * t;
    float t5 = t2 * t2 * t;
    float ih2 = ih * ih;
    float ih3 = ih2 * ih;
    float n3 = kSigmaW * ih3;
    W = n3 * t5 * t * (1.0f + q * (3.0f + q * (35.0f / 12.0f)));
    dWr = n3 * ih2 * t5 * (-14.0f / 3.0f) * (1.0f + 2.5f * q);
}

// W, (dW/dr)/r and (d[(dW/dr)/r]/dr)/r = 495/(256 pi h^7) 35 (1 - q/2)^4 (zero beyond 2h)
__device__ __forceinline__ void wendland2(float r2, float hij, float &W, float &dWr, float &ddWr) {
    float r = r2 * rsqrt_normal(fmaxf(r2, 1e-30f));
    float ih = div_normal(1.0f, hij);
    float q = r * ih;
    float t = fmaxf(1.0f - 0.5f * q, 0.0f);
    float t2 = t * t;
    float t4 = t2 * t2;
    float ih2 = ih * ih;
    float n3 = kSigmaW * ih2 * ih;
    W = n3 * t4 * t2 * (1.0f + q * (3.0f + q * (35.0f / 12.0f)));
    dWr = n3 * ih2 * t4 * t * (-14.0f / 3.0f) * (1.0f + 2.5f * q);
    ddWr = n3 * ih2 * ih2 * 35.0f * t4;
}

// ------------------------------------------------------------------ stages
// Each stage defines Rec (one kernel-order record, also the shared-memory
// entry), gather (build Rec of particle p), box_cut (pruning radius of a
// candidate against the i-group box), I (per-lane state), init, interact and
// finish.

struct GravP {
    const float *m;
    float *a3;
    float rc2, eps2;
    float c[6];
    int64_t n;
    unsigned long long *count;
    unsigned long long *swept;  // counting runs: candidate pair evaluations (tiles and lists), may be NULL
};

struct GravStage {
    static constexpr bool kHalfWarp = true;
    static constexpr bool kGasOnly = false;
    static constexpr bool kAllVariants = true;
    using P = GravP;
    struct Rec {
        float x, y, z, m;
    };
    struct I {
        float ax, ay, az;
        int cnt;
    };
    __device__ static Rec gather(const P &p, int32_t orig, float4 ps) { return {ps.x, ps.y, ps.z, p.m[orig]}; }
    static constexpr bool kCons = false;
    __device__ static float box_cut(const P &p, float, const Rec &) { return sqrtf(p.rc2); }
    __device__ static float leaf_cut(const P &p, float, float) { return sqrtf(p.rc2); }
    __device__ static void shift(Rec &r, float sx, float sy, float sz) { r.x += sx; r.y += sy; r.z += sz; }
    __device__ static void init(const P &, I &s, const Rec &, int64_t, int, int, int32_t) { s.ax = s.ay = s.az = 0.f; s.cnt = 0; }
    template <bool kCount>
    __device__ static void interact(const P &p, I &s, const Rec &ri, const Rec &rj) {
        float dx = rj.x - ri.x, dy = rj.y - ri.y, dz = rj.z - ri.z;
        float r2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
        float rinv = rsqrt_normal(r2 + p.eps2);
        float r3 = rinv * rinv * rinv;
        float poly = fmaf(fmaf(fmaf(fmaf(fmaf(p.c[5], r2, p.c[4]), r2, p.c[3]), r2, p.c[2]), r2, p.c[1]), r2, p.c[0]);
        bool in = r2 < p.rc2;
        float f = in ? rj.m * (r3 - poly) : 0.0f;
        s.ax = fmaf(f, dx, s.ax);
        s.ay = fmaf(f, dy, s.ay);
        s.az = fmaf(f, dz, s.az);
        if (kCount) s.cnt += in;
    }
    __device__ static void finish(const P &p, I &s, const Rec &, int32_t orig, int64_t) {
        p.a3[orig] = s.ax;
        p.a3[p.n + orig] = s.ay;
        p.a3[2 * p.n + orig] = s.az;
    }
    __device__ static void finish_other(const P &, int32_t) {}

    // Two candidates per lane step with packed FP32 (f32x2) arithmetic: the
    // same operations and roundings per pair as interact, half the
    // instructions.  Rec2 holds two candidates field-interleaved, so each
    // field pair is one register pair.
    static constexpr bool kPair = true;
    struct __align__(16) Rec2 {
        float2 x, y, z, m;
    };
    struct I2 {
        float2 nx, ny, nz;  // -x_i, broadcast
        float2 ax, ay, az;
        int cnt;
    };
    __device__ static void put2(Rec2 *b, int c, const Rec &r) {
        float *d = reinterpret_cast<float *>(b + (c >> 1)) + (c & 1);
        d[0] = r.x; d[2] = r.y; d[4] = r.z; d[6] = r.m;
    }
    __device__ static Rec far_dummy(float fx, float fy, float fz) { return {fx, fy, fz, 0.0f}; }
    __device__ static void init2(const P &, I2 &s, const Rec &ri) {
        s.nx = make_float2(-ri.x, -ri.x);
        s.ny = make_float2(-ri.y, -ri.y);
        s.nz = make_float2(-ri.z, -ri.z);
        s.ax = s.ay = s.az = make_float2(0.f, 0.f);
        s.cnt = 0;
    }
    template <bool kCount>
    __device__ static void interact2(const P &p, I2 &s, const Rec2 &rj) {
        const float2 dx = __fadd2_rn(rj.x, s.nx), dy = __fadd2_rn(rj.y, s.ny), dz = __fadd2_rn(rj.z, s.nz);
        const float2 r2 = __ffma2_rn(dx, dx, __ffma2_rn(dy, dy, __fmul2_rn(dz, dz)));
        const float2 t = __fadd2_rn(r2, make_float2(p.eps2, p.eps2));
        const float2 rinv = make_float2(rsqrt_normal(t.x), rsqrt_normal(t.y));
        const float2 r3 = __fmul2_rn(__fmul2_rn(rinv, rinv), rinv);
        // -P5(r^2) by Horner with negated coefficients (negation is exact)
        float2 np = __ffma2_rn(make_float2(-p.c[5], -p.c[5]), r2, make_float2(-p.c[4], -p.c[4]));
        np = __ffma2_rn(np, r2, make_float2(-p.c[3], -p.c[3]));
        np = __ffma2_rn(np, r2, make_float2(-p.c[2], -p.c[2]));
        np = __ffma2_rn(np, r2, make_float2(-p.c[1], -p.c[1]));
        np = __ffma2_rn(np, r2, make_float2(-p.c[0], -p.c[0]));
        const float2 g = __fmul2_rn(rj.m, __fadd2_rn(r3, np));
        const bool in0 = r2.x < p.rc2, in1 = r2.y < p.rc2;
        const float2 f = make_float2(in0 ? g.x : 0.0f, in1 ? g.y : 0.0f);
        s.ax = __ffma2_rn(f, dx, s.ax);
        s.ay = __ffma2_rn(f, dy, s.ay);
        s.az = __ffma2_rn(f, dz, s.az);
        if (kCount) s.cnt += (int)in0 + (int)in1;
    }
    // Cell sweeps: the candidate buffer is in planes of float4 over candidate pairs, (x0, x1, y0, y1)
    // and (z0, z1, m0, m1), so that a pair's fields load as register pairs.
    static constexpr int kPlanes = 2;
    __device__ static void putc(float4 (*b)[kCellPairs], int c, const Rec &r) {
        float *a = reinterpret_cast<float *>(b[0] + (c >> 1)) + (c & 1), *d = reinterpret_cast<float *>(b[1] + (c >> 1)) + (c & 1);
        a[0] = r.x; a[2] = r.y; d[0] = r.z; d[2] = r.m;
    }
    __device__ static Rec2 getc(const float4 (*b)[kCellPairs], int k) {
        const float4 a = b[0][k], d = b[1][k];
        return {make_float2(a.x, a.y), make_float2(a.z, a.w), make_float2(d.x, d.y), make_float2(d.z, d.w)};
    }
    // adds the sums of lane ^ o
    __device__ static void addc(I2 &s, int o) {
        float2 *a[3] = {&s.ax, &s.ay, &s.az};
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            a[k]->x += __shfl_xor_sync(CRK_FULL_MASK, a[k]->x, o);
            a[k]->y += __shfl_xor_sync(CRK_FULL_MASK, a[k]->y, o);
        }
    }
    // partial sums of one i from one leaf-pair tile (half-warp arms): added atomically
    __device__ static void flush(const P &p, const I &s, const Rec &, int32_t o) {
        atomicAdd(&p.a3[o], s.ax);
        atomicAdd(&p.a3[p.n + o], s.ay);
        atomicAdd(&p.a3[2 * p.n + o], s.az);
    }
    static void zero_outputs(const P &p, cudaStream_t st) { cudaMemsetAsync(p.a3, 0, sizeof(float) * 3 * p.n, st); }
    __device__ static void finish2(const P &p, I2 &s, int32_t orig) {
        p.a3[orig] = s.ax.x + s.ax.y;
        p.a3[p.n + orig] = s.ay.x + s.ay.y;
        p.a3[2 * p.n + orig] = s.az.x + s.az.y;
    }
};

struct GravAdjP {
    const float *m, *abar;
    float *gx3, *gm;
    float rc2, eps2;
    float c[6];
    int64_t n;
    unsigned long long *count;
    unsigned long long *swept;  // counting runs: candidate pair evaluations (tiles and lists), may be NULL
};

struct GravAdjStage {
    static constexpr bool kHalfWarp = true;
    static constexpr bool kGasOnly = false;
    static constexpr bool kAllVariants = true;
    using P = GravAdjP;
    struct __align__(16) Rec {
        float x, y, z, m;
        float bx, by, bz, pad;
    };
    struct I {
        float gx, gy, gz, gm;
        int cnt;
    };
    __device__ static Rec gather(const P &p, int32_t o, float4 ps) {
        return {ps.x, ps.y, ps.z, p.m[o], p.abar[o], p.abar[p.n + o], p.abar[2 * p.n + o], 0.f};
    }
    static constexpr bool kCons = false;
    __device__ static float box_cut(const P &p, float, const Rec &) { return sqrtf(p.rc2); }
    __device__ static float leaf_cut(const P &p, float, float) { return sqrtf(p.rc2); }
    __device__ static void shift(Rec &r, float sx, float sy, float sz) { r.x += sx; r.y += sy; r.z += sz; }
    __device__ static void init(const P &, I &s, const Rec &, int64_t, int, int, int32_t) { s.gx = s.gy = s.gz = s.gm = 0.f; s.cnt = 0; }
    template <bool kCount>
    __device__ static void interact(const P &p, I &s, const Rec &ri, const Rec &rj) {
        float dx = rj.x - ri.x, dy = rj.y - ri.y, dz = rj.z - ri.z;  // d_ij = x_j - x_i
        float r2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
        float rinv = rsqrt_normal(r2 + p.eps2);
        float ri2 = rinv * rinv;
        float r3 = ri2 * rinv;
        float poly = fmaf(fmaf(fmaf(fmaf(fmaf(p.c[5], r2, p.c[4]), r2, p.c[3]), r2, p.c[2]), r2, p.c[1]), r2, p.c[0]);
        float dpoly = fmaf(fmaf(fmaf(fmaf(5.0f * p.c[5], r2, 4.0f * p.c[4]), r2, 3.0f * p.c[3]), r2, 2.0f * p.c[2]),
                           r2, p.c[1]);
        bool in = r2 < p.rc2;
        float g = in ? r3 - poly : 0.0f;
        float dg2 = in ? 2.0f * fmaf(-1.5f * r3, ri2, -dpoly) : 0.0f;
        float wx = ri.m * rj.bx - rj.m * ri.bx;
        float wy = ri.m * rj.by - rj.m * ri.by;
        float wz = ri.m * rj.bz - rj.m * ri.bz;
        float dw = fmaf(dx, wx, fmaf(dy, wy, dz * wz));
        float k = dg2 * dw;
        s.gx = fmaf(g, wx, fmaf(k, dx, s.gx));
        s.gy = fmaf(g, wy, fmaf(k, dy, s.gy));
        s.gz = fmaf(g, wz, fmaf(k, dz, s.gz));
        s.gm = fmaf(-g, fmaf(rj.bx, dx, fmaf(rj.by, dy, rj.bz * dz)), s.gm);
        if (kCount) s.cnt += in;
    }
    __device__ static void finish(const P &p, I &s, const Rec &, int32_t o, int64_t) {
        p.gx3[o] = s.gx;
        p.gx3[p.n + o] = s.gy;
        p.gx3[2 * p.n + o] = s.gz;
        p.gm[o] = s.gm;
    }
    __device__ static void finish_other(const P &, int32_t) {}

    // Two candidates per lane step with packed FP32 (f32x2) arithmetic (see GravStage).
    static constexpr bool kPair = true;
    struct __align__(16) Rec2 {
        float2 x, y, z, m;
        float2 bx, by, bz, pad;
    };
    struct I2 {
        float2 nx, ny, nz;         // -x_i, broadcast
        float2 mi, nbx, nby, nbz;  // m_i, -abar_i, broadcast
        // sum_j g w_j = m_i sum_j g abar_j - abar_i sum_j g m_j (w = m_i abar_j - m_j abar_i), so the
        // pair loop accumulates the two sums and k d; sg accumulates g (abar_j . d) (gm = -sg)
        float2 kx, ky, kz, s1x, s1y, s1z, s2, sg;
        int cnt;
    };
    __device__ static void put2(Rec2 *b, int c, const Rec &r) {
        float *d = reinterpret_cast<float *>(b + (c >> 1)) + (c & 1);
        d[0] = r.x; d[2] = r.y; d[4] = r.z; d[6] = r.m;
        d[8] = r.bx; d[10] = r.by; d[12] = r.bz; d[14] = 0.0f;
    }
    __device__ static Rec far_dummy(float fx, float fy, float fz) { return {fx, fy, fz, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f}; }
    __device__ static void init2(const P &, I2 &s, const Rec &ri) {
        s.nx = make_float2(-ri.x, -ri.x);
        s.ny = make_float2(-ri.y, -ri.y);
        s.nz = make_float2(-ri.z, -ri.z);
        s.mi = make_float2(ri.m, ri.m);
        s.nbx = make_float2(-ri.bx, -ri.bx);
        s.nby = make_float2(-ri.by, -ri.by);
        s.nbz = make_float2(-ri.bz, -ri.bz);
        s.kx = s.ky = s.kz = s.s1x = s.s1y = s.s1z = s.s2 = s.sg = make_float2(0.f, 0.f);
        s.cnt = 0;
    }
    template <bool kCount>
    __device__ static void interact2(const P &p, I2 &s, const Rec2 &rj) {
        const float2 dx = __fadd2_rn(rj.x, s.nx), dy = __fadd2_rn(rj.y, s.ny), dz = __fadd2_rn(rj.z, s.nz);
        const float2 r2 = __ffma2_rn(dx, dx, __ffma2_rn(dy, dy, __fmul2_rn(dz, dz)));
        const float2 t = __fadd2_rn(r2, make_float2(p.eps2, p.eps2));
        const float2 rinv = make_float2(rsqrt_normal(t.x), rsqrt_normal(t.y));
        const float2 ri2 = __fmul2_rn(rinv, rinv);
        const float2 r3 = __fmul2_rn(ri2, rinv);
        float2 np = __ffma2_rn(make_float2(-p.c[5], -p.c[5]), r2, make_float2(-p.c[4], -p.c[4]));
        np = __ffma2_rn(np, r2, make_float2(-p.c[3], -p.c[3]));
        np = __ffma2_rn(np, r2, make_float2(-p.c[2], -p.c[2]));
        np = __ffma2_rn(np, r2, make_float2(-p.c[1], -p.c[1]));
        np = __ffma2_rn(np, r2, make_float2(-p.c[0], -p.c[0]));  // -P5
        // -2 P5' with doubled coefficients (scaling by 2 is exact)
        const float c5 = -10.0f * p.c[5], c4 = -8.0f * p.c[4], c3 = -6.0f * p.c[3], c2 = -4.0f * p.c[2];
        float2 ndp = __ffma2_rn(make_float2(c5, c5), r2, make_float2(c4, c4));
        ndp = __ffma2_rn(ndp, r2, make_float2(c3, c3));
        ndp = __ffma2_rn(ndp, r2, make_float2(c2, c2));
        ndp = __ffma2_rn(ndp, r2, make_float2(-2.0f * p.c[1], -2.0f * p.c[1]));
        const bool in0 = r2.x < p.rc2, in1 = r2.y < p.rc2;
        const float2 gv = __fadd2_rn(r3, np);
        // 2 g'(s) = 2 (-1.5 r^-5 - P5')
        const float2 dv = __ffma2_rn(__fmul2_rn(make_float2(-3.0f, -3.0f), r3), ri2, ndp);
        const float2 g = make_float2(in0 ? gv.x : 0.0f, in1 ? gv.y : 0.0f);
        const float2 dg2 = make_float2(in0 ? dv.x : 0.0f, in1 ? dv.y : 0.0f);
        // abar_j . d and -abar_i . d, then d . w = m_i (abar_j . d) - m_j (abar_i . d)
        const float2 dbj = __ffma2_rn(rj.bx, dx, __ffma2_rn(rj.by, dy, __fmul2_rn(rj.bz, dz)));
        const float2 ndbi = __ffma2_rn(s.nbx, dx, __ffma2_rn(s.nby, dy, __fmul2_rn(s.nbz, dz)));
        const float2 dw = __ffma2_rn(s.mi, dbj, __fmul2_rn(rj.m, ndbi));
        const float2 k = __fmul2_rn(dg2, dw);
        s.kx = __ffma2_rn(k, dx, s.kx);
        s.ky = __ffma2_rn(k, dy, s.ky);
        s.kz = __ffma2_rn(k, dz, s.kz);
        s.s1x = __ffma2_rn(g, rj.bx, s.s1x);
        s.s1y = __ffma2_rn(g, rj.by, s.s1y);
        s.s1z = __ffma2_rn(g, rj.bz, s.s1z);
        s.s2 = __ffma2_rn(g, rj.m, s.s2);
        s.sg = __ffma2_rn(g, dbj, s.sg);
        if (kCount) s.cnt += (int)in0 + (int)in1;
    }
    // Cell sweeps: planes (x0, x1, y0, y1), (z0, z1, m0, m1), (bx0, bx1, by0, by1), (bz0, bz1, -, -).
    static constexpr int kPlanes = 4;
    __device__ static void putc(float4 (*b)[kCellPairs], int c, const Rec &r) {
        const float v[7] = {r.x, r.y, r.z, r.m, r.bx, r.by, r.bz};
#pragma unroll
        for (int k = 0; k < 7; ++k)
            (reinterpret_cast<float *>(b[k >> 1] + (c >> 1)) + (c & 1))[2 * (k & 1)] = v[k];
    }
    __device__ static Rec2 getc(const float4 (*b)[kCellPairs], int k) {
        const float4 a = b[0][k], d = b[1][k], e = b[2][k];
        const float2 f = *reinterpret_cast<const float2 *>(&b[3][k]);
        return {make_float2(a.x, a.y), make_float2(a.z, a.w), make_float2(d.x, d.y), make_float2(d.z, d.w),
                make_float2(e.x, e.y), make_float2(e.z, e.w), f, f};
    }
    // adds the sums of lane ^ o
    __device__ static void addc(I2 &s, int o) {
        float2 *a[8] = {&s.kx, &s.ky, &s.kz, &s.s1x, &s.s1y, &s.s1z, &s.s2, &s.sg};
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            a[k]->x += __shfl_xor_sync(CRK_FULL_MASK, a[k]->x, o);
            a[k]->y += __shfl_xor_sync(CRK_FULL_MASK, a[k]->y, o);
        }
    }
    // partial sums of one i from one leaf-pair tile (half-warp arms): added atomically
    __device__ static void flush(const P &p, const I &s, const Rec &, int32_t o) {
        atomicAdd(&p.gx3[o], s.gx);
        atomicAdd(&p.gx3[p.n + o], s.gy);
        atomicAdd(&p.gx3[2 * p.n + o], s.gz);
        atomicAdd(&p.gm[o], s.gm);
    }
    static void zero_outputs(const P &p, cudaStream_t st) {
        cudaMemsetAsync(p.gx3, 0, sizeof(float) * 3 * p.n, st);
        cudaMemsetAsync(p.gm, 0, sizeof(float) * p.n, st);
    }
    __device__ static void finish2(const P &p, I2 &s, int32_t o) {
        const float mi = s.mi.x, nbx = s.nbx.x, nby = s.nby.x, nbz = s.nbz.x;
        const float s2 = s.s2.x + s.s2.y;
        p.gx3[o] = fmaf(mi, s.s1x.x + s.s1x.y, fmaf(nbx, s2, s.kx.x + s.kx.y));
        p.gx3[p.n + o] = fmaf(mi, s.s1y.x + s.s1y.y, fmaf(nby, s2, s.ky.x + s.ky.y));
        p.gx3[2 * p.n + o] = fmaf(mi, s.s1z.x + s.s1z.y, fmaf(nbz, s2, s.kz.x + s.kz.y));
        p.gm[o] = -(s.sg.x + s.sg.y);
    }
};

struct GeomP {
    const float *m;
    float *V, *rho;
    int64_t n;
    unsigned long long *count;
    unsigned long long *swept;  // counting runs: candidate pair evaluations (tiles and lists), may be NULL
};

struct GeomStage {
    static constexpr bool kPair = false;
    static constexpr bool kGasOnly = true;
    static constexpr bool kCons = false;
    static constexpr bool kAllVariants = true;
    using P = GeomP;
    struct Rec {
        float x, y, z, h;
    };
    struct I {
        float s, c;
        int cnt;
    };
    __device__ static Rec gather(const P &, int32_t, float4 ps) { return {ps.x, ps.y, ps.z, ps.w}; }
    __device__ static float box_cut(const P &, float hmax_i, const Rec &rj) { return hmax_i + rj.h; }
    __device__ static float leaf_cut(const P &, float hmax_i, float hmax_j) { return hmax_i + hmax_j; }
    __device__ static void shift(Rec &r, float sx, float sy, float sz) { r.x += sx; r.y += sy; r.z += sz; }
    __device__ static void init(const P &, I &s, const Rec &, int64_t, int, int, int32_t) { s.s = s.c = 0.f; s.cnt = 0; }
    template <bool kCount>
    __device__ static void interact(const P &, I &s, const Rec &ri, const Rec &rj) {
        float dx = ri.x - rj.x, dy = ri.y - rj.y, dz = ri.z - rj.z;
        float r2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
        float hs = ri.h + rj.h;
        bool in = r2 < hs * hs;
        float W, dWr;
        wendland(r2, 0.5f * hs, W, dWr);
        kahan_add(s.s, s.c, in ? W : 0.0f);
        if (kCount) s.cnt += in;
    }
    __device__ static void finish(const P &p, I &s, const Rec &, int32_t o, int64_t) {
        float sum = s.s - s.c;
        float V = 1.0f / sum;
        p.V[o] = V;
        p.rho[o] = p.m[o] * sum;
    }
    __device__ static void finish_other(const P &p, int32_t o) {
        p.V[o] = 0.f;
        p.rho[o] = 0.f;
    }
};

struct GeomAdjP {
    const float *m, *V, *rhobar, *Vbar;
    float *gx3, *gm;
    int64_t n;
    unsigned long long *count;
    unsigned long long *swept;  // counting runs: candidate pair evaluations (tiles and lists), may be NULL
};

struct GeomAdjStage {
    static constexpr bool kPair = false;
    static constexpr bool kGasOnly = true;
    static constexpr bool kCons = false;
    static constexpr bool kAllVariants = true;
    using P = GeomAdjP;
    struct __align__(16) Rec {
        float x, y, z, h;
        float sbar, pad0, pad1, pad2;
        static constexpr int kWords = 5;
    };
    struct I {
        float gx, gy, gz;
        int cnt;
    };
    __device__ static Rec gather(const P &p, int32_t o, float4 ps) {
        float V = p.V[o];
        float sb = p.rhobar[o] * p.m[o] - (p.Vbar ? p.Vbar[o] * V * V : 0.0f);
        return {ps.x, ps.y, ps.z, ps.w, sb, 0.f, 0.f, 0.f};
    }
    __device__ static float box_cut(const P &, float hmax_i, const Rec &rj) { return hmax_i + rj.h; }
    __device__ static float leaf_cut(const P &, float hmax_i, float hmax_j) { return hmax_i + hmax_j; }
    __device__ static void shift(Rec &r, float sx, float sy, float sz) { r.x += sx; r.y += sy; r.z += sz; }
    __device__ static void init(const P &, I &s, const Rec &, int64_t, int, int, int32_t) { s.gx = s.gy = s.gz = 0.f; s.cnt = 0; }
    template <bool kCount>
    __device__ static void interact(const P &, I &s, const Rec &ri, const Rec &rj) {
        float dx = ri.x - rj.x, dy = ri.y - rj.y, dz = ri.z - rj.z;  // x_kj
        float r2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
        float hs = ri.h + rj.h;
        bool in = r2 < hs * hs;
        float W, dWr;
        wendland(r2, 0.5f * hs, W, dWr);
        float k = in ? (ri.sbar + rj.sbar) * dWr : 0.0f;
        s.gx = fmaf(k, dx, s.gx);
        s.gy = fmaf(k, dy, s.gy);
        s.gz = fmaf(k, dz, s.gz);
        if (kCount) s.cnt += in;
    }
    __device__ static void finish(const P &p, I &s, const Rec &, int32_t o, int64_t) {
        p.gx3[o] = s.gx;
        p.gx3[p.n + o] = s.gy;
        p.gx3[2 * p.n + o] = s.gz;
        p.gm[o] = p.rhobar[o] / p.V[o];
    }
    __device__ static void finish_other(const P &p, int32_t o) {
        p.gx3[o] = 0.f;
        p.gx3[p.n + o] = 0.f;
        p.gx3[2 * p.n + o] = 0.f;
        p.gm[o] = 0.f;
    }
};

struct CorrP {
    const float *V;
    float *A, *B, *gA, *gB;
    int32_t *n_singular;
    int64_t n;
    unsigned long long *count;
    unsigned long long *swept;  // counting runs: candidate pair evaluations (tiles and lists), may be NULL
};

struct CorrStage {
    static constexpr bool kPair = false;
    static constexpr bool kGasOnly = true;
    static constexpr bool kCons = false;
    static constexpr bool kAllVariants = true;
    using P = CorrP;
    struct __align__(16) Rec {
        float x, y, z, h;
        float V, pad0, pad1, pad2;
        static constexpr int kWords = 5;
    };
    struct I {
        float m0, c0;
        float m1[3], c1[3];
        float m2[6], c2[6];  // xx xy xz yy yz zz
        // Gradient moments.  With w = V_j W and d_g(V_j W) = V_j dWr x_g, the g-derivatives of
        // m1_a and m2_ab are delta_ag m0 + V_j dWr x_a x_g and delta_ag m1_b + delta_bg m1_a +
        // V_j dWr x_a x_b x_g: only the symmetric dWr sums s2 (second order) and s3 (third
        // order) are accumulated, the delta terms come from m0 and m1 in finish.
        float dm0[3];
        float s2[6];   // xx xy xz yy yz zz
        float s3[10];  // xxx xxy xxz xyy xyz xzz yyy yyz yzz zzz
        int cnt;
    };
    // packed index of (a <= b) among xx xy xz yy yz zz
    __host__ __device__ static constexpr int idx2(int a, int b) { return a * (5 - a) / 2 + b; }
    // packed index of (a <= b <= c) among xxx xxy xxz xyy xyz xzz yyy yyz yzz zzz
    __host__ __device__ static constexpr int idx3(int a, int b, int c) {
        return a == 0 ? (b == 0 ? c : (b == 1 ? 2 + c : 5)) : (a == 1 ? (b == 1 ? 5 + c : 8) : 9);
    }
    // The solve of one particle.  With q = m0 + B.m1 = 1/A, T = s3 B (the symmetric matrix
    // sum_b s3_abg B_b) and U = s2 + T,
    //   dm1_g + dm2_g B = q e_g + U_g + B_g m1  (U_g: column g)  and  m2^-1 m1 = -B, so
    //   dB_g = -m2^-1 (U_g + q e_g) + B_g B,
    //   dm0_g + 2 B.dm1_g + B^T dm2_g B = dm0_g + 2 q B_g + ((2 s2 + T) B)_g.
    // Matrices are packed xx xy xz yy yz zz; Uq is U with q added on its diagonal.
    // T = Two: lengths in units of a power of two near sqrt(tr m2), which keeps the FP32 exponents
    // in range.  FP64 runs at 1/64 of the FP32 rate here: with it the solve took a third of the kernel
    // (2x64^3: 164 us, now 127; 2x128^3 in the kernel order 1.15 ms, now 0.90; the reverse's
    // preparation 295 us, now 254).  Only a particle that is close to singular (det m2 < 1e-6 tr^3,
    // where 47 bits could show) or out of range goes through FP64.
    template <class T>
    struct Solved {
        using F = typename beside<T>::type;
        T Mi[6], m1[3], B[3], q, A, U[6], Uq[6], K[3];
        F s3[10], f1, g1;  // third sums in scaled lengths; scale of a length and its inverse
    };
    template <class T>
    __device__ static T at(const T m[6], int a, int b) { return m[a <= b ? idx2(a, b) : idx2(b, a)]; }
    // row a of the symmetric matrix m times v
    template <class T>
    __device__ static T row(const T m[6], int a, const T v[3]) {
        return dot3(at(m, a, 0), v[0], at(m, a, 1), v[1], at(m, a, 2), v[2]);
    }
    __device__ static void scale_of(float tr, double &f1, double &g1) { f1 = g1 = 1.0; }
    __device__ static void scale_of(float tr, float &f1, float &g1) {
        const int half = max((((__float_as_int(tr) >> 23) & 255) - 127) >> 1, -63);
        f1 = __int_as_float((127 - half) << 23);
        g1 = __int_as_float((127 + half) << 23);
    }
    // is det m2 large enough for T, in scaled lengths
    __device__ static bool regular(double det, double tr, float) { return det > 1e-12 * tr * tr * tr; }
    __device__ static bool regular(Two det, Two tr, float m0) {
        return det.h > 1e-6f * tr.h * tr.h * tr.h && m0 > 1e-12f && m0 < 1e12f;
    }
    // false for a singular particle (FP64) or one that needs FP64 (Two)
    template <class T, class Sums>
    __device__ static bool solve(const Sums &s, Solved<T> &r) {
        using F = typename beside<T>::type;
        scale_of(s.m2[0] + s.m2[3] + s.m2[5], r.f1, r.g1);
        const F f1 = r.f1, f2 = f1 * f1;
        T M[6];
#pragma unroll
        for (int k = 0; k < 6; ++k) difference((F)s.m2[k] * f2, (F)s.c2[k] * f2, M[k]);
        // cofactors of the symmetric matrix
        r.Mi[0] = mad(M[3], M[5], -(M[4] * M[4]));
        r.Mi[1] = mad(M[2], M[4], -(M[1] * M[5]));
        r.Mi[2] = mad(M[1], M[4], -(M[2] * M[3]));
        r.Mi[3] = mad(M[0], M[5], -(M[2] * M[2]));
        r.Mi[4] = mad(M[1], M[2], -(M[0] * M[4]));
        r.Mi[5] = mad(M[0], M[3], -(M[1] * M[1]));
        const T det = dot3(M[0], r.Mi[0], M[1], r.Mi[1], M[2], r.Mi[2]);
        if (!regular(det, M[0] + M[3] + M[5], s.m0)) return false;
        const T id = inverse(det);
#pragma unroll
        for (int k = 0; k < 6; ++k) r.Mi[k] = r.Mi[k] * id;
#pragma unroll
        for (int a = 0; a < 3; ++a) difference((F)s.m1[a] * f1, (F)s.c1[a] * f1, r.m1[a]);
#pragma unroll
        for (int a = 0; a < 3; ++a) r.B[a] = -row(r.Mi, a, r.m1);
        T m0;
        difference((F)s.m0, (F)s.c0, m0);
        r.q = m0 + dot3(r.B[0], r.m1[0], r.B[1], r.m1[1], r.B[2], r.m1[2]);
        r.A = inverse(r.q);
        T W[6];
#pragma unroll
        for (int k = 0; k < 10; ++k) r.s3[k] = (F)s.s3[k] * f1;
        const int ia[6] = {0, 0, 0, 1, 1, 2}, ib[6] = {0, 1, 2, 1, 2, 2};
#pragma unroll
        for (int k = 0; k < 6; ++k) {
            const T t = dot3(r.B[0], r.s3[sorted3(ia[k], ib[k], 0)], r.B[1], r.s3[sorted3(ia[k], ib[k], 1)], r.B[2],
                             r.s3[sorted3(ia[k], ib[k], 2)]);
            r.U[k] = t + (F)s.s2[k];
            r.Uq[k] = ia[k] == ib[k] ? r.U[k] + r.q : r.U[k];
            W[k] = r.U[k] + (F)s.s2[k];  // 2 s2 + T
        }
#pragma unroll
        for (int g = 0; g < 3; ++g) r.K[g] = mad(twice(r.q), r.B[g], row(W, g, r.B)) + (F)s.dm0[g] * r.g1;
        return true;
    }
    // packed index of the sorted axes of (a <= b) and c
    __host__ __device__ static constexpr int sorted3(int a, int b, int c) {
        return c >= b ? idx3(a, b, c) : (c >= a ? idx3(a, c, b) : idx3(c, a, b));
    }
    __device__ static Rec gather(const P &p, int32_t o, float4 ps) { return {ps.x, ps.y, ps.z, ps.w, p.V[o], 0, 0, 0}; }
    __device__ static float box_cut(const P &, float hmax_i, const Rec &rj) { return hmax_i + rj.h; }
    __device__ static float leaf_cut(const P &, float hmax_i, float hmax_j) { return hmax_i + hmax_j; }
    __device__ static void shift(Rec &r, float sx, float sy, float sz) { r.x += sx; r.y += sy; r.z += sz; }
    __device__ static void init(const P &, I &s, const Rec &, int64_t, int, int, int32_t) {
        s.m0 = s.c0 = 0.f;
#pragma unroll
        for (int a = 0; a < 3; ++a) s.m1[a] = s.c1[a] = s.dm0[a] = 0.f;
#pragma unroll
        for (int a = 0; a < 6; ++a) s.m2[a] = s.c2[a] = 0.f;
#pragma unroll
        for (int a = 0; a < 6; ++a) s.s2[a] = 0.f;
#pragma unroll
        for (int a = 0; a < 10; ++a) s.s3[a] = 0.f;
        s.cnt = 0;
    }
    template <bool kCount>
    __device__ static void interact(const P &, I &s, const Rec &ri, const Rec &rj) {
        float x[3] = {ri.x - rj.x, ri.y - rj.y, ri.z - rj.z};  // x_ij
        float r2 = fmaf(x[0], x[0], fmaf(x[1], x[1], x[2] * x[2]));
        float hs = ri.h + rj.h;
        bool in = r2 < hs * hs;
        float W, dWr;
        wendland(r2, 0.5f * hs, W, dWr);
        float w = in ? rj.V * W : 0.0f;
        float vd = in ? rj.V * dWr : 0.0f;
        float wx[3] = {w * x[0], w * x[1], w * x[2]};
        float dW[3] = {vd * x[0], vd * x[1], vd * x[2]};  // V_j d_g W
        kahan_add(s.m0, s.c0, w);
#pragma unroll
        for (int a = 0; a < 3; ++a) kahan_add(s.m1[a], s.c1[a], wx[a]);
        const int ia[6] = {0, 0, 0, 1, 1, 2}, ib[6] = {0, 1, 2, 1, 2, 2};
        float xx[6];
#pragma unroll
        for (int q = 0; q < 6; ++q) {
            xx[q] = x[ia[q]] * x[ib[q]];
            kahan_add(s.m2[q], s.c2[q], wx[ia[q]] * x[ib[q]]);
            s.s2[q] = fmaf(xx[q], vd, s.s2[q]);
        }
#pragma unroll
        for (int g = 0; g < 3; ++g) s.dm0[g] += dW[g];
        // s3[abc] += x_a x_b (V_j dWr x_c) for a <= b <= c
        const int k3q[10] = {0, 0, 0, 1, 1, 2, 3, 3, 4, 5}, k3c[10] = {0, 1, 2, 1, 2, 2, 1, 2, 2, 2};
#pragma unroll
        for (int k = 0; k < 10; ++k) s.s3[k] = fmaf(xx[k3q[k]], dW[k3c[k]], s.s3[k]);
        if (kCount) s.cnt += in;
    }
    // false if the particle's sums cannot be worked on in T
    template <class T>
    __device__ static bool finish_in(const P &p, const I &s, int32_t o) {
        using F = typename beside<T>::type;
        const int64_t n = p.n;
        Solved<T> r;
        if (!solve(s, r)) return false;
        float sum = 0.0f;  // NaN once a result is not finite
        auto put = [&](float *out, float v) {
            *out = v;
            sum = fmaf(v, 0.0f, sum);
        };
        put(p.A + o, rounded(r.A));
#pragma unroll
        for (int a = 0; a < 3; ++a) put(p.B + a * n + o, rounded(r.B[a] * r.f1));
#pragma unroll
        for (int g = 0; g < 3; ++g) {
            put(p.gA + g * n + o, rounded(-(r.A * r.K[g]) * r.A * r.f1));
            const T u[3] = {at(r.Uq, 0, g), at(r.Uq, 1, g), at(r.Uq, 2, g)};
#pragma unroll
            for (int a = 0; a < 3; ++a)
                put(p.gB + (3 * g + a) * n + o, rounded(mad(r.B[a], r.B[g], -row(r.Mi, a, u)) * (r.f1 * r.f1)));
        }
        return std::is_same<T, double>::value || sum == 0.0f;
    }
    __device__ static void finish(const P &p, I &s, const Rec &, int32_t o, int64_t) {
        if (finish_in<Two>(p, s, o) || finish_in<double>(p, s, o)) return;
        const int64_t n = p.n;
        const float nan = __int_as_float(0x7fc00000);
        p.A[o] = nan;
        for (int a = 0; a < 3; ++a) { p.B[a * n + o] = nan; p.gA[a * n + o] = nan; }
        for (int a = 0; a < 9; ++a) p.gB[a * n + o] = nan;
        if (p.n_singular) atomicAdd(p.n_singular, 1);
    }
    __device__ static void finish_other(const P &p, int32_t o) {
        const int64_t n = p.n;
        p.A[o] = 0.f;
        for (int a = 0; a < 3; ++a) { p.B[a * n + o] = 0.f; p.gA[a * n + o] = 0.f; }
        for (int a = 0; a < 9; ++a) p.gB[a * n + o] = 0.f;
    }
};

// Reverse mode of Corrections (not in the paper).  Pair (i, j) enters i's
// moments as V_j t(x_ij); with i's moment cotangents (from those of A, B, dA,
// dB by the closed-form reverse of the per-particle step) the weighted terms
// are T_i(x) = S0_i(x) W + S1_i(x) dWr, S0 a quadratic and S1 a cubic
// polynomial in x.  The preparation sweep recomputes the moments and writes
// each particle's 29 polynomial coefficients
//   [c0, l0 (3), q0 (6: xx xy xz yy yz zz), l1 (3), q1 (6), k (10: xxx xxy xxz
//    xyy xyz xzz yyy yyz yzz zzz)],
// S0 = c0 + l0.x + q0(x), S1 = l1.x + q1(x) + k(x); the gradient sweep gathers
//   xbar_i = sum_j V_j grad T_i(x_ij) - V_i grad T_j(x_ji),
//   Vbar_i = sum_j T_j(x_ji)          (j = i included).
constexpr int kCorrCoef = 29;

struct CorrAdjP : CorrP {
    const float *Abar, *Bbar, *gAbar, *gBbar;  // cotangents: A [n], B [3][n], dA [3][n], dB [9][n] (3g+a)
    float *coef;                               // out: [29][n] (kernel order when korder, else caller)
};

struct CorrAdjPrepStage : CorrStage {
    static constexpr bool kAllVariants = false;
    using P = CorrAdjP;
    // Reverse of CorrStage's Solved, in the sums m0, m1, m2, dm0, s2, s3 themselves, whose cotangents
    // are the polynomial coefficients.  H_ga: the cotangent of dB_g^a (row g).  The sweep is CorrStage's, with
    // the very sums of the forward pass: through the chain the gradients in the positions are 4% nearer to 64
    // bits than through the 30 unreduced sums dm1, dm2 (by themselves, for cotangents of dA, 1-2% farther off).
    // This finish (2,500 FP32 instructions in float pairs) is half of the kernel's time: 422 -> 295 us on
    // the 2x64^3 box against the unreduced sums, then 254 us in float pairs.
    // The reverse is linear in the cotangents, and a float pair holds its 47 bits only while its low word is a
    // normal number: it works on them (in scaled lengths) in units u of a power of two near the largest, c = 1/u.
    // False where the unit or the lengths are so far from 1 that products of the scales leave the FP32 range.
    __device__ static bool unit_of(const float *, double, double &c, double &u) {
        c = u = 1.0;
        return true;
    }
    __device__ static bool unit_of(const float cot[16], float f1, float &c, float &u) {
        float m[3] = {fabsf(cot[0]), 0.0f, 0.0f};
#pragma unroll
        for (int k = 1; k < 7; ++k) m[1] = fmaxf(m[1], fabsf(cot[k]));
#pragma unroll
        for (int k = 7; k < 16; ++k) m[2] = fmaxf(m[2], fabsf(cot[k]));
        c = u = 1.0f;
        if (fmaxf(m[0], fmaxf(m[1], m[2])) == 0.0f) return true;
        const float most = fmaxf(m[0], fmaxf(m[1], m[2] * f1) * f1);
        if (!(most > 0x1p-60f && most < 0x1p60f && f1 > 0x1p-30f && f1 < 0x1p30f)) return false;
        const int e = __float_as_int(most) >> 23;  // exponent + 127
        c = __int_as_float((254 - e) << 23);
        u = __int_as_float(e << 23);
        return true;
    }
    template <class T>
    __device__ static bool finish_in(const P &p, const I &s, int32_t o) {
        using F = typename beside<T>::type;
        const int64_t n = p.n;
        Solved<T> r;
        if (!solve(s, r)) return false;
        const F f1 = r.f1;
        float cot[16];  // A, B, dA, dB (3g+a)
        cot[0] = p.Abar[o];
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            cot[1 + k] = p.Bbar[k * n + o];
            cot[4 + k] = p.gAbar[k * n + o];
        }
#pragma unroll
        for (int k = 0; k < 9; ++k) cot[7 + k] = p.gBbar[k * n + o];
        F c0, u0;
        if (!unit_of(cot, f1, c0, u0)) return false;
        const F c1 = c0 * f1, c2 = c1 * f1, u1 = u0 * f1, u2 = u1 * f1, v1 = u0 * r.g1;
        float sum = 0.0f;  // NaN once a result is not finite
        auto put = [&](int k, float v) {
            p.coef[k * n + o] = v;
            sum = fmaf(v, 0.0f, sum);
        };
        T H[3][3], Kb[3], Bb[3], Ab, qb;
        difference(cot[0] * c0, (F)0, Ab);
#pragma unroll
        for (int g = 0; g < 3; ++g) {
            T gAb;
#pragma unroll
            for (int a = 0; a < 3; ++a) difference(cot[7 + 3 * g + a] * c2, (F)0, H[g][a]);
            difference(cot[4 + g] * c1, (F)0, gAb);
            difference(cot[1 + g] * c1, (F)0, Bb[g]);
            const T Ag = -(r.A * gAb);
            Kb[g] = r.A * Ag;
            Ab = mad(twice(Ag), r.K[g], Ab);
            put(10 + g, rounded(Kb[g] * v1));  // l1: dm0
        }
        // dB_g^a = B_a B_g - (Mi Uq)_ag and K_g = dm0_g + 2 q B_g + ((2 s2 + T) B)_g
        T Mib[3][3], Uqb[3][3];
#pragma unroll
        for (int a = 0; a < 3; ++a)
#pragma unroll
            for (int b = 0; b < 3; ++b) {
                Mib[a][b] = -dot3(H[0][a], at(r.Uq, b, 0), H[1][a], at(r.Uq, b, 1), H[2][a], at(r.Uq, b, 2));
                Uqb[a][b] = -row(r.Mi, a, H[b]);
            }
        qb = Uqb[0][0] + Uqb[1][1] + Uqb[2][2] + twice(dot3(Kb[0], r.B[0], Kb[1], r.B[1], Kb[2], r.B[2]));
#pragma unroll
        for (int a = 0; a < 3; ++a) {
#pragma unroll
            for (int g = 0; g < 3; ++g) {
                Bb[a] = mad(H[g][a] + H[a][g], r.B[g], Bb[a]);
                // 2 s2 + T = s2 + U
                Bb[a] = mad(Kb[g], at(r.U, a, g) + (F)s.s2[a <= g ? idx2(a, g) : idx2(g, a)], Bb[a]);
            }
            Bb[a] = mad(twice(r.q), Kb[a], Bb[a]);
        }
        // s2 and T cotangents, one entry per monomial x_a x_b (both orders of an off-diagonal pair)
        T Tb[6];
        const int ia[6] = {0, 0, 0, 1, 1, 2}, ib[6] = {0, 1, 2, 1, 2, 2};
#pragma unroll
        for (int k = 0; k < 6; ++k) {
            const int a = ia[k], b = ib[k];
            const T w = a == b ? Kb[a] * r.B[a] : mad(Kb[a], r.B[b], Kb[b] * r.B[a]);
            Tb[k] = (a == b ? Uqb[a][a] : Uqb[a][b] + Uqb[b][a]) + w;
            put(13 + k, rounded((Tb[k] + w) * u0));  // q1: s2
        }
        // T = s3 B: Bb_c += sum_ab Tb_ab s3_abc, and s3's coefficients are those of (x^T Tb x)(B.x)
#pragma unroll
        for (int c = 0; c < 3; ++c)
#pragma unroll
            for (int k = 0; k < 6; ++k) Bb[c] = mad(Tb[k], r.s3[sorted3(ia[k], ib[k], c)], Bb[c]);
        const T *B = r.B;
        put(19, rounded(Tb[0] * B[0] * u1));
        put(20, rounded(mad(Tb[0], B[1], Tb[1] * B[0]) * u1));
        put(21, rounded(mad(Tb[0], B[2], Tb[2] * B[0]) * u1));
        put(22, rounded(mad(Tb[1], B[1], Tb[3] * B[0]) * u1));
        put(23, rounded(dot3(Tb[1], B[2], Tb[2], B[1], Tb[4], B[0]) * u1));
        put(24, rounded(mad(Tb[2], B[2], Tb[5] * B[0]) * u1));
        put(25, rounded(Tb[3] * B[1] * u1));
        put(26, rounded(mad(Tb[3], B[2], Tb[4] * B[1]) * u1));
        put(27, rounded(mad(Tb[4], B[2], Tb[5] * B[1]) * u1));
        put(28, rounded(Tb[5] * B[2] * u1));
        // A = 1/q, q = m0 + B.m1, B = -Mi m1, Mi = m2^-1
        qb = mad(-(r.A * Ab), r.A, qb);
        put(0, rounded(qb * u0));  // c0: m0
#pragma unroll
        for (int a = 0; a < 3; ++a) Bb[a] = mad(qb, r.m1[a], Bb[a]);
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            put(1 + a, rounded(mad(qb, r.B[a], -row(r.Mi, a, Bb)) * u1));  // l0: m1
#pragma unroll
            for (int b = 0; b < 3; ++b) Mib[a][b] = mad(-Bb[a], r.m1[b], Mib[a][b]);
        }
        // m2's cotangent -Mi Mib Mi, per monomial: -Mi (Mib + Mib^T) Mi off the diagonal, half of it on it
        T S[6], Y[3][3];
#pragma unroll
        for (int k = 0; k < 6; ++k) S[k] = ia[k] == ib[k] ? twice(Mib[ia[k]][ia[k]]) : Mib[ia[k]][ib[k]] + Mib[ib[k]][ia[k]];
#pragma unroll
        for (int a = 0; a < 3; ++a)
#pragma unroll
            for (int b = 0; b < 3; ++b) {
                const T c[3] = {at(r.Mi, 0, b), at(r.Mi, 1, b), at(r.Mi, 2, b)};
                Y[a][b] = row(S, a, c);
            }
#pragma unroll
        for (int k = 0; k < 6; ++k) {
            const T c[3] = {Y[0][ib[k]], Y[1][ib[k]], Y[2][ib[k]]};
            put(4 + k, rounded(row(r.Mi, ia[k], c) * ((ia[k] == ib[k] ? (F)-0.5 : (F)-1.0) * u2)));  // q0: m2
        }
        return std::is_same<T, double>::value || sum == 0.0f;
    }
    __device__ static void finish(const P &p, I &s, const Rec &, int32_t o, int64_t) {
        if (finish_in<Two>(p, s, o) || finish_in<double>(p, s, o)) return;
        for (int k = 0; k < kCorrCoef; ++k) p.coef[k * p.n + o] = 0.f;  // singular: contributes nothing
        if (p.n_singular) atomicAdd(p.n_singular, 1);
    }
    __device__ static void finish_other(const P &p, int32_t o) {
        for (int k = 0; k < kCorrCoef; ++k) p.coef[k * p.n + o] = 0.f;
    }
};

struct CorrAdjSweepP {
    const float *V, *coef;
    float *xbar3, *Vbar;
    int64_t n;
    unsigned long long *count;
    unsigned long long *swept;
};

// value and gradient of T(x) = S0 W + S1 dWr for coefficients c (layout above)
__device__ __forceinline__ float corr_term(const float *c, const float x[3], float W, float dWr, float ddWr,
                                           float g[3]) {
    const float X = x[0], Y = x[1], Z = x[2];
    const float q0 = fmaf(c[4] * X, X, fmaf(c[5] * X, Y, fmaf(c[6] * X, Z, fmaf(c[7] * Y, Y, fmaf(c[8] * Y, Z, c[9] * Z * Z)))));
    const float S0 = c[0] + fmaf(c[1], X, fmaf(c[2], Y, c[3] * Z)) + q0;
    const float g0x = c[1] + fmaf(2.0f * c[4], X, fmaf(c[5], Y, c[6] * Z));
    const float g0y = c[2] + fmaf(c[5], X, fmaf(2.0f * c[7], Y, c[8] * Z));
    const float g0z = c[3] + fmaf(c[6], X, fmaf(c[8], Y, 2.0f * c[9] * Z));
    const float *k = c + 19;
    const float XX = X * X, XY = X * Y, XZ = X * Z, YY = Y * Y, YZ = Y * Z, ZZ = Z * Z;
    const float q1 = fmaf(c[13], XX, fmaf(c[14], XY, fmaf(c[15], XZ, fmaf(c[16], YY, fmaf(c[17], YZ, c[18] * ZZ)))));
    const float cub = fmaf(k[0] * XX, X, fmaf(k[1] * XX, Y, fmaf(k[2] * XX, Z, fmaf(k[3] * YY, X, fmaf(k[4] * XY, Z,
                      fmaf(k[5] * ZZ, X, fmaf(k[6] * YY, Y, fmaf(k[7] * YY, Z, fmaf(k[8] * ZZ, Y, k[9] * ZZ * Z)))))))));
    const float S1 = fmaf(c[10], X, fmaf(c[11], Y, c[12] * Z)) + q1 + cub;
    const float g1x = c[10] + fmaf(2.0f * c[13], X, fmaf(c[14], Y, c[15] * Z)) +
                      fmaf(3.0f * k[0], XX, fmaf(2.0f * k[1], XY, fmaf(2.0f * k[2], XZ, fmaf(k[3], YY, fmaf(k[4], YZ, k[5] * ZZ)))));
    const float g1y = c[11] + fmaf(c[14], X, fmaf(2.0f * c[16], Y, c[17] * Z)) +
                      fmaf(k[1], XX, fmaf(2.0f * k[3], XY, fmaf(k[4], XZ, fmaf(3.0f * k[6], YY, fmaf(2.0f * k[7], YZ, k[8] * ZZ)))));
    const float g1z = c[12] + fmaf(c[15], X, fmaf(c[17], Y, 2.0f * c[18] * Z)) +
                      fmaf(k[2], XX, fmaf(k[4], XY, fmaf(2.0f * k[5], XZ, fmaf(k[7], YY, fmaf(2.0f * k[8], YZ, 3.0f * k[9] * ZZ)))));
    const float a = fmaf(S0, dWr, S1 * ddWr);
    g[0] = fmaf(g0x, W, fmaf(g1x, dWr, a * X));
    g[1] = fmaf(g0y, W, fmaf(g1y, dWr, a * Y));
    g[2] = fmaf(g0z, W, fmaf(g1z, dWr, a * Z));
    return fmaf(S0, W, S1 * dWr);
}

struct CorrAdjStage {
    static constexpr bool kPair = false;
    static constexpr bool kGasOnly = true;
    static constexpr bool kCons = false;
    static constexpr bool kAllVariants = false;
    using P = CorrAdjSweepP;
    struct __align__(16) Rec {
        float x, y, z, h;
        float V, c[kCorrCoef], pad[2];
        static constexpr bool kWhole = true;
    };
    struct I {
        float gx, gy, gz, Vb;
        int cnt;
    };
    __device__ static Rec gather(const P &p, int32_t o, float4 ps) {
        Rec r;
        r.x = ps.x; r.y = ps.y; r.z = ps.z; r.h = ps.w;
        r.V = p.V[o];
#pragma unroll
        for (int k = 0; k < kCorrCoef; ++k) r.c[k] = p.coef[k * p.n + o];
        r.pad[0] = r.pad[1] = 0.f;
        return r;
    }
    __device__ static float box_cut(const P &, float hmax_i, const Rec &rj) { return hmax_i + rj.h; }
    __device__ static float leaf_cut(const P &, float hmax_i, float hmax_j) { return hmax_i + hmax_j; }
    __device__ static void shift(Rec &r, float sx, float sy, float sz) { r.x += sx; r.y += sy; r.z += sz; }
    __device__ static void init(const P &, I &s, const Rec &, int64_t, int, int, int32_t) {
        s.gx = s.gy = s.gz = s.Vb = 0.f;
        s.cnt = 0;
    }
    template <bool kCount>
    __device__ static void interact(const P &, I &s, const Rec &ri, const Rec &rj) {
        float x[3] = {ri.x - rj.x, ri.y - rj.y, ri.z - rj.z};  // x_ij
        float r2 = fmaf(x[0], x[0], fmaf(x[1], x[1], x[2] * x[2]));
        float hs = ri.h + rj.h;
        bool in = r2 < hs * hs;
        float W, dWr, ddWr;
        wendland2(r2, 0.5f * hs, W, dWr, ddWr);
        W = in ? W : 0.0f;
        dWr = in ? dWr : 0.0f;
        ddWr = in ? ddWr : 0.0f;
        float gi[3], gj[3];
        const float xm[3] = {-x[0], -x[1], -x[2]};
        corr_term(ri.c, x, W, dWr, ddWr, gi);
        const float Tj = corr_term(rj.c, xm, W, dWr, ddWr, gj);
        s.gx += rj.V * gi[0] - ri.V * gj[0];
        s.gy += rj.V * gi[1] - ri.V * gj[1];
        s.gz += rj.V * gi[2] - ri.V * gj[2];
        s.Vb += Tj;
        if (kCount) s.cnt += in;
    }
    __device__ static void finish(const P &p, I &s, const Rec &, int32_t o, int64_t) {
        p.xbar3[o] = s.gx;
        p.xbar3[p.n + o] = s.gy;
        p.xbar3[2 * p.n + o] = s.gz;
        p.Vbar[o] = s.Vb;
    }
    __device__ static void finish_other(const P &p, int32_t o) {
        p.xbar3[o] = 0.f;
        p.xbar3[p.n + o] = 0.f;
        p.xbar3[2 * p.n + o] = 0.f;
        p.Vbar[o] = 0.f;
    }
};

struct HydroP {
    const float *m, *v3, *u, *V, *rho, *A, *B, *gA, *gB;
    float *dv3, *du;
    double *cons;
    float gamma, alpha, beta, eta2;
    int64_t n;
    unsigned long long *count;
    const float *dvg;  // limited viscosity: velocity gradient [9][n], dv^a/dx^b at 3a+b
    unsigned long long *swept;  // counting runs: candidate pair evaluations, may be NULL
    const float *vstar;         // Energy pass: time-centred velocities [3][n]
    unsigned int *vsig_h;       // Acceleration pass: atomic max of vsig_i / h_i (FP32 bits), may be NULL
    float sig_beta;             // Acceleration pass: vsig_ij = c_i + c_j - sig_beta min(0, v_ij.x_ij / r)
};

struct HydroRec {
    float x, y, z, h;
    float vx, vy, vz, P;
    float c, rho, V, A;
    float B[3], gA0;
    float gA1, gA2, gB0, gB1;
    float gB[7];  // gB[2..8]
    float pad;    // limited viscosity: G[0]; hydro adjoint: the particle's identity
};
struct HydroRecLim : HydroRec {
    float G8[8];  // velocity gradient, dv^a/dx^b at 3a+b, entries 1..8 (entry 0 in pad)
};
template <class Base>
struct HydroRecVstar : Base {
    float wx, wy, wz, u;  // time-centred velocity v* and specific internal energy
};

// kLim: the viscosity sees both velocities reconstructed linearly to the pair
// midpoint, s = (dv) x, with the van Leer limiter
// phi = 4 r/(1+r)^2, r = (x.s_i)/(x.s_j), written 4 a_i a_j/(a_i + a_j)^2 for
// a_i a_j > 0 (else 0): the same value without a division by a_j alone.
//
// kPass (Sec. 5: Acceleration and Energy; Sec. 5.4: each runs twice a step):
//   kHydroBoth    dv/dt and du/dt with the equal split of the pair work on v;
//   kHydroAccel   dv/dt only, plus the signal velocity
//                 vsig_i = max_j (c_i + c_j - sig_beta min(0, v_ij.x_ij / r))
//                 (j = i gives 2 c_i), folded into one FP32 atomic max of
//                 vsig_i / h_i (Sec. 5.1: floating-point atomic max);
//   kHydroEnergy  du/dt with the compatible split: the pair heat
//                 dE_ij = -f_ij.(v*_i - v*_j) goes to i with the share
//                 w_ij = 1/2 (1 + sgn(dE) (u_j - u_i) / (|u_j - u_i| + (u_i + u_j)/2))
//                 (1/2 when u_i = u_j), so that sum_i m_i du_i = -sum_i f_i.v*_i.
constexpr int kHydroBoth = 0, kHydroAccel = 1, kHydroEnergy = 2;

template <bool kLim, int kPass = kHydroBoth, bool kWholeRec = kPass != kHydroEnergy>
struct HydroStageT {
    static constexpr bool kPair = false;
    static constexpr bool kGasOnly = true;
    static constexpr bool kCons = true;
    static constexpr bool kAllVariants = kPass == kHydroBoth;  // the step passes: lists and tiles only
    using P = HydroP;
    using Base = std::conditional_t<kLim, HydroRecLim, HydroRec>;
    struct __align__(16) Rec : std::conditional_t<kPass == kHydroEnergy, HydroRecVstar<Base>, Base> {
        static constexpr bool kWhole = kWholeRec;
    };
    struct I {
        float fx, fy, fz, e;
        int cnt;
    };
    __device__ static Rec gather(const P &p, int32_t o, float4 ps) {
        const int64_t n = p.n;
        Rec r;
        r.x = ps.x; r.y = ps.y; r.z = ps.z; r.h = ps.w;
        r.vx = p.v3[o]; r.vy = p.v3[n + o]; r.vz = p.v3[2 * n + o];
        float rho = p.rho[o], u = p.u[o];
        r.P = (p.gamma - 1.0f) * rho * u;
        r.c = sqrtf(p.gamma * (p.gamma - 1.0f) * u);
        r.rho = rho;
        r.V = p.V[o];
        r.A = p.A[o];
        r.B[0] = p.B[o]; r.B[1] = p.B[n + o]; r.B[2] = p.B[2 * n + o];
        r.gA0 = p.gA[o]; r.gA1 = p.gA[n + o]; r.gA2 = p.gA[2 * n + o];
        r.gB0 = p.gB[o]; r.gB1 = p.gB[n + o];
        for (int k = 0; k < 7; ++k) r.gB[k] = p.gB[(2 + k) * n + o];
        r.pad = 0.f;
        if constexpr (kLim) {
            r.pad = p.dvg[o];
            for (int k = 1; k < 9; ++k) r.G8[k - 1] = p.dvg[k * n + o];
        }
        if constexpr (kPass == kHydroEnergy) {
            r.wx = p.vstar[o]; r.wy = p.vstar[n + o]; r.wz = p.vstar[2 * n + o];
            r.u = u;
        }
        return r;
    }
    __device__ static float box_cut(const P &, float hmax_i, const Rec &rj) { return hmax_i + rj.h; }
    __device__ static float leaf_cut(const P &, float hmax_i, float hmax_j) { return hmax_i + hmax_j; }
    __device__ static void shift(Rec &r, float sx, float sy, float sz) { r.x += sx; r.y += sy; r.z += sz; }
    __device__ static void init(const P &, I &s, const Rec &, int64_t, int, int, int32_t) { s.fx = s.fy = s.fz = s.e = 0.f; s.cnt = 0; }
    // grad W^R of record r at separation x (x = x_r - x_other): gA (1 + B.x) W + A (gB.x + B) W + A (1 + B.x) dWr x
    template <class R>
    __device__ static void grad_wr(const R &r, const float x[3], float W, float dWr, float g[3]) {
        float Bx = fmaf(r.B[0], x[0], fmaf(r.B[1], x[1], r.B[2] * x[2]));
        float gb[9] = {r.gB0, r.gB1, r.gB[0], r.gB[1], r.gB[2], r.gB[3], r.gB[4], r.gB[5], r.gB[6]};
        float gA[3] = {r.gA0, r.gA1, r.gA2};
        float k1 = (1.0f + Bx) * W;
        float k3 = r.A * (1.0f + Bx) * dWr;
        float AW = r.A * W;
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            float gBx = fmaf(gb[3 * q], x[0], fmaf(gb[3 * q + 1], x[1], gb[3 * q + 2] * x[2]));
            g[q] = fmaf(gA[q], k1, fmaf(AW, gBx + r.B[q], k3 * x[q]));
        }
    }
    template <bool kCount>
    __device__ static void interact(const P &p, I &s, const Rec &ri, const Rec &rj) {
        float x[3] = {ri.x - rj.x, ri.y - rj.y, ri.z - rj.z};  // x_ij
        float r2 = fmaf(x[0], x[0], fmaf(x[1], x[1], x[2] * x[2]));
        float hs = ri.h + rj.h;
        bool in = r2 < hs * hs;
        float hij = 0.5f * hs;
        float W, dWr;
        wendland(r2, hij, W, dWr);
        float gi[3], gj[3];
        grad_wr(ri, x, W, dWr, gi);
        float xm[3] = {-x[0], -x[1], -x[2]};
        grad_wr(rj, xm, W, dWr, gj);
        float vij[3] = {ri.vx - rj.vx, ri.vy - rj.vy, ri.vz - rj.vz};
        float vx;
        if constexpr (kLim) {
            const float Gi[9] = {ri.pad, ri.G8[0], ri.G8[1], ri.G8[2], ri.G8[3], ri.G8[4], ri.G8[5], ri.G8[6], ri.G8[7]};
            const float Gj[9] = {rj.pad, rj.G8[0], rj.G8[1], rj.G8[2], rj.G8[3], rj.G8[4], rj.G8[5], rj.G8[6], rj.G8[7]};
            float si[3], sj[3];
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                si[a] = fmaf(Gi[3 * a], x[0], fmaf(Gi[3 * a + 1], x[1], Gi[3 * a + 2] * x[2]));
                sj[a] = fmaf(Gj[3 * a], x[0], fmaf(Gj[3 * a + 1], x[1], Gj[3 * a + 2] * x[2]));
            }
            const float ai = fmaf(x[0], si[0], fmaf(x[1], si[1], x[2] * si[2]));
            const float aj = fmaf(x[0], sj[0], fmaf(x[1], sj[1], x[2] * sj[2]));
            const float aa = ai * aj, as = ai + aj;
            const float phi = aa > 0.0f ? __fdividef(4.0f * aa, as * as) : 0.0f;
            const float hp = 0.5f * phi;
            float vs[3];
#pragma unroll
            for (int a = 0; a < 3; ++a) vs[a] = fmaf(-hp, si[a] + sj[a], vij[a]);
            vx = fmaf(vs[0], x[0], fmaf(vs[1], x[1], vs[2] * x[2]));
        } else {
            vx = fmaf(vij[0], x[0], fmaf(vij[1], x[1], vij[2] * x[2]));
        }
        float mu = vx < 0.0f ? div_normal(hij * vx, fmaf(p.eta2 * hij, hij, r2)) : 0.0f;
        float Q = 0.5f * (ri.rho + rj.rho) * mu * fmaf(-p.alpha * 0.5f, ri.c + rj.c, p.beta * mu);
        float pre = in ? -0.5f * ri.V * rj.V * (ri.P + rj.P + Q) : 0.0f;
        float f[3] = {pre * (gi[0] - gj[0]), pre * (gi[1] - gj[1]), pre * (gi[2] - gj[2])};
        s.fx += f[0];
        s.fy += f[1];
        s.fz += f[2];
        if constexpr (kPass == kHydroBoth) {
            s.e = fmaf(-0.5f, fmaf(vij[0], f[0], fmaf(vij[1], f[1], vij[2] * f[2])), s.e);
        } else if constexpr (kPass == kHydroAccel) {
            // approach speed on the true velocities (the limiter shapes only the viscosity)
            const float w = fmaf(vij[0], x[0], fmaf(vij[1], x[1], vij[2] * x[2])) * (r2 > 0.0f ? rsqrtf(r2) : 0.0f);
            const float vs = fmaf(-p.sig_beta, fminf(w, 0.0f), ri.c + rj.c);
            s.e = in ? fmaxf(s.e, vs) : s.e;
        } else {
            const float dE = -fmaf(ri.wx - rj.wx, f[0], fmaf(ri.wy - rj.wy, f[1], (ri.wz - rj.wz) * f[2]));
            const float du = rj.u - ri.u;
            // (u_j - u_i) / (|u_j - u_i| + (u_i + u_j)/2): the same magnitude for i and j, opposite sign
            const float t = du != 0.0f ? __fdividef(du, fabsf(du) + 0.5f * (ri.u + rj.u)) : 0.0f;
            const float w = 0.5f + 0.5f * (dE > 0.0f ? t : -t);
            s.e = fmaf(w, dE, s.e);
        }
        if (kCount) s.cnt += in;
    }
    __device__ static void finish(const P &p, I &s, const Rec &ri, int32_t o, int64_t) {
        float mi = p.m[o];
        if constexpr (kPass != kHydroEnergy) {
            p.dv3[o] = s.fx / mi;
            p.dv3[p.n + o] = s.fy / mi;
            p.dv3[2 * p.n + o] = s.fz / mi;
        }
        if constexpr (kPass != kHydroAccel) p.du[o] = s.e / mi;
        if constexpr (kPass == kHydroAccel) {
            if (p.vsig_h) {
                // vsig / h >= 0: its FP32 bit pattern orders like the value; one atomic per
                // converged set of lanes
                const unsigned q = __float_as_uint(__fdividef(s.e, ri.h));
                const unsigned mask = __activemask();
                const unsigned qm = __reduce_max_sync(mask, q);
                if ((int)(threadIdx.x & 31) == __ffs(mask) - 1) atomicMax(p.vsig_h, qm);
            }
        }
    }
    // FP64 conservation terms of one gas particle: m dv (3) and m (v.dv + du), with
    // v = v* in the Energy pass (the compatible balance) and du = 0 in the Acceleration pass
    __device__ static void cons_terms(const P &p, const I &s, const Rec &ri, int32_t o, double c[4]) {
        double mi = (double)p.m[o];
        double dvx = (double)(s.fx / p.m[o]), dvy = (double)(s.fy / p.m[o]), dvz = (double)(s.fz / p.m[o]);
        double du = kPass == kHydroAccel ? 0.0 : (double)(s.e / p.m[o]);
        double wx = ri.vx, wy = ri.vy, wz = ri.vz;
        if constexpr (kPass == kHydroEnergy) { wx = ri.wx; wy = ri.wy; wz = ri.wz; }
        c[0] = mi * dvx;
        c[1] = mi * dvy;
        c[2] = mi * dvz;
        c[3] = mi * (wx * dvx + wy * dvy + wz * dvz + du);
    }
    __device__ static void finish_other(const P &p, int32_t o) {
        if constexpr (kPass != kHydroEnergy) {
            p.dv3[o] = 0.f;
            p.dv3[p.n + o] = 0.f;
            p.dv3[2 * p.n + o] = 0.f;
        }
        if constexpr (kPass != kHydroAccel) p.du[o] = 0.f;
    }

    // Half-warp arms (Sec. 5.3): partial sums of one i from one leaf-pair tile are added
    // to the zeroed outputs with atomics (the Energy pass also adds its recomputed force
    // to p.dv3 when given, for the conservation sums); the signal-velocity maximum goes
    // straight to the one atomic max of vsig_i / h_i (a max of partial maxima).
    static constexpr bool kHalfWarp = true;
    __device__ static void flush(const P &p, const I &s, const Rec &ri, int32_t o) {
        const float mi = p.m[o];
        if (p.dv3) {
            atomicAdd(&p.dv3[o], s.fx / mi);
            atomicAdd(&p.dv3[p.n + o], s.fy / mi);
            atomicAdd(&p.dv3[2 * p.n + o], s.fz / mi);
        }
        if constexpr (kPass != kHydroAccel) atomicAdd(&p.du[o], s.e / mi);
        if constexpr (kPass == kHydroAccel) {
            if (p.vsig_h) atomicMax(p.vsig_h, __float_as_uint(__fdividef(s.e, ri.h)));
        }
    }
    // outside every cut (r^2 ~ 1e30 against (h_i + h_j)^2) with zero fields: exact zeros
    __device__ static Rec far_dummy(float fx, float fy, float fz) {
        Rec r{};
        r.x = fx; r.y = fy; r.z = fz; r.h = 1.0f;
        return r;
    }
    static void zero_outputs(const P &p, cudaStream_t st) {
        if (p.dv3) cudaMemsetAsync(p.dv3, 0, sizeof(float) * 3 * p.n, st);
        if (kPass != kHydroAccel && p.du) cudaMemsetAsync(p.du, 0, sizeof(float) * p.n, st);
    }
    // the conservation terms of cons_terms from the finished outputs of gas particle o
    __device__ static void cons_of(const P &p, int32_t o, double c[4]) {
        const int64_t n = p.n;
        const double mi = (double)p.m[o];
        const double dvx = p.dv3[o], dvy = p.dv3[n + o], dvz = p.dv3[2 * n + o];
        const double du = kPass == kHydroAccel ? 0.0 : (double)p.du[o];
        const float *w = kPass == kHydroEnergy ? p.vstar : p.v3;
        c[0] = mi * dvx;
        c[1] = mi * dvy;
        c[2] = mi * dvz;
        c[3] = mi * ((double)w[o] * dvx + (double)w[n + o] * dvy + (double)w[2 * n + o] * dvz + du);
    }
};


using HydroStage = HydroStageT<false>;
using HydroLimStage = HydroStageT<true>;
// Reverse mode of the hydro pair force (Monaghan viscosity, equal split; not
// in the paper) for cotangents dvbar, dubar, with every input independent.
// With a_i = dvbar_i/m_i, b_i = dubar_i/m_i the loss is a sum over unordered
// pairs i != j of l_ij = z.f_ij, z = (a_i - a_j) - (b_i + b_j) v_ij / 2
// (f_ji = -f_ij, e_ji = e_ij; the self pair has f_ii = 0 for all of i's
// inputs), so each i gathers dl_ij/d(i's inputs) over its neighbours: one-sided,
// nothing per pair stored, no atomics.  m enters through a and b only:
// mbar_i = -(a_i.F_i + b_i E_i)/m_i with the recomputed sums F, E.
struct HydroAdjP {
    const float *m, *v3, *u, *V, *rho, *A, *B, *gA, *gB, *dvbar3, *dubar;
    float *xbar3, *vbar3, *ubar, *mbar, *Vbar, *rhobar, *Abar, *Bbar3, *gAbar3, *gBbar9;
    float gamma, alpha, beta, eta2;
    int64_t n;
    unsigned long long *count;
    unsigned long long *swept;
};

// sum_q c_q dG_q/dy_p for the corrected-kernel gradient G(y) of a record (see grad_wr), and the
// cotangents of its A, B, dA, dB when kParams
template <bool kParams, class R>
__device__ __forceinline__ void grad_wr_vjp(const R &r, const float y[3], float W, float dWr, float ddWr,
                                            const float c[3], float out[3], float *Ab, float *Bb, float *gAb,
                                            float *gBb) {
    const float gb[9] = {r.gB0, r.gB1, r.gB[0], r.gB[1], r.gB[2], r.gB[3], r.gB[4], r.gB[5], r.gB[6]};
    const float gA[3] = {r.gA0, r.gA1, r.gA2};
    const float By = fmaf(r.B[0], y[0], fmaf(r.B[1], y[1], r.B[2] * y[2]));
    const float cy = fmaf(c[0], y[0], fmaf(c[1], y[1], c[2] * y[2]));
    const float cgA = fmaf(c[0], gA[0], fmaf(c[1], gA[1], c[2] * gA[2]));
    const float cB = fmaf(c[0], r.B[0], fmaf(c[1], r.B[1], c[2] * r.B[2]));
    float cgBy = 0.0f;
#pragma unroll
    for (int q = 0; q < 3; ++q) cgBy = fmaf(c[q], fmaf(gb[3 * q], y[0], fmaf(gb[3 * q + 1], y[1], gb[3 * q + 2] * y[2])), cgBy);
    const float opB = 1.0f + By;
    const float kB = fmaf(W, cgA, r.A * dWr * cy);
    const float ky = fmaf(cgA * opB, dWr, r.A * fmaf(dWr, cgBy + cB, opB * ddWr * cy));
    const float AW = r.A * W, kc = r.A * opB * dWr;
#pragma unroll
    for (int pp = 0; pp < 3; ++pp) {
        const float gBtc = fmaf(c[0], gb[pp], fmaf(c[1], gb[3 + pp], c[2] * gb[6 + pp]));
        out[pp] = fmaf(r.B[pp], kB, fmaf(y[pp], ky, fmaf(AW, gBtc, kc * c[pp])));
    }
    if constexpr (kParams) {
        *Ab += fmaf(W, cgBy + cB, opB * dWr * cy);
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            gAb[q] = fmaf(c[q] * opB, W, gAb[q]);
            Bb[q] = fmaf(y[q], kB, fmaf(AW, c[q], Bb[q]));
#pragma unroll
            for (int a = 0; a < 3; ++a) gBb[3 * q + a] = fmaf(c[q] * AW, y[a], gBb[3 * q + a]);
        }
    }
}

template <bool kWholeRec>
struct HydroAdjStage {
    static constexpr bool kPair = false;
    static constexpr bool kGasOnly = true;
    static constexpr bool kCons = false;
    static constexpr bool kAllVariants = false;
    using P = HydroAdjP;
    struct __align__(16) Rec : HydroRec {
        float ax, ay, az, b;  // dvbar/m, dubar/m
        static constexpr bool kWhole = kWholeRec;
    };
    struct I {
        float xb[3], vb[3], Vb, Pb, cb, rb, Ab, Bb[3], gAb[3], gBb[9], F[3], E;
        int cnt;
    };
    __device__ static Rec gather(const P &p, int32_t o, float4 ps) {
        const int64_t n = p.n;
        Rec r;
        r.x = ps.x; r.y = ps.y; r.z = ps.z; r.h = ps.w;
        r.vx = p.v3[o]; r.vy = p.v3[n + o]; r.vz = p.v3[2 * n + o];
        const float rho = p.rho[o], u = p.u[o];
        r.P = (p.gamma - 1.0f) * rho * u;
        r.c = sqrtf(p.gamma * (p.gamma - 1.0f) * u);
        r.rho = rho;
        r.V = p.V[o];
        r.A = p.A[o];
        r.B[0] = p.B[o]; r.B[1] = p.B[n + o]; r.B[2] = p.B[2 * n + o];
        r.gA0 = p.gA[o]; r.gA1 = p.gA[n + o]; r.gA2 = p.gA[2 * n + o];
        r.gB0 = p.gB[o]; r.gB1 = p.gB[n + o];
        for (int k = 0; k < 7; ++k) r.gB[k] = p.gB[(2 + k) * n + o];
        r.pad = __int_as_float(o);  // particle identity: the self pair is skipped
        const float im = __fdividef(1.0f, p.m[o]);
        r.ax = p.dvbar3[o] * im; r.ay = p.dvbar3[n + o] * im; r.az = p.dvbar3[2 * n + o] * im;
        r.b = p.dubar[o] * im;
        return r;
    }
    __device__ static float box_cut(const P &, float hmax_i, const Rec &rj) { return hmax_i + rj.h; }
    __device__ static float leaf_cut(const P &, float hmax_i, float hmax_j) { return hmax_i + hmax_j; }
    __device__ static void shift(Rec &r, float sx, float sy, float sz) { r.x += sx; r.y += sy; r.z += sz; }
    __device__ static void init(const P &, I &s, const Rec &, int64_t, int, int, int32_t) {
#pragma unroll
        for (int a = 0; a < 3; ++a) s.xb[a] = s.vb[a] = s.Bb[a] = s.gAb[a] = s.F[a] = 0.f;
#pragma unroll
        for (int a = 0; a < 9; ++a) s.gBb[a] = 0.f;
        s.Vb = s.Pb = s.cb = s.rb = s.Ab = s.E = 0.f;
        s.cnt = 0;
    }
    template <bool kCount>
    __device__ static void interact(const P &p, I &s, const Rec &ri, const Rec &rj) {
        float x[3] = {ri.x - rj.x, ri.y - rj.y, ri.z - rj.z};  // x_ij
        float r2 = fmaf(x[0], x[0], fmaf(x[1], x[1], x[2] * x[2]));
        float hs = ri.h + rj.h;
        const bool in = r2 < hs * hs && __float_as_int(ri.pad) != __float_as_int(rj.pad);
        float hij = 0.5f * hs;
        float W, dWr, ddWr;
        wendland2(r2, hij, W, dWr, ddWr);
        W = in ? W : 0.0f;  // every term below is then zero
        dWr = in ? dWr : 0.0f;
        ddWr = in ? ddWr : 0.0f;
        float gi[3], gj[3];
        HydroStage::grad_wr(ri, x, W, dWr, gi);
        const float xm[3] = {-x[0], -x[1], -x[2]};
        HydroStage::grad_wr(rj, xm, W, dWr, gj);
        const float vij[3] = {ri.vx - rj.vx, ri.vy - rj.vy, ri.vz - rj.vz};
        const float vx = fmaf(vij[0], x[0], fmaf(vij[1], x[1], vij[2] * x[2]));
        const float den = fmaf(p.eta2 * hij, hij, r2);
        const bool visc = vx < 0.0f && in;
        const float mu = visc ? div_normal(hij * vx, den) : 0.0f;
        const float rbar = 0.5f * (ri.rho + rj.rho), cbar = 0.5f * (ri.c + rj.c);
        const float Q = rbar * mu * fmaf(-p.alpha, cbar, p.beta * mu);
        const float Pi = ri.P + rj.P + Q;
        const float VV = ri.V * rj.V;
        const float pre = -0.5f * VV * Pi;
        const float d[3] = {gi[0] - gj[0], gi[1] - gj[1], gi[2] - gj[2]};
        const float sb = ri.b + rj.b;
        const float z[3] = {fmaf(-0.5f * sb, vij[0], ri.ax - rj.ax), fmaf(-0.5f * sb, vij[1], ri.ay - rj.ay),
                            fmaf(-0.5f * sb, vij[2], ri.az - rj.az)};
        const float D = fmaf(z[0], d[0], fmaf(z[1], d[1], z[2] * d[2]));
#pragma unroll
        for (int c = 0; c < 3; ++c) s.F[c] = fmaf(pre, d[c], s.F[c]);
        s.E = fmaf(-0.5f * pre, fmaf(vij[0], d[0], fmaf(vij[1], d[1], vij[2] * d[2])), s.E);
        const float Pib = -0.5f * VV * D;
        s.Vb = fmaf(-0.5f * rj.V * Pi, D, s.Vb);
        s.Pb += Pib;
        if (visc) {
            const float mub = Pib * rbar * fmaf(-p.alpha, cbar, 2.0f * p.beta * mu);
            s.rb = fmaf(Pib * 0.5f * mu, fmaf(-p.alpha, cbar, p.beta * mu), s.rb);
            s.cb = fmaf(Pib * rbar * mu, -0.5f * p.alpha, s.cb);
            const float vxb = div_normal(mub * hij, den);
            const float r2b2 = -2.0f * vxb * div_normal(vx, den);
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                s.xb[c] = fmaf(vxb, vij[c], fmaf(r2b2, x[c], s.xb[c]));
                s.vb[c] = fmaf(vxb, x[c], s.vb[c]);
            }
        }
        const float dbar[3] = {pre * z[0], pre * z[1], pre * z[2]};
#pragma unroll
        for (int c = 0; c < 3; ++c) s.vb[c] = fmaf(-0.5f * sb * pre, d[c], s.vb[c]);
        float o1[3], o2[3];
        grad_wr_vjp<true>(ri, x, W, dWr, ddWr, dbar, o1, &s.Ab, s.Bb, s.gAb, s.gBb);
        grad_wr_vjp<false>(rj, xm, W, dWr, ddWr, dbar, o2, nullptr, nullptr, nullptr, nullptr);
#pragma unroll
        for (int c = 0; c < 3; ++c) s.xb[c] += o1[c] + o2[c];
        if (kCount) s.cnt += in;
    }
    __device__ static void finish(const P &p, I &s, const Rec &ri, int32_t o, int64_t) {
        const int64_t n = p.n;
        const float u = p.u[o], rho = p.rho[o], g1 = p.gamma - 1.0f;
        const float ub = fmaf(s.Pb * g1, rho, ri.c > 0.0f ? __fdividef(s.cb * p.gamma * g1, 2.0f * ri.c) : 0.0f);
        const float rb = fmaf(s.Pb * g1, u, s.rb);
        const float mb = -__fdividef(fmaf(ri.ax, s.F[0], fmaf(ri.ay, s.F[1], fmaf(ri.az, s.F[2], ri.b * s.E))), p.m[o]);
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            p.xbar3[c * n + o] = s.xb[c];
            p.vbar3[c * n + o] = s.vb[c];
            p.Bbar3[c * n + o] = s.Bb[c];
            p.gAbar3[c * n + o] = s.gAb[c];
        }
#pragma unroll
        for (int c = 0; c < 9; ++c) p.gBbar9[c * n + o] = s.gBb[c];
        p.ubar[o] = ub;
        p.mbar[o] = mb;
        p.Vbar[o] = s.Vb;
        p.rhobar[o] = rb;
        p.Abar[o] = s.Ab;
    }
    __device__ static void finish_other(const P &p, int32_t o) {
        const int64_t n = p.n;
        for (int c = 0; c < 3; ++c) {
            p.xbar3[c * n + o] = 0.f;
            p.vbar3[c * n + o] = 0.f;
            p.Bbar3[c * n + o] = 0.f;
            p.gAbar3[c * n + o] = 0.f;
        }
        for (int c = 0; c < 9; ++c) p.gBbar9[c * n + o] = 0.f;
        p.ubar[o] = p.mbar[o] = p.Vbar[o] = p.rhobar[o] = p.Abar[o] = 0.f;
    }
};

template <bool kLim>
using HydroAccelStage = HydroStageT<kLim, kHydroAccel>;
template <bool kLim, bool kWholeRec = false>
using HydroEnergyStage = HydroStageT<kLim, kHydroEnergy, kWholeRec>;

// Extras (Sec. 5: the density and state gradients), over gas j including j = i:
//   rhoR_i = sum_j m_j W^R_ij,   dv_i[3a+b] = sum_j V_j (v_j^a - v_i^a) (grad_i W^R_ij)^b
// with W^R_ij = A_i (1 + B_i.x_ij) W_ij and grad_i W^R_ij as in the hydro stage.
struct ExtrasP {
    const float *m, *v3, *V, *A, *B, *gA, *gB;
    float *rhoR, *dvg;
    int64_t n;
    unsigned long long *count;
    unsigned long long *swept;  // counting runs: candidate pair evaluations (tiles and lists), may be NULL
};

struct ExtrasStage {
    static constexpr bool kPair = false;
    static constexpr bool kGasOnly = true;
    static constexpr bool kCons = false;
    static constexpr bool kAllVariants = true;
    using P = ExtrasP;
    struct __align__(16) Rec {
        float x, y, z, h;
        float V, m, vx, vy;
        float vz, pad0, pad1, pad2;
        static constexpr int kWords = 9;
    };
    struct I {
        float A, B[3], gA[3], gB[9];  // the i particle's corrections (gB[3g+a] = d_g B^a)
        float rho, crho;              // compensated sum
        float G[9];
        int cnt;
    };
    __device__ static Rec gather(const P &p, int32_t o, float4 ps) {
        const int64_t n = p.n;
        return {ps.x, ps.y, ps.z, ps.w, p.V[o], p.m[o], p.v3[o], p.v3[n + o], p.v3[2 * n + o], 0.f, 0.f, 0.f};
    }
    __device__ static float box_cut(const P &, float hmax_i, const Rec &rj) { return hmax_i + rj.h; }
    __device__ static float leaf_cut(const P &, float hmax_i, float hmax_j) { return hmax_i + hmax_j; }
    __device__ static void shift(Rec &r, float sx, float sy, float sz) { r.x += sx; r.y += sy; r.z += sz; }
    __device__ static void init(const P &p, I &s, const Rec &, int64_t, int, int, int32_t o) {
        const int64_t n = p.n;
        s.A = p.A[o];
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            s.B[a] = p.B[a * n + o];
            s.gA[a] = p.gA[a * n + o];
        }
#pragma unroll
        for (int a = 0; a < 9; ++a) {
            s.gB[a] = p.gB[a * n + o];
            s.G[a] = 0.f;
        }
        s.rho = s.crho = 0.f;
        s.cnt = 0;
    }
    template <bool kCount>
    __device__ static void interact(const P &, I &s, const Rec &ri, const Rec &rj) {
        float x[3] = {ri.x - rj.x, ri.y - rj.y, ri.z - rj.z};  // x_ij
        float r2 = fmaf(x[0], x[0], fmaf(x[1], x[1], x[2] * x[2]));
        float hs = ri.h + rj.h;
        bool in = r2 < hs * hs;
        float W, dWr;
        wendland(r2, 0.5f * hs, W, dWr);
        W = in ? W : 0.0f;
        dWr = in ? dWr : 0.0f;
        const float Bx = fmaf(s.B[0], x[0], fmaf(s.B[1], x[1], s.B[2] * x[2]));
        const float k1 = (1.0f + Bx) * W;
        kahan_add(s.rho, s.crho, rj.m * (s.A * k1));
        // grad_i W^R_ij = gA (1 + B.x) W + A (gB.x + B) W + A (1 + B.x) dWr x
        const float AW = s.A * W, k3 = s.A * (1.0f + Bx) * dWr;
        float g[3];
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            float gBx = fmaf(s.gB[3 * q], x[0], fmaf(s.gB[3 * q + 1], x[1], s.gB[3 * q + 2] * x[2]));
            g[q] = fmaf(s.gA[q], k1, fmaf(AW, gBx + s.B[q], k3 * x[q]));
        }
        const float dv[3] = {rj.V * (rj.vx - ri.vx), rj.V * (rj.vy - ri.vy), rj.V * (rj.vz - ri.vz)};
#pragma unroll
        for (int a = 0; a < 3; ++a)
#pragma unroll
            for (int b = 0; b < 3; ++b) s.G[3 * a + b] = fmaf(dv[a], g[b], s.G[3 * a + b]);
        if (kCount) s.cnt += in;
    }
    __device__ static void finish(const P &p, I &s, const Rec &, int32_t o, int64_t) {
        p.rhoR[o] = s.rho;
#pragma unroll
        for (int k = 0; k < 9; ++k) p.dvg[k * p.n + o] = s.G[k];
    }
    __device__ static void finish_other(const P &p, int32_t o) {
        p.rhoR[o] = 0.f;
#pragma unroll
        for (int k = 0; k < 9; ++k) p.dvg[k * p.n + o] = 0.f;
    }
};

// Builds the exact neighbour lists of every i-group (count pass, then fill
// pass): gas pairs (r < h_i + h_j) or gravity pairs (r < r_cut).  A group's
// lists index a table of the distinct j the group needs (the union over its
// lanes, in the order the sweep meets them), so that a pair kernel stages each
// j of the group once and every lane reads its j from that table.
struct ListP {
    uint16_t *list;                    // per-lane table indices, k-major rows of 32 (written when non-null)
    uint32_t *ucode;                   // table entries (written when non-null)
    const int32_t *gstart, *goff, *uoff;
    int32_t *cnt;                      // list length per kernel-order position (written when non-null)
    int32_t *ucnt;                     // table size per group (written when non-null)
    int32_t *umax;                     // largest table (atomicMax), may be null
    int32_t *overflow;                 // set when a list or a table exceeds its capacity, may be null
    int cap_rows, cap_table;           // capacity of one lane's list and of one group's table
    float rc2;
};

// --------------------------------------------------------------- framework
template <class S>
__global__ void gather_kernel(int64_t n, const float4 *__restrict__ pos, const int32_t *__restrict__ kperm,
                              typename S::P p, void *__restrict__ rec, int korder) {
    int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= n) return;
    const float4 ps = pos[q];
    const int32_t o = korder ? (int32_t)q : kperm[q];
    if (S::kGasOnly && ps.w == 0.0f) {  // dark matter (h = 0): never read by gas-pair stages
        S::finish_other(p, o);           // its gas-only outputs are zero
        return;
    }
    Planes<typename S::Rec>::store(rec, n, q, S::gather(p, o, ps));
}

// Work of one warp on one i-group (tiles): the kernel-order particles
// g0 .. min(g0 + 32, hi) - 1 of i-leaf a (first particle lo) against every j
// of the leaf's images.  Each j within the cut of the group's box is
// ballot-compacted into the warp's shared-memory buffer; all lanes sweep the
// buffer (broadcast reads), each accumulating its own i.
template <class S, bool kCount>
__device__ __forceinline__ void tile_group(const LeafView &lv, const typename S::P &p,
                                           RecView<typename S::Rec> rec, typename S::Rec *buf,
                                           int64_t a, int lo, int g0, int hi, int lane, double cons_acc[4]) {
    using Rec = typename S::Rec;
    const unsigned below = lanemask_lt();
    const int ib = lv.img_start[a], ie = ib + lv.img_cnt[a];
    const int i = g0 + lane;
    const bool act = i < hi;
    const Rec ri = rec[act ? i : g0];
    typename S::I st;
    S::init(p, st, ri, a, (g0 - lo) >> 5, lane, stage_index(lv, act ? i : g0));
    // i-group box and largest h (inactive lanes repeat lane 0's particle)
    float bl0 = ri.x, bl1 = ri.y, bl2 = ri.z, bh0 = ri.x, bh1 = ri.y, bh2 = ri.z;
    float hm = lv.pos[act ? i : g0].w;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        bl0 = fminf(bl0, __shfl_xor_sync(CRK_FULL_MASK, bl0, o));
        bl1 = fminf(bl1, __shfl_xor_sync(CRK_FULL_MASK, bl1, o));
        bl2 = fminf(bl2, __shfl_xor_sync(CRK_FULL_MASK, bl2, o));
        bh0 = fmaxf(bh0, __shfl_xor_sync(CRK_FULL_MASK, bh0, o));
        bh1 = fmaxf(bh1, __shfl_xor_sync(CRK_FULL_MASK, bh1, o));
        bh2 = fmaxf(bh2, __shfl_xor_sync(CRK_FULL_MASK, bh2, o));
        hm = fmaxf(hm, __shfl_xor_sync(CRK_FULL_MASK, hm, o));
    }
    int cnt = 0;
    unsigned long long swept = 0;  // counting runs: candidates swept
    for (int e = ib; e < ie; ++e) {
        const crk_image im = lv.img[e];
        const int jlo = lv.leaf_start[im.b];
        const int jhi = S::kGasOnly ? jlo + lv.leaf_ngas[im.b] : lv.leaf_start[im.b + 1];
        // whole j-leaf against the i-group box (warp-uniform)
        {
            const float *bb = lv.bbox + 6 * (int64_t)im.b;
            float gx = fmaxf(fmaxf(im.sx - bh0, bl0 - (im.sx + (bb[3] - bb[0]))), 0.f);
            float gy = fmaxf(fmaxf(im.sy - bh1, bl1 - (im.sy + (bb[4] - bb[1]))), 0.f);
            float gz = fmaxf(fmaxf(im.sz - bh2, bl2 - (im.sz + (bb[5] - bb[2]))), 0.f);
            float cut = S::leaf_cut(p, hm, lv.hmax[im.b]);
            if (!(fmaf(gx, gx, fmaf(gy, gy, gz * gz)) <= cut * cut * 1.0001f + 1e-6f)) continue;
        }
        for (int j0 = jlo; j0 < jhi; j0 += 32) {
            const int j = j0 + lane;
            const bool jv = j < jhi;
            Rec rj;
            bool keep = false;
            if (jv) {
                rj = rec[j];
                S::shift(rj, im.sx, im.sy, im.sz);
                float dx = fmaxf(fmaxf(bl0 - rj.x, rj.x - bh0), 0.f);
                float dy = fmaxf(fmaxf(bl1 - rj.y, rj.y - bh1), 0.f);
                float dz = fmaxf(fmaxf(bl2 - rj.z, rj.z - bh2), 0.f);
                float cut = S::box_cut(p, hm, rj);
                keep = fmaf(dx, dx, fmaf(dy, dy, dz * dz)) <= cut * cut * 1.0001f + 1e-6f;
            }
            const unsigned m = __ballot_sync(CRK_FULL_MASK, keep);
            if (keep) buf[cnt + __popc(m & below)] = rj;
            cnt += __popc(m);
            if (cnt >= 32) {
                __syncwarp();
                for (int k = 0; k < cnt; ++k) S::template interact<kCount>(p, st, ri, buf[k]);
                if (kCount) swept += cnt;
                cnt = 0;
                __syncwarp();
            }
        }
    }
    __syncwarp();
    for (int k = 0; k < cnt; ++k) S::template interact<kCount>(p, st, ri, buf[k]);
    if (kCount) swept += cnt;
    __syncwarp();
    if (act) S::finish(p, st, ri, lv.korder ? i : lv.kperm[i], i);
    if constexpr (S::kCons) {
        double c[4] = {0.0, 0.0, 0.0, 0.0};
        if (act) S::cons_terms(p, st, ri, lv.korder ? i : lv.kperm[i], c);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) c[k] += __shfl_xor_sync(CRK_FULL_MASK, c[k], o);
            cons_acc[k] += c[k];
        }
    }
    if (kCount) {
        int c = act ? st.cnt - 1 : 0;  // the self pair (r = 0) is always in range
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(CRK_FULL_MASK, c, o);
        if (lane == 0 && c) atomicAdd(p.count, (unsigned long long)c);
        // candidate evaluations: every active lane evaluated every swept candidate
        const unsigned long long na = __popc(__ballot_sync(CRK_FULL_MASK, act));
        if (lane == 0 && p.swept) atomicAdd(p.swept, swept * na);
    }
}

// Cell sweeps (the TILES and SPLIT8 variants of the gravity kernels).  A warp
// takes G consecutive particles of a leaf (G = 16 or 8; in RCB leaves of at most
// 128 an RCB cell of the gravity kernel order, in larger leaves and mesh cells a
// part of a cell of 32) and all candidates within r_c of their box:
//   1. The j side is walked in cells of 32 (the groups of the kernel order).
//      Their boxes are tested 32 at a time, one per lane, before any particle
//      is loaded; the particles of a cell near enough are tested one per lane,
//      loaded one cell ahead, and those kept are compacted into shared memory.
//   2. A full buffer is swept: lane l evaluates candidate pairs k 32/G + l/G
//      (k = 0, 1, ..) against particle l % G with packed FP32 (f32x2)
//      arithmetic, so each row of the sweep reads 32/G pairs and every lane
//      works.  The sums of the 32/G streams are added by shuffles at the end
//      (fixed order, no atomics: deterministic).
// The FP32 pipe bounds it (56% busy; DRAM below 1%), on swept pairs: of those
// 0.43 are in range with G = 16 on the clustered boxes and 0.54 with G = 8, whose
// candidate tests cost more than the pairs they save.  2x128^3 box, gravity /
// adjoint: 2.92 / 5.49 ms (G = 8: 3.56 / 6.33), against 3.27 / 6.01 for a warp
// per group of 32 that walked the leaf images one by one.  The same holds where
// units are not RCB cells (2x48^3, that form -> G = 16, us: leaves of 256 340 /
// 541 -> 217 / 379, of 1024 844 / 1032 -> 231 / 389; mesh cells of 128 on the
// lattice box of 2x64^3 551 / 920 -> 454 / 852).
template <class S, bool kCount, int G, int kW>
__global__ void __launch_bounds__(32 * kW) cell_kernel(LeafView lv, typename S::P p, RecView<typename S::Rec> rec,
                                                       int units, int log_cpl, int full) {
    using Rec = typename S::Rec;
    constexpr int T = 32 / G;  // streams: candidate pairs per row
    __shared__ float4 buf[kW][S::kPlanes][kCellPairs];
    __shared__ float4 cells[kW][32];  // one round's cells: shift, first particle
    __shared__ int cell_n[kW][32];    // and particles
    __shared__ int64_t slot;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, str = lane / G;
    const unsigned below = lanemask_lt();
    const float cut = S::leaf_cut(p, 0.0f, 0.0f), cut2 = cut * cut * 1.0001f + 1e-6f;
    const int cmask = (1 << log_cpl) - 1;
    // block b takes units b kW .. b kW + kW - 1; a unit is G consecutive particles of one leaf
    for (int64_t b = next_leaf(lv, -1, &slot); b * kW < lv.n_leaves * units; b = next_leaf(lv, b, &slot)) {
        const int64_t unit = b * kW + warp;
        const int64_t a = unit / units;
        if (a >= lv.n_leaves) continue;
        const int lo = lv.leaf_start[a], hi = lv.leaf_start[a + 1];
        const int ib = lv.img_start[a], ie = ib + lv.img_cnt[a];
        // (a rebuilt chaining-mesh cell may hold more units than the launch counted: strided)
        for (int c0 = lo + G * (int)(unit - a * units); c0 < hi; c0 += G * units) {
            const int i = c0 + lane % G;
            const bool act = i < hi;
            typename S::I2 st;
            float ul[3], uh[3];  // the unit's box
            {
                const Rec ri = rec[act ? i : hi - 1];
                S::init2(p, st, ri);
                // leaf-relative coordinates are >= 0 (-0 + 0 = 0): their bits order like the values
                const unsigned x[3] = {__float_as_uint(ri.x + 0.0f), __float_as_uint(ri.y + 0.0f),
                                       __float_as_uint(ri.z + 0.0f)};
#pragma unroll
                for (int k = 0; k < 3; ++k) {
                    ul[k] = __uint_as_float(__reduce_min_sync(CRK_FULL_MASK, x[k]));
                    uh[k] = __uint_as_float(__reduce_max_sync(CRK_FULL_MASK, x[k]));
                }
            }
            unsigned long long swept = 0;  // counting runs: candidates swept
            int cnt = 0, e0 = ib, q = lane & cmask;  // q: this lane's cell of its image's leaf
            unsigned todo = 0;
            Rec rn;        // this lane's particle of the next cell, loaded one cell ahead
            float4 cl;     // that cell's shift
            int nn = 0;    // and its particles
            auto next = [&]() {
                const int src = __ffs(todo) - 1;
                cl = cells[warp][src];
                nn = cell_n[warp][src];
                if (lane < nn) rn = rec[__float_as_int(cl.w) + lane];
            };
            bool done = false;
            while (!done) {
                // ---- 1. fill the buffer
                while (cnt < full) {
                    if (!todo) {
                        if (e0 >= ie) {
                            done = true;
                            break;
                        }
                        const int e = e0 + (lane >> log_cpl);
                        bool pass = false, more = false;
                        if (e < ie) {
                            const crk_image im = lv.img[e];
                            const int jlo = lv.leaf_start[im.b], jhi = lv.leaf_start[im.b + 1];
                            const int jb = jlo + 32 * q;
                            more = jhi - jb > 32 * (cmask + 1);
                            if (jb < jhi) {
                                const float4 *gb = lv.gcell + 2 * ((int64_t)(jlo >> 5) + im.b + q);
                                const float4 l = gb[0], h = gb[1];
                                const float gx = fmaxf(fmaxf(im.sx + l.x - uh[0], ul[0] - (im.sx + h.x)), 0.f);
                                const float gy = fmaxf(fmaxf(im.sy + l.y - uh[1], ul[1] - (im.sy + h.y)), 0.f);
                                const float gz = fmaxf(fmaxf(im.sz + l.z - uh[2], ul[2] - (im.sz + h.z)), 0.f);
                                pass = fmaf(gx, gx, fmaf(gy, gy, gz * gz)) <= cut2;
                                cells[warp][lane] = make_float4(im.sx, im.sy, im.sz, __int_as_float(jb));
                                cell_n[warp][lane] = min(jhi - jb, 32);
                            }
                        }
                        todo = __ballot_sync(CRK_FULL_MASK, pass);
                        if (__any_sync(CRK_FULL_MASK, more)) {  // a leaf with more cells than its lanes: once more
                            q += cmask + 1;
                        } else {
                            q = lane & cmask;
                            e0 += 32 >> log_cpl;
                        }
                        if (!todo) continue;
                        __syncwarp();
                        next();
                    }
                    Rec rj = rn;
                    const bool jv = lane < nn;
                    S::shift(rj, cl.x, cl.y, cl.z);
                    todo &= todo - 1;
                    if (todo) next();
                    const float dx = fmaxf(fmaxf(ul[0] - rj.x, rj.x - uh[0]), 0.f);
                    const float dy = fmaxf(fmaxf(ul[1] - rj.y, rj.y - uh[1]), 0.f);
                    const float dz = fmaxf(fmaxf(ul[2] - rj.z, rj.z - uh[2]), 0.f);
                    const bool keep = jv && fmaf(dx, dx, fmaf(dy, dy, dz * dz)) <= cut2;
                    const unsigned m = __ballot_sync(CRK_FULL_MASK, keep);
                    if (keep) S::putc(buf[warp], cnt + __popc(m & below), rj);
                    cnt += __popc(m);
                }
                // ---- 2. sweep the whole rows; what is left over goes to the front (at the end: padded
                // with a massless dummy outside every cut, which adds exact zeros)
                if (done) {
                    const float far = 2.0f * cut + 1.0f;
                    const Rec dummy = S::far_dummy(uh[0] + far, uh[1] + far, uh[2] + far);
                    const int pad = -cnt & (2 * T - 1);
                    if (kCount) swept += cnt;
                    if (lane < pad) S::putc(buf[warp], cnt + lane, dummy);
                    cnt += pad;
                }
                __syncwarp();
                const int rows = cnt / (2 * T);
#pragma unroll 8
                for (int k = 0; k < rows; ++k) S::template interact2<kCount>(p, st, S::getc(buf[warp], k * T + str));
                if (!done) {
                    if (kCount) swept += rows * 2 * T;
                    cnt -= rows * 2 * T;
                    __syncwarp();
                    if (lane < T * S::kPlanes) {  // at most T pairs (rows > 1: the two ranges do not overlap)
                        const int k = lane % T, w = lane / T;
                        buf[warp][w][k] = buf[warp][w][rows * T + k];
                    }
                }
                __syncwarp();
            }
#pragma unroll
            for (int o = G; o < 32; o <<= 1) S::addc(st, o);
            if (act && str == 0) S::finish2(p, st, stage_index(lv, i));
            if (kCount) {
                int cn = act ? st.cnt - (str == 0) : 0;  // the self pair (r = 0) is always in range
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) cn += __shfl_xor_sync(CRK_FULL_MASK, cn, o);
                if (lane == 0 && cn) atomicAdd(p.count, (unsigned long long)cn);
                if (lane == 0 && p.swept) atomicAdd(p.swept, swept * min(G, hi - c0));
            }
        }
    }
}

template <class S, bool kCount, int G>
void launch_cells_g(const crk_ctx *ctx, const crk_leaves *lv, const LeafView &v, const typename S::P &p,
                    RecView<typename S::Rec> rec, bool persistent, int warps) {
    const int most = lv->max_leaf_size > 0 ? lv->max_leaf_size : 1;
    const int units = (most + G - 1) / G;
    int log_cpl = 0;  // cells of 32 per leaf, rounded up to a power of two (at most 32: one per lane)
    while ((32 << log_cpl) < most && log_cpl < 5) ++log_cpl;
    const int kw = warps == 2 ? 2 : 4;
    int64_t grid = (lv->n_leaves * units + kw - 1) / kw;
    if (grid < 1) grid = 1;
    if (grid > 2147483647LL) grid = 2147483647LL;
    if (persistent) grid = std::min<int64_t>(grid, (int64_t)ctx->num_sms * (kw == 2 ? 8 : 4));
    const int full = v.depth + 64;  // at most 160: 32 more fit, and a padded row
    if (kw == 2) cell_kernel<S, kCount, G, 2><<<(unsigned)grid, 64, 0, ctx->stream>>>(v, p, rec, units, log_cpl, full);
    else cell_kernel<S, kCount, G, 4><<<(unsigned)grid, 128, 0, ctx->stream>>>(v, p, rec, units, log_cpl, full);
}

// TILES: 16 particles per warp, SPLIT8: 8, at every size: the split decides the order of an i's sums, and
// a box of a batch gives the same bits as the box alone.  (8 would be faster where units of 16 are fewer
// than the warps the GPU holds: a box of 8192 particles takes 42 / 52 us, gravity / adjoint, against
// 35 / 43 with 8, one of 30,011 47 / 68 against 43 / 70, one of 65,536 80 / 129 against 80 / 125.)
template <class S, bool kCount>
void launch_cells(const crk_ctx *ctx, const crk_leaves *lv, const LeafView &v, const typename S::P &p,
                  RecView<typename S::Rec> rec, bool persistent, int warps, bool split8) {
    if (split8) launch_cells_g<S, kCount, 8>(ctx, lv, v, p, rec, persistent, warps);
    else launch_cells_g<S, kCount, 16>(ctx, lv, v, p, rec, persistent, warps);
}

// The paper's "half-warp" leaf-pair scheme (Sec. 5.3), as autotuner arms for
// the gravity stages.  Lanes 0-15 hold 16 particles of leaf A, lanes 16-31 16
// particles of leaf B (shifted into A's frame); in step s lane l and lane
// 16 + (l ^ s) exchange their particles and each evaluates the interaction on
// its own particle, so every A-B pair is evaluated once in each direction in
// the same step.  Each unordered leaf-pair image is visited once (entries with
// b > a, or b = a with a positive shift, and the leaf with itself); the
// partial sums of each tile are added to the outputs atomically, so the
// result is exact up to the order of the FP32 additions.  kEx selects how the
// partner's particle reaches a lane: 0 register shuffle, 1 shared memory,
// 2 a second load of the partner's record.
template <class Rec>
__device__ __forceinline__ Rec shfl_rec(const Rec &r, int src) {
    Rec o;
    const float *a = reinterpret_cast<const float *>(&r);
    float *b = reinterpret_cast<float *>(&o);
#pragma unroll
    for (int k = 0; k < (int)(sizeof(Rec) / sizeof(float)); ++k) b[k] = __shfl_sync(CRK_FULL_MASK, a[k], src);
    return o;
}

__device__ __forceinline__ bool positive_shift(float sx, float sy, float sz) {
    return sx > 0.f || (sx == 0.f && (sy > 0.f || (sy == 0.f && sz > 0.f)));
}

// Gas stages (the Acceleration and Energy passes) use the gas prefix of each
// leaf and the tile cut h_max(A slice) + h_max(B slice); their conservation
// sums are taken afterwards from the finished outputs (halfwarp_cons_kernel).
template <class S, bool kCount, int kEx>
__global__ void __launch_bounds__(kThreads) pair_kernel_halfwarp(LeafView lv, typename S::P p,
                                                                 RecView<typename S::Rec> rec,
                                                                 double *__restrict__) {
    using Rec = typename S::Rec;
    static_assert(S::kHalfWarp, "half-warp arms: stages with atomic partial sums");
    __shared__ __align__(16) Rec xbuf[kWarps][32];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, half = lane >> 4, hl = lane & 15;
    const float rc = S::leaf_cut(p, 0.f, 0.f);
    __shared__ int64_t leaf_slot;
    for (int64_t a = next_leaf(lv, -1, &leaf_slot); a < lv.n_leaves; a = next_leaf(lv, a, &leaf_slot)) {
        const int alo = lv.leaf_start[a];
        const int ahi = S::kGasOnly ? alo + lv.leaf_ngas[a] : lv.leaf_start[a + 1];
        const int nsa = (ahi - alo + 15) >> 4;
        const int ib = lv.img_start[a], ie = ib + lv.img_cnt[a];
        int t0 = warp;  // tiles are dealt to the block's warps in turn across the leaf's entries
        for (int e = ib; e < ie; ++e) {
            const crk_image im = lv.img[e];
            const int b = im.b;
            const bool self = b == a && im.sx == 0.f && im.sy == 0.f && im.sz == 0.f;
            if (b < a || (b == a && !self && !positive_shift(im.sx, im.sy, im.sz))) continue;
            const int blo = lv.leaf_start[b];
            const int bhi = S::kGasOnly ? blo + lv.leaf_ngas[b] : lv.leaf_start[b + 1];
            const int nsb = (bhi - blo + 15) >> 4;
            const int ntile = nsa * nsb;
            int t = t0;
            for (; t < ntile; t += kWarps) {
                const int u = t / nsb, v = t - u * nsb;
                if (self && v < u) continue;
                const bool diag = self && u == v;  // the same 16 particles in both halves: only A accumulates
                const int idx = half ? blo + 16 * v + hl : alo + 16 * u + hl;
                const bool valid = idx < (half ? bhi : ahi);
                Rec r = rec[valid ? idx : (half ? blo : alo)];
                if (half) S::shift(r, im.sx, im.sy, im.sz);
                // slice boxes (valid lanes only), then the whole tile against the cut (warp-uniform)
                float l0 = valid ? r.x : INFINITY, l1 = valid ? r.y : INFINITY, l2 = valid ? r.z : INFINITY;
                float h0 = valid ? r.x : -INFINITY, h1 = valid ? r.y : -INFINITY, h2 = valid ? r.z : -INFINITY;
#pragma unroll
                for (int o = 1; o < 16; o <<= 1) {
                    l0 = fminf(l0, __shfl_xor_sync(CRK_FULL_MASK, l0, o));
                    l1 = fminf(l1, __shfl_xor_sync(CRK_FULL_MASK, l1, o));
                    l2 = fminf(l2, __shfl_xor_sync(CRK_FULL_MASK, l2, o));
                    h0 = fmaxf(h0, __shfl_xor_sync(CRK_FULL_MASK, h0, o));
                    h1 = fmaxf(h1, __shfl_xor_sync(CRK_FULL_MASK, h1, o));
                    h2 = fmaxf(h2, __shfl_xor_sync(CRK_FULL_MASK, h2, o));
                }
                float cut = rc;
                if constexpr (S::kGasOnly) {  // h_max of each slice: the cut is their sum
                    float hs = valid ? lv.pos[idx].w : 0.0f;
#pragma unroll
                    for (int o = 1; o < 16; o <<= 1) hs = fmaxf(hs, __shfl_xor_sync(CRK_FULL_MASK, hs, o));
                    cut = S::leaf_cut(p, hs, __shfl_xor_sync(CRK_FULL_MASK, hs, 16));
                }
                const float ol0 = __shfl_xor_sync(CRK_FULL_MASK, l0, 16), ol1 = __shfl_xor_sync(CRK_FULL_MASK, l1, 16),
                            ol2 = __shfl_xor_sync(CRK_FULL_MASK, l2, 16), oh0 = __shfl_xor_sync(CRK_FULL_MASK, h0, 16),
                            oh1 = __shfl_xor_sync(CRK_FULL_MASK, h1, 16), oh2 = __shfl_xor_sync(CRK_FULL_MASK, h2, 16);
                const float gx = fmaxf(fmaxf(ol0 - h0, l0 - oh0), 0.f), gy = fmaxf(fmaxf(ol1 - h1, l1 - oh1), 0.f),
                            gz = fmaxf(fmaxf(ol2 - h2, l2 - oh2), 0.f);
                // empty halves give NaN/inf gaps: those tiles are skipped too
                if (!(fmaf(gx, gx, fmaf(gy, gy, gz * gz)) <= cut * cut * 1.0001f + 1e-6f)) continue;
                if (!valid) {  // a particle outside every cut that contributes exact zeros
                    r = S::far_dummy(1e15f, 1e15f, 1e15f);
                }
                if constexpr (kEx == 1) {
                    __syncwarp();
                    xbuf[warp][lane] = r;
                    __syncwarp();
                }
                typename S::I st;
                S::init(p, st, r, a, 0, lane, 0);
                const bool acc = valid && !(diag && half);
#pragma unroll 2
                for (int s = 0; s < 16; ++s) {
                    const int pl = half ? (hl ^ s) : 16 + (hl ^ s);
                    Rec q;
                    if constexpr (kEx == 0) {
                        q = shfl_rec(r, pl);
                    } else if constexpr (kEx == 1) {
                        q = xbuf[warp][pl];
                    } else {
                        const int pi = pl < 16 ? alo + 16 * u + pl : (diag ? alo + 16 * u : blo + 16 * v) + (pl - 16);
                        const bool pv = pi < (pl < 16 || diag ? ahi : bhi);
                        if (pv) {
                            q = rec[pi];
                            if (pl >= 16 && !diag) S::shift(q, im.sx, im.sy, im.sz);
                        } else {
                            q = S::far_dummy(1e15f, 1e15f, 1e15f);
                        }
                    }
                    if (acc) S::template interact<kCount>(p, st, r, q);
                }
                if (acc) S::flush(p, st, r, stage_index(lv, idx));
                if (kCount) {
                    int c = acc ? st.cnt - (diag ? 1 : 0) : 0;  // the self pair of a diagonal tile
#pragma unroll
                    for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(CRK_FULL_MASK, c, o);
                    if (lane == 0 && c) atomicAdd(p.count, (unsigned long long)c);
                }
            }
            t0 = t - ntile;  // continue the round robin in the next entry
        }
    }
}

// Per-block partial of the FP64 conservation sums in a fixed order (reduced by
// cons_reduce_kernel: deterministic for a fixed assignment of work to blocks).
__device__ __forceinline__ void cons_block_sum(double (*cons_sh)[4], double *__restrict__ cons_part) {
    __syncthreads();
    if (threadIdx.x == 0)
        for (int k = 0; k < 4; ++k) {
            double t = 0.0;
            for (int w = 0; w < kWarps; ++w) t += cons_sh[w][k];
            cons_part[4 * (int64_t)blockIdx.x + k] = t;
        }
}

__device__ __forceinline__ void cons_block_partial(double (*cons_sh)[4], const double cons_acc[4],
                                                   double *__restrict__ cons_part) {
    if ((threadIdx.x & 31) == 0)
        for (int k = 0; k < 4; ++k) cons_sh[threadIdx.x >> 5][k] = cons_acc[k];
    cons_block_sum(cons_sh, cons_part);
}

// The warp's sum of c[lane / 8]: the lanes halve the values between them on the way, 6 FP64 additions
// (16 cycles of an SM each) instead of 20.
__device__ __forceinline__ double cons_warp_sum(const double c[4], int lane) {
    const bool h = lane & 16, q = lane & 8;
    const double a0 = (h ? c[2] : c[0]) + __shfl_xor_sync(CRK_FULL_MASK, h ? c[0] : c[2], 16);
    const double a1 = (h ? c[3] : c[1]) + __shfl_xor_sync(CRK_FULL_MASK, h ? c[1] : c[3], 16);
    double a = (q ? a1 : a0) + __shfl_xor_sync(CRK_FULL_MASK, q ? a0 : a1, 8);
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) a += __shfl_xor_sync(CRK_FULL_MASK, a, o);
    return a;
}

// Tiles, one block per i-leaf (or leaves from the persistent queue); the
// block's warps take the leaf's groups in turn (gas stages; the gravity
// stages run cell_kernel).
template <class S, bool kCount>
__global__ void __launch_bounds__(kThreads) pair_kernel(LeafView lv, typename S::P p, RecView<typename S::Rec> rec,
                                                        double *__restrict__ cons_part) {
    using Rec = typename S::Rec;
    static_assert(!S::kPair, "gravity stages sweep sub-cells");
    __shared__ __align__(16) Rec buf[kWarps][kCap];
    __shared__ double cons_sh[kWarps][4];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    double cons_acc[4] = {0.0, 0.0, 0.0, 0.0};
    __shared__ int64_t leaf_slot;
    for (int64_t a = next_leaf(lv, -1, &leaf_slot); a < lv.n_leaves; a = next_leaf(lv, a, &leaf_slot)) {
        const int lo = lv.leaf_start[a];
        const int hi = S::kGasOnly ? lo + lv.leaf_ngas[a] : lv.leaf_start[a + 1];
        for (int g0 = lo + warp * 32; g0 < hi; g0 += kWarps * 32)
            tile_group<S, kCount>(lv, p, rec, buf[warp], a, lo, g0, hi, lane, cons_acc);
    }
    if constexpr (S::kCons) {
        if (cons_part) cons_block_partial(cons_sh, cons_acc, cons_part);
    }
}

// Group table of one set of leaves: groups of 32 consecutive kernel-order
// particles (gas only for gas stages), numbered leaf by leaf.
struct GroupTable {
    const int32_t *gstart;   // [n_leaves + 1] first group of each leaf
    const int32_t *gleaf;    // [groups] leaf of each group
    int64_t groups;          // capacity of the group arrays
    const int32_t *dgroups;  // device: the groups of this build (<= groups), or NULL for all
};

// groups of a build: the device count when the arrays have room for more
__device__ __forceinline__ int64_t group_count(int64_t cap, const int32_t *dgroups) {
    if (!dgroups) return cap;
    const int64_t g = *dgroups;
    return g < cap ? g : cap;
}

// Builds the neighbour lists, one warp per i-group.  The j cells of 32 are
// culled 32 at a time, one per lane, by their boxes (and largest h), the
// particles of a cell near enough are tested against the group's box and
// compacted; then every lane tests 32 buffered candidates against its own i in
// straight-line packed FP32 (the kernels' own arithmetic, so the lists hold
// exactly the pairs they would find in range) and keeps the answers as bits.
// The union of the lanes' bits gives the candidates their table entries, and
// each lane writes the entries of its own bits.  A ballot, a counter and two
// predicated stores for every candidate, as before, kept the issue slots busy.
// 2x256^3 box 11.2 -> 6.9 ms, 2x64^3 230 -> 142 us, 2x32^3 90 -> 43 us.
template <bool kGas>
__global__ void __launch_bounds__(kThreads) list_build_kernel(LeafView lv, ListP p, GroupTable gt,
                                                              const float4 *__restrict__ cellbox, int log_cpl) {
    __shared__ float4 buf[kWarps][2][32];  // candidate pairs: (x0, x1, y0, y1), (z0, z1, h0, h1)
    __shared__ uint32_t code[kWarps][64];
    __shared__ float4 cells[kWarps][32];   // one round's cells: shift, first particle
    __shared__ int2 cell_n[kWarps][32];    // particles, code of the first
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const unsigned below = lanemask_lt();
    const int cmask = (1 << log_cpl) - 1;
    const float rc = sqrtf(p.rc2);
    const int64_t ngroups = group_count(gt.groups, gt.dgroups);
    for (int64_t grp = next_group(lv, -1, lane); grp < ngroups; grp = next_group(lv, grp, lane)) {
        const int64_t a = gt.gleaf[grp];
        const int lo = lv.leaf_start[a];
        const int hi = kGas ? lo + lv.leaf_ngas[a] : lv.leaf_start[a + 1];
        const int g0 = lo + 32 * (int)(grp - gt.gstart[a]), i = g0 + lane;
        const bool act = i < hi;
        const float4 ri = lv.pos[act ? i : g0];
        // leaf-relative coordinates and h are >= 0 (-0 + 0 = 0): their bits order like the values
        const unsigned x[3] = {__float_as_uint(ri.x + 0.0f), __float_as_uint(ri.y + 0.0f), __float_as_uint(ri.z + 0.0f)};
        float bl[3], bh[3];
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            bl[k] = __uint_as_float(__reduce_min_sync(CRK_FULL_MASK, x[k]));
            bh[k] = __uint_as_float(__reduce_max_sync(CRK_FULL_MASK, x[k]));
        }
        const float hm = __uint_as_float(__reduce_max_sync(CRK_FULL_MASK, __float_as_uint(ri.w)));
        const float2 nx = make_float2(-ri.x, -ri.x), ny = make_float2(-ri.y, -ri.y), nz = make_float2(-ri.z, -ri.z),
                     h2 = make_float2(ri.w, ri.w);
        uint16_t *const out = p.list ? p.list + (size_t)p.goff[grp] * 32 + lane : nullptr;
        uint32_t *const uout = p.ucode ? p.ucode + p.uoff[grp] : nullptr;
        int c = 0, u = 0, cnt = 0;  // this lane's list length; table size and candidates (warp-uniform)
        // the first `m` (at most 32) candidates
        auto test = [&](int m) {
            __syncwarp();
            unsigned in = 0u;
#pragma unroll
            for (int k = 0; k < 16; ++k) {
                const float4 q0 = buf[warp][0][k], q1 = buf[warp][1][k];
                const float2 dx = __fadd2_rn(make_float2(q0.x, q0.y), nx), dy = __fadd2_rn(make_float2(q0.z, q0.w), ny),
                             dz = __fadd2_rn(make_float2(q1.x, q1.y), nz);
                const float2 r2 = __ffma2_rn(dx, dx, __ffma2_rn(dy, dy, __fmul2_rn(dz, dz)));
                float2 c2 = make_float2(p.rc2, p.rc2);
                if constexpr (kGas) {
                    const float2 hs = __fadd2_rn(h2, make_float2(q1.z, q1.w));
                    c2 = __fmul2_rn(hs, hs);
                }
                if (r2.x < c2.x) in |= 1u << (2 * k);
                if (r2.y < c2.y) in |= 2u << (2 * k);
            }
            if (m < 32) in &= (1u << m) - 1u;
            if (!act) in = 0u;
            const unsigned used = __reduce_or_sync(CRK_FULL_MASK, in);
            if (uout && (used >> lane & 1u)) {
                const int at = u + __popc(used & below);
                if (at < p.cap_table) uout[at] = code[warp][lane];
            }
            while (in) {
                const unsigned low = in & (0u - in);
                const int at = u + __popc(used & (low - 1u));
                if (out && c < p.cap_rows && at < p.cap_table) out[(size_t)c * 32] = (uint16_t)at;
                ++c;
                in ^= low;
            }
            u += __popc(used);
            __syncwarp();
        };
        const int ib = lv.img_start[a], ie = ib + lv.img_cnt[a];
        int q = lane & cmask;  // this lane's cell of its image's leaf
        for (int e0 = ib; e0 < ie;) {
            const int e = e0 + (lane >> log_cpl);
            bool pass = false, more = false;
            if (e < ie) {
                const crk_image im = lv.img[e];
                const int jlo = lv.leaf_start[im.b], jhi = kGas ? jlo + lv.leaf_ngas[im.b] : lv.leaf_start[im.b + 1];
                const int jb = jlo + 32 * q;
                more = jhi - jb > 32 * (cmask + 1);
                if (jb < jhi) {
                    const float4 *gb = cellbox + 2 * ((int64_t)(jlo >> 5) + im.b + q);
                    const float4 l = gb[0], h = gb[1];
                    const float gx = fmaxf(fmaxf(im.sx + l.x - bh[0], bl[0] - (im.sx + h.x)), 0.f);
                    const float gy = fmaxf(fmaxf(im.sy + l.y - bh[1], bl[1] - (im.sy + h.y)), 0.f);
                    const float gz = fmaxf(fmaxf(im.sz + l.z - bh[2], bl[2] - (im.sz + h.z)), 0.f);
                    const float cut = kGas ? hm + l.w : rc;
                    pass = fmaf(gx, gx, fmaf(gy, gy, gz * gz)) <= cut * cut * 1.0001f + 1e-6f;
                    cells[warp][lane] = make_float4(im.sx, im.sy, im.sz, __int_as_float(jb));
                    cell_n[warp][lane] = make_int2(min(jhi - jb, 32), ((e - ib) << 10) | (jb - jlo));
                }
            }
            unsigned todo = __ballot_sync(CRK_FULL_MASK, pass);
            if (__any_sync(CRK_FULL_MASK, more)) {  // a leaf with more cells than its lanes: once more
                q += cmask + 1;
            } else {
                q = lane & cmask;
                e0 += 32 >> log_cpl;
            }
            __syncwarp();
            float4 cl = make_float4(0.f, 0.f, 0.f, 0.f), rn = cl;  // the next cell, loaded one ahead
            int2 nn = make_int2(0, 0);
            auto next = [&]() {
                const int src = __ffs(todo) - 1;
                cl = cells[warp][src];
                nn = cell_n[warp][src];
                if (lane < nn.x) rn = lv.pos[__float_as_int(cl.w) + lane];
            };
            if (todo) next();
            while (todo) {
                const float4 rj = make_float4(rn.x + cl.x, rn.y + cl.y, rn.z + cl.z, rn.w);
                const bool jv = lane < nn.x;
                const uint32_t cd = (uint32_t)(nn.y + lane);
                todo &= todo - 1;
                if (todo) next();
                const float dx = fmaxf(fmaxf(bl[0] - rj.x, rj.x - bh[0]), 0.f);
                const float dy = fmaxf(fmaxf(bl[1] - rj.y, rj.y - bh[1]), 0.f);
                const float dz = fmaxf(fmaxf(bl[2] - rj.z, rj.z - bh[2]), 0.f);
                const float cut = kGas ? hm + rj.w : rc;
                const bool keep = jv && fmaf(dx, dx, fmaf(dy, dy, dz * dz)) <= cut * cut * 1.0001f + 1e-6f;
                const unsigned m = __ballot_sync(CRK_FULL_MASK, keep);
                if (keep) {
                    const int at = cnt + __popc(m & below);
                    float *d0 = reinterpret_cast<float *>(&buf[warp][0][at >> 1]) + (at & 1);
                    float *d1 = reinterpret_cast<float *>(&buf[warp][1][at >> 1]) + (at & 1);
                    d0[0] = rj.x; d0[2] = rj.y; d1[0] = rj.z; d1[2] = rj.w;
                    code[warp][at] = cd;
                }
                cnt += __popc(m);
                if (cnt >= 32) {
                    test(32);
                    cnt -= 32;  // the rest (at most 31) goes to the front
                    buf[warp][lane >> 4][lane & 15] = buf[warp][lane >> 4][16 + (lane & 15)];
                    code[warp][lane] = code[warp][32 + lane];
                    __syncwarp();
                }
            }
            __syncwarp();
        }
        if (cnt) test(cnt);
        if (p.cnt && act) p.cnt[i] = c;
        const int cmax = (int)__reduce_max_sync(CRK_FULL_MASK, (unsigned)c);
        if (lane == 0) {
            if (p.overflow && (cmax > p.cap_rows || u > p.cap_table)) atomicOr(p.overflow, 1);
            if (p.ucnt) p.ucnt[grp] = u;
            if (p.umax) atomicMax(p.umax, u);
        }
        __syncwarp();
    }
}

template <bool kGas>
void launch_list_build(crk_ctx *ctx, const crk_leaves *lv, const LeafView &v, const ListP &p, const GroupTable &gt,
                       int64_t groups) {
    int log_cpl = 0;  // cells of 32 per leaf, rounded up to a power of two (at most 32: one per lane)
    while ((32 << log_cpl) < lv->max_leaf_size && log_cpl < 5) ++log_cpl;
    const unsigned grid = (unsigned)std::max<int64_t>(1, (groups + kWarps - 1) / kWarps);
    list_build_kernel<kGas><<<grid, kThreads, 0, ctx->stream>>>(v, p, gt, kGas ? lv->hcell : lv->gcell, log_cpl);
    ++ctx->launches;
}

// Tiles with sub-warp i-groups: the warp's 32 i-particles form 32/G groups of
// G consecutive particles of the kernel order, each with its own box and its own
// compacted candidate buffer; lane l sweeps the buffer of group l/G.  Smaller
// groups have smaller boxes, so a larger share of the swept pairs is in range.
// Within one 8-lane phase of a shared-memory load every lane reads the same
// record (G >= 8), so the sweep stays a broadcast.
template <class S, int G, bool kCount>
__global__ void __launch_bounds__(kThreads) pair_kernel_sub(LeafView lv, typename S::P p,
                                                            RecView<typename S::Rec> rec,
                                                            double *__restrict__ cons_part) {
    using Rec = typename S::Rec;
    constexpr int NS = 32 / G;
    __shared__ Rec buf[kWarps][NS][kCap];
    __shared__ double cons_sh[kWarps][4];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, sg = lane / G;
    const unsigned below = lanemask_lt();
    double cons_acc[4] = {0.0, 0.0, 0.0, 0.0};
    __shared__ int64_t leaf_slot;
    for (int64_t a = next_leaf(lv, -1, &leaf_slot); a < lv.n_leaves; a = next_leaf(lv, a, &leaf_slot)) {
        const int lo = lv.leaf_start[a];
        const int hi = S::kGasOnly ? lo + lv.leaf_ngas[a] : lv.leaf_start[a + 1];
        const int ib = lv.img_start[a], ie = ib + lv.img_cnt[a];
        for (int g0 = lo + warp * 32; g0 < hi; g0 += kWarps * 32) {
            const int i = g0 + lane;
            const bool act = i < hi;
            const Rec ri = rec[act ? i : g0];
            typename S::I st;
            S::init(p, st, ri, a, (g0 - lo) >> 5, lane, stage_index(lv, act ? i : g0));
            // group boxes (empty for groups without active lanes) and largest h
            float l0 = act ? ri.x : INFINITY, l1 = act ? ri.y : INFINITY, l2 = act ? ri.z : INFINITY;
            float h0 = act ? ri.x : -INFINITY, h1 = act ? ri.y : -INFINITY, h2 = act ? ri.z : -INFINITY;
            float hm = act ? lv.pos[i].w : 0.0f;
#pragma unroll
            for (int o = G / 2; o > 0; o >>= 1) {
                l0 = fminf(l0, __shfl_xor_sync(CRK_FULL_MASK, l0, o));
                l1 = fminf(l1, __shfl_xor_sync(CRK_FULL_MASK, l1, o));
                l2 = fminf(l2, __shfl_xor_sync(CRK_FULL_MASK, l2, o));
                h0 = fmaxf(h0, __shfl_xor_sync(CRK_FULL_MASK, h0, o));
                h1 = fmaxf(h1, __shfl_xor_sync(CRK_FULL_MASK, h1, o));
                h2 = fmaxf(h2, __shfl_xor_sync(CRK_FULL_MASK, h2, o));
                hm = fmaxf(hm, __shfl_xor_sync(CRK_FULL_MASK, hm, o));
            }
            float bl[NS][3], bh[NS][3], bhm[NS];
            float ul0 = INFINITY, ul1 = INFINITY, ul2 = INFINITY, uh0 = -INFINITY, uh1 = -INFINITY, uh2 = -INFINITY,
                  uhm = 0.0f;
#pragma unroll
            for (int t = 0; t < NS; ++t) {
                bl[t][0] = __shfl_sync(CRK_FULL_MASK, l0, t * G);
                bl[t][1] = __shfl_sync(CRK_FULL_MASK, l1, t * G);
                bl[t][2] = __shfl_sync(CRK_FULL_MASK, l2, t * G);
                bh[t][0] = __shfl_sync(CRK_FULL_MASK, h0, t * G);
                bh[t][1] = __shfl_sync(CRK_FULL_MASK, h1, t * G);
                bh[t][2] = __shfl_sync(CRK_FULL_MASK, h2, t * G);
                bhm[t] = __shfl_sync(CRK_FULL_MASK, hm, t * G);
                ul0 = fminf(ul0, bl[t][0]); ul1 = fminf(ul1, bl[t][1]); ul2 = fminf(ul2, bl[t][2]);
                uh0 = fmaxf(uh0, bh[t][0]); uh1 = fmaxf(uh1, bh[t][1]); uh2 = fmaxf(uh2, bh[t][2]);
                uhm = fmaxf(uhm, bhm[t]);
            }
            int cnt[NS];
#pragma unroll
            for (int t = 0; t < NS; ++t) cnt[t] = 0;
            auto sweep = [&]() {
                __syncwarp();
                int kmax = 0, mine = 0;
#pragma unroll
                for (int t = 0; t < NS; ++t) {
                    kmax = max(kmax, cnt[t]);
                    if (t == sg) mine = cnt[t];
                }
                for (int k = 0; k < kmax; ++k)
                    if (k < mine) S::template interact<kCount>(p, st, ri, buf[warp][sg][k]);
#pragma unroll
                for (int t = 0; t < NS; ++t) cnt[t] = 0;
                __syncwarp();
            };
            for (int e = ib; e < ie; ++e) {
                const crk_image im = lv.img[e];
                const int jlo = lv.leaf_start[im.b];
                const int jhi = S::kGasOnly ? jlo + lv.leaf_ngas[im.b] : lv.leaf_start[im.b + 1];
                {
                    const float *bb = lv.bbox + 6 * (int64_t)im.b;
                    float gx = fmaxf(fmaxf(im.sx - uh0, ul0 - (im.sx + (bb[3] - bb[0]))), 0.f);
                    float gy = fmaxf(fmaxf(im.sy - uh1, ul1 - (im.sy + (bb[4] - bb[1]))), 0.f);
                    float gz = fmaxf(fmaxf(im.sz - uh2, ul2 - (im.sz + (bb[5] - bb[2]))), 0.f);
                    float cut = S::leaf_cut(p, uhm, lv.hmax[im.b]);
                    if (!(fmaf(gx, gx, fmaf(gy, gy, gz * gz)) <= cut * cut * 1.0001f + 1e-6f)) continue;
                }
                for (int j0 = jlo; j0 < jhi; j0 += 32) {
                    const int j = j0 + lane;
                    const bool jv = j < jhi;
                    Rec rj;
                    if (jv) {
                        rj = rec[j];
                        S::shift(rj, im.sx, im.sy, im.sz);
                    }
                    bool full = false;
#pragma unroll
                    for (int t = 0; t < NS; ++t) {
                        bool keep = false;
                        if (jv) {
                            float dx = fmaxf(fmaxf(bl[t][0] - rj.x, rj.x - bh[t][0]), 0.f);
                            float dy = fmaxf(fmaxf(bl[t][1] - rj.y, rj.y - bh[t][1]), 0.f);
                            float dz = fmaxf(fmaxf(bl[t][2] - rj.z, rj.z - bh[t][2]), 0.f);
                            float cut = S::box_cut(p, bhm[t], rj);
                            keep = fmaf(dx, dx, fmaf(dy, dy, dz * dz)) <= cut * cut * 1.0001f + 1e-6f;
                        }
                        const unsigned m = __ballot_sync(CRK_FULL_MASK, keep);
                        if (keep) buf[warp][t][cnt[t] + __popc(m & below)] = rj;
                        cnt[t] += __popc(m);
                        full |= cnt[t] >= 32;
                    }
                    if (full) sweep();
                }
            }
            sweep();
            if (act) S::finish(p, st, ri, lv.korder ? i : lv.kperm[i], i);
            if constexpr (S::kCons) {
                double cc[4] = {0.0, 0.0, 0.0, 0.0};
                if (act) S::cons_terms(p, st, ri, lv.korder ? i : lv.kperm[i], cc);
#pragma unroll
                for (int k = 0; k < 4; ++k) {
#pragma unroll
                    for (int o = 16; o > 0; o >>= 1) cc[k] += __shfl_xor_sync(CRK_FULL_MASK, cc[k], o);
                    cons_acc[k] += cc[k];
                }
            }
            if (kCount) {
                int cn = act ? st.cnt - 1 : 0;
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) cn += __shfl_xor_sync(CRK_FULL_MASK, cn, o);
                if (lane == 0 && cn) atomicAdd(p.count, (unsigned long long)cn);
            }
        }
    }
    if constexpr (S::kCons) {
        if (cons_part) {
            if (lane == 0)
                for (int k = 0; k < 4; ++k) cons_sh[warp][k] = cons_acc[k];
            __syncthreads();
            if (threadIdx.x == 0)
                for (int k = 0; k < 4; ++k) {
                    double t = 0.0;
                    for (int w = 0; w < kWarps; ++w) t += cons_sh[w][k];
                    cons_part[4 * (int64_t)blockIdx.x + k] = t;
                }
        }
    }
}


// Tiles with two 16-particle i-groups per warp for the packed gravity stages
// (kPair): each half-warp's group (an RCB cell of its leaf) has its own box
// and its own buffer of field-interleaved candidate pairs, swept two
// candidates per lane step with f32x2 arithmetic; an odd tail is padded with
// a massless dummy outside every cut.  A 16-particle cell prunes ~22% more of
// the candidates than its 32-particle parent at r_c = 3.
template <class S, bool kCount>
__global__ void __launch_bounds__(kThreads) pair_kernel_sub_pair(LeafView lv, typename S::P p,
                                                                 RecView<typename S::Rec> rec,
                                                                 double *__restrict__ cons_part) {
    using Rec = typename S::Rec;
    using Rec2 = typename S::Rec2;
    constexpr int G = 16, NS = 2;
    __shared__ __align__(16) Rec2 buf[kWarps][NS][kCap / 2];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, sg = lane / G;
    const unsigned below = lanemask_lt();
    (void)cons_part;
    __shared__ int64_t leaf_slot;
    for (int64_t a = next_leaf(lv, -1, &leaf_slot); a < lv.n_leaves; a = next_leaf(lv, a, &leaf_slot)) {
        const int lo = lv.leaf_start[a];
        const int hi = lv.leaf_start[a + 1];
        const int ib = lv.img_start[a], ie = ib + lv.img_cnt[a];
        for (int g0 = lo + warp * 32; g0 < hi; g0 += kWarps * 32) {
            const int i = g0 + lane;
            const bool act = i < hi;
            const Rec ri = rec[act ? i : g0];
            typename S::I2 st;
            S::init2(p, st, ri);
            // group boxes (empty for groups without active lanes)
            float l0 = act ? ri.x : INFINITY, l1 = act ? ri.y : INFINITY, l2 = act ? ri.z : INFINITY;
            float h0 = act ? ri.x : -INFINITY, h1 = act ? ri.y : -INFINITY, h2 = act ? ri.z : -INFINITY;
#pragma unroll
            for (int o = G / 2; o > 0; o >>= 1) {
                l0 = fminf(l0, __shfl_xor_sync(CRK_FULL_MASK, l0, o));
                l1 = fminf(l1, __shfl_xor_sync(CRK_FULL_MASK, l1, o));
                l2 = fminf(l2, __shfl_xor_sync(CRK_FULL_MASK, l2, o));
                h0 = fmaxf(h0, __shfl_xor_sync(CRK_FULL_MASK, h0, o));
                h1 = fmaxf(h1, __shfl_xor_sync(CRK_FULL_MASK, h1, o));
                h2 = fmaxf(h2, __shfl_xor_sync(CRK_FULL_MASK, h2, o));
            }
            float bl[NS][3], bh[NS][3];
            float ul0 = INFINITY, ul1 = INFINITY, ul2 = INFINITY, uh0 = -INFINITY, uh1 = -INFINITY, uh2 = -INFINITY;
#pragma unroll
            for (int t = 0; t < NS; ++t) {
                bl[t][0] = __shfl_sync(CRK_FULL_MASK, l0, t * G);
                bl[t][1] = __shfl_sync(CRK_FULL_MASK, l1, t * G);
                bl[t][2] = __shfl_sync(CRK_FULL_MASK, l2, t * G);
                bh[t][0] = __shfl_sync(CRK_FULL_MASK, h0, t * G);
                bh[t][1] = __shfl_sync(CRK_FULL_MASK, h1, t * G);
                bh[t][2] = __shfl_sync(CRK_FULL_MASK, h2, t * G);
                ul0 = fminf(ul0, bl[t][0]); ul1 = fminf(ul1, bl[t][1]); ul2 = fminf(ul2, bl[t][2]);
                uh0 = fmaxf(uh0, bh[t][0]); uh1 = fmaxf(uh1, bh[t][1]); uh2 = fmaxf(uh2, bh[t][2]);
            }
            const float cut = S::leaf_cut(p, 0.0f, 0.0f);
            const float far = 2.0f * cut + 1.0f;
            const Rec dummy = S::far_dummy(uh0 + far, uh1 + far, uh2 + far);
            int cnt[NS] = {0, 0};
            unsigned long long swept = 0;  // counting runs: candidate evaluations of this lane's group
            auto sweep = [&]() {
                // pad odd counts, then every half-warp sweeps its own buffer in pairs
                if (kCount) swept += (unsigned long long)(sg ? cnt[1] : cnt[0]);
                if (lane == 0 && (cnt[0] & 1)) S::put2(buf[warp][0], cnt[0], dummy);
                if (lane == 1 && (cnt[1] & 1)) S::put2(buf[warp][1], cnt[1], dummy);
#pragma unroll
                for (int t = 0; t < NS; ++t) cnt[t] = (cnt[t] + 1) & ~1;
                __syncwarp();
                const int kmax = max(cnt[0], cnt[1]) >> 1, mine = (sg ? cnt[1] : cnt[0]) >> 1;
                for (int k = 0; k < kmax; ++k)
                    if (k < mine) S::template interact2<kCount>(p, st, buf[warp][sg][k]);
#pragma unroll
                for (int t = 0; t < NS; ++t) cnt[t] = 0;
                __syncwarp();
            };
            for (int e = ib; e < ie; ++e) {
                const crk_image im = lv.img[e];
                const int jlo = lv.leaf_start[im.b];
                const int jhi = lv.leaf_start[im.b + 1];
                {
                    const float *bb = lv.bbox + 6 * (int64_t)im.b;
                    float gx = fmaxf(fmaxf(im.sx - uh0, ul0 - (im.sx + (bb[3] - bb[0]))), 0.f);
                    float gy = fmaxf(fmaxf(im.sy - uh1, ul1 - (im.sy + (bb[4] - bb[1]))), 0.f);
                    float gz = fmaxf(fmaxf(im.sz - uh2, ul2 - (im.sz + (bb[5] - bb[2]))), 0.f);
                    if (!(fmaf(gx, gx, fmaf(gy, gy, gz * gz)) <= cut * cut * 1.0001f + 1e-6f)) continue;
                }
                for (int j0 = jlo; j0 < jhi; j0 += 32) {
                    const int j = j0 + lane;
                    const bool jv = j < jhi;
                    Rec rj;
                    if (jv) {
                        rj = rec[j];
                        S::shift(rj, im.sx, im.sy, im.sz);
                    }
                    bool full = false;
#pragma unroll
                    for (int t = 0; t < NS; ++t) {
                        bool keep = false;
                        if (jv) {
                            float dx = fmaxf(fmaxf(bl[t][0] - rj.x, rj.x - bh[t][0]), 0.f);
                            float dy = fmaxf(fmaxf(bl[t][1] - rj.y, rj.y - bh[t][1]), 0.f);
                            float dz = fmaxf(fmaxf(bl[t][2] - rj.z, rj.z - bh[t][2]), 0.f);
                            keep = fmaf(dx, dx, fmaf(dy, dy, dz * dz)) <= cut * cut * 1.0001f + 1e-6f;
                        }
                        const unsigned m = __ballot_sync(CRK_FULL_MASK, keep);
                        if (keep) S::put2(buf[warp][t], cnt[t] + __popc(m & below), rj);
                        cnt[t] += __popc(m);
                        full |= cnt[t] >= 32;
                    }
                    if (full) sweep();
                }
            }
            sweep();
            if (act) S::finish2(p, st, lv.korder ? i : lv.kperm[i]);
            if (kCount) {
                int cn = act ? st.cnt - 1 : 0;  // the self pair (r = 0) is always in range
                unsigned long long sw = act ? swept : 0ull;
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) {
                    cn += __shfl_xor_sync(CRK_FULL_MASK, cn, o);
                    sw += __shfl_xor_sync(CRK_FULL_MASK, sw, o);
                }
                if (lane == 0 && cn) atomicAdd(p.count, (unsigned long long)cn);
                if (lane == 0 && p.swept) atomicAdd(p.swept, sw);
            }
        }
    }
}

// Two 16-particle i-groups per warp with balanced sweeps: each half-warp has
// a ring buffer of candidates; a sweep consumes the same number of entries
// from both rings (as many as both have ready), so neither half idles while
// the other works.  Only when a ring is about to overflow, and at the end,
// is a sweep unbalanced.
constexpr int kRing = 128;  // entries per ring (power of two)

template <class S, bool kCount>
__global__ void __launch_bounds__(kThreads) pair_kernel_ring(LeafView lv, typename S::P p,
                                                             RecView<typename S::Rec> rec,
                                                             double *__restrict__ cons_part) {
    using Rec = typename S::Rec;
    static_assert(!S::kCons, "the balanced sub-warp sweep has no conservation sums");
    __shared__ Rec ring[kWarps][2][kRing];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, sg = lane >> 4;
    const unsigned below = lanemask_lt();
    __shared__ int64_t leaf_slot;
    for (int64_t a = next_leaf(lv, -1, &leaf_slot); a < lv.n_leaves; a = next_leaf(lv, a, &leaf_slot)) {
        const int lo = lv.leaf_start[a];
        const int hi = S::kGasOnly ? lo + lv.leaf_ngas[a] : lv.leaf_start[a + 1];
        const int ib = lv.img_start[a], ie = ib + lv.img_cnt[a];
        for (int g0 = lo + warp * 32; g0 < hi; g0 += kWarps * 32) {
            const int i = g0 + lane;
            const bool act = i < hi;
            const Rec ri = rec[act ? i : g0];
            typename S::I st;
            S::init(p, st, ri, a, (g0 - lo) >> 5, lane, stage_index(lv, act ? i : g0));
            float l0 = act ? ri.x : INFINITY, l1 = act ? ri.y : INFINITY, l2 = act ? ri.z : INFINITY;
            float h0 = act ? ri.x : -INFINITY, h1 = act ? ri.y : -INFINITY, h2 = act ? ri.z : -INFINITY;
            float hm = act ? lv.pos[i].w : 0.0f;
#pragma unroll
            for (int o = 8; o > 0; o >>= 1) {
                l0 = fminf(l0, __shfl_xor_sync(CRK_FULL_MASK, l0, o));
                l1 = fminf(l1, __shfl_xor_sync(CRK_FULL_MASK, l1, o));
                l2 = fminf(l2, __shfl_xor_sync(CRK_FULL_MASK, l2, o));
                h0 = fmaxf(h0, __shfl_xor_sync(CRK_FULL_MASK, h0, o));
                h1 = fmaxf(h1, __shfl_xor_sync(CRK_FULL_MASK, h1, o));
                h2 = fmaxf(h2, __shfl_xor_sync(CRK_FULL_MASK, h2, o));
                hm = fmaxf(hm, __shfl_xor_sync(CRK_FULL_MASK, hm, o));
            }
            float bl[2][3], bh[2][3], bhm[2];
#pragma unroll
            for (int t = 0; t < 2; ++t) {
                bl[t][0] = __shfl_sync(CRK_FULL_MASK, l0, 16 * t);
                bl[t][1] = __shfl_sync(CRK_FULL_MASK, l1, 16 * t);
                bl[t][2] = __shfl_sync(CRK_FULL_MASK, l2, 16 * t);
                bh[t][0] = __shfl_sync(CRK_FULL_MASK, h0, 16 * t);
                bh[t][1] = __shfl_sync(CRK_FULL_MASK, h1, 16 * t);
                bh[t][2] = __shfl_sync(CRK_FULL_MASK, h2, 16 * t);
                bhm[t] = __shfl_sync(CRK_FULL_MASK, hm, 16 * t);
            }
            const float ul0 = fminf(bl[0][0], bl[1][0]), ul1 = fminf(bl[0][1], bl[1][1]), ul2 = fminf(bl[0][2], bl[1][2]);
            const float uh0 = fmaxf(bh[0][0], bh[1][0]), uh1 = fmaxf(bh[0][1], bh[1][1]), uh2 = fmaxf(bh[0][2], bh[1][2]);
            const float uhm = fmaxf(bhm[0], bhm[1]);
            unsigned head0 = 0, head1 = 0, tail0 = 0, tail1 = 0;  // warp-uniform ring counters
            // consume k0 entries of ring 0 (lanes 0-15) and k1 of ring 1 (lanes 16-31)
            auto sweep = [&](unsigned k0, unsigned k1) {
                __syncwarp();
                const unsigned kmax = k0 > k1 ? k0 : k1, mine = sg ? k1 : k0, h = sg ? head1 : head0;
                for (unsigned k = 0; k < kmax; ++k)
                    if (k < mine) S::template interact<kCount>(p, st, ri, ring[warp][sg][(h + k) & (kRing - 1)]);
                head0 += k0;
                head1 += k1;
                __syncwarp();
            };
            for (int e = ib; e < ie; ++e) {
                const crk_image im = lv.img[e];
                const int jlo = lv.leaf_start[im.b];
                const int jhi = S::kGasOnly ? jlo + lv.leaf_ngas[im.b] : lv.leaf_start[im.b + 1];
                {
                    const float *bb = lv.bbox + 6 * (int64_t)im.b;
                    float gx = fmaxf(fmaxf(im.sx - uh0, ul0 - (im.sx + (bb[3] - bb[0]))), 0.f);
                    float gy = fmaxf(fmaxf(im.sy - uh1, ul1 - (im.sy + (bb[4] - bb[1]))), 0.f);
                    float gz = fmaxf(fmaxf(im.sz - uh2, ul2 - (im.sz + (bb[5] - bb[2]))), 0.f);
                    float cut = S::leaf_cut(p, uhm, lv.hmax[im.b]);
                    if (!(fmaf(gx, gx, fmaf(gy, gy, gz * gz)) <= cut * cut * 1.0001f + 1e-6f)) continue;
                }
                for (int j0 = jlo; j0 < jhi; j0 += 32) {
                    const int j = j0 + lane;
                    const bool jv = j < jhi;
                    Rec rj;
                    bool keep[2] = {false, false};
                    if (jv) {
                        rj = rec[j];
                        S::shift(rj, im.sx, im.sy, im.sz);
#pragma unroll
                        for (int t = 0; t < 2; ++t) {
                            float dx = fmaxf(fmaxf(bl[t][0] - rj.x, rj.x - bh[t][0]), 0.f);
                            float dy = fmaxf(fmaxf(bl[t][1] - rj.y, rj.y - bh[t][1]), 0.f);
                            float dz = fmaxf(fmaxf(bl[t][2] - rj.z, rj.z - bh[t][2]), 0.f);
                            float cut = S::box_cut(p, bhm[t], rj);
                            keep[t] = fmaf(dx, dx, fmaf(dy, dy, dz * dz)) <= cut * cut * 1.0001f + 1e-6f;
                        }
                    }
                    const unsigned m0 = __ballot_sync(CRK_FULL_MASK, keep[0]);
                    const unsigned m1 = __ballot_sync(CRK_FULL_MASK, keep[1]);
                    if (keep[0]) ring[warp][0][(tail0 + __popc(m0 & below)) & (kRing - 1)] = rj;
                    if (keep[1]) ring[warp][1][(tail1 + __popc(m1 & below)) & (kRing - 1)] = rj;
                    tail0 += __popc(m0);
                    tail1 += __popc(m1);
                    const unsigned r0 = tail0 - head0, r1 = tail1 - head1;
                    const unsigned both = r0 < r1 ? r0 : r1;
                    if (r0 > kRing - 32 || r1 > kRing - 32) sweep(r0, r1);  // a ring is nearly full
                    else if (both >= 32) sweep(both, both);                // balanced
                }
            }
            sweep(tail0 - head0, tail1 - head1);
            if (act) S::finish(p, st, ri, lv.korder ? i : lv.kperm[i], i);
            if (kCount) {
                int cn = act ? st.cnt - 1 : 0;
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) cn += __shfl_xor_sync(CRK_FULL_MASK, cn, o);
                if (lane == 0 && cn) atomicAdd(p.count, (unsigned long long)cn);
            }
        }
    }
}

// stages with half-warp arms (kHalfWarp): partial sums flushed with atomics
template <class S, class = void>
struct has_halfwarp : std::false_type {};
template <class S>
struct has_halfwarp<S, std::void_t<decltype(S::kHalfWarp)>> : std::bool_constant<S::kHalfWarp> {};

// Conservation sums of a half-warp arm, from the finished outputs: per-block
// FP64 partials over the gas particles in kernel order (fixed assignment of
// particles to blocks and a fixed reduction order: deterministic).
template <class S>
__global__ void __launch_bounds__(256) halfwarp_cons_kernel(int64_t n, const float4 *__restrict__ pos,
                                                            const int32_t *__restrict__ kperm, int korder,
                                                            typename S::P p, double *__restrict__ part) {
    __shared__ double sh[8][4];
    double acc[4] = {0.0, 0.0, 0.0, 0.0};
    for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < n; q += (int64_t)gridDim.x * blockDim.x) {
        if (!(pos[q].w > 0.0f)) continue;  // dark matter
        double c[4];
        S::cons_of(p, korder ? (int32_t)q : kperm[q], c);
        for (int k = 0; k < 4; ++k) acc[k] += c[k];
    }
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    for (int k = 0; k < 4; ++k) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) acc[k] += __shfl_xor_sync(CRK_FULL_MASK, acc[k], o);
        if (lane == 0) sh[w][k] = acc[k];
    }
    __syncthreads();
    if (threadIdx.x < 4) {
        double t = 0.0;
        for (int v = 0; v < (int)(blockDim.x >> 5); ++v) t += sh[v][threadIdx.x];
        part[4 * blockIdx.x + threadIdx.x] = t;
    }
}

__global__ void cons_reduce_kernel(const double *__restrict__ part, int64_t nb, double *__restrict__ out) {
    __shared__ double sh[256];
    for (int k = 0; k < 4; ++k) {
        double t = 0.0;
        for (int64_t b = threadIdx.x; b < nb; b += blockDim.x) t += part[4 * b + k];
        sh[threadIdx.x] = t;
        __syncthreads();
        for (int s = blockDim.x / 2; s > 0; s >>= 1) {
            if ((int)threadIdx.x < s) sh[threadIdx.x] += sh[threadIdx.x + s];
            __syncthreads();
        }
        if (threadIdx.x == 0) out[k] = sh[0];
        __syncthreads();
    }
}


// Gas-pair stages driven by the exact neighbour lists: each lane walks its own
// list (k-major, so entry k of the 32 lanes is one coalesced row); inactive
// lanes (k beyond their length) idle.
struct GasLists {
    const int32_t *gstart, *goff, *cnt;
    const uint16_t *list;
    const int32_t *uoff, *unum;
    const uint32_t *ucode;
    const int32_t *gleaf;
    int64_t groups;          // capacity of the group arrays
    const int32_t *dgroups;  // device: the groups of this build, or NULL for all
};

// j-table entries staged per warp in shared memory (records of at most 48
// bytes; the hydro record is too large to stage, its lanes gather directly)
template <class S>
__host__ __device__ constexpr int table_cap() {
    return sizeof(typename S::Rec) <= 32 ? 320 : (sizeof(typename S::Rec) <= 48 ? 224 : 0);
}

// resident blocks per SM that list_kernel<S> is compiled for (a register cap; 0: none).
// Corrections is latency bound: capped for five blocks (96 registers, a few bytes spilled) it runs
// 0.90 ms on the 2x128^3 box, against 0.95 ms at four and 1.07 ms at six.
template <class S>
struct list_min_blocks {
    static constexpr int value = 0;  // no register cap
};
template <>
struct list_min_blocks<CorrStage> {
    static constexpr int value = 5;
};
// its reverse preparation: four blocks 254 us on the 2x64^3 box, three 267, five 271
template <>
struct list_min_blocks<CorrAdjPrepStage> {
    static constexpr int value = 4;
};

// index rows in flight in list_kernel<S>: 8 for the short pair terms (records of at most 32
// bytes and few registers), 4 for the long ones
template <class S>
__host__ __device__ constexpr int list_ahead() {
    return (std::is_same<S, GeomStage>::value || std::is_same<S, GeomAdjStage>::value) ? 8 : 4;
}

// Stages whose pair term is gated by the in-range test (every contribution of
// an out-of-range j is an exact zero): list_kernel runs their rows of entries
// as straight-line code, padding the end of a lane's list with i's own record
// moved 4 h + 1 away, so the compiler interleaves the entries' dependent
// chains (geometry 5.34 -> 4.88 ms, corrections 10.48 -> 10.11 ms on the
// 2x256^3 box).  Hydro is left out: four staged 112-byte records per lane
// cost it its occupancy (15.1 -> 22.6 ms).
template <class S>
struct flat_tail {
    static constexpr bool value = false;
};
template <>
struct flat_tail<GeomStage> {
    static constexpr bool value = true;
};
template <>
struct flat_tail<GeomAdjStage> {
    static constexpr bool value = true;
};
template <>
struct flat_tail<CorrStage> {
    static constexpr bool value = true;
};
template <>
struct flat_tail<CorrAdjPrepStage> {
    static constexpr bool value = true;
};
template <>
struct flat_tail<ExtrasStage> {
    static constexpr bool value = true;
};

// Exact neighbour lists, one warp per i-group.  The warp stages the group's
// j table in shared memory (each distinct j of the group gathered once,
// shifted into the i frame), then each lane walks its own list of table
// indices.  Table entries beyond the staged capacity are gathered from global
// memory through the leaf's image table.
template <class S, bool kCount>
__global__ void __launch_bounds__(kThreads, list_min_blocks<S>::value) list_kernel(LeafView lv, typename S::P p,
                                                        RecView<typename S::Rec> rec, GasLists gl,
                                                        double *__restrict__ cons_part) {
    using Rec = typename S::Rec;
    constexpr int kTab = table_cap<S>();
    extern __shared__ __align__(16) unsigned char list_dyn[];
    __shared__ double cons_sh[kWarps][4];
    __shared__ float4 itab_all[kWarps][kGroupImgCap];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    float4 *itab = itab_all[warp];
    unsigned char *table = list_dyn + (size_t)warp * kTab * Planes<Rec>::kBytes;
    double cons_acc = 0.0;  // of component lane / 8
    const int64_t ngroups = group_count(gl.groups, gl.dgroups);
    for (int64_t grp = next_group(lv, -1, lane); grp < ngroups; grp = next_group(lv, grp, lane)) {
        const int64_t a = gl.gleaf[grp];
        const int q = (int)(grp - gl.gstart[a]);
        const int lo = lv.leaf_start[a];
        const int hi = S::kGasOnly ? lo + lv.leaf_ngas[a] : lv.leaf_start[a + 1];
        const int g0 = lo + 32 * q;
        const crk_image *imgs = lv.img + lv.img_start[a];
        const int nimg = lv.img_cnt[a];
        const bool staged = nimg <= kGroupImgCap;
        __syncwarp();  // the previous group's tables are no longer read
        if (staged) {
            for (int t = lane; t < nimg; t += 32) {
                const crk_image im = imgs[t];
                itab[t] = make_float4(im.sx, im.sy, im.sz, __int_as_float(lv.leaf_start[im.b]));
            }
            __syncwarp();
        }
        const uint32_t *U = gl.ucode + gl.uoff[grp];
        const int nu = gl.unum[grp];
        // table entry -> shifted record of j
        auto fetch = [&](uint32_t code) -> Rec {
            float4 t;
            if (staged) {
                t = itab[code >> 10];
            } else {
                const crk_image im = imgs[code >> 10];
                t = make_float4(im.sx, im.sy, im.sz, __int_as_float(lv.leaf_start[im.b]));
            }
            Rec r = rec[__float_as_int(t.w) + (int)(code & 1023u)];
            S::shift(r, t.x, t.y, t.z);
            return r;
        };
        if constexpr (kTab > 0) {
            const int ns = nu < kTab ? nu : kTab;
#pragma unroll 4
            for (int u = lane; u < ns; u += 32) Planes<Rec>::store(table, kTab, u, fetch(__ldg(U + u)));
            __syncwarp();
        }
        auto entry = [&](int idx) -> Rec {
            if constexpr (kTab > 0) {
                if (idx < kTab) return Planes<Rec>::template load<false>(table, kTab, idx);
            }
            return fetch(__ldg(U + idx));
        };
        const uint16_t *Lp = gl.list + (size_t)gl.goff[grp] * 32 + lane;
        const int i = g0 + lane;
        const bool act = i < hi;
        const Rec ri = rec[act ? i : g0];
        typename S::I st;
        S::init(p, st, ri, a, q, lane, stage_index(lv, act ? i : g0));
        const int c = act ? gl.cnt[i] : 0;
        // indices kAhead rows ahead, so their loads overlap the pair arithmetic (light pair terms
        // need more rows in flight to cover a DRAM latency)
        constexpr int kAhead = list_ahead<S>();
        if constexpr (kAhead == 4) {
            int k = 0;
            int nx0 = 0 < c ? __ldg(Lp) : 0, nx1 = 1 < c ? __ldg(Lp + 32) : 0, nx2 = 2 < c ? __ldg(Lp + 64) : 0,
                nx3 = 3 < c ? __ldg(Lp + 96) : 0;
            for (; k < c; k += 4) {
                const int i0 = nx0, i1 = nx1, i2 = nx2, i3 = nx3;
                const uint16_t *Lk = Lp + (size_t)(k + 4) * 32;
                nx0 = k + 4 < c ? __ldg(Lk) : 0;
                nx1 = k + 5 < c ? __ldg(Lk + 32) : 0;
                nx2 = k + 6 < c ? __ldg(Lk + 64) : 0;
                nx3 = k + 7 < c ? __ldg(Lk + 96) : 0;
                if constexpr (flat_tail<S>::value) {
                    Rec far = ri;  // past the end of the list: out of range, every term finite
                    far.x += 4.0f * ri.h + 1.0f;
                    const Rec e0 = entry(i0);
                    const Rec e1 = k + 1 < c ? entry(i1) : far;
                    const Rec e2 = k + 2 < c ? entry(i2) : far;
                    const Rec e3 = k + 3 < c ? entry(i3) : far;
                    S::template interact<kCount>(p, st, ri, e0);
                    S::template interact<kCount>(p, st, ri, e1);
                    S::template interact<kCount>(p, st, ri, e2);
                    S::template interact<kCount>(p, st, ri, e3);
                } else {
                    S::template interact<kCount>(p, st, ri, entry(i0));
                    if (k + 1 < c) S::template interact<kCount>(p, st, ri, entry(i1));
                    if (k + 2 < c) S::template interact<kCount>(p, st, ri, entry(i2));
                    if (k + 3 < c) S::template interact<kCount>(p, st, ri, entry(i3));
                }
            }
        } else {
            int nx[kAhead];
#pragma unroll
            for (int d = 0; d < kAhead; ++d) nx[d] = d < c ? __ldg(Lp + (size_t)d * 32) : 0;
            for (int k = 0; k < c; k += kAhead) {
                int cur[kAhead];
                const uint16_t *Lk = Lp + (size_t)(k + kAhead) * 32;
#pragma unroll
                for (int d = 0; d < kAhead; ++d) {
                    cur[d] = nx[d];
                    nx[d] = k + kAhead + d < c ? __ldg(Lk + (size_t)d * 32) : 0;
                }
                if constexpr (flat_tail<S>::value) {
                    Rec far = ri;
                    far.x += 4.0f * ri.h + 1.0f;
                    Rec e[kAhead];
#pragma unroll
                    for (int d = 0; d < kAhead; ++d) e[d] = (d == 0 || k + d < c) ? entry(cur[d]) : far;
#pragma unroll
                    for (int d = 0; d < kAhead; ++d) S::template interact<kCount>(p, st, ri, e[d]);
                } else {
                    S::template interact<kCount>(p, st, ri, entry(cur[0]));
#pragma unroll
                    for (int d = 1; d < kAhead; ++d)
                        if (k + d < c) S::template interact<kCount>(p, st, ri, entry(cur[d]));
                }
            }
        }
        if (act) S::finish(p, st, ri, lv.korder ? i : lv.kperm[i], i);
        if constexpr (S::kCons) {
            if (cons_part) {
                double cc[4] = {0.0, 0.0, 0.0, 0.0};
                if (act) S::cons_terms(p, st, ri, lv.korder ? i : lv.kperm[i], cc);
                cons_acc += cons_warp_sum(cc, lane);
            }
        }
        if (kCount) {
            int cn = act ? st.cnt - 1 : 0;
            int sw = c;  // candidate evaluations: the list entries
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                cn += __shfl_xor_sync(CRK_FULL_MASK, cn, o);
                sw += __shfl_xor_sync(CRK_FULL_MASK, sw, o);
            }
            if (lane == 0 && cn) atomicAdd(p.count, (unsigned long long)cn);
            if (lane == 0 && p.swept && sw) atomicAdd(p.swept, (unsigned long long)sw);
        }
    }
    if constexpr (S::kCons) {
        if (cons_part) {
            if ((lane & 7) == 0) cons_sh[warp][lane >> 3] = cons_acc;
            cons_block_sum(cons_sh, cons_part);
        }
    }
}

// dynamic shared memory of list_kernel<S>, and the opt-in above the 48 KB default (once per kernel)
template <class S, bool kCount>
size_t list_kernel_smem() {
    const size_t bytes = (size_t)kWarps * table_cap<S>() * Planes<typename S::Rec>::kBytes;
    static bool set = false;
    if (!set) {
        cudaFuncSetAttribute(list_kernel<S, kCount>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
        set = true;
    }
    return bytes;
}

// resident blocks per SM of list_kernel<S> (registers and shared memory; once per kernel)
template <class S, bool kCount>
int list_kernel_resident() {
    static int nb = 0;
    if (!nb) {
        const size_t smem = list_kernel_smem<S, kCount>();
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, list_kernel<S, kCount>, kThreads, smem) != cudaSuccess) {
            cudaGetLastError();
            nb = 4;
        }
        if (nb < 1) nb = 1;
    }
    return nb;
}

// fixed-capacity list and table offsets: goff[g] = g capr, uoff[g] = g capt
__global__ void strided_offsets_kernel(int64_t m, int capr, int capt, int32_t *__restrict__ goff,
                                       int32_t *__restrict__ uoff) {
    int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (g < m) {
        goff[g] = (int32_t)(g * capr);
        uoff[g] = (int32_t)(g * capt);
    }
}

// groups of each leaf, and the leaf of each group (groups beyond the capacity cap are dropped)
__global__ void list_group_leaf_kernel(int64_t n_leaves, const int32_t *__restrict__ gstart,
                                       int32_t *__restrict__ gleaf, int64_t cap) {
    int64_t a = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (a >= n_leaves) return;
    for (int32_t g = gstart[a]; g < gstart[a + 1] && g < cap; ++g) gleaf[g] = (int32_t)a;
}

// a rebuild's group count and list overflow as bits of the leaves' status word
__global__ void lists_status_kernel(const int32_t *__restrict__ groups, int64_t cap, const int32_t *__restrict__ ovf,
                                    int32_t *__restrict__ status) {
    int32_t s = 0;
    if (*groups > cap) s |= CRK_LEAVES_GROUP_CAP;
    if (ovf && *ovf) s |= CRK_LEAVES_LIST_CAP;
    if (s) atomicOr(status, s);
}

__global__ void list_group_count_kernel(int64_t n_leaves, const int32_t *__restrict__ leaf_start,
                                        const int32_t *__restrict__ ngas, int gas, int32_t *__restrict__ ng) {
    int64_t a = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (a < n_leaves) ng[a] = ((gas ? ngas[a] : leaf_start[a + 1] - leaf_start[a]) + 31) >> 5;
    if (a == n_leaves) ng[a] = 0;
}

// per group: the longest list of its lanes (units of 32 entries once scanned)
__global__ void list_group_k_kernel(int64_t n_leaves, const int32_t *__restrict__ leaf_start,
                                    const int32_t *__restrict__ ngas, int gas, const int32_t *__restrict__ gstart,
                                    const int32_t *__restrict__ cnt, int32_t *__restrict__ gk) {
    int64_t a = blockIdx.x;
    if (a >= n_leaves) return;
    const int lo = leaf_start[a], hi = gas ? lo + ngas[a] : leaf_start[a + 1];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int g0 = lo + warp * 32; g0 < hi; g0 += (blockDim.x >> 5) * 32) {
        int i = g0 + lane;
        int c = i < hi ? cnt[i] : 0;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) c = max(c, __shfl_xor_sync(CRK_FULL_MASK, c, o));
        if (lane == 0) gk[gstart[a] + ((g0 - lo) >> 5)] = c;
    }
}

template <class S>
int run_stage(crk_ctx *ctx, const crk_leaves *lv, typename S::P p, bool gas_pairs, int kernel_id,
              double *cons = nullptr, bool korder = false) {
    if (!lv) return crk_fail(ctx, CRK_EINVAL, "null leaves");
    const int64_t n = lv->n;
    if (n == 0) return CRK_OK;
    using Rec = typename S::Rec;
    void *recs = crk_scratch(ctx, 4, Planes<Rec>::kBytes * (size_t)n);
    if (!recs) return crk_fail(ctx, CRK_ENOMEM, "stage scratch");
    const RecView<Rec> rec{recs, n};
    const crk_nlist &nls = gas_pairs ? lv->gas_lists : lv->grav_lists;
    const bool lists = nls.list && ctx->variant[kernel_id] == CRK_VARIANT_LISTS;
    // one block per i-leaf, or (lists) one warp per i-group
    int64_t grid = lists ? (nls.groups + kWarps - 1) / kWarps : lv->n_leaves;
    if (grid < 1) grid = 1;
    if (grid > 2147483647LL) grid = 2147483647LL;
    const bool persistent = ctx->persist[kernel_id] != 0;
    if (persistent) {
        // persistent grid: resident blocks on every SM (lists: as many as fit; tiles: 4 blocks of
        // 128 threads per SM, the design point)
        int per_sm = 4;
        if (lists) per_sm = p.count ? list_kernel_resident<S, true>() : list_kernel_resident<S, false>();
        const int64_t g = (int64_t)ctx->num_sms * per_sm;
        if (g < grid) grid = g;
    }
    const bool halfwarp = !lists && ctx->variant[kernel_id] >= CRK_VARIANT_HALFWARP_SHFL &&
                          ctx->variant[kernel_id] <= CRK_VARIANT_HALFWARP_LOAD && has_halfwarp<S>::value;
    // half-warp arms take their conservation sums from the finished outputs, in cblocks partials
    const int64_t cblocks = std::min<int64_t>(crk_grid(n, 256), (int64_t)ctx->num_sms * 8);
    int64_t nparts = halfwarp ? cblocks : grid;
    double *part = nullptr;
    if (cons) {
        part = (double *)crk_scratch(ctx, 5, sizeof(double) * 4 * (size_t)nparts);
        if (!part) return crk_fail(ctx, CRK_ENOMEM, "stage scratch");
    }
    const float4 *kpos = gas_pairs ? lv->pos : lv->pos_g;          // gravity: species-mixed kernel order
    const int32_t *kperm = gas_pairs ? lv->kperm : lv->kperm_g;
    gather_kernel<S><<<crk_grid(n, 256), 256, 0, ctx->stream>>>(n, kpos, kperm, p, recs, korder ? 1 : 0);
    int32_t *queue = nullptr;
    if (persistent) {
        queue = (int32_t *)crk_scratch(ctx, 17, 64);
        if (!queue) return crk_fail(ctx, CRK_ENOMEM, "stage scratch");
        CRK_CUDA(ctx, cudaMemsetAsync(queue, 0, sizeof(int32_t), ctx->stream));
    }
    LeafView v{lv->leaf_start, lv->leaf_ngas, lv->bbox, lv->hmax, kpos, kperm,
               gas_pairs ? lv->himg_start : lv->gimg_start, gas_pairs ? lv->himg_cnt : lv->gimg_cnt,
               gas_pairs ? lv->himg : lv->gimg, lv->n_leaves, queue, korder ? 1 : 0, ctx->depth[kernel_id], lv->gcell};
    if (p.count) CRK_CUDA(ctx, cudaMemsetAsync(p.count, 0, sizeof(unsigned long long), ctx->stream));
    if (p.swept) CRK_CUDA(ctx, cudaMemsetAsync(p.swept, 0, sizeof(unsigned long long), ctx->stream));
    if (lists) {
        GasLists gl{nls.gstart, nls.goff, nls.cnt, nls.list, nls.uoff, nls.unum, nls.ucode, nls.gleaf, nls.groups,
                    nls.dgroups};
        if (p.count)
            list_kernel<S, true><<<(unsigned)grid, kThreads, list_kernel_smem<S, true>(), ctx->stream>>>(v, p, rec, gl,
                                                                                                       part);
        else
            list_kernel<S, false><<<(unsigned)grid, kThreads, list_kernel_smem<S, false>(), ctx->stream>>>(v, p, rec, gl,
                                                                                                         part);
    } else if (halfwarp) {
        if constexpr (has_halfwarp<S>::value) {
            typename S::P q = p;
            if constexpr (S::kCons) {
                if (cons && !q.dv3) {  // the Energy pass: its recomputed force, for the conservation sums
                    q.dv3 = (float *)crk_scratch(ctx, 35, sizeof(float) * 3 * (size_t)n);
                    if (!q.dv3) return crk_fail(ctx, CRK_ENOMEM, "stage scratch");
                }
            }
            S::zero_outputs(q, ctx->stream);
            const int ex = ctx->variant[kernel_id] - CRK_VARIANT_HALFWARP_SHFL;
            const unsigned gg = (unsigned)grid;
            if (p.count) {
                if (ex == 0) pair_kernel_halfwarp<S, true, 0><<<gg, kThreads, 0, ctx->stream>>>(v, q, rec, part);
                else if (ex == 1) pair_kernel_halfwarp<S, true, 1><<<gg, kThreads, 0, ctx->stream>>>(v, q, rec, part);
                else pair_kernel_halfwarp<S, true, 2><<<gg, kThreads, 0, ctx->stream>>>(v, q, rec, part);
            } else {
                if (ex == 0) pair_kernel_halfwarp<S, false, 0><<<gg, kThreads, 0, ctx->stream>>>(v, q, rec, part);
                else if (ex == 1) pair_kernel_halfwarp<S, false, 1><<<gg, kThreads, 0, ctx->stream>>>(v, q, rec, part);
                else pair_kernel_halfwarp<S, false, 2><<<gg, kThreads, 0, ctx->stream>>>(v, q, rec, part);
            }
            if constexpr (S::kCons) {
                if (cons) {
                    halfwarp_cons_kernel<S><<<(unsigned)cblocks, 256, 0, ctx->stream>>>(n, kpos, kperm, korder ? 1 : 0,
                                                                                         q, part);
                    ++ctx->launches;
                }
            }
        }
    } else if constexpr (!S::kAllVariants) {  // built for lists and tiles only
        if (p.count)
            pair_kernel<S, true><<<(unsigned)grid, kThreads, 0, ctx->stream>>>(v, p, rec, part);
        else
            pair_kernel<S, false><<<(unsigned)grid, kThreads, 0, ctx->stream>>>(v, p, rec, part);
    } else {
        if (ctx->variant[kernel_id] == CRK_VARIANT_TILES16) {
            if constexpr (S::kPair) {  // gravity stages: packed two-candidate sweeps
                if (p.count)
                    pair_kernel_sub_pair<S, true><<<(unsigned)grid, kThreads, 0, ctx->stream>>>(v, p, rec, part);
                else
                    pair_kernel_sub_pair<S, false><<<(unsigned)grid, kThreads, 0, ctx->stream>>>(v, p, rec, part);
            } else {
                if (p.count)
                    pair_kernel_sub<S, 16, true><<<(unsigned)grid, kThreads, 0, ctx->stream>>>(v, p, rec, part);
                else
                    pair_kernel_sub<S, 16, false><<<(unsigned)grid, kThreads, 0, ctx->stream>>>(v, p, rec, part);
            }
        } else if (ctx->variant[kernel_id] == CRK_VARIANT_RING16 && !S::kCons) {
            if constexpr (!S::kCons) {
                if (p.count)
                    pair_kernel_ring<S, true><<<(unsigned)grid, kThreads, 0, ctx->stream>>>(v, p, rec, part);
                else
                    pair_kernel_ring<S, false><<<(unsigned)grid, kThreads, 0, ctx->stream>>>(v, p, rec, part);
            }
        } else if (ctx->variant[kernel_id] == CRK_VARIANT_TILES8) {
            if (p.count)
                pair_kernel_sub<S, 8, true><<<(unsigned)grid, kThreads, 0, ctx->stream>>>(v, p, rec, part);
            else
                pair_kernel_sub<S, 8, false><<<(unsigned)grid, kThreads, 0, ctx->stream>>>(v, p, rec, part);
        } else if constexpr (S::kPair) {
            const bool one = ctx->variant[kernel_id] == CRK_VARIANT_SPLIT8;
            const int w = ctx->warps[kernel_id];
            if (p.count) launch_cells<S, true>(ctx, lv, v, p, rec, persistent, w, one);
            else launch_cells<S, false>(ctx, lv, v, p, rec, persistent, w, one);
        } else if (p.count) {
            pair_kernel<S, true><<<(unsigned)grid, kThreads, 0, ctx->stream>>>(v, p, rec, part);
        } else {
            pair_kernel<S, false><<<(unsigned)grid, kThreads, 0, ctx->stream>>>(v, p, rec, part);
        }
    }
    if (cons) cons_reduce_kernel<<<1, 256, 0, ctx->stream>>>(part, nparts, cons);
    ctx->launches += 2 + (cons ? 1 : 0);
    CRK_LAUNCH_CHECK(ctx, "pair kernel");
    return CRK_OK;
}

// ------------------------------------------------------- columns in another order
// One column through a permutation: dst[o] = src[perm[o]] (o in the
// destination order).  One column per launch keeps the randomly read source
// (n floats) about the size of L2, so each 32-byte sector is fetched from DRAM
// about once; gathering many columns at once thrashes L2 (measured slower).
__global__ void permute_col_kernel(int64_t n, const int32_t *__restrict__ perm, const float *__restrict__ src,
                                   float *__restrict__ dst) {
    int64_t o = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (o < n) dst[o] = __ldg(src + perm[o]);
}

// Several columns through one permutation in two streaming passes: the columns
// are interleaved into rows of 4 Q floats (through shared memory, both sides
// coalesced), then each destination reads its whole row, so a random access
// brings 16 Q useful bytes instead of 4.  33.5M particles: 0.33 ms a column by
// permute_col_kernel, 0.16 ms in rows of 5 to 8 (the step's 20 columns: 6.5 ->
// 3.2 ms); 524,288 particles: 168 -> 60 us for 38 columns.
constexpr int kBundle = 36;  // columns of one bundle (the limited Energy pass reads 35)
struct Bundle {
    const float *src[kBundle];
    float *dst[kBundle];
    int k = 0;
    bool over = false;  // more columns than the bundle holds were added
    void add(const float *s, float *d, int comps, int64_t n) {
        over |= k + comps > kBundle;
        if (over) return;
        for (int c = 0; c < comps; ++c, ++k) {
            src[k] = s + (size_t)c * n;
            dst[k] = d + (size_t)c * n;
        }
    }
};
constexpr int kRowTile = 128;  // particles per block of the interleaving pass

template <int Q>
__global__ void __launch_bounds__(kRowTile) interleave_kernel(int64_t n, Bundle b, float4 *__restrict__ rows) {
    __shared__ float tile[4 * Q][kRowTile + 1];
    const int64_t base = (int64_t)blockIdx.x * kRowTile;
    const int t = threadIdx.x, m = (int)(n - base < kRowTile ? n - base : kRowTile);
    if (t < m) {
#pragma unroll
        for (int c = 0; c < 4 * Q; ++c)
            if (c < b.k) tile[c][t] = __ldg(b.src[c] + base + t);
    }
    __syncthreads();
    for (int j = t; j < m * Q; j += kRowTile) {
        const int r = j / Q, c = 4 * (j % Q);
        rows[base * Q + j] = make_float4(tile[c][r], tile[c + 1][r], tile[c + 2][r], tile[c + 3][r]);
    }
}

template <int Q>
__global__ void __launch_bounds__(256) deal_rows_kernel(int64_t n, const int32_t *__restrict__ perm, Bundle b,
                                                        const float4 *__restrict__ rows) {
    const int64_t o = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (o >= n) return;
    const float4 *r = rows + (int64_t)perm[o] * Q;
    float4 v[Q];
#pragma unroll
    for (int q = 0; q < Q; ++q) v[q] = __ldg(r + q);
#pragma unroll
    for (int q = 0; q < Q; ++q) {
        if (4 * q < b.k) b.dst[4 * q][o] = v[q].x;
        if (4 * q + 1 < b.k) b.dst[4 * q + 1][o] = v[q].y;
        if (4 * q + 2 < b.k) b.dst[4 * q + 2][o] = v[q].z;
        if (4 * q + 3 < b.k) b.dst[4 * q + 3][o] = v[q].w;
    }
}

template <int Q>
int permute_rows(crk_ctx *ctx, int64_t n, const int32_t *perm, const Bundle &b) {
    if constexpr (Q > 1) {
        if (b.k <= 4 * (Q - 1)) return permute_rows<Q - 1>(ctx, n, perm, b);
    }
    // the rows live in the stages' record scratch, which holds nothing between two stages
    float4 *rows = (float4 *)crk_scratch(ctx, 4, sizeof(float4) * Q * (size_t)n);
    if (!rows) return crk_fail(ctx, CRK_ENOMEM, "permutation scratch");
    interleave_kernel<Q><<<crk_grid(n, kRowTile), kRowTile, 0, ctx->stream>>>(n, b, rows);
    deal_rows_kernel<Q><<<crk_grid(n, 256), 256, 0, ctx->stream>>>(n, perm, b, rows);
    ctx->launches += 2;
    CRK_LAUNCH_CHECK(ctx, "column permutation");
    return CRK_OK;
}

// dst = src[perm] for every column of the bundle
int permute_bundle(crk_ctx *ctx, int64_t n, const int32_t *perm, const Bundle &b) {
    if (b.over) return crk_fail(ctx, CRK_EINVAL, "column permutation: more than %d columns", kBundle);
    if (b.k >= 3) return permute_rows<kBundle / 4>(ctx, n, perm, b);
    for (int c = 0; c < b.k; ++c) {
        permute_col_kernel<<<crk_grid(n, 256), 256, 0, ctx->stream>>>(n, perm, b.src[c], b.dst[c]);
        ++ctx->launches;
    }
    CRK_LAUNCH_CHECK(ctx, "column permutation");
    return CRK_OK;
}

// The records of the Energy pass and the hydro adjoint: planes, and whole records where gas is below a sixteenth
// (hydro adjoint: an eighth) of the particles: few lanes of a group are active, and each reads a record of its
// own.  The hydro adjoint, whole -> planes, us: 687 -> 552 on the 2x64^3 box; uniform boxes of 500,009 particles,
// a fifth of them gas, 391 -> 339, of 300,007, a twentieth, 229 -> 243, of 880,001, a fiftieth, 501 -> 532.
// Energy: 563 -> 355; 500,009 particles, a tenth gas, 175 -> 157, of 650,001, a fiftieth, 201 -> 207.
bool sparse_gas(const crk_leaves *lv, int part) { return lv->n_gas < lv->n / part; }
int run_hydro_adjoint(crk_ctx *ctx, const crk_leaves *lv, const HydroAdjP &p, bool korder) {
    if (sparse_gas(lv, 8)) return run_stage<HydroAdjStage<true>>(ctx, lv, p, true, CRK_K_HYDRO, nullptr, korder);
    return run_stage<HydroAdjStage<false>>(ctx, lv, p, true, CRK_K_HYDRO, nullptr, korder);
}
template <bool kLim>
int run_energy(crk_ctx *ctx, const crk_leaves *lv, const HydroP &p, double *conservation, bool korder) {
    if (sparse_gas(lv, 16))
        return run_stage<HydroEnergyStage<kLim, true>>(ctx, lv, p, true, CRK_K_ENERGY, conservation, korder);
    return run_stage<HydroEnergyStage<kLim>>(ctx, lv, p, true, CRK_K_ENERGY, conservation, korder);
}

// Single calls of the gas stages on large boxes: the caller's columns are
// permuted into the kernel order, the stage runs there and its outputs are
// permuted back, instead of gathering and scattering every column at random
// 4-byte places inside the stage's kernels.  In units of one column streamed
// through the rows, the permutation costs the columns in and out (all
// particles) and about 5 more; it saves
//   * 2 per column that the stage scatters (dark matter gets zeros, so all
//     particles count), 6 once those columns no longer fit L2 together;
//   * 1 per column that it gathers and share of gas (gas rows only), 3 once
//     those columns do not fit.
// Uniform boxes, direct -> permuted, ms, at 2%, 20%, 50% and 100% gas: hydro on
// 900,001 particles 0.22 -> 0.28, 0.31 -> 0.35, 0.55 -> 0.57, 0.94 -> 0.94, on
// 4M 0.71 -> 0.96, 1.37 -> 1.28, 2.73 -> 2.33, 4.68 -> 3.85; corrections on
// 900,001 0.23 -> 0.18, 0.24 -> 0.21, 0.32 -> 0.30, 0.45 -> 0.48, on 4M 1.85 ->
// 0.62, 1.94 -> 1.19 at 50%; Extras on 4M 1.11 -> 0.78, 2.16 -> 1.64 at 50%.
// Where the permuted form is taken it is at most 6% slower than the direct one
// (corrections without dark matter near 1M); the rule errs towards the direct
// form.  The gravity calls, four columns each way, gain nothing: 8.33 -> 8.42 ms
// on 4.19M, 68.3 -> 68.1 on 33.5M.
constexpr int64_t kKorderMin = 900000;
constexpr int64_t kKorderL2 = 128 << 20;
bool kernel_order_pays(int64_t n, int64_t n_gas, int in, int out, int scattered) {
    const int64_t written = (4 * scattered * n > kKorderL2 ? 6 : 2) * scattered * n;
    const int64_t read = (4 * in * n > kKorderL2 ? 3 : 1) * in * n_gas;
    return n >= kKorderMin && written + read >= (in + out + 5) * n;
}
struct KernelOrder {
    crk_ctx *ctx;
    const crk_leaves *lv;
    bool on;
    float *next = nullptr;
    int left;  // columns not yet taken
    Bundle in, out;
    // ni, no: columns the call reads and writes; scattered: columns that its kernels write in the
    // caller's order (its intermediate ones among them); record: bytes of its stage's largest record
    KernelOrder(crk_ctx *c, const crk_leaves *l, int ni, int no, int scattered, size_t record)
        : ctx(c), lv(l), left(ni + no) {
        on = kernel_order_pays(lv->n, lv->n_gas, ni, no, scattered);
        if (!on) return;
        // never in a captured call: its columns may not exist yet (no allocation there), and a graph must not
        // hold scratch that a later call may grow
        cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
        if (cudaStreamIsCapturing(ctx->stream, &cs) != cudaSuccess) cudaGetLastError();
        if (cs != cudaStreamCaptureStatusNone) {
            on = false;
            return;
        }
        // the columns, and the rows they pass through (later the records), before anything runs; without room:
        // the direct form
        const size_t row = std::max(sizeof(float4) * (size_t)((std::max(ni, no) + 3) / 4), record);
        next = (float *)crk_scratch(ctx, crk_ctx::kColumns, sizeof(float) * (size_t)(ni + no) * (size_t)lv->n);
        on = ctx->columns_live = next != nullptr;
        if (on && !crk_scratch(ctx, 4, row * (size_t)lv->n)) {
            crk_scratch_drop(ctx, crk_ctx::kColumns);
            on = ctx->columns_live = false;
        }
    }
    ~KernelOrder() { ctx->columns_live = false; }
    KernelOrder(const KernelOrder &) = delete;
    float *take(int comps) {
        float *r = next;
        left -= comps;
        if (left >= 0) next += (size_t)comps * lv->n;
        return r;
    }
    const float *input(const float *p, int comps) {
        if (!on || !p) return p;
        float *r = take(comps);
        in.add(p, r, comps, lv->n);
        return r;
    }
    float *output(float *p, int comps) {
        if (!on || !p) return p;
        float *r = take(comps);
        out.add(r, p, comps, lv->n);
        return r;
    }
    int begin() {
        if (!on) return CRK_OK;
        if (left < 0 || in.over || out.over) return crk_fail(ctx, CRK_EINVAL, "more columns than the call reserved");
        return permute_bundle(ctx, lv->n, lv->kperm, in);
    }
    int end(int rc) { return rc || !on ? rc : permute_bundle(ctx, lv->n, lv->kinv, out); }
};

template <class... S>
constexpr size_t record_bytes() {
    size_t most = 0;
    ((most = std::max(most, (size_t)Planes<typename S::Rec>::kBytes)), ...);
    return most;
}

}  // namespace

int grav_short(crk_ctx *ctx, const crk_leaves *lv, const crk_grav_params *gp, const float *m, float *a3,
               int64_t *pair_count) {
    if (!ctx) return CRK_EINVAL;
    if (!lv || !gp) return crk_fail(ctx, CRK_EINVAL, "null argument");
    if (lv->n > 0 && (!m || !a3)) return crk_fail(ctx, CRK_EINVAL, "null array");
    if (gp->r_cut != lv->r_cut_grav) return crk_fail(ctx, CRK_ESTATE, "r_cut differs from the leaves' r_cut_grav");
    GravP p{};
    p.m = m;
    p.a3 = a3;
    p.rc2 = gp->r_cut * gp->r_cut;
    p.eps2 = gp->eps * gp->eps;
    for (int k = 0; k < 6; ++k) p.c[k] = gp->poly[k];
    p.n = lv->n;
    p.count = (unsigned long long *)pair_count;
    return run_stage<GravStage>(ctx, lv, p, false, CRK_K_GRAVITY);
}

int grav_short_adjoint(crk_ctx *ctx, const crk_leaves *lv, const crk_grav_params *gp, const float *m,
                       const float *abar3, float *gx3, float *gm) {
    if (!ctx) return CRK_EINVAL;
    if (!lv || !gp) return crk_fail(ctx, CRK_EINVAL, "null argument");
    if (lv->n > 0 && (!m || !abar3 || !gx3 || !gm)) return crk_fail(ctx, CRK_EINVAL, "null array");
    if (gp->r_cut != lv->r_cut_grav) return crk_fail(ctx, CRK_ESTATE, "r_cut differs from the leaves' r_cut_grav");
    GravAdjP p{};
    p.m = m;
    p.abar = abar3;
    p.gx3 = gx3;
    p.gm = gm;
    p.rc2 = gp->r_cut * gp->r_cut;
    p.eps2 = gp->eps * gp->eps;
    for (int k = 0; k < 6; ++k) p.c[k] = gp->poly[k];
    p.n = lv->n;
    p.count = nullptr;
    return run_stage<GravAdjStage>(ctx, lv, p, false, CRK_K_GRAVITY_ADJOINT);
}

int crk_geometry(crk_ctx *ctx, const crk_leaves *lv, const float *m, float *V, float *rho, int64_t *pair_count) {
    if (!ctx) return CRK_EINVAL;
    if (!lv) return crk_fail(ctx, CRK_EINVAL, "null leaves");
    if (lv->n > 0 && (!m || !V || !rho)) return crk_fail(ctx, CRK_EINVAL, "null array");
    GeomP p{m, V, rho, lv->n, (unsigned long long *)pair_count};
    return run_stage<GeomStage>(ctx, lv, p, true, CRK_K_GEOMETRY);
}

int crk_geometry_adjoint(crk_ctx *ctx, const crk_leaves *lv, const float *m, const float *V, const float *rhobar,
                         const float *Vbar, float *gx3, float *gm) {
    if (!ctx) return CRK_EINVAL;
    if (!lv) return crk_fail(ctx, CRK_EINVAL, "null leaves");
    if (lv->n > 0 && (!m || !V || !rhobar || !gx3 || !gm)) return crk_fail(ctx, CRK_EINVAL, "null array");
    KernelOrder ko(ctx, lv, Vbar ? 4 : 3, 4, 4, record_bytes<GeomAdjStage>());
    GeomAdjP p{ko.input(m, 1), ko.input(V, 1), ko.input(rhobar, 1), ko.input(Vbar, 1), ko.output(gx3, 3),
               ko.output(gm, 1), lv->n, nullptr};
    const int rc = ko.begin();
    return rc ? rc : ko.end(run_stage<GeomAdjStage>(ctx, lv, p, true, CRK_K_GEOMETRY_ADJOINT, nullptr, ko.on));
}

int crk_corrections(crk_ctx *ctx, const crk_leaves *lv, const float *V, float *A, float *B, float *gradA,
                    float *gradB, int32_t *n_singular) {
    if (!ctx) return CRK_EINVAL;
    if (!lv) return crk_fail(ctx, CRK_EINVAL, "null leaves");
    if (lv->n > 0 && (!V || !A || !B || !gradA || !gradB)) return crk_fail(ctx, CRK_EINVAL, "null array");
    if (n_singular) CRK_CUDA(ctx, cudaMemsetAsync(n_singular, 0, sizeof(int32_t), ctx->stream));
    KernelOrder ko(ctx, lv, 1, 16, 16, record_bytes<CorrStage>());
    CorrP p{ko.input(V, 1), ko.output(A, 1), ko.output(B, 3), ko.output(gradA, 3), ko.output(gradB, 9), n_singular,
            lv->n, nullptr};
    const int rc = ko.begin();
    return rc ? rc : ko.end(run_stage<CorrStage>(ctx, lv, p, true, CRK_K_CORRECTIONS, nullptr, ko.on));
}

int crk_hydro(crk_ctx *ctx, const crk_leaves *lv, const crk_hydro_params *hp, const float *m, const float *v3,
              const float *u, const float *V, const float *rho, const float *A, const float *B, const float *gradA,
              const float *gradB, float *dvdt3, float *dudt, double *conservation, int64_t *pair_count) {
    if (!ctx) return CRK_EINVAL;
    if (!lv || !hp) return crk_fail(ctx, CRK_EINVAL, "null argument");
    if (lv->n > 0 && (!m || !v3 || !u || !V || !rho || !A || !B || !gradA || !gradB || !dvdt3 || !dudt))
        return crk_fail(ctx, CRK_EINVAL, "null array");
    KernelOrder ko(ctx, lv, 23, 4, 4, record_bytes<HydroStage>());
    HydroP p{ko.input(m, 1), ko.input(v3, 3), ko.input(u, 1), ko.input(V, 1), ko.input(rho, 1), ko.input(A, 1), ko.input(B, 3),
             ko.input(gradA, 3), ko.input(gradB, 9), ko.output(dvdt3, 3), ko.output(dudt, 1), conservation,
             hp->gamma, hp->alpha, hp->beta, hp->eta2, lv->n, (unsigned long long *)pair_count};
    const int rc = ko.begin();
    return rc ? rc : ko.end(run_stage<HydroStage>(ctx, lv, p, true, CRK_K_HYDRO, conservation, ko.on));
}

int crk_extras(crk_ctx *ctx, const crk_leaves *lv, const float *m, const float *v3, const float *V, const float *A,
               const float *B, const float *gradA, const float *gradB, float *rho_r, float *dvdx,
               int64_t *pair_count) {
    if (!ctx) return CRK_EINVAL;
    if (!lv) return crk_fail(ctx, CRK_EINVAL, "null argument");
    if (lv->n > 0 && (!m || !v3 || !V || !A || !B || !gradA || !gradB || !rho_r || !dvdx))
        return crk_fail(ctx, CRK_EINVAL, "null array");
    KernelOrder ko(ctx, lv, 21, 10, 10, record_bytes<ExtrasStage>());
    ExtrasP p{ko.input(m, 1), ko.input(v3, 3), ko.input(V, 1), ko.input(A, 1), ko.input(B, 3), ko.input(gradA, 3),
              ko.input(gradB, 9), ko.output(rho_r, 1), ko.output(dvdx, 9), lv->n, (unsigned long long *)pair_count};
    const int rc = ko.begin();
    return rc ? rc : ko.end(run_stage<ExtrasStage>(ctx, lv, p, true, CRK_K_EXTRAS, nullptr, ko.on));
}

int crk_hydro_limited(crk_ctx *ctx, const crk_leaves *lv, const crk_hydro_params *hp, const float *m,
                      const float *v3, const float *u, const float *V, const float *rho, const float *A,
                      const float *B, const float *gradA, const float *gradB, const float *dvdx, float *dvdt3,
                      float *dudt, double *conservation, int64_t *pair_count) {
    if (!ctx) return CRK_EINVAL;
    if (!lv || !hp) return crk_fail(ctx, CRK_EINVAL, "null argument");
    if (lv->n > 0 && (!m || !v3 || !u || !V || !rho || !A || !B || !gradA || !gradB || !dvdx || !dvdt3 || !dudt))
        return crk_fail(ctx, CRK_EINVAL, "null array");
    KernelOrder ko(ctx, lv, 32, 4, 4, record_bytes<HydroLimStage>());
    HydroP p{ko.input(m, 1), ko.input(v3, 3), ko.input(u, 1), ko.input(V, 1), ko.input(rho, 1), ko.input(A, 1), ko.input(B, 3),
             ko.input(gradA, 3), ko.input(gradB, 9), ko.output(dvdt3, 3), ko.output(dudt, 1), conservation,
             hp->gamma, hp->alpha, hp->beta, hp->eta2, lv->n, (unsigned long long *)pair_count, ko.input(dvdx, 9)};
    const int rc = ko.begin();
    return rc ? rc : ko.end(run_stage<HydroLimStage>(ctx, lv, p, true, CRK_K_HYDRO, conservation, ko.on));
}

int crk_hydro_accel(crk_ctx *ctx, const crk_leaves *lv, const crk_hydro_params *hp, const float *m, const float *v3,
                    const float *u, const float *V, const float *rho, const float *A, const float *B,
                    const float *gradA, const float *gradB, const float *dvdx, float sig_beta, float *dvdt3,
                    uint32_t *vsig_h_max, double *conservation, int64_t *pair_count) {
    if (!ctx) return CRK_EINVAL;
    if (!lv || !hp) return crk_fail(ctx, CRK_EINVAL, "null argument");
    if (lv->n > 0 && (!m || !v3 || !u || !V || !rho || !A || !B || !gradA || !gradB || !dvdt3))
        return crk_fail(ctx, CRK_EINVAL, "null array");
    if (!(sig_beta >= 0.0f)) return crk_fail(ctx, CRK_EINVAL, "sig_beta must be >= 0");
    KernelOrder ko(ctx, lv, dvdx ? 32 : 23, 3, 3, record_bytes<HydroAccelStage<true>>());
    HydroP p{ko.input(m, 1), ko.input(v3, 3), ko.input(u, 1), ko.input(V, 1), ko.input(rho, 1), ko.input(A, 1), ko.input(B, 3),
             ko.input(gradA, 3), ko.input(gradB, 9), ko.output(dvdt3, 3), nullptr, conservation,
             hp->gamma, hp->alpha, hp->beta, hp->eta2, lv->n, (unsigned long long *)pair_count, ko.input(dvdx, 9)};
    p.vsig_h = vsig_h_max;
    p.sig_beta = sig_beta;
    const int rc = ko.begin();
    if (rc) return rc;
    if (dvdx) return ko.end(run_stage<HydroAccelStage<true>>(ctx, lv, p, true, CRK_K_ACCEL, conservation, ko.on));
    return ko.end(run_stage<HydroAccelStage<false>>(ctx, lv, p, true, CRK_K_ACCEL, conservation, ko.on));
}

int crk_hydro_energy(crk_ctx *ctx, const crk_leaves *lv, const crk_hydro_params *hp, const float *m, const float *v3,
                     const float *u, const float *V, const float *rho, const float *A, const float *B,
                     const float *gradA, const float *gradB, const float *dvdx, const float *vstar3, float *dudt,
                     double *conservation, int64_t *pair_count) {
    if (!ctx) return CRK_EINVAL;
    if (!lv || !hp) return crk_fail(ctx, CRK_EINVAL, "null argument");
    if (lv->n > 0 && (!m || !v3 || !u || !V || !rho || !A || !B || !gradA || !gradB || !vstar3 || !dudt))
        return crk_fail(ctx, CRK_EINVAL, "null array");
    KernelOrder ko(ctx, lv, 23 + (dvdx ? 9 : 0) + (vstar3 == v3 ? 0 : 3), 1, 1, record_bytes<HydroEnergyStage<true, true>>());
    HydroP p{ko.input(m, 1), ko.input(v3, 3), ko.input(u, 1), ko.input(V, 1), ko.input(rho, 1), ko.input(A, 1), ko.input(B, 3),
             ko.input(gradA, 3), ko.input(gradB, 9), nullptr, ko.output(dudt, 1), conservation,
             hp->gamma, hp->alpha, hp->beta, hp->eta2, lv->n, (unsigned long long *)pair_count, ko.input(dvdx, 9)};
    p.vstar = vstar3 == v3 ? p.v3 : ko.input(vstar3, 3);
    const int rc = ko.begin();
    if (rc) return rc;
    if (dvdx) return ko.end(run_energy<true>(ctx, lv, p, conservation, ko.on));
    return ko.end(run_energy<false>(ctx, lv, p, conservation, ko.on));
}

int crk_corrections_adjoint(crk_ctx *ctx, const crk_leaves *lv, const float *V, const float *Abar,
                            const float *Bbar, const float *gradAbar, const float *gradBbar, float *xbar3,
                            float *Vbar, int32_t *n_singular) {
    if (!ctx) return CRK_EINVAL;
    if (!lv) return crk_fail(ctx, CRK_EINVAL, "null argument");
    if (lv->n > 0 && (!V || !Abar || !Bbar || !gradAbar || !gradBbar || !xbar3 || !Vbar))
        return crk_fail(ctx, CRK_EINVAL, "null array");
    const int64_t n = lv->n;
    if (n_singular) CRK_CUDA(ctx, cudaMemsetAsync(n_singular, 0, sizeof(int32_t), ctx->stream));
    if (n == 0) return CRK_OK;
    float *coef = (float *)crk_scratch(ctx, 33, sizeof(float) * kCorrCoef * (size_t)n);
    if (!coef) return crk_fail(ctx, CRK_ENOMEM, "adjoint scratch");
    KernelOrder ko(ctx, lv, 17, 4, 4 + kCorrCoef, record_bytes<CorrAdjPrepStage, CorrAdjStage>());
    CorrAdjP p{};
    p.V = ko.input(V, 1);
    p.n_singular = n_singular;
    p.n = n;
    p.Abar = ko.input(Abar, 1);
    p.Bbar = ko.input(Bbar, 3);
    p.gAbar = ko.input(gradAbar, 3);
    p.gBbar = ko.input(gradBbar, 9);
    p.coef = coef;
    CorrAdjSweepP q{p.V, coef, ko.output(xbar3, 3), ko.output(Vbar, 1), n, nullptr, nullptr};
    int rc = ko.begin();
    if (!rc) rc = run_stage<CorrAdjPrepStage>(ctx, lv, p, true, CRK_K_CORRECTIONS, nullptr, ko.on);
    if (!rc) rc = run_stage<CorrAdjStage>(ctx, lv, q, true, CRK_K_CORRECTIONS, nullptr, ko.on);
    return ko.end(rc);
}

int crk_hydro_adjoint(crk_ctx *ctx, const crk_leaves *lv, const crk_hydro_params *hp, const float *m, const float *v3,
                      const float *u, const float *V, const float *rho, const float *A, const float *B,
                      const float *gradA, const float *gradB, const float *dvbar3, const float *dubar, float *xbar3,
                      float *vbar3, float *ubar, float *mbar, float *Vbar, float *rhobar, float *Abar, float *Bbar3,
                      float *gradAbar3, float *gradBbar9) {
    if (!ctx) return CRK_EINVAL;
    if (!lv || !hp) return crk_fail(ctx, CRK_EINVAL, "null argument");
    if (lv->n > 0 && (!m || !v3 || !u || !V || !rho || !A || !B || !gradA || !gradB || !dvbar3 || !dubar || !xbar3 ||
                      !vbar3 || !ubar || !mbar || !Vbar || !rhobar || !Abar || !Bbar3 || !gradAbar3 || !gradBbar9))
        return crk_fail(ctx, CRK_EINVAL, "null array");
    KernelOrder ko(ctx, lv, 27, 26, 26, record_bytes<HydroAdjStage<true>>());
    HydroAdjP p{ko.input(m, 1), ko.input(v3, 3), ko.input(u, 1), ko.input(V, 1), ko.input(rho, 1), ko.input(A, 1), ko.input(B, 3),
                ko.input(gradA, 3), ko.input(gradB, 9),
                ko.input(dvbar3, 3), ko.input(dubar, 1), ko.output(xbar3, 3), ko.output(vbar3, 3), ko.output(ubar, 1),
                ko.output(mbar, 1), ko.output(Vbar, 1), ko.output(rhobar, 1), ko.output(Abar, 1), ko.output(Bbar3, 3),
                ko.output(gradAbar3, 3), ko.output(gradBbar9, 9), hp->gamma, hp->alpha, hp->beta, hp->eta2, lv->n,
                nullptr, nullptr};
    const int rc = ko.begin();
    return rc ? rc : ko.end(run_hydro_adjoint(ctx, lv, p, ko.on));
}

template <bool kGas>
static LeafView list_view(const crk_leaves *lv) {
    return LeafView{lv->leaf_start, lv->leaf_ngas, lv->bbox, lv->hmax, kGas ? lv->pos : lv->pos_g,
                    kGas ? lv->kperm : lv->kperm_g, kGas ? lv->himg_start : lv->gimg_start,
                    kGas ? lv->himg_cnt : lv->gimg_cnt, kGas ? lv->himg : lv->gimg, lv->n_leaves, nullptr, 0, 32, nullptr};
}

// groups of each leaf and their number, into gstart and lv->dev[1] (gas) or [2]
template <bool kGas>
static int list_groups(crk_ctx *ctx, crk_leaves *lv, int32_t *gstart) {
    const int64_t nl = lv->n_leaves;
    int32_t *ng = (int32_t *)crk_scratch(ctx, 6, sizeof(int32_t) * (size_t)(nl + 1));
    if (!ng) return crk_fail(ctx, CRK_ENOMEM, "neighbour list allocation");
    list_group_count_kernel<<<crk_grid(nl + 1, 256), 256, 0, ctx->stream>>>(nl, lv->leaf_start, lv->leaf_ngas, kGas, ng);
    ++ctx->launches;
    return crk_exclusive_scan_i32(ctx, ng, gstart, nl + 1, lv->dev + (kGas ? 1 : 2));
}

static bool no_lists(const crk_leaves *lv, bool gas) { return lv->n_leaves == 0 || lv->n == 0 || (gas && lv->n_gas == 0); }

bool crk_wants_gas_lists(const crk_ctx *ctx) {
    for (int k : {CRK_K_GEOMETRY, CRK_K_CORRECTIONS, CRK_K_HYDRO, CRK_K_GEOMETRY_ADJOINT, CRK_K_EXTRAS, CRK_K_ACCEL,
                  CRK_K_ENERGY})
        if (ctx->variant[k] == CRK_VARIANT_LISTS) return true;
    return false;
}

int crk_gas_groups(crk_ctx *ctx, crk_leaves *lv) {
    if (lv->n_leaves == 0 || lv->n == 0) return CRK_OK;
    crk_nlist &out = lv->gas_lists;
    out.gstart = (int32_t *)crk_leaves_alloc(ctx, lv, sizeof(int32_t) * (size_t)(lv->n_leaves + 1));
    if (!out.gstart) return crk_fail(ctx, CRK_ENOMEM, "neighbour list allocation");
    return list_groups<true>(ctx, lv, out.gstart);
}

// One pass into fixed capacities (a lane's list and a group's table), which the adaptive
// smoothing lengths keep well above the largest counts; room for 1/8 more groups than this build
// holds (a rebuild of moved particles reuses the buffers).
int crk_gas_lists_onepass(crk_ctx *ctx, crk_leaves *lv, int32_t ngroups) {
    if (no_lists(lv, true)) return CRK_OK;
    crk_nlist &out = lv->gas_lists;
    const int64_t nl = lv->n_leaves, n = lv->n;
    const int capr = kGasListCapRows, capt = kGasTableCap;
    const int64_t capg = (int64_t)ngroups + ngroups / 8 + 64;
    cudaStream_t st = ctx->stream;
    if (capg * capt >= 2147483647LL) {  // 32-bit offsets: the exact build
        CRK_CUDA(ctx, cudaMemsetAsync(lv->dev + 3, 1, sizeof(int32_t), st));
        return CRK_OK;
    }
    if (!out.list) {  // (a second attempt of the pair lists keeps the first's buffers)
        // room for the records of the light stages, so that the first pair kernel need not allocate
        if (!crk_scratch(ctx, 4, 32 * (size_t)n)) return crk_fail(ctx, CRK_ENOMEM, "neighbour list scratch");
        out.cnt = (int32_t *)crk_leaves_alloc(ctx, lv, sizeof(int32_t) * (size_t)n);
        out.gleaf = (int32_t *)crk_leaves_alloc(ctx, lv, sizeof(int32_t) * (size_t)capg);
        out.unum = (int32_t *)crk_leaves_alloc(ctx, lv, sizeof(int32_t) * (size_t)(capg + 1));
        out.goff = (int32_t *)crk_leaves_alloc(ctx, lv, sizeof(int32_t) * (size_t)(capg + 1));
        out.uoff = (int32_t *)crk_leaves_alloc(ctx, lv, sizeof(int32_t) * (size_t)(capg + 1));
        out.ucode = (uint32_t *)crk_leaves_alloc(ctx, lv, sizeof(uint32_t) * (size_t)capg * capt);
        out.list = (uint16_t *)crk_leaves_alloc(ctx, lv, sizeof(uint16_t) * (size_t)capg * capr * 32);
        if (!out.cnt || !out.gleaf || !out.unum || !out.goff || !out.uoff || !out.list || !out.ucode)
            return crk_fail(ctx, CRK_ENOMEM, "neighbour list allocation");
    }
    out.groups = capg;
    out.dgroups = lv->dev + 1;
    out.onepass = true;
    out.entries = capg * capr * 32;
    out.table = capg * capt;
    const LeafView v = list_view<true>(lv);
    list_group_leaf_kernel<<<crk_grid(nl, 256), 256, 0, st>>>(nl, out.gstart, out.gleaf, capg);
    strided_offsets_kernel<<<crk_grid(capg + 1, 256), 256, 0, st>>>(capg + 1, capr, capt, out.goff, out.uoff);
    ListP pf{out.list, out.ucode, out.gstart, out.goff, out.uoff, out.cnt, out.unum, nullptr, lv->dev + 3, capr, capt,
             lv->r_cut_grav * lv->r_cut_grav};
    launch_list_build<true>(ctx, lv, v, pf, GroupTable{out.gstart, out.gleaf, ngroups, nullptr}, ngroups);
    ctx->launches += 2;
    CRK_LAUNCH_CHECK(ctx, "neighbour lists");
    return CRK_OK;
}

// reuse: a rebuild of one-pass gas lists into the buffers of the first build; no host
// synchronisation, overflows go to the leaves' status word.  Otherwise the exact two-pass build
// (count, scan, fill): gravity lists, and gas lists beyond the one-pass capacities.
template <bool kGas>
static int build_lists(crk_ctx *ctx, crk_leaves *lv, crk_nlist &out, bool reuse) {
    const int64_t nl = lv->n_leaves, n = lv->n;
    if (no_lists(lv, kGas)) return CRK_OK;
    if (reuse && (!kGas || !out.onepass)) return crk_fail(ctx, CRK_ESTATE, "rebuild: lists without fixed capacities");
    cudaStream_t st = ctx->stream;
    const LeafView v = list_view<kGas>(lv);
    const float rc2 = lv->r_cut_grav * lv->r_cut_grav;
    int32_t *dgroups = lv->dev + (kGas ? 1 : 2);  // this build's group count, for the kernels
    int rc;
    if (reuse) {
        if ((rc = list_groups<kGas>(ctx, lv, out.gstart))) return rc;
        const int64_t capg = out.groups;
        list_group_leaf_kernel<<<crk_grid(nl, 256), 256, 0, st>>>(nl, out.gstart, out.gleaf, capg);
        ListP pf{out.list, out.ucode, out.gstart, out.goff, out.uoff, out.cnt, out.unum, nullptr, lv->dev + 3,
                 kGasListCapRows, kGasTableCap, rc2};
        launch_list_build<kGas>(ctx, lv, v, pf, GroupTable{out.gstart, out.gleaf, capg, dgroups}, capg);
        lists_status_kernel<<<1, 1, 0, st>>>(dgroups, capg, lv->dev + 3, lv->dev);
        ctx->launches += 2;
        CRK_LAUNCH_CHECK(ctx, "neighbour lists");
        return CRK_OK;
    }
    if (kGas && ctx->trace) fprintf(stderr, "[crk] gas lists: a list or table exceeded its capacity, exact build\n");
    out = crk_nlist{};
    int32_t *gstart = (int32_t *)crk_leaves_alloc(ctx, lv, sizeof(int32_t) * (size_t)(nl + 1));
    int32_t *cnt = (int32_t *)crk_leaves_alloc(ctx, lv, sizeof(int32_t) * (size_t)n);
    int32_t *tot = (int32_t *)crk_scratch(ctx, 7, 64);  // [1] rows, [2] table entries, [4] largest table
    if (!gstart || !cnt || !tot) return crk_fail(ctx, CRK_ENOMEM, "neighbour list allocation");
    if ((rc = list_groups<kGas>(ctx, lv, gstart))) return rc;
    int32_t ngroups = 0;
    CRK_CUDA(ctx, cudaMemcpyAsync(&ngroups, dgroups, sizeof(int32_t), cudaMemcpyDeviceToHost, st));
    CRK_CUDA(ctx, cudaStreamSynchronize(st));
    int32_t *gleaf = (int32_t *)crk_leaves_alloc(ctx, lv, sizeof(int32_t) * (size_t)std::max(ngroups, 1));
    int32_t *ucnt = (int32_t *)crk_leaves_alloc(ctx, lv, sizeof(int32_t) * (size_t)(ngroups + 1));
    int32_t *goff = (int32_t *)crk_leaves_alloc(ctx, lv, sizeof(int32_t) * (size_t)(ngroups + 1));
    int32_t *uoff = (int32_t *)crk_leaves_alloc(ctx, lv, sizeof(int32_t) * (size_t)(ngroups + 1));
    int32_t *gk = (int32_t *)crk_scratch(ctx, 8, sizeof(int32_t) * (size_t)(ngroups + 1));
    if (!gleaf || !ucnt || !goff || !uoff || !gk) return crk_fail(ctx, CRK_ENOMEM, "neighbour list allocation");
    list_group_leaf_kernel<<<crk_grid(nl, 256), 256, 0, st>>>(nl, gstart, gleaf, ngroups);
    const GroupTable gt{gstart, gleaf, ngroups, nullptr};
    CRK_CUDA(ctx, cudaMemsetAsync(ucnt, 0, sizeof(int32_t) * (size_t)(ngroups + 1), st));
    CRK_CUDA(ctx, cudaMemsetAsync(tot + 4, 0, sizeof(int32_t), st));
    ListP pc{nullptr, nullptr, gstart, nullptr, nullptr, cnt, ucnt, tot + 4, nullptr, 2147483647, 2147483647,
             rc2};
    launch_list_build<kGas>(ctx, lv, v, pc, gt, ngroups);
    CRK_LAUNCH_CHECK(ctx, "neighbour counts");
    CRK_CUDA(ctx, cudaMemsetAsync(gk, 0, sizeof(int32_t) * (size_t)(ngroups + 1), st));
    list_group_k_kernel<<<(unsigned)nl, kThreads, 0, st>>>(nl, lv->leaf_start, lv->leaf_ngas, kGas, gstart, cnt, gk);
    ctx->launches += 2;
    rc = crk_exclusive_scan_i32(ctx, gk, goff, ngroups + 1, tot + 1);
    if (rc) return rc;
    rc = crk_exclusive_scan_i32(ctx, ucnt, uoff, ngroups + 1, tot + 2);
    if (rc) return rc;
    int32_t sizes[5] = {0, 0, 0, 0, 0};
    CRK_CUDA(ctx, cudaMemcpyAsync(sizes, tot, sizeof(sizes), cudaMemcpyDeviceToHost, st));
    CRK_CUDA(ctx, cudaStreamSynchronize(st));
    const int32_t rows = sizes[1], umax = sizes[4];
    const int64_t tsize = (int64_t)(uint32_t)sizes[2];
    // table indices are 16-bit, and the offsets 32-bit: without lists the kernels use tiles
    if (umax > 65535 || rows < 0 || sizes[2] < 0) {
        if (ctx->trace)
            fprintf(stderr, "[crk] %s lists skipped (largest group table %d)\n", kGas ? "gas" : "gravity", umax);
        return CRK_OK;
    }
    const int64_t entries = (int64_t)rows * 32;
    uint16_t *list = (uint16_t *)crk_leaves_alloc(ctx, lv, sizeof(uint16_t) * (size_t)(entries > 0 ? entries : 1));
    uint32_t *ucode = (uint32_t *)crk_leaves_alloc(ctx, lv, sizeof(uint32_t) * (size_t)(tsize > 0 ? tsize : 1));
    if (!list || !ucode)
        return crk_fail(ctx, CRK_ENOMEM, "neighbour list allocation (%lld entries)", (long long)entries);
    ListP pf{list, ucode, gstart, goff, uoff, nullptr, nullptr, nullptr, nullptr, 2147483647, 2147483647,
             rc2};
    launch_list_build<kGas>(ctx, lv, v, pf, gt, ngroups);
    CRK_LAUNCH_CHECK(ctx, "neighbour lists");
    out.unum = ucnt;
    out.uoff = uoff;
    out.ucode = ucode;
    out.table = tsize;
    out.gstart = gstart;
    out.gleaf = gleaf;
    out.goff = goff;
    out.cnt = cnt;
    out.list = list;
    out.groups = ngroups;
    out.dgroups = dgroups;
    out.onepass = false;
    out.entries = entries;
    return CRK_OK;
}

int crk_build_lists(crk_ctx *ctx, crk_leaves *lv, bool gas, bool reuse) {
    return gas ? build_lists<true>(ctx, lv, lv->gas_lists, reuse) : build_lists<false>(ctx, lv, lv->grav_lists, reuse);
}

// ---------------------------------------------------------------------------
// Allocation-free short-range gravity (no counterpart in the paper).
//
// Some callers cannot let a library call cudaMalloc: an application whose own
// pool already owns the device memory, or a time-stepping loop that must not
// pay the device synchronisation that cudaMalloc/cudaFree can imply.  This
// entry point runs the same gravity kernels as grav_short, but its only
// scratch (the kernel-order particle records, 16 bytes per particle) lives in
// the file-scope array below, which every GPU that loads libcrk holds until
// the process exits: CRK_NOALLOC_MAX_PARTICLES x 16 bytes = 32 MiB.
namespace {
__device__ __align__(256) GravStage::Rec g_noalloc_rec[CRK_NOALLOC_MAX_PARTICLES];

constexpr int kNoAllocMaxDevices = 64;
void *g_noalloc_ptr[kNoAllocMaxDevices] = {};  // device address of g_noalloc_rec, per device
std::mutex g_noalloc_mu;
}  // namespace

int grav_short_noalloc(crk_ctx *ctx, const crk_leaves *lv, const crk_grav_params *gp, const float *m, float *a3) {
    if (!ctx || !lv || !gp) return CRK_EINVAL;
    const int64_t n = lv->n;
    if (n > CRK_NOALLOC_MAX_PARTICLES) return CRK_ETOOLARGE;
    if (n > 0 && (!m || !a3)) return CRK_EINVAL;
    if (gp->r_cut != lv->r_cut_grav) return CRK_ESTATE;
    if (n == 0) return CRK_OK;
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev != ctx->device || dev < 0 || dev >= kNoAllocMaxDevices) {
        cudaGetLastError();
        return CRK_ESTATE;  // the context's device must be current
    }
    // set-up, once per device, with that device current: the host-side name of a
    // __device__ array is not a device address, so ask the runtime for it
    void *base = nullptr;
    {
        std::lock_guard<std::mutex> lock(g_noalloc_mu);
        if (!g_noalloc_ptr[dev]) {
            void *ptr = nullptr;
            if (cudaGetSymbolAddress(&ptr, g_noalloc_rec) != cudaSuccess || !ptr) {
                cudaGetLastError();
                return CRK_ECUDA;
            }
            g_noalloc_ptr[dev] = ptr;
        }
        base = g_noalloc_ptr[dev];
    }
    const RecView<GravStage::Rec> rec{base, n};
    GravP p{};
    p.m = m;
    p.a3 = a3;
    p.rc2 = gp->r_cut * gp->r_cut;
    p.eps2 = gp->eps * gp->eps;
    for (int k = 0; k < 6; ++k) p.c[k] = gp->poly[k];
    p.n = n;
    p.count = nullptr;
    // every record is rewritten before it is read, so nothing needs clearing
    gather_kernel<GravStage><<<crk_grid(n, 256), 256, 0, ctx->stream>>>(n, lv->pos_g, lv->kperm_g, p, base, 0);
    LeafView v{lv->leaf_start, lv->leaf_ngas, lv->bbox, lv->hmax, lv->pos_g, lv->kperm_g, lv->gimg_start,
               lv->gimg_cnt, lv->gimg, lv->n_leaves, nullptr, 0, 32, lv->gcell};
    const crk_nlist &nls = lv->grav_lists;
    if (nls.list && ctx->variant[CRK_K_GRAVITY] == CRK_VARIANT_LISTS) {
        GasLists gl{nls.gstart, nls.goff, nls.cnt, nls.list, nls.uoff, nls.unum, nls.ucode, nls.gleaf, nls.groups,
                    nls.dgroups};
        const int64_t lgrid = (nls.groups + kWarps - 1) / kWarps;
        list_kernel<GravStage, false><<<(unsigned)(lgrid > 0 ? lgrid : 1), kThreads,
                                        list_kernel_smem<GravStage, false>(), ctx->stream>>>(v, p, rec, gl, nullptr);
    } else {
        launch_cells<GravStage, false>(ctx, lv, v, p, rec, false, 4, false);
    }
    ctx->launches += 2;
    return cudaGetLastError() == cudaSuccess ? CRK_OK : CRK_ECUDA;
}

// ---------------------------------------------------------------------------
// Whole step with kernel-order intermediates.  The step's inputs are permuted
// into the two kernel orders once; every intermediate (V, rho, A, B, dA, dB,
// a, the cotangents) stays in kernel order, so it is written and read
// coalesced instead of being scattered to the caller's order and gathered
// back by the next kernel; the outputs the caller asked for are gathered back
// to the caller's order once at the end.
namespace {

__global__ void cotangent_kernel(int64_t n, const float *__restrict__ a_g, const float4 *__restrict__ pos,
                                 float *__restrict__ abar_g, float *__restrict__ rhob_k) {
    int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= n) return;
    if (abar_g)
        for (int c = 0; c < 3; ++c) abar_g[c * n + q] = 2.0f * a_g[c * n + q];
    if (rhob_k) rhob_k[q] = pos[q].w > 0.0f ? 1.0f : 0.0f;
}

}  // namespace

int crk_stage_forces(crk_ctx *ctx, const crk_leaves *lv, const crk_grav_params *gp, const crk_hydro_params *hp,
                     int limited, int gravity, float sig_beta, const float *m, const float *v3, const float *u,
                     uint32_t *vsig_h, int32_t *n_singular, float *w) {
    namespace K = crk_stage_cols;
    const int64_t n = lv->n;
    if (n == 0) return CRK_OK;
    auto C = [&](int k) { return w + (size_t)k * n; };
    int rc;
    Bundle in, in_g;
    in.add(m, C(K::m), 1, n);
    in.add(v3, C(K::v), 3, n);
    in.add(u, C(K::u), 1, n);
    if (gravity) in_g.add(m, C(K::mg), 1, n);
    if ((rc = permute_bundle(ctx, n, lv->kperm, in)) || (rc = permute_bundle(ctx, n, lv->kperm_g, in_g))) return rc;
    {
        GeomP p{C(K::m), C(K::V), C(K::rho), n, nullptr, nullptr};
        if ((rc = run_stage<GeomStage>(ctx, lv, p, true, CRK_K_GEOMETRY, nullptr, true))) return rc;
    }
    {
        if (n_singular) CRK_CUDA(ctx, cudaMemsetAsync(n_singular, 0, sizeof(int32_t), ctx->stream));
        CorrP p{C(K::V), C(K::A), C(K::B), C(K::gA), C(K::gB), n_singular, n, nullptr};
        if ((rc = run_stage<CorrStage>(ctx, lv, p, true, CRK_K_CORRECTIONS, nullptr, true))) return rc;
    }
    if (limited) {
        ExtrasP p{C(K::m), C(K::v), C(K::V), C(K::A), C(K::B), C(K::gA), C(K::gB), C(K::rhoR), C(K::dvdx), n, nullptr};
        if ((rc = run_stage<ExtrasStage>(ctx, lv, p, true, CRK_K_EXTRAS, nullptr, true))) return rc;
    }
    {
        HydroP p{C(K::m), C(K::v), C(K::u), C(K::V), C(limited ? K::rhoR : K::rho), C(K::A), C(K::B), C(K::gA),
                 C(K::gB), C(K::dv), nullptr, nullptr, hp->gamma, hp->alpha, hp->beta, hp->eta2, n, nullptr,
                 limited ? C(K::dvdx) : nullptr};
        p.vsig_h = vsig_h;
        p.sig_beta = sig_beta;
        if (limited) rc = run_stage<HydroAccelStage<true>>(ctx, lv, p, true, CRK_K_ACCEL, nullptr, true);
        else rc = run_stage<HydroAccelStage<false>>(ctx, lv, p, true, CRK_K_ACCEL, nullptr, true);
        if (rc) return rc;
    }
    if (gravity) {
        if (gp->r_cut != lv->r_cut_grav) return crk_fail(ctx, CRK_ESTATE, "r_cut differs from the leaves' r_cut_grav");
        GravP p{};
        p.m = C(K::mg);
        p.a3 = C(K::ag);
        p.rc2 = gp->r_cut * gp->r_cut;
        p.eps2 = gp->eps * gp->eps;
        for (int k = 0; k < 6; ++k) p.c[k] = gp->poly[k];
        p.n = n;
        if ((rc = run_stage<GravStage>(ctx, lv, p, false, CRK_K_GRAVITY, nullptr, true))) return rc;
    }
    return CRK_OK;
}

int crk_stage_energy(crk_ctx *ctx, const crk_leaves *lv, const crk_hydro_params *hp, int limited,
                     const float *vstar3, float *w, double *conservation) {
    namespace K = crk_stage_cols;
    const int64_t n = lv->n;
    if (n == 0) return CRK_OK;
    auto C = [&](int k) { return w + (size_t)k * n; };
    const float *vs = C(K::v);
    if (vstar3) {
        Bundle in;
        in.add(vstar3, C(K::vs), 3, n);
        const int rc = permute_bundle(ctx, n, lv->kperm, in);
        if (rc) return rc;
        vs = C(K::vs);
    }
    HydroP p{C(K::m), C(K::v), C(K::u), C(K::V), C(limited ? K::rhoR : K::rho), C(K::A), C(K::B), C(K::gA),
             C(K::gB), nullptr, C(K::du), conservation, hp->gamma, hp->alpha, hp->beta, hp->eta2, n, nullptr,
             limited ? C(K::dvdx) : nullptr};
    p.vstar = vs;
    if (limited) return run_energy<true>(ctx, lv, p, conservation, true);
    return run_energy<false>(ctx, lv, p, conservation, true);
}

namespace {
// out[i] = a[i] + b[i] (+ c[i] when c is given), over cols columns of n
__global__ void add_cols_kernel(int64_t n, int cols, float *__restrict__ out, const float *__restrict__ a,
                                const float *__restrict__ b, const float *__restrict__ c) {
    const int64_t total = n * cols;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x)
        out[i] = c ? a[i] + b[i] + c[i] : a[i] + b[i];
}
}  // namespace

int crk_hydro_chain_adjoint(crk_ctx *ctx, const crk_leaves *lv, const crk_hydro_params *hp,
                            const crk_chain_adjoint_io *io) {
    if (!ctx) return CRK_EINVAL;
    if (!lv || !hp || !io) return crk_fail(ctx, CRK_EINVAL, "null argument");
    const int64_t n = lv->n;
    if (io->n_singular) CRK_CUDA(ctx, cudaMemsetAsync(io->n_singular, 0, sizeof(int32_t), ctx->stream));
    if (n == 0) return CRK_OK;
    if (!io->m || !io->v3 || !io->u || !io->dvbar3 || !io->dubar) return crk_fail(ctx, CRK_EINVAL, "null array");
    // kernel-order columns
    enum : int {
        cm = 0, cv = 1, cu = 4, cdvb = 5, cdub = 8, cV = 9, crho = 10, cA = 11, cB = 12, cgA = 15, cgB = 18,
        cdv = 27, cdu = 30, cxh = 31, cvb = 34, cub = 37, cmh = 38, cVh = 39, crhob = 40, cAb = 41, cBb = 42,
        cgAb = 45, cgBb = 48, ccoef = 57, cxc = ccoef + kCorrCoef, cVc = cxc + 3, cxg = cVc + 1, cmg = cxg + 3,
        cols = cmg + 1
    };
    float *w = (float *)crk_scratch(ctx, 34, sizeof(float) * cols * (size_t)n);
    if (!w) return crk_fail(ctx, CRK_ENOMEM, "chain scratch");
    auto C = [&](int k) { return w + (size_t)k * n; };
    cudaStream_t st = ctx->stream;
    const int g = crk_grid(n, 256);
    int rc;
    Bundle in, outs;
    in.add(io->m, C(cm), 1, n);
    in.add(io->u, C(cu), 1, n);
    in.add(io->dubar, C(cdub), 1, n);
    in.add(io->v3, C(cv), 3, n);
    in.add(io->dvbar3, C(cdvb), 3, n);
    if ((rc = permute_bundle(ctx, n, lv->kperm, in))) return rc;
    {
        GeomP p{C(cm), C(cV), C(crho), n, nullptr, nullptr};
        if ((rc = run_stage<GeomStage>(ctx, lv, p, true, CRK_K_GEOMETRY, nullptr, true))) return rc;
    }
    {
        CorrP p{C(cV), C(cA), C(cB), C(cgA), C(cgB), io->n_singular, n, nullptr};
        if ((rc = run_stage<CorrStage>(ctx, lv, p, true, CRK_K_CORRECTIONS, nullptr, true))) return rc;
    }
    if (io->dvdt3 || io->dudt) {
        HydroP p{C(cm), C(cv), C(cu), C(cV), C(crho), C(cA), C(cB), C(cgA), C(cgB), C(cdv), C(cdu), nullptr,
                 hp->gamma, hp->alpha, hp->beta, hp->eta2, n, nullptr};
        if ((rc = run_stage<HydroStage>(ctx, lv, p, true, CRK_K_HYDRO, nullptr, true))) return rc;
    }
    {
        HydroAdjP p{C(cm),  C(cv),  C(cu),   C(cV),   C(crho),   C(cA),  C(cB),  C(cgA),     C(cgB),
                    C(cdvb), C(cdub), C(cxh), C(cvb), C(cub), C(cmh), C(cVh), C(crhob), C(cAb),
                    C(cBb), C(cgAb), C(cgBb), hp->gamma, hp->alpha, hp->beta, hp->eta2, n, nullptr, nullptr};
        if ((rc = run_hydro_adjoint(ctx, lv, p, true))) return rc;
    }
    {
        CorrAdjP p{};
        p.V = C(cV);
        p.n = n;
        p.Abar = C(cAb);
        p.Bbar = C(cBb);
        p.gAbar = C(cgAb);
        p.gBbar = C(cgBb);
        p.coef = C(ccoef);
        if ((rc = run_stage<CorrAdjPrepStage>(ctx, lv, p, true, CRK_K_CORRECTIONS, nullptr, true))) return rc;
        CorrAdjSweepP q{C(cV), C(ccoef), C(cxc), C(cVc), n, nullptr, nullptr};
        if ((rc = run_stage<CorrAdjStage>(ctx, lv, q, true, CRK_K_CORRECTIONS, nullptr, true))) return rc;
    }
    const int ge = g < 8 * ctx->num_sms ? g : 8 * ctx->num_sms;
    add_cols_kernel<<<ge, 256, 0, st>>>(n, 1, C(cVh), C(cVh), C(cVc), nullptr);  // Vbar = hydro + corrections
    ++ctx->launches;
    {
        GeomAdjP p{C(cm), C(cV), C(crhob), C(cVh), C(cxg), C(cmg), n, nullptr};
        if ((rc = run_stage<GeomAdjStage>(ctx, lv, p, true, CRK_K_GEOMETRY_ADJOINT, nullptr, true))) return rc;
    }
    add_cols_kernel<<<ge, 256, 0, st>>>(n, 3, C(cxh), C(cxh), C(cxc), C(cxg));  // xbar
    add_cols_kernel<<<ge, 256, 0, st>>>(n, 1, C(cmh), C(cmh), C(cmg), nullptr);  // mbar
    ctx->launches += 2;
    CRK_LAUNCH_CHECK(ctx, "chain sums");
    if (io->dvdt3) outs.add(C(cdv), io->dvdt3, 3, n);
    if (io->dudt) outs.add(C(cdu), io->dudt, 1, n);
    if (io->xbar3) outs.add(C(cxh), io->xbar3, 3, n);
    if (io->mbar) outs.add(C(cmh), io->mbar, 1, n);
    if (io->vbar3) outs.add(C(cvb), io->vbar3, 3, n);
    if (io->ubar) outs.add(C(cub), io->ubar, 1, n);
    return permute_bundle(ctx, n, lv->kinv, outs);
}

int crk_step_fused(crk_ctx *ctx, const crk_leaves *lv, const crk_grav_params *gp, const crk_hydro_params *hp,
                   const crk_step_io *io) {
    const int64_t n = lv->n;
    if (n == 0) return CRK_OK;
    if (!io->m || !io->v3 || !io->u) return crk_fail(ctx, CRK_EINVAL, "step inputs m, v3, u are required");
    if (gp->r_cut != lv->r_cut_grav) return crk_fail(ctx, CRK_ESTATE, "r_cut differs from the leaves' r_cut_grav");
    float *buf = (float *)crk_scratch(ctx, 18, sizeof(float) * 58 * (size_t)n);
    if (!buf) return crk_fail(ctx, CRK_ENOMEM, "step scratch");
    float *cur = buf;
    auto take = [&](int k) { float *r = cur; cur += (size_t)k * n; return r; };
    float *m_k = take(1), *v_k = take(3), *u_k = take(1), *V_k = take(1), *rho_k = take(1), *A_k = take(1);
    float *B_k = take(3), *gA_k = take(3), *gB_k = take(9), *dv_k = take(3), *du_k = take(1), *rhob_k = take(1);
    float *Vb_k = take(1), *gx2_k = take(3), *gm2_k = take(1);
    float *m_g = take(1), *a_g = take(3), *abar_g = take(3), *gx_g = take(3), *gm_g = take(1);
    float *rhoR_k = take(1), *dvdx_k = take(9);
    cudaStream_t st = ctx->stream;
    const int g = crk_grid(n, 256);
    crk_step_mark(ctx, 0);
    int rc;
    {
        // inputs into the two kernel orders: m, v, u (gas order) and m (gravity order), with the
        // caller's cotangents
        Bundle in, in_g;
        in.add(io->m, m_k, 1, n);
        in.add(io->v3, v_k, 3, n);
        in.add(io->u, u_k, 1, n);
        if (io->rhobar) in.add(io->rhobar, rhob_k, 1, n);
        if (io->Vbar) in.add(io->Vbar, Vb_k, 1, n);
        in_g.add(io->m, m_g, 1, n);
        if (io->abar3) in_g.add(io->abar3, abar_g, 3, n);
        if ((rc = permute_bundle(ctx, n, lv->kperm, in)) || (rc = permute_bundle(ctx, n, lv->kperm_g, in_g))) return rc;
    }
    unsigned long long *cnt = (unsigned long long *)io->pair_count;
    unsigned long long *swc = cnt ? (unsigned long long *)io->swept_count : nullptr;
    {
        GeomP p{m_k, V_k, rho_k, n, cnt ? cnt + 0 : nullptr, swc ? swc + 0 : nullptr};
        if ((rc = run_stage<GeomStage>(ctx, lv, p, true, CRK_K_GEOMETRY, nullptr, true))) return rc;
    }
    crk_step_mark(ctx, 1);
    {
        if (io->n_singular) CRK_CUDA(ctx, cudaMemsetAsync(io->n_singular, 0, sizeof(int32_t), st));
        CorrP p{V_k, A_k, B_k, gA_k, gB_k, io->n_singular, n, nullptr};
        if ((rc = run_stage<CorrStage>(ctx, lv, p, true, CRK_K_CORRECTIONS, nullptr, true))) return rc;
    }
    if (io->extras) {
        ExtrasP p{m_k, v_k, V_k, A_k, B_k, gA_k, gB_k, rhoR_k, dvdx_k, n, nullptr};
        if ((rc = run_stage<ExtrasStage>(ctx, lv, p, true, CRK_K_EXTRAS, nullptr, true))) return rc;
    }
    crk_step_mark(ctx, 2);
    if (io->extras) {
        HydroP p{m_k, v_k, u_k, V_k, rhoR_k, A_k, B_k, gA_k, gB_k, dv_k, du_k, io->conservation,
                 hp->gamma, hp->alpha, hp->beta, hp->eta2, n, cnt ? cnt + 1 : nullptr, dvdx_k,
                 swc ? swc + 1 : nullptr};
        if ((rc = run_stage<HydroLimStage>(ctx, lv, p, true, CRK_K_HYDRO, io->conservation, true))) return rc;
    } else {
        HydroP p{m_k, v_k, u_k, V_k, rho_k, A_k, B_k, gA_k, gB_k, dv_k, du_k, io->conservation,
                 hp->gamma, hp->alpha, hp->beta, hp->eta2, n, cnt ? cnt + 1 : nullptr, nullptr,
                 swc ? swc + 1 : nullptr};
        if ((rc = run_stage<HydroStage>(ctx, lv, p, true, CRK_K_HYDRO, io->conservation, true))) return rc;
    }
    crk_step_mark(ctx, 3);
    {
        GravP p{};
        p.m = m_g;
        p.a3 = a_g;
        p.rc2 = gp->r_cut * gp->r_cut;
        p.eps2 = gp->eps * gp->eps;
        for (int k = 0; k < 6; ++k) p.c[k] = gp->poly[k];
        p.n = n;
        p.count = cnt ? cnt + 2 : nullptr;
        p.swept = swc ? swc + 2 : nullptr;
        if ((rc = run_stage<GravStage>(ctx, lv, p, false, CRK_K_GRAVITY, nullptr, true))) return rc;
    }
    crk_step_mark(ctx, 4);
    // cotangents not given by the caller: those of sum |a|^2 + sum_gas rho
    if (!io->abar3 || !io->rhobar) {
        cotangent_kernel<<<g, 256, 0, st>>>(n, a_g, lv->pos, io->abar3 ? nullptr : abar_g, io->rhobar ? nullptr : rhob_k);
        ++ctx->launches;
    }
    CRK_LAUNCH_CHECK(ctx, "step cotangents");
    {
        GravAdjP p{};
        p.m = m_g;
        p.abar = abar_g;
        p.gx3 = gx_g;
        p.gm = gm_g;
        p.rc2 = gp->r_cut * gp->r_cut;
        p.eps2 = gp->eps * gp->eps;
        for (int k = 0; k < 6; ++k) p.c[k] = gp->poly[k];
        p.n = n;
        p.count = nullptr;
        if ((rc = run_stage<GravAdjStage>(ctx, lv, p, false, CRK_K_GRAVITY_ADJOINT, nullptr, true))) return rc;
    }
    crk_step_mark(ctx, 5);
    {
        GeomAdjP p{m_k, V_k, rhob_k, io->Vbar ? Vb_k : nullptr, gx2_k, gm2_k, n, nullptr};
        if ((rc = run_stage<GeomAdjStage>(ctx, lv, p, true, CRK_K_GEOMETRY_ADJOINT, nullptr, true))) return rc;
    }
    crk_step_mark(ctx, 6);
    // outputs back to the caller's order (only those asked for)
    {
        Bundle out[3];
        auto give = [&](Bundle &b, const float *src, float *dst, int comps) {
            if (dst) b.add(src, dst, comps, n);
        };
        give(out[0], V_k, io->V, 1);
        give(out[0], rho_k, io->rho, 1);
        give(out[0], A_k, io->A, 1);
        give(out[0], B_k, io->B, 3);
        give(out[0], gA_k, io->gradA, 3);
        give(out[0], gB_k, io->gradB, 9);
        give(out[0], dv_k, io->dvdt3, 3);
        give(out[0], du_k, io->dudt, 1);
        give(out[0], gx2_k, io->gx3_geom, 3);
        give(out[0], gm2_k, io->gm_geom, 1);
        if (io->extras) {
            give(out[1], rhoR_k, io->rho_r, 1);
            give(out[1], dvdx_k, io->dvdx, 9);
        }
        give(out[2], a_g, io->a3, 3);
        give(out[2], gx_g, io->gx3_grav, 3);
        give(out[2], gm_g, io->gm_grav, 1);
        for (int k = 0; k < 3; ++k)
            if ((rc = permute_bundle(ctx, n, k < 2 ? lv->kinv : lv->kinv_g, out[k]))) return rc;
    }
    crk_step_mark(ctx, 7);
    return CRK_OK;
}
