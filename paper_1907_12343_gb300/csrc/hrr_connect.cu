// Connection evaluation: the step after the culling (the connections it keeps are what a
// bidirectional path tracer then evaluates).
//
// Every accepted pair (eye j, light id) carries the Russian-roulette weight
// (I / max(d^2, 1e-4)) / p_ij, with d^2 and p_ij the acceptance rule's own float32 values,
// times the visibility of the open segment eye -> light against a triangle scene. The
// per-eye sums of the weights are unbiased estimates of the eyes' unculled sums.
//
// The scene is a bounding-volume hierarchy over the triangles: the Morton order of their
// centroids, the binary radix tree over it and the box pass of the light hierarchies (with
// triangle boxes, widened so that floating-point slab tests can never reject a box that holds a
// crossing) give a binary tree, and every three levels of it become one node of eight children
// whose boxes are stored in seven bits a side, rounded outwards (Scene nodes, below). Each lane of
// a persistent grid traces one pair's shadow segment at a time (any hit ends it) and takes the
// next pair when it is done.
#include <algorithm>
#include <new>

#include "hrr_boxes.cuh"
#include "hrr_internal.cuh"
#include "hrr_order.cuh"
#include "hrr_sort.cuh"

struct hrr_scene {
    int device = 0;
    uint32_t n = 0;
    bool large = false;         // a node of more than kLargeNode a side
    uint32_t *nodes = nullptr;  // n - 1 nodes of kNodeWords words (below); one when n == 1
    float *tris = nullptr;     // sorted triangles, 16 floats each: v0, e1 = v1 - v0, e2 = v2 - v0, pad
};

namespace {

constexpr int kThreads = 256;
constexpr int kTriFloats = 16;  // a sorted triangle's stride (64 bytes: aligned 256-bit loads)

// Scene nodes. Node g holds the up to eight nodes or triangles three levels below binary node g
// (a leaf met on the way stands for itself), in one 128-byte line of which 96 bytes are read:
//   words 0-2   origin o of the node's box grid
//   word 3      bytes: exponents of S = 2^(k-127) per axis (x, y, z), mask of the children there are
//   words 4-15  per axis: 8 low sides, 8 high sides, a byte 0x80 | q each; the side lies at
//               o + q S / 128, so 1 + q / 128 is one byte permutation away from a float
//   words 16-23 children: a triangle (bit 31 set) or a node
// (Wide nodes with quantised boxes are a published method: Ylitie, Karras and Laine, "Efficient
// Incoherent Ray Traversal on GPUs Through Compressed Wide BVHs", HPG 2017.) A binary walk over
// 64-byte nodes was bound by its scattered loads (93% of the L1 data pipe, 87 loads a segment);
// this one is bound by instructions (70% of the issue slots at 32 warps per SM, L1 at 53%). 8.3e6
// segments against 2^18 triangles, scene build included: 6.35 ms, now 4.20 to 4.48.
constexpr uint32_t kNodeWords = 32;
constexpr uint32_t kTriangle = 0x80000000u;
// A direction component counts as at least 1e-30 (the margin of the triangles' boxes covers the
// difference), so an eye inside a node of S up to 2^27 has slab times up to 2 S 1e30, finite.
constexpr uint32_t kLargeNode = 127 + 27;  // exponent of the largest such S
constexpr int kSharedStack = 24;   // entries of a segment's stack in shared memory
constexpr int kLocalStack = 232;   // ... and below them: 7 per level of at most 33, and a margin

__global__ void __launch_bounds__(kThreads) centroid_kernel(const float *__restrict__ tri, uint32_t n,
                                                             float *cx, float *cy, float *cz, unsigned long long *flags) {
    const uint32_t i = blockIdx.x * kThreads + threadIdx.x;
    if (i >= n) return;
    const float *t = tri + 9 * (size_t)i;
    float s[3];
    for (int c = 0; c < 3; ++c) {
        const float a = t[c], b = t[3 + c], d = t[6 + c];
        if (!isfinite(a) || !isfinite(b) || !isfinite(d)) atomicOr(flags, HRR_FLAG_NONFINITE);
        s[c] = (a + b + d) * (1.0f / 3.0f);
    }
    if (!isfinite(s[0]) || !isfinite(s[1]) || !isfinite(s[2])) atomicOr(flags, HRR_FLAG_NONFINITE);
    cx[i] = s[0];
    cy[i] = s[1];
    cz[i] = s[2];
}

// A box that surely holds a triangle: its vertices' bounds widened by 2^-16 of the
// larger of their magnitude and the box's extent (float32 rounding in the slab and
// triangle tests is below 2^-20 of those).
__device__ __forceinline__ void tri_box(const float *t, float lo[3], float hi[3]) {
    for (int c = 0; c < 3; ++c) {
        const float a = fminf(fminf(t[c], t[3 + c]), t[6 + c]);
        const float b = fmaxf(fmaxf(t[c], t[3 + c]), t[6 + c]);
        const float m = fmaxf(fmaxf(fabsf(a), fabsf(b)), b - a) * 1.52587890625e-05f + 1e-30f;
        lo[c] = a - m;
        hi[c] = b + m;
    }
}

// Sorted triangles (v0 and the edges e1, e2, the segment test's first six roundings, done once
// here, so that one 256-bit load and one 32-bit load fetch a triangle) and their boxes.
__global__ void __launch_bounds__(kThreads) triangles_kernel(const float *__restrict__ tri, const uint32_t *__restrict__ perm,
                                                             uint32_t n, float *__restrict__ sorted,
                                                             float4 *__restrict__ box, const unsigned long long *flags) {
    const uint32_t i = blockIdx.x * kThreads + threadIdx.x;
    if (i >= n || (*flags & HRR_FLAG_WAIT)) return;  // no permutation
    const float *t = tri + 9 * (size_t)(perm ? perm[i] : i);
    float v[9];
    for (int c = 0; c < 9; ++c) v[c] = t[c];
    float4 *o = reinterpret_cast<float4 *>(sorted + kTriFloats * (size_t)i);
    store32(o, make_float4(v[0], v[1], v[2], __fsub_rn(v[3], v[0])),
            make_float4(__fsub_rn(v[4], v[1]), __fsub_rn(v[5], v[2]), __fsub_rn(v[6], v[0]), __fsub_rn(v[7], v[1])));
    store32(o + 2, make_float4(__fsub_rn(v[8], v[2]), 0.f, 0.f, 0.f), make_float4(0.f, 0.f, 0.f, 0.f));
    float lo[3], hi[3];
    tri_box(v, lo, hi);
    if (box) store32(box + 2 * (size_t)i, make_float4(lo[0], lo[1], lo[2], 0.f), make_float4(hi[0], hi[1], hi[2], 0.f));
}

// Leaves that are boxes.
struct BoxLeaves {
    static constexpr bool kOwnNodes = true;
    const float4 *box;
    __device__ __forceinline__ Box operator()(uint32_t i) const { return box_of(box[2 * (size_t)i], box[2 * (size_t)i + 1]); }
};

// One node of eight children per binary node (those that no traversal reaches as well: they are
// cheaper made than told apart). The grid's step s = S / 128 leaves the box 124 steps, its origin
// lies a 64th of a step below the box, and every side moves outwards by a 128th of a step before
// it is rounded outwards: more than the rounding of the segment's slab arithmetic on a grid near
// the eye (2^-16 of the grid; far from it the slab test's own widening covers it).
__global__ void __launch_bounds__(kThreads) collapse_kernel(const float4 *__restrict__ nodes, uint32_t n,
                                                            uint32_t *__restrict__ out, unsigned long long *flags) {
    const uint32_t g = blockIdx.x * kThreads + threadIdx.x;
    if (g >= n - 1 || (*flags & (HRR_FLAG_NONFINITE | HRR_FLAG_UNSORTED | HRR_FLAG_TOPOLOGY))) return;
    float4 lo[8], hi[8];
    uint32_t f[8], l[8], id[8];  // ranges and node numbers; an empty place has f > l
    for (int k = 0; k < 8; ++k) {
        f[k] = 1;
        l[k] = 0;
        id[k] = 0;
        lo[k] = hi[k] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
    {
        const uint32_t other = __float_as_uint(nodes[4 * (size_t)g + 3].w);
        f[0] = min(g, other);
        l[0] = max(g, other);
        id[0] = g;
    }
#pragma unroll
    for (int step = 4; step >= 1; step >>= 1) {  // places 0, 2 step, 4 step, ... split into two
#pragma unroll
        for (int k = 0; k < 8; k += 2 * step) {
            if (f[k] >= l[k]) continue;  // empty, or a leaf: it keeps its place
            const float4 *r = nodes + 4 * (size_t)id[k];
            const float4 r1 = r[1];
            const uint32_t split = __float_as_uint(r1.w);
            lo[k + step] = r[2];
            hi[k + step] = r[3];
            f[k + step] = split + 1u;
            l[k + step] = l[k];
            id[k + step] = split + 1u;
            lo[k] = r[0];
            hi[k] = r1;
            l[k] = split;
            id[k] = split;
        }
    }
    float a[3] = {1e38f, 1e38f, 1e38f}, b[3] = {-1e38f, -1e38f, -1e38f};
    for (int k = 0; k < 8; ++k)
        if (f[k] <= l[k]) {
            a[0] = fminf(a[0], lo[k].x); a[1] = fminf(a[1], lo[k].y); a[2] = fminf(a[2], lo[k].z);
            b[0] = fmaxf(b[0], hi[k].x); b[1] = fmaxf(b[1], hi[k].y); b[2] = fmaxf(b[2], hi[k].z);
        }
    uint32_t w[24];
    w[3] = 0;
    for (int c = 0; c < 3; ++c) {
        // s = 2^m, the least with 124 s >= the extent, at least 2^-112; past 2^119 (and for a box
        // that is not finite) the axis gets S = infinity, whose sides are no numbers, and the slab
        // test goes by the other axes
        int m = min((int)((__float_as_uint(fmaxf((b[c] - a[c]) * (1.0f / 124.0f), 0x1p-113f)) >> 23) & 255u) - 126, 119);
        float s, o;
        for (;; ++m) {
            s = __uint_as_float((uint32_t)(m + 127) << 23);
            o = __fsub_rd(a[c], s * 0.015625f);
            if (__fsub_ru(b[c], o) <= 126.0f * s || m >= 119) break;
        }
        const bool covered = __fsub_ru(b[c], o) <= 126.0f * s;
        w[c] = covered ? __float_as_uint(o) : 0u;
        w[3] |= (covered ? (uint32_t)(m + 7 + 127) : 255u) << (8 * c);
        if (!covered || (uint32_t)(m + 7 + 127) > kLargeNode) atomicOr(flags, HRR_FLAG_LARGE);
        const float inv = __uint_as_float((uint32_t)(127 - m) << 23);
        uint32_t ql[2] = {0, 0}, qh[2] = {0, 0};
        for (int k = 0; k < 8; ++k) {
            const float x = c == 0 ? lo[k].x : c == 1 ? lo[k].y : lo[k].z, y = c == 0 ? hi[k].x : c == 1 ? hi[k].y : hi[k].z;
            const float u = fminf(fmaxf(floorf(__fsub_rd(x, o) * inv - 0.0078125f), 0.0f), 127.0f);
            const float v = fminf(fmaxf(ceilf(__fsub_ru(y, o) * inv + 0.0078125f), 0.0f), 127.0f);
            ql[k >> 2] |= (0x80u | (uint32_t)u) << (8 * (k & 3));
            qh[k >> 2] |= (0x80u | (uint32_t)v) << (8 * (k & 3));
        }
        w[4 + 4 * c] = ql[0];
        w[5 + 4 * c] = ql[1];
        w[6 + 4 * c] = qh[0];
        w[7 + 4 * c] = qh[1];
    }
    for (int k = 0; k < 8; ++k) {
        if (f[k] <= l[k]) w[3] |= 1u << (24 + k);
        w[16 + k] = f[k] == l[k] ? kTriangle | f[k] : id[k];
    }
    float4 *to = reinterpret_cast<float4 *>(out + kNodeWords * (size_t)g);
    for (int k = 0; k < 3; ++k)
        store32(to + 2 * k,
                make_float4(__uint_as_float(w[8 * k]), __uint_as_float(w[8 * k + 1]), __uint_as_float(w[8 * k + 2]),
                            __uint_as_float(w[8 * k + 3])),
                make_float4(__uint_as_float(w[8 * k + 4]), __uint_as_float(w[8 * k + 5]), __uint_as_float(w[8 * k + 6]),
                            __uint_as_float(w[8 * k + 7])));
}

// Open segment e -> e + D, t in (1e-4, 1 - 1e-4), against the closed triangle (v0, v1, v2),
// stored as v0, e1 = v1 - v0, e2 = v2 - v0: Moller-Trumbore with every product and sum
// rounded separately (no fused operations), dot products summed x + y then + z, one
// correctly rounded reciprocal of det.
__device__ __forceinline__ bool segment_hits(const float e[3], const float D[3], const float *__restrict__ tri) {
    float v0x, v0y, v0z, e1x, e1y, e1z, e2x, e2y;
    asm("ld.global.nc.L1::no_allocate.v8.f32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
        : "=f"(v0x), "=f"(v0y), "=f"(v0z), "=f"(e1x), "=f"(e1y), "=f"(e1z), "=f"(e2x), "=f"(e2y)
        : "l"(tri));
    const float e2z = __ldg(tri + 8);
    const float Px = __fsub_rn(__fmul_rn(D[1], e2z), __fmul_rn(D[2], e2y));
    const float Py = __fsub_rn(__fmul_rn(D[2], e2x), __fmul_rn(D[0], e2z));
    const float Pz = __fsub_rn(__fmul_rn(D[0], e2y), __fmul_rn(D[1], e2x));
    const float det = __fadd_rn(__fadd_rn(__fmul_rn(e1x, Px), __fmul_rn(e1y, Py)), __fmul_rn(e1z, Pz));
    if (det == 0.0f) return false;
    const float inv = __frcp_rn(det);
    const float Tx = __fsub_rn(e[0], v0x), Ty = __fsub_rn(e[1], v0y), Tz = __fsub_rn(e[2], v0z);
    const float u = __fmul_rn(__fadd_rn(__fadd_rn(__fmul_rn(Tx, Px), __fmul_rn(Ty, Py)), __fmul_rn(Tz, Pz)), inv);
    if (!(u >= 0.0f && u <= 1.0f)) return false;
    const float Qx = __fsub_rn(__fmul_rn(Ty, e1z), __fmul_rn(Tz, e1y));
    const float Qy = __fsub_rn(__fmul_rn(Tz, e1x), __fmul_rn(Tx, e1z));
    const float Qz = __fsub_rn(__fmul_rn(Tx, e1y), __fmul_rn(Ty, e1x));
    const float v = __fmul_rn(__fadd_rn(__fadd_rn(__fmul_rn(D[0], Qx), __fmul_rn(D[1], Qy)), __fmul_rn(D[2], Qz)), inv);
    if (!(v >= 0.0f && __fadd_rn(u, v) <= 1.0f)) return false;
    const float t = __fmul_rn(__fadd_rn(__fadd_rn(__fmul_rn(e2x, Qx), __fmul_rn(e2y, Qy)), __fmul_rn(e2z, Qz)), inv);
    return t > 1e-4f && t < 1.0f - 1e-4f;
}

// 32 bytes of a node as one 256-bit read-only load that does not allocate in L1 (scattered
// nodes are rarely reused from L1; filling it would cost L1 data-pipe cycles).
__device__ __forceinline__ void load8(const uint32_t *p, uint32_t (&v)[8]) {
    asm("ld.global.nc.L1::no_allocate.v8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7])
        : "l"(p));
}
// min(a, b, c) in one instruction; a NaN operand is ignored.
__device__ __forceinline__ float min3(float a, float b, float c) {
    float d;
    asm("min.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
    return d;
}
// Times at which the segment passes one axis' near and far sides of child k (k & 3 in the words).
__device__ __forceinline__ void sides(uint32_t near, uint32_t far, int k, hrr_f2 slope, hrr_f2 start, float &tn, float &tf) {
    // bytes (0, 0, 0x80 | q, 0x3f): 1 + q / 128
    const uint32_t sel = 0x7044u | ((uint32_t)k << 8);
    const hrr_f2 v = hrr_pack2(__uint_as_float(__byte_perm(near, 0x3F000000u, sel)),
                               __uint_as_float(__byte_perm(far, 0x3F000000u, sel)));
    hrr_f2 t;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(t) : "l"(v), "l"(slope), "l"(start));
    hrr_unpack2(t, tn, tf);
}
// The children of a node that the segment's [0, 1] meets (slab test, widened by 2^-18). LARGE: the
// start of an axis may overflow (a zero or nearly zero component on a node of more than 2^27), which
// would put both sides at the same infinity, even around an eye inside the node; 0 b + b makes such a
// start no number, which the minima and maxima ignore, and the axis rejects nothing. The three
// operations took 2% of the walk, so scenes without such nodes have a kernel without them.
template <bool LARGE>
__device__ __forceinline__ uint32_t meets(const uint32_t (&h)[8], const uint32_t (&q)[8], const float (&e)[3],
                                          const float (&inv)[3]) {
    hrr_f2 slope[3], start[3];
    uint32_t near[3][2], far[3][2];
    const uint32_t side[3][4] = {{h[4], h[5], h[6], h[7]}, {q[0], q[1], q[2], q[3]}, {q[4], q[5], q[6], q[7]}};
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const float S = __uint_as_float(((h[3] >> (8 * c)) & 255u) << 23);
        const float a = S * inv[c];
        float b = ((__uint_as_float(h[c]) - S) - e[c]) * inv[c];
        if (LARGE) b = __fmaf_rn(b, 0.0f, b);
        slope[c] = hrr_pack2(a, a);
        start[c] = hrr_pack2(b, b);
        const bool back = inv[c] < 0.0f;
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            near[c][k] = back ? side[c][2 + k] : side[c][k];
            far[c][k] = back ? side[c][k] : side[c][2 + k];
        }
    }
    uint32_t mask = 0;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        float xn, xf, yn, yf, zn, zf;
        sides(near[0][k >> 2], far[0][k >> 2], k & 3, slope[0], start[0], xn, xf);
        sides(near[1][k >> 2], far[1][k >> 2], k & 3, slope[1], start[1], yn, yf);
        sides(near[2][k >> 2], far[2][k >> 2], k & 3, slope[2], start[2], zn, zf);
        const float tn = fmaxf(hrr_max3(xn, yn, zn), 0.0f), tf = fminf(min3(xf, yf, zf), 1.0f);
        if (tn <= tf * (1.0f + 0x1p-18f)) mask |= 1u << k;
    }
    return mask & (h[3] >> 24);
}

struct ConnectArgs {
    hrr_eyes eyes;
    uint32_t n_eyes;
    hrr_lights lights;
    uint32_t n_lights;
    float tau;
    const uint2 *pairs;
    unsigned long long n_pairs;
    const uint32_t *nodes;  // scene, or NULL
    const float *tris;    // sorted triangles, kTriFloats each
    uint32_t n_tris;
    float *weight;        // per pair, or NULL
    uint8_t *visible;     // per pair, or NULL
    float *eye_sum;       // per eye
    unsigned long long *flags;   // without a scene: a host word, written only by a bad pair
    unsigned long long *cursor;  // next pair to trace (starts at 0)
};

#ifndef HRR_CONNECT_REFILL_BELOW
#define HRR_CONNECT_REFILL_BELOW 24
#endif
constexpr uint32_t kRefillBelow = HRR_CONNECT_REFILL_BELOW;  // refill idle lanes once fewer are busy

// The outputs of pair k (eye j): weight times visibility, the visibility bit, the eye's sum.
__device__ __forceinline__ void finish(const ConnectArgs &A, unsigned long long k, uint32_t j, float w, bool vis) {
    const float out = vis ? w : 0.0f;
    if (A.weight) A.weight[k] = out;
    if (A.visible) A.visible[k] = vis ? 1 : 0;
    if (out != 0.0f) atomicAdd(&A.eye_sum[j], out);
}

// Lights as float4 by id, so that a pair's light is one scattered load.
__global__ void __launch_bounds__(kThreads) pack_lights_kernel(hrr_lights l, uint32_t n, float4 *packed) {
    for (size_t i = blockIdx.x * kThreads + threadIdx.x; i < n; i += gridDim.x * kThreads)  // n may be up to 2^32 - 1
        packed[i] = make_float4(l.x[i], l.y[i], l.z[i], l.intensity[i]);
}

// Without a scene every connection is visible: a pass over the pairs, 4 x 32 of them per warp and
// iteration. What bounds it is the scattered loads of the lights (requests for single lines leave
// L2 at 2.9e11 a second), so calls with many pairs per light read them packed, one request a pair
// instead of four; and the culling writes runs of one eye's pairs, so a warp sums each run before
// the atomic: 1.35e8 pairs of 2^20 lights took 2.61 ms with four gathers and an atomic per pair,
// now 0.76 ms (the pairs alone are 0.16 ms of memory traffic).
constexpr int kWeightItems = 4;
template <bool PACKED>
__global__ void __launch_bounds__(kThreads) weights_kernel(const ConnectArgs A, const float4 *__restrict__ packed) {
    const uint32_t lane = threadIdx.x & 31u;
    const unsigned long long warps = (unsigned long long)gridDim.x * (kThreads / 32);
    constexpr unsigned long long kChunk = 32 * kWeightItems;
    for (unsigned long long c = (unsigned long long)blockIdx.x * (kThreads / 32) + threadIdx.x / 32; c * kChunk < A.n_pairs;
         c += warps) {
        uint2 pr[kWeightItems];
        float4 l[kWeightItems];
        float ex[kWeightItems], ey[kWeightItems], ez[kWeightItems];
        bool ok[kWeightItems];
#pragma unroll
        for (int t = 0; t < kWeightItems; ++t) {
            const unsigned long long k = c * kChunk + 32u * t + lane;
            pr[t] = k < A.n_pairs ? __ldcs(&A.pairs[k]) : make_uint2(0xFFFFFFFFu, 0u);
            ok[t] = k < A.n_pairs;
        }
#pragma unroll
        for (int t = 0; t < kWeightItems; ++t) {
            if (ok[t] && (pr[t].x >= A.n_eyes || pr[t].y >= A.n_lights)) {
                __stcs(A.flags, (unsigned long long)HRR_FLAG_RANGE);
                ok[t] = false;
            }
            if (!ok[t]) continue;
            const uint32_t i = pr[t].y;
            l[t] = PACKED ? __ldg(&packed[i])
                          : make_float4(A.lights.x[i], A.lights.y[i], A.lights.z[i], A.lights.intensity[i]);
            ex[t] = A.eyes.x[pr[t].x];
            ey[t] = A.eyes.y[pr[t].x];
            ez[t] = A.eyes.z[pr[t].x];
        }
#pragma unroll
        for (int t = 0; t < kWeightItems; ++t) {
            float w = 0.0f;
            if (ok[t]) {
                const float dx = __fsub_rn(l[t].x, ex[t]);
                const float dy = __fsub_rn(l[t].y, ey[t]);
                const float dz = __fsub_rn(l[t].z, ez[t]);
                float d2 = __fmul_rn(dx, dx);
                d2 = __fadd_rn(d2, __fmul_rn(dy, dy));
                d2 = __fadd_rn(d2, __fmul_rn(dz, dz));
                const float den = fmaxf(d2, 1e-4f);
                const float p = fminf(1.0f, __fdiv_rn(__fmul_rn(A.tau, l[t].w), den));
                w = __fdiv_rn(__fdiv_rn(l[t].w, den), p);
                const unsigned long long k = c * kChunk + 32u * t + lane;
                if (A.weight) A.weight[k] = w;
                if (A.visible) A.visible[k] = 1;
            }
            // each run of one eye, summed into its first lane
            const uint32_t j = ok[t] ? pr[t].x : 0xFFFFFFFFu;
            const uint32_t left = __shfl_up_sync(0xFFFFFFFFu, j, 1);
            const bool head = lane == 0u || left != j;
            const unsigned heads = __ballot_sync(0xFFFFFFFFu, head);
            const uint32_t end = lane == 31u || (heads >> (lane + 1u)) == 0u ? 32u : lane + __ffs(heads >> (lane + 1u));
#pragma unroll
            for (uint32_t d = 1; d < 32; d <<= 1) {
                const float o = __shfl_down_sync(0xFFFFFFFFu, w, d);
                if (lane + d < end) w = __fadd_rn(w, o);
            }
            if (head && ok[t] && w != 0.0f) atomicAdd(&A.eye_sum[j], w);
        }
    }
}

// Persistent segments: each lane traces one pair's segment, at most one node and one triangle per
// step, and a warp refills its idle lanes from the global pair cursor (one atomic per refill), so
// lanes do not idle behind the warp's longest segment. A segment ends at its first crossing
// (occluded) or when its stack runs dry (visible). The stack's first entries are in shared memory,
// interleaved by lane (no bank conflicts whatever the depths). Letting nodes and triangles take
// turns warp by warp (triangles only when 8, 12, 16 or 20 lanes had one) left too many lanes
// waiting: 5.1 to 6.0 ms against 4.5; refilling below 16 or 28 busy lanes 4.6 and 4.8 ms.
template <bool LARGE>
__global__ void __launch_bounds__(kThreads) connect_kernel(const ConnectArgs A) {
    __shared__ uint32_t stack_all[kSharedStack][kThreads];
    uint32_t deep[kLocalStack];
    const int lane = threadIdx.x & 31;
    const unsigned lt = (1u << lane) - 1u;
    bool alive = false, more = true;
    unsigned long long k = 0;
    uint32_t j = 0, cur = 0, steps = 0;
    int sp = 0;
    float w = 0.0f;
    float e[3] = {0.f, 0.f, 0.f}, D[3] = {0.f, 0.f, 0.f}, inv[3] = {0.f, 0.f, 0.f};
    auto pop = [&]() {
        --sp;
        return sp < kSharedStack ? stack_all[sp][threadIdx.x] : deep[sp - kSharedStack];
    };
    for (;;) {
        unsigned alive_mask = __ballot_sync(0xFFFFFFFFu, alive);
        if (more && (uint32_t)__popc(alive_mask) < kRefillBelow) {
            const unsigned idle = ~alive_mask;
            unsigned long long base = 0;
            if (lane == 0) base = atomicAdd(A.cursor, (unsigned long long)__popc(idle));
            base = __shfl_sync(0xFFFFFFFFu, base, 0);
            if (base + __popc(idle) >= A.n_pairs) more = false;
            if (!alive) {
                k = base + __popc(idle & lt);
                if (k < A.n_pairs) {
                    const uint2 pr = A.pairs[k];
                    if (pr.x >= A.n_eyes || pr.y >= A.n_lights) {
                        atomicOr(A.flags, HRR_FLAG_RANGE);
                    } else {
                        j = pr.x;
                        e[0] = A.eyes.x[j]; e[1] = A.eyes.y[j]; e[2] = A.eyes.z[j];
                        const float l0 = A.lights.x[pr.y], l1 = A.lights.y[pr.y], l2 = A.lights.z[pr.y];
                        const float inten = A.lights.intensity[pr.y];
                        D[0] = __fsub_rn(l0, e[0]); D[1] = __fsub_rn(l1, e[1]); D[2] = __fsub_rn(l2, e[2]);
                        // the weight: the acceptance rule's d^2 and p, then (I / den) / p
                        float d2 = __fmul_rn(D[0], D[0]);
                        d2 = __fadd_rn(d2, __fmul_rn(D[1], D[1]));
                        d2 = __fadd_rn(d2, __fmul_rn(D[2], D[2]));
                        const float den = fmaxf(d2, 1e-4f);
                        const float p = fminf(1.0f, __fdiv_rn(__fmul_rn(A.tau, inten), den));
                        w = __fdiv_rn(__fdiv_rn(inten, den), p);
                        // a component below 1e-30 is taken as that: its slab then admits exactly
                        // the boxes whose range holds e (up to 1e-30, a conservative margin)
                        for (int c = 0; c < 3; ++c) inv[c] = __frcp_rn(fabsf(D[c]) < 1e-30f ? copysignf(1e-30f, D[c]) : D[c]);
                        cur = A.n_tris == 1 ? kTriangle : 0u;
                        sp = 0;
                        steps = 0;
                        alive = true;
                    }
                }
            }
            alive_mask = __ballot_sync(0xFFFFFFFFu, alive);
        }
        if (alive_mask == 0u && !more) break;
        if (!alive) continue;
        bool have = true, hit = false;  // cur is still to be looked at; the segment is blocked
        if (!(cur & kTriangle)) {
            // corrupt nodes: out-of-range links, an impossible depth, or more steps than there
            // are nodes
            if (cur >= A.n_tris - 1u || ++steps >= A.n_tris || sp > kSharedStack + kLocalStack - 8) {
                atomicOr(A.flags, HRR_FLAG_TOPOLOGY);
                alive = false;
                continue;
            }
            uint32_t h[8], q[8], ref[8];
            const uint32_t *node = A.nodes + kNodeWords * (size_t)cur;
            load8(node, h);
            load8(node + 8, q);
            load8(node + 16, ref);
            const uint32_t mask = meets<LARGE>(h, q, e, inv);
            if (sp <= kSharedStack - 8) {
                uint32_t *at = &stack_all[sp][threadIdx.x];
#pragma unroll
                for (int c = 0; c < 8; ++c)
                    if ((mask >> c) & 1u) {
                        *at = ref[c];
                        at += kThreads;
                    }
            } else {
                int s = sp;
#pragma unroll
                for (int c = 0; c < 8; ++c)
                    if ((mask >> c) & 1u) {
                        if (s < kSharedStack) stack_all[s][threadIdx.x] = ref[c];
                        else deep[s - kSharedStack] = ref[c];
                        ++s;
                    }
            }
            sp += __popc(mask);
            have = sp > 0;
            if (have) cur = pop();
        }
        if (have && (cur & kTriangle)) {
            const uint32_t i = cur & ~kTriangle;
            if (i >= A.n_tris) {
                atomicOr(A.flags, HRR_FLAG_TOPOLOGY);
                alive = false;
                continue;
            }
            hit = segment_hits(e, D, A.tris + kTriFloats * (size_t)i);
            have = sp > 0;
            if (have && !hit) cur = pop();
        }
        if (hit || !have) {
            finish(A, k, j, w, !hit);
            alive = false;
        }
    }
}

// Sorts by the key bits from `shift` up, as the light builder does. All that is done with before the
// binary nodes are collapsed is kept in the memory of the nodes they become (106 of its 128 bytes
// a triangle), so a build takes 256 bytes a triangle at most, not 362.
int scene_attempt(hrr_ctx *ctx, const float *tris, uint32_t n, hrr_scene *sc, int shift) {
    cudaStream_t st = ctx->stream;
    const size_t un = n;
    unsigned long long *flags = ctx->counters + 2;
    const size_t work = 3 * pad256(sizeof(float) * un) + 2 * pad256(sizeof(uint64_t) * un) + 2 * pad256(sizeof(uint32_t) * un) +
                        pad256(sort_scratch_bytes(un)) + pad256(sizeof(float4) * un) + pad256(2 * sizeof(float4) * un) +
                        box_scratch_bytes(n);
    const bool fits = work <= sizeof(uint32_t) * kNodeWords * (un - 1);  // few triangles: the padding does not
    char *scratch = nullptr;
    HRR_CUDA(ctx, hrr_alloc(ctx, &scratch, pad256(sizeof(hrr_node) * un) + (fits ? 0 : work)));
    char *p = scratch;
    hrr_node *nodes = carve<hrr_node>(p, un);
    if (fits) p = reinterpret_cast<char *>(sc->nodes);
    float *cx = carve<float>(p, un), *cy = carve<float>(p, un), *cz = carve<float>(p, un);
    uint64_t *keys0 = carve<uint64_t>(p, un), *keys1 = carve<uint64_t>(p, un);
    uint32_t *vals0 = carve<uint32_t>(p, un), *perm = carve<uint32_t>(p, un);
    const SortScratch ss = carve_sort(p, un);
    float4 *spos = carve<float4>(p, un), *box = carve<float4>(p, 2 * un);
    const BoxScratch bs = carve_boxes(p, n);
    const unsigned g = (unsigned)((un + kThreads - 1) / kThreads);
    cudaError_t e = cudaMemsetAsync(flags, 0, sizeof(unsigned long long), st);
    if (e == cudaSuccess) e = cudaMemsetAsync(ss.hist, 0, sort_scratch_bytes(un), st);
    if (e == cudaSuccess) {
        centroid_kernel<<<g, kThreads, 0, st>>>(tris, n, cx, cy, cz, flags);
        const int passes = sort_passes(shift);
        morton_kernel<<<morton_grid(n), kThreads, 0, st>>>(cx, cy, cz, cx, n, keys0, shift, passes, ss.hist, flags);
        sort_enqueue(keys0, vals0, keys1, perm, n, shift, ss, flags, st);
        launch_chained(shift ? gather_sorted_kernel<true> : gather_sorted_kernel<false>, g, kThreads, st,
            cx, cy, cz, cx, keys0, vals0, n, keys1, perm, spos, bs, flags);
        launch_chained(topology_kernel, g, kThreads, st, keys1, n, nodes, bs.leaf_parent, bs.int_parent, flags);
        triangles_kernel<<<g, kThreads, 0, st>>>(tris, perm, n, sc->tris, box, flags);
        boxes_enqueue(BoxLeaves{box}, n, nodes, {nullptr, nullptr}, bs, flags, st);
        collapse_kernel<<<g, kThreads, 0, st>>>(reinterpret_cast<const float4 *>(nodes), n, sc->nodes, flags);
        ctx->launches += 8 + passes;
        e = cudaGetLastError();
    }
    cudaFreeAsync(scratch, st);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(&ctx->host_counters[2], flags, sizeof(unsigned long long), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) return hrr_cuda_fail(ctx, e, "scene build");
    const unsigned long long f = ctx->host_counters[2];
    if (f & HRR_FLAG_NONFINITE) return hrr_fail(ctx, HRR_ERR_INVALID_ARG, "a triangle vertex is not finite");
    if ((f & HRR_FLAG_RUNS) && shift) return scene_attempt(ctx, tris, n, sc, 0);
    if (f & HRR_FLAG_WAIT) return hrr_fail(ctx, HRR_ERR_TIMEOUT, "a wait of the sort ran out");
    if (f & HRR_FLAG_TOPOLOGY) return hrr_fail(ctx, HRR_ERR_DEVICE, "scene links");
    sc->large = (f & HRR_FLAG_LARGE) != 0;
    return HRR_OK;
}

// A scene of one triangle: no nodes, the triangle alone.
int scene_of_one(hrr_ctx *ctx, const float *tris, hrr_scene *sc) {
    cudaStream_t st = ctx->stream;
    unsigned long long *flags = ctx->counters + 2;
    float *cen = nullptr;
    HRR_CUDA(ctx, hrr_alloc(ctx, &cen, 3 * sizeof(float)));
    cudaError_t e = cudaMemsetAsync(flags, 0, sizeof(unsigned long long), st);
    if (e == cudaSuccess) {
        centroid_kernel<<<1, kThreads, 0, st>>>(tris, 1u, cen, cen + 1, cen + 2, flags);
        triangles_kernel<<<1, kThreads, 0, st>>>(tris, nullptr, 1u, sc->tris, nullptr, flags);
        ctx->launches += 2;
        e = cudaGetLastError();
    }
    cudaFreeAsync(cen, st);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(&ctx->host_counters[2], flags, sizeof(unsigned long long), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) return hrr_cuda_fail(ctx, e, "scene build");
    if (ctx->host_counters[2] & HRR_FLAG_NONFINITE)
        return hrr_fail(ctx, HRR_ERR_INVALID_ARG, "a triangle vertex is not finite");
    return HRR_OK;
}

}  // namespace

extern "C" {

int hrr_build_scene(hrr_ctx *ctx, const float *dev_tris, uint32_t n_tris, hrr_scene **out) {
    if (!ctx) return HRR_ERR_INVALID_ARG;
    if (!out) return hrr_fail(ctx, HRR_ERR_INVALID_ARG, "out is NULL");
    *out = nullptr;
    if (!dev_tris || n_tris == 0 || n_tris > 0x7FFFFFFFu)
        return hrr_fail(ctx, HRR_ERR_INVALID_ARG, "need 1 .. 2^31 - 1 triangles");
    DeviceGuard g(ctx->device);
    hrr_scene *sc = new (std::nothrow) hrr_scene();
    if (!sc) return hrr_fail(ctx, HRR_ERR_OOM, "host allocation of the scene");
    sc->device = ctx->device;
    sc->n = n_tris;
    cudaError_t e = hrr_alloc(ctx, &sc->tris, sizeof(float) * kTriFloats * (size_t)n_tris);
    if (e == cudaSuccess) e = hrr_alloc(ctx, &sc->nodes, sizeof(uint32_t) * kNodeWords * (size_t)std::max(n_tris - 1u, 1u));
    const int rc = e != cudaSuccess ? hrr_cuda_fail(ctx, e, "scene allocation")
                   : n_tris == 1    ? scene_of_one(ctx, dev_tris, sc)
                                    : scene_attempt(ctx, dev_tris, n_tris, sc, kTopShift);
    if (rc != HRR_OK) {
        const std::string err = ctx->err;
        hrr_free_scene(ctx, sc);
        ctx->err = err;
        return rc;
    }
    *out = sc;
    return HRR_OK;
}

int hrr_free_scene(hrr_ctx *ctx, hrr_scene *scene) {
    if (!ctx || !scene) return HRR_ERR_INVALID_ARG;
    DeviceGuard g(ctx->device);
    if (scene->nodes) cudaFreeAsync(scene->nodes, ctx->stream);
    if (scene->tris) cudaFreeAsync(scene->tris, ctx->stream);
    delete scene;
    return HRR_OK;
}

int hrr_connect(hrr_ctx *ctx, hrr_eyes eyes, uint32_t n_eyes, hrr_lights lights, uint32_t n_lights, float tau,
                const uint32_t *dev_pairs, uint64_t n_pairs, const hrr_scene *scene, float *dev_weight,
                uint8_t *dev_visible, float *dev_eye_sum) {
    if (!ctx) return HRR_ERR_INVALID_ARG;
    if (!(tau >= 0.0f) || !(tau < __builtin_huge_valf())) return hrr_fail(ctx, HRR_ERR_INVALID_ARG, "tau must be finite and >= 0");
    if (n_pairs && (!dev_pairs || !eyes.x || !eyes.y || !eyes.z || !lights.x || !lights.y || !lights.z ||
                    !lights.intensity))
        return hrr_fail(ctx, HRR_ERR_INVALID_ARG, "a pair, eye or light array is NULL");
    if (n_eyes && !dev_eye_sum) return hrr_fail(ctx, HRR_ERR_INVALID_ARG, "dev_eye_sum is NULL");
    if (((uintptr_t)dev_pairs & 7u) != 0) return hrr_fail(ctx, HRR_ERR_INVALID_ARG, "dev_pairs must be 8-byte aligned");
    if (scene && scene->device != ctx->device) return hrr_fail(ctx, HRR_ERR_INVALID_ARG, "scene lives on another device");
    DeviceGuard g(ctx->device);
    cudaStream_t st = ctx->stream;
    unsigned long long *flags = scene ? ctx->counters + 2 : &ctx->host_counters[2];
    ctx->host_counters[2] = 0;
    if (scene) HRR_CUDA(ctx, cudaMemsetAsync(flags, 0, 2 * sizeof(unsigned long long), st));  // flags, pair cursor
    if (n_eyes) HRR_CUDA(ctx, cudaMemsetAsync(dev_eye_sum, 0, sizeof(float) * (size_t)n_eyes, st));
    if (n_pairs) {
        ConnectArgs A{};
        A.eyes = eyes;
        A.n_eyes = n_eyes;
        A.lights = lights;
        A.n_lights = n_lights;
        A.tau = tau;
        A.pairs = reinterpret_cast<const uint2 *>(dev_pairs);
        A.n_pairs = n_pairs;
        A.nodes = scene ? scene->nodes : nullptr;
        A.tris = scene ? scene->tris : nullptr;
        A.n_tris = scene ? scene->n : 0;
        A.weight = dev_weight;
        A.visible = dev_visible;
        A.eye_sum = dev_eye_sum;
        A.flags = flags;
        A.cursor = ctx->counters + 3;
        // packing pays from a few pairs per light on (its pass reads and writes 32 bytes a light; a
        // pair saves three requests) and where the extra launch is small beside the rest
        float4 *packed = nullptr;
        if (!scene && n_lights && n_pairs >= (1u << 20) && n_pairs / 4 >= n_lights &&
            hrr_alloc(ctx, &packed, sizeof(float4) * (size_t)n_lights) != cudaSuccess) {
            cudaGetLastError();
            packed = nullptr;  // no memory for it: gather from the arrays
        }
        const auto walk = scene && scene->large ? connect_kernel<true> : connect_kernel<false>;
        const void *fn = scene ? reinterpret_cast<const void *>(walk)
                               : packed ? reinterpret_cast<const void *>(weights_kernel<true>)
                                        : reinterpret_cast<const void *>(weights_kernel<false>);
        int per_sm = 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, kThreads, 0) != cudaSuccess || per_sm < 1)
            per_sm = 1;
        const unsigned long long per_block = scene ? kThreads : kThreads * kWeightItems;
        const unsigned long long want = (n_pairs + per_block - 1) / per_block;
        const unsigned grid = (unsigned)std::min<unsigned long long>(want, (unsigned long long)per_sm * ctx->sm_count);
        hrr_timing_begin(ctx);
        if (packed) {
            pack_lights_kernel<<<(unsigned)std::min<size_t>(((size_t)n_lights + kThreads - 1) / kThreads, ctx->sm_count * 8), kThreads,
                                 0, st>>>(lights, n_lights, packed);
            ++ctx->launches;
        }
        if (scene) walk<<<grid, kThreads, 0, st>>>(A);
        else if (packed) weights_kernel<true><<<grid, kThreads, 0, st>>>(A, packed);
        else weights_kernel<false><<<grid, kThreads, 0, st>>>(A, nullptr);
        hrr_timing_end(ctx);
        ++ctx->launches;
        if (packed) cudaFreeAsync(packed, st);
        HRR_CUDA(ctx, cudaGetLastError());
    }
    if (scene)
        HRR_CUDA(ctx, cudaMemcpyAsync(&ctx->host_counters[2], flags, sizeof(unsigned long long), cudaMemcpyDeviceToHost, st));
    HRR_CUDA(ctx, cudaStreamSynchronize(st));
    if (ctx->host_counters[2] & HRR_FLAG_RANGE) return hrr_fail(ctx, HRR_ERR_INVALID_ARG, "a pair's eye or light index is out of range");
    if (ctx->host_counters[2] & (HRR_FLAG_STACK | HRR_FLAG_TOPOLOGY))
        return hrr_fail(ctx, HRR_ERR_DEVICE, "corrupt scene records");
    return HRR_OK;
}

}  // extern "C"
