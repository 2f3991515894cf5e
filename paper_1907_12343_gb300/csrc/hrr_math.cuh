// Device-side definitions shared by the library's kernels: the flags the kernels raise and
// the method's arithmetic (range minimum, node bound, leaf test).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

// Device flags reported through counters[2]
enum : unsigned long long {
    HRR_FLAG_STACK = 1ull,     // traversal stack spill area would overflow (not seen for any tree)
    HRR_FLAG_NONFINITE = 2ull, // a light position or intensity is not finite
    HRR_FLAG_TOPOLOGY = 4ull,  // a node record or parent link is out of range
    HRR_FLAG_RANGE = 8ull,     // an input index (a pair's eye or light) is out of range
    HRR_FLAG_RUNS = 16ull,     // a build's keys have long runs of equal upper halves: sort them fully
    HRR_FLAG_WAIT = 32ull,     // a bounded wait of the sort ran out (cannot happen)
    // keys and values are not what the kernels after the sort take: in no order, or not written
    HRR_FLAG_UNSORTED = HRR_FLAG_RUNS | HRR_FLAG_WAIT,
    HRR_FLAG_LARGE = 64ull,    // a scene has nodes on which slab times can overflow (no error)
};

// ------------------------------------------------------------------------------------
// Device math
// ------------------------------------------------------------------------------------

// Range minimum of the shifted radical inverse, closed form.
//
// With T = (2^32 - r) mod 2^32 (the threshold 1 - r of Sec. 2), the minimum of
// (brev(i) + r) mod 2^32 over [a,b) sits at the smallest brev(i) >= T if any (cases one
// and two of Sec. 2's split), else at the smallest brev(i) (case three, Alg. 1). The
// values brev(i) form a binary trie whose level-k digit is bit k of i, and a level-k
// prefix p is present iff a + ((p - a) mod 2^k) < b. With c = brev(T) (the paper's k_r),
// D = c - a and L = b - a, every quantity of the successor walk is an O(1) bit
// expression:
//   * c is in the range (case one)               iff D < L;
//   * the right sibling of T's path at level k   exists iff bit k of c is 0 and
//     ((D xor 2^k) mod 2^(k+1)) < L;
//   * with h = fls(L), that holds for every zero bit k < h of c, for k = h iff bit h of D
//     is set or (D mod 2^h) < L - 2^h, and above h only for K = h + 1 + ctz(D >> (h+1))
//     when (D mod 2^(h+1)) < L.
// The deepest such level k* fixes the low k*+1 bits of the answer; its members form the
// progression i0, i0 + 2^(k*+1), ... <= b - 1, and by the identity
// Phi_2(l + n 2^d) = 2^-d Phi_2(n) + Phi_2(l) (Sec. 4) the smallest value among them is at
// the multiplier with the most trailing zeros: for s in [x, y], x >= 1, that is y with
// its bits below fls((x-1) xor y) cleared (the same rule, on [a,b), gives case three).
__device__ __forceinline__ uint32_t hrr_most_trailing_zeros(uint32_t x, uint32_t y) {
    // the number in [x, y] with the most trailing zero bits
    if (x == 0u) return 0u;
    const uint32_t h = 31u - __clz((x - 1u) ^ y);
    return y & ~((1u << h) - 1u);
}

__device__ __forceinline__ uint32_t hrr_rangemin_closed(uint32_t a, uint32_t b, uint32_t r,
                                                        uint32_t *argmin) {
    const uint32_t T = 0u - r;
    const uint32_t c = __brev(T);
    const uint32_t L = b - a;
    const uint32_t D = c - a;
    uint32_t k;
    if (D < L) {
        k = c;
    } else {
        const int h = 31 - __clz(L);
        int ks = -1;
        const uint32_t lowD = D & ((2u << h) - 1u);  // 2u << 31 wraps to 0: mask = all ones
        if (lowD < L) {                               // only possible when h <= 30
            const int K = h + __ffs(D >> (h + 1));    // h + 1 + ctz; D >> (h+1) != 0 here
            if (!((c >> K) & 1u)) ks = K;
        }
        if (ks < 0 && !((c >> h) & 1u)) {
            if (((D >> h) & 1u) || (D & ((1u << h) - 1u)) < L - (1u << h)) ks = h;
        }
        if (ks < 0) {
            const uint32_t low = ~c & ((1u << h) - 1u);
            if (low) ks = 31 - __clz(low);
        }
        if (ks >= 0) {
            const uint32_t mask = (2u << ks) - 1u;
            const uint32_t i0 = a + ((D ^ (1u << ks)) & mask);
            const uint32_t s_lo = (i0 >> ks) >> 1;
            const uint32_t s_hi = s_lo + (((b - 1u - i0) >> ks) >> 1);
            const uint32_t s = hrr_most_trailing_zeros(s_lo, s_hi);
            k = ((s << ks) << 1) | (i0 & mask);
        } else {
            k = hrr_most_trailing_zeros(a, b - 1u);
        }
    }
    *argmin = k;
    return __brev(k) + r;
}

// The same minimum without branches, as the smallest of three candidates, for warps whose
// lanes take different cases. With h = fls(L), an interval of L >= 2^h indices holds every
// residue mod 2^h once or twice, and the low h bits of i are the top h bits of brev(i).
// Measured from T = 2^32 - r upward (cyclically), brev(i) + r is the distance of brev(i) from
// T, so:
//   * the indices with c's low h bits (c = brev(T)) share T's top h bits: one at or above T is
//     the minimum, one below T wraps round to the far end. There are one or two of them, i0 =
//     a + ((c - a) mod 2^h) and i0 + 2^h, and both are candidates;
//   * if neither is at or above T the minimum has the next value of the top h bits, i.e. the
//     low h bits of c2 = brev(T + 2^(32-h)), and all of those are above T. There are again
//     one or two, i1 and i1 + 2^h, and the smaller brev has bit h zero: i1 + 2^h when bit h
//     of i1 is set and i1 + 2^h is in the range, else i1.
// The unsigned minimum of the candidates' brev(i) + r is the answer in every case (a wrapped
// or a later candidate is larger). About 27 operations, against about 45 for the successor
// walk above evaluated without branches, which this replaced: the traversals are bound by
// instruction issue and compute one per node visit (two per sample-visit in the several-
// samples form). Build, cull and weights of 1920x1080 eyes and 2^20 lights: 112.8 ms before,
// 100.3 ms with it; four samples of 480x270 eyes and 2^17 lights: 10.75 and 7.87 ms. The
// argmin is brev(v - r).
__device__ __forceinline__ uint32_t hrr_range_min_value(uint32_t a, uint32_t L, uint32_t r, uint32_t T, uint32_t c) {
    const uint32_t s = (uint32_t)__clz((int)L);   // h = 31 - s
    const uint32_t mh = 0x7FFFFFFFu >> s;         // 2^h - 1
    const uint32_t c2 = __brev(T + (2u << s));    // 2 << 31 = 0: h = 0 has one residue
    const uint32_t x0 = (c - a) & mh, x1 = (c2 - a) & mh;
    const uint32_t rem = L & mh;                  // residues below rem (from a) occur twice
    const uint32_t i0 = a + x0, i1 = a + x1;
    const uint32_t j0 = x0 < rem ? i0 + mh + 1u : i0;
    const uint32_t k1 = (x1 < rem && (i1 & (mh + 1u)) != 0u) ? i1 + mh + 1u : i1;
    return __vimin3_u32(__brev(i0) + r, __brev(j0) + r, __brev(k1) + r);
}

// The same for the leaves [a, z] of a hierarchy (a <= z < 2^31, so nothing below overflows): a
// candidate past the end may be replaced by any index of the range, so the second index of
// either class is clamped to z instead of tested, and both of the second class are tried.
__device__ __forceinline__ uint32_t hrr_range_min_leaves(uint32_t a, uint32_t z, uint32_t r, uint32_t T, uint32_t c) {
    uint32_t s;  // 31 - floor(log2(z - a + 1))
    asm("bfind.shiftamt.u32 %0, %1;" : "=r"(s) : "r"(z - a + 1u));
    const uint32_t mh = 0x7FFFFFFFu >> s;
    const uint32_t c2 = __brev(T + (2u << s));
    const uint32_t i0 = a + ((c - a) & mh), i1 = a + ((c2 - a) & mh);
    const uint32_t j0 = min(i0 + mh + 1u, z), j1 = min(i1 + mh + 1u, z);
    return min(__vimin3_u32(__brev(i0) + r, __brev(j0) + r, __brev(i1) + r), __brev(j1) + r);
}

// Exact per-pair test (round to nearest, canonical order, no FMA): accept iff
// xi < ceil(p 2^32), p = min(1, (tau I) / max(d2, 1e-4)). For 0 < p < 1, p 2^32 is an
// exact float below 2^32, so its ceiling fits in 32 bits. The traversals ask it only about
// lights that the node test on the light alone (a box of one point, whose range minimum is
// the light's xi) leaves undecided; that test is sound, so the accepted set is this rule's.
__device__ __forceinline__ bool hrr_pair_accepts(uint32_t xi, float tau, float lx, float ly, float lz, float inten,
                                                 float ex, float ey, float ez) {
    const float dx = __fsub_rn(lx, ex);
    const float dy = __fsub_rn(ly, ey);
    const float dz = __fsub_rn(lz, ez);
    float d2 = __fmul_rn(dx, dx);
    d2 = __fadd_rn(d2, __fmul_rn(dy, dy));
    d2 = __fadd_rn(d2, __fmul_rn(dz, dz));
    const float den = fmaxf(d2, 1e-4f);
    const float num = __fmul_rn(tau, inten);
    const float p = fminf(1.0f, __fdiv_rn(num, den));
    if (p >= 1.0f) return true;
    if (!(p > 0.0f)) return false;
    return xi < __float2uint_ru(__fmul_rn(p, 4294967296.0f));
}

// max(a, b, c) in one instruction (three-operand max of sm_100 and later; a NaN operand
// is ignored as in fmaxf). Exact, so the same as fmaxf(a, fmaxf(b, c)).
__device__ __forceinline__ float hrr_max3(float a, float b, float c) {
    float d;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
    return d;
}

// The node test's scale for a frame's tau: RU(tau 2^32 (1 + 2^-22)); tau 2^32 is exact (a
// power-of-two scaling), infinite when it overflows.
__device__ __forceinline__ float hrr_node_scale(float tau) {
    return __fmul_ru(tau * 4294967296.0f, 1.0f + 0x1p-22f);
}

// Conservative cull test of a node with box [lo, hi] and maximum intensity imax, for an eye
// at e, with the scale s = hrr_node_scale(tau):
//   den = max(d2, 1e-4), d2 = RD(gz^2 + RD(gy^2 + RD(gx^2))) (fused, rounded down) with
//         per-axis gaps g = max(0, RD(lo - e), RD(e - hi)): at most the float32 max(d^2, 1e-4)
//         of any light in the box;
//   rhs = RU(s imax) >= 2^32 tau imax (1 + 2^-22) >= 2^32 RN(tau I) (1 + 2^-24)(1 + 2^-23) of
//         every light with 0 < I <= imax, when tau I is a normal float.
// The node is culled at range minimum v iff RD(RD(v) den) >= rhs. Then for every such light,
// v den_i >= 2^32 RN(tau I_i) (1 + 2^-23) >= 2^32 RN(RN(tau I_i) / den_i), so v is at least
// its threshold ceil(p_i 2^32). The cases outside that chain are sound as well: rhs <= 0
// (tau imax <= 0: no light below has p > 0) culls at any v, v = 0 included, and otherwise
// v = 0 never culls; if tau I is subnormal the light's threshold is at most 1 and a cull
// needs v >= 1 (rhs > 0); rhs = +inf or NaN (tau 2^32 overflows) never culls.
__device__ __forceinline__ void hrr_node_bound(float scale, float lox, float loy, float loz,
                                               float hix, float hiy, float hiz, float imax,
                                               float ex, float ey, float ez, float &den,
                                               float &rhs) {
    const float gx = hrr_max3(0.0f, __fsub_rd(lox, ex), __fsub_rd(ex, hix));
    const float gy = hrr_max3(0.0f, __fsub_rd(loy, ey), __fsub_rd(ey, hiy));
    const float gz = hrr_max3(0.0f, __fsub_rd(loz, ez), __fsub_rd(ez, hiz));
    float d2 = __fmul_rd(gx, gx);
    d2 = __fmaf_rd(gy, gy, d2);
    d2 = __fmaf_rd(gz, gz, d2);
    den = fmaxf(d2, 1e-4f);
    rhs = __fmul_ru(scale, imax);
}

__device__ __forceinline__ bool hrr_node_culls(uint32_t v, float den, float rhs) {
    return __fmul_rd(__uint2float_rd(v), den) >= rhs;
}

// The node test of two boxes at once (the children of a binary node), on the packed pairs of
// a traversal record: nlo and nhi hold the negated box corners of both, one axis per pair. The
// same operations on the same values as hrr_node_bound, rounded alike (e - lo rounded up is
// the negated lo - e rounded down), two per instruction: packed 32-bit float arithmetic
// halves the issue slots of everything but the three-operand maxima.
using hrr_f2 = unsigned long long;  // two floats, the first in the low word

__device__ __forceinline__ hrr_f2 hrr_pack2(float a, float b) {
    hrr_f2 d;
    asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(a), "f"(b));
    return d;
}
__device__ __forceinline__ void hrr_unpack2(hrr_f2 d, float &a, float &b) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(d));
}
__device__ __forceinline__ hrr_f2 hrr_gap2(hrr_f2 nlo, hrr_f2 nhi, hrr_f2 e) {
    hrr_f2 up, dn;
    asm("add.rp.f32x2 %0, %1, %2;" : "=l"(up) : "l"(e), "l"(nlo));
    asm("add.rm.f32x2 %0, %1, %2;" : "=l"(dn) : "l"(e), "l"(nhi));
    float u0, u1, d0, d1;
    hrr_unpack2(up, u0, u1);
    hrr_unpack2(dn, d0, d1);
    return hrr_pack2(hrr_max3(0.0f, -u0, d0), hrr_max3(0.0f, -u1, d1));
}
// Both boxes' sides of the cull test (hrr_node_bound).
__device__ __forceinline__ void hrr_bound2(hrr_f2 nlox, hrr_f2 nloy, hrr_f2 nloz, hrr_f2 nhix, hrr_f2 nhiy, hrr_f2 nhiz,
                                           hrr_f2 imax, hrr_f2 ex, hrr_f2 ey, hrr_f2 ez, float scale, hrr_f2 &den,
                                           hrr_f2 &rhs) {
    const hrr_f2 gx = hrr_gap2(nlox, nhix, ex), gy = hrr_gap2(nloy, nhiy, ey), gz = hrr_gap2(nloz, nhiz, ez);
    hrr_f2 d2;
    asm("mul.rm.f32x2 %0, %1, %1;" : "=l"(d2) : "l"(gx));
    asm("fma.rm.f32x2 %0, %1, %1, %0;" : "+l"(d2) : "l"(gy));
    asm("fma.rm.f32x2 %0, %1, %1, %0;" : "+l"(d2) : "l"(gz));
    float a, b;
    hrr_unpack2(d2, a, b);
    den = hrr_pack2(fmaxf(a, 1e-4f), fmaxf(b, 1e-4f));
    asm("mul.rp.f32x2 %0, %1, %2;" : "=l"(rhs) : "l"(imax), "l"(hrr_pack2(scale, scale)));
}
// Whether each box survives (is not culled) at range minima v0, v1, where `ok`.
__device__ __forceinline__ void hrr_survive2(hrr_f2 den, hrr_f2 rhs, uint32_t v0, uint32_t v1, bool ok, bool &s0, bool &s1) {
    hrr_f2 lhs;
    asm("mul.rm.f32x2 %0, %1, %2;"
        : "=l"(lhs)
        : "l"(hrr_pack2(__uint2float_rd(v0), __uint2float_rd(v1))), "l"(den));
    float l0, l1, r0, r1;
    hrr_unpack2(lhs, l0, l1);
    hrr_unpack2(rhs, r0, r1);
    s0 = ok && !(l0 >= r0);
    s1 = ok && !(l1 >= r1);
}

// The paired form (hrr_tree::pairs) of a binary record, for trees without paired records.
__device__ __forceinline__ void hrr_load_binary(const float4 *p, hrr_f2 &nlox, hrr_f2 &nloy, hrr_f2 &nloz, hrr_f2 &nhix,
                                                hrr_f2 &nhiy, hrr_f2 &nhiz, hrr_f2 &imax, hrr_f2 &links) {
    float4 q[4];
#pragma unroll
    for (int k = 0; k < 4; k += 2)
        asm("ld.global.nc.L1::no_allocate.v8.f32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
            : "=f"(q[k].x), "=f"(q[k].y), "=f"(q[k].z), "=f"(q[k].w), "=f"(q[k + 1].x), "=f"(q[k + 1].y), "=f"(q[k + 1].z),
              "=f"(q[k + 1].w)
            : "l"(p + k));
    nlox = hrr_pack2(-q[0].x, -q[2].x);
    nloy = hrr_pack2(-q[0].y, -q[2].y);
    nloz = hrr_pack2(-q[0].z, -q[2].z);
    nhix = hrr_pack2(-q[1].x, -q[3].x);
    nhiy = hrr_pack2(-q[1].y, -q[3].y);
    nhiz = hrr_pack2(-q[1].z, -q[3].z);
    imax = hrr_pack2(q[0].w, q[2].w);
    links = hrr_pack2(q[1].w, q[3].w);
}
