// wide.cuh -- traversal of the tree's four-wide form: the walk that answers closest-hit queries
// wherever nothing asks for the hit/miss links themselves (gsp_dev_scene decides).
//
// A wide node stands for a binary node of even depth and holds its up to four grandchildren (a
// child that is a leaf stands for itself): their boxes as centres and half extents, plane by
// plane, and a reference per child -- eight float4, 128 bytes, one cache line:
//   {c.x}x4 {h.x}x4 | {c.y}x4 {h.y}x4 | {c.z}x4 {h.z}x4 | {ref}x4, unused
// ref >= 0 is a wide node, < 0 is ~(leaf word); an absent child is a leaf of no triangles behind a box
// that no ray meets unless its distances overflow on every axis (an origin at 1e10 with a direction of
// length 1e-29, an infinite direction), so that a walk which goes there goes on after it. Leaves are the
// binary tree's, and the hit is the lexicographic (t, index) minimum of the same triangle tests. A box is
// passed over only when it begins more than 2^-19 of the best t behind it (gsp_reach, gsp_wide_keep), which
// covers the rounding of a triangle's t where that is well conditioned: the hit does not depend on the order
// of the walk then, coincident surfaces included.
//
// What bounds a walk is the chain of dependent node fetches and the instructions per box. The links
// visit 53 boxes for a bounce ray of the 247,234-triangle scene (two per fetch at best) and need six
// copies of the nodes; the wide form makes 13 node fetches for the same ray from one copy (20 MB
// instead of 123 MB for a million triangles, so that it stays in L2). Four children rather than
// eight: eight would make 9 fetches but test 72 boxes for 52, and the trees fill 3.1 of 4 slots but
// 3.4 of 8. Measured against the links when it came: 4,194,304 rays over 1,003,520 triangles 815 -> 596 us,
// 262,147 rays over 247,234 triangles 138 -> 86 us, 1,021 rays 64 -> 24 us (with the last ray of a warp
// walked by all lanes, below), a 512x512 pass 1.30 -> 1.00 ms, a 131x97 one 752 -> 430 us. With what
// followed (four lanes to a ray at the end, the stack's upper entries in shared memory, fewer launches,
// path pools): 570, 67 and 18 us, 0.82 ms and 252 us.
#pragma once

#include "launch.h"
#include "persist.cuh"

#ifndef GSP_WIDE_KEEP
#define GSP_WIDE_KEEP 1
#endif
#ifndef GSP_WIDE_KEEP_TRACE
#define GSP_WIDE_KEEP_TRACE 2
#endif
#ifndef GSP_WIDE_TOP_TRACE
#define GSP_WIDE_TOP_TRACE 12
#endif
#ifndef GSP_WIDE_KEEP_LONG
#define GSP_WIDE_KEEP_LONG 3
#endif
#ifndef GSP_WIDE_CHUNK
#define GSP_WIDE_CHUNK 32
#endif
#ifndef GSP_WIDE_LEAF_BATCH
#define GSP_WIDE_LEAF_BATCH 12
#endif

namespace gspd {

constexpr int kWideLeafBatch = GSP_WIDE_LEAF_BATCH;  // lanes at a leaf that trigger a warp-wide leaf test

// Slab interval of the box c +- h along one axis: tc = (c - o) inv, tc -+ h |inv|. With unit
// roundoff u and an inverse good to 2u, either end is off by at most 5u |tc| + 3u h |inv|. Where
// |tc| <= 2 h |inv| that is below the 32u h |inv| by which gsp_wide_box widens h; else
// both ends have the sign of tc and a relative error of at most 13u, which gsp_reach's 32u cover: the
// test is conservative on both sides of the origin. (A pad of 64u |tmin| for negative tmin, which this
// once had, lets every box through when |tmin| is large against the scene: 683 instead of 14 nodes per
// line through 2,000 triangles at tmin = -FLT_MAX.) Two operations of the half-rate min/max pipe fewer
// per axis and box than min and max over the two planes: that pipe was the busiest at 57-61 % of its cycles.

// BEHIND: the form of the rules for rays with a negative tmin (gsp_reach, gsp_wide_order, gsp_wide_keep). A warp of the
// closest-hit kernel changes to it with its first such ray; the rays beside and after that one may be of either
// kind. In one form for all, the far end would cost every ray an operation per box (an FMA has no absolute value
// of its own; 4,194,304 rays 575 -> 581 us) and the order of negative distances two; the two forms chosen anew
// in every round of the loop cost 2 % (577 -> 590). Without that order, rays behind their origin visited their
// boxes farthest first and dropped none from the stack: 1,048,576 lines through 20,000 triangles 1,338 us, with
// it 684 (917 along the links), through 1,003,520 triangles 608 and 450 (722).

// 1 / d to 1 ulp (2u): all that the slab test needs.
__device__ __forceinline__ float wide_inv(float d) {
    float r;
    asm("rcp.approx.f32 %0, %1;" : "=f"(r) : "f"(fabsf(d) < 1e-30f ? copysignf(1e-30f, d) : d));
    return r;
}

__device__ __forceinline__ void wide_ray(float3 o, float3 d, float tmin, float tmax, RayHit& st) {
    st.o = o;
    st.d = d;
    st.inv = make_float3(wide_inv(d.x), wide_inv(d.y), wide_inv(d.z));
    st.tmin = tmin;
    st.tbest = tmax;
    st.best = -1;
    st.slot = -1;
}

// One ray's walk: the node or leaf it is at (kWalkDone: the walk is over) and the children still
// to visit, each with its key (entry distance; the two low bits hold the child number).
// The stack is beside it, so that passing its address on does not hold these in memory.
struct WideWalk {
    int32_t cur, sp;
};

// Entries [0, K) of a lane's stack are in shared memory, an entry of the warp's lanes side by side (`top`
// points to the lane's first), the others in the lane's local memory. The closest-hit kernel pops 1.5
// times per node it tests, for four lanes of a warp at once; lanes at different depths make a local access
// two L1 wavefronts a lane, beside the nodes' in a pipe that is busy 65 % of the time, but meet no bank
// conflict in shared memory. K = 12 (the 96 KB of an SM's 32 warps come out of the L1 cache):
// 4,194,304 rays 643 -> 625 us, the random half alone 496 -> 474 us, 1,048,576 rays in host memory
// 288 -> 279 us; 4 entries give 650 us, 8 628, 16 628, 20 633. The path kernels, whose path pools have
// taken that shared memory, keep K = 0: with 4 or 8 a 512x512 pass is level and a 131x97 one 6 % slower.
template <int K>
struct WideStack {
    int2 *deep, *top;

    __device__ __forceinline__ int2 get(int i) const {
        if (K > 0 && i < K) return top[32 * i];
        return deep[i - K];
    }
    __device__ __forceinline__ void set(int i, int2 e) const {
        if (K > 0 && i < K)
            top[32 * i] = e;
        else
            deep[i - K] = e;
    }
};

__device__ __forceinline__ void wide_init(WideWalk& w) {
    w.cur = 0;
    w.sp = 0;
}

constexpr int32_t kWideMiss = 0x7fffffff;  // sorts behind every key

template <bool BEHIND, class Stack>
__device__ __forceinline__ int32_t wide_pop(const RayHit& st, WideWalk& w, const Stack& stk) {
    while (w.sp > 0) {
        const int2 e = stk.get(--w.sp);
        if (gsp_wide_keep<BEHIND>(e.x, st.tbest)) return e.y;
    }
    return kWalkDone;
}

// Key of child i: its entry distance as an integer in the same order, with the child number in the two low
// bits, or kWideMiss.
template <bool BEHIND>
__device__ __forceinline__ int32_t wide_key(const RayHit& st, float cx, float hx, float cy, float hy, float cz,
                                            float hz, int i) {
    const float tx = __fmul_rn(cx - st.o.x, st.inv.x), ty = __fmul_rn(cy - st.o.y, st.inv.y),
                tz = __fmul_rn(cz - st.o.z, st.inv.z);
    const float ax = fabsf(st.inv.x), ay = fabsf(st.inv.y), az = fabsf(st.inv.z);
    const float tn = max3f(__fmaf_rn(-hx, ax, tx), __fmaf_rn(-hy, ay, ty), fmaxf(__fmaf_rn(-hz, az, tz), st.tmin));
    const float tf = min3f(__fmaf_rn(hx, ax, tx), __fmaf_rn(hy, ay, ty), __fmaf_rn(hz, az, tz));
    return tn <= gsp_reach<BEHIND>(fminf(st.tbest, tf)) ? ((gsp_wide_order<BEHIND>(tn) & ~3) | i) : kWideMiss;
}

template <class Stack>
__device__ __forceinline__ void wide_push(WideWalk& w, const Stack& stk, int32_t key, int32_t nearest, int32_t ref) {
    if (key != kWideMiss && key != nearest) stk.set(w.sp++, make_int2(key, ref));
}

// Moves to the nearest of the children hit; the others go on the stack as they come (sorting them
// too saves under 1 % of the visits and costs more).
template <bool BEHIND, class Stack>
__device__ __forceinline__ void wide_next(int32_t k0, int32_t k1, int32_t k2, int32_t k3, int4 ref, const RayHit& st,
                                          WideWalk& w, const Stack& stk) {
    const int32_t k = min(min(k0, k1), min(k2, k3));
    if (k == kWideMiss) {
        w.cur = wide_pop<BEHIND>(st, w, stk);
        return;
    }
    wide_push(w, stk, k0, k, ref.x);
    wide_push(w, stk, k1, k, ref.y);
    wide_push(w, stk, k2, k, ref.z);
    wide_push(w, stk, k3, k, ref.w);
    const int32_t a = k & 1 ? ref.y : ref.x, b = k & 1 ? ref.w : ref.z;
    w.cur = k & 2 ? b : a;
}

// Tests the four children of node w.cur and moves on.
template <bool BEHIND, class Stack>
__device__ __forceinline__ void wide_node(const float4* __restrict__ nodes, const RayHit& st, WideWalk& w,
                                          const Stack& stk) {
    const float4* p = nodes + 8 * (int64_t)w.cur;
    float4 cx, hx, cy, hy, cz, hz;
    ldg32(p, cx, hx);
    ldg32(p + 2, cy, hy);
    ldg32(p + 4, cz, hz);
    const int4 ref = __ldg((const int4*)(p + 6));
    const int32_t k0 = wide_key<BEHIND>(st, cx.x, hx.x, cy.x, hy.x, cz.x, hz.x, 0);
    const int32_t k1 = wide_key<BEHIND>(st, cx.y, hx.y, cy.y, hy.y, cz.y, hz.y, 1);
    const int32_t k2 = wide_key<BEHIND>(st, cx.z, hx.z, cy.z, hy.z, cz.z, hz.z, 2);
    const int32_t k3 = wide_key<BEHIND>(st, cx.w, hx.w, cy.w, hy.w, cz.w, hz.w, 3);
    wide_next<BEHIND>(k0, k1, k2, k3, ref, st, w, stk);
}

// Walks the warp's active lanes until no more than `keep` quarters of them still walk: what follows a
// walk then runs for many lanes at once. A path kernel's shading is long (1 of 4; 8.0 ms per eight
// 512x512 passes, against 8.07 with 2 and 8.33 with 3), a ray's end in the closest-hit kernel short:
// 3 in calls that list hits for refinement (4,194,304 rays 574 us, 572 with 3; random ones alone 474 and
// 463), 2 in shorter ones, which end sooner (262,147 rays 67.4 us, 68.1 with 3), and for rays read over
// the link (4,194,304 of them 4,607 Mrays/s, 4,514 with 3).
// Lanes at a leaf wait until kWideLeafBatch of them are, or no lane
// has a node left to test, and test their leaves together (12; 8 costs 1-2 %, 4 costs 5 %).
template <bool BEHIND, class Stack>
__device__ __forceinline__ void wide_steps(const float4* __restrict__ wide, const float4* __restrict__ tris, RayHit& st,
                                           WideWalk& w, const Stack& stk, bool active, int keep) {
    const int stop = (__popc(__ballot_sync(0xffffffffu, active)) * keep) >> 2;
    uint32_t nm, lm;
    do {
        if (active && w.cur >= 0) wide_node<BEHIND>(wide, st, w, stk);
        const bool leaf = active && w.cur < 0 && w.cur != kWalkDone;
        lm = __ballot_sync(0xffffffffu, leaf);
        nm = __ballot_sync(0xffffffffu, active && w.cur >= 0);
        if (lm && (!nm || __popc(lm) >= kWideLeafBatch)) {
            if (leaf) {
                trav_leaf(tris, st, (~w.cur) >> 3, (~w.cur) & 7);
                w.cur = wide_pop<BEHIND>(st, w, stk);
            }
            lm = __ballot_sync(0xffffffffu, active && w.cur != kWalkDone);
        }
    } while (__popc(lm | nm) > stop);
}

// ---- the last rays of a warp, four lanes to a ray --------------------------------------------
// Once a warp's queue is exhausted and no more than eight rays are left, each is handed to four
// lanes, which hold the same state and keep the same stack: a lane tests one child of a node, or one
// triangle of a leaf, and the four exchange what they found. The chain of dependent steps that a
// short launch, or the end of a long one, waits for is then a quarter as long in instructions:
// 262,147 rays 87 -> 76 us, one bounce per pass 1.84 -> 1.69 ms, the batch of 16 scenes 6.26 -> 6.04 ms.
// The last ray of all goes on with the whole warp (coop_wide): left to four lanes, 1,021 single rays
// take 30 us instead of 23 and a 131x97 pass 473 us instead of 392.
constexpr int kQuadRays = 8;

// The lane whose ray this lane's group of four takes over, given the lanes that have one; -1: none.
__device__ __forceinline__ int quad_source(uint32_t lanes) {
    const uint32_t s = __fns(lanes, 0, ((threadIdx.x & 31) >> 2) + 1);
    return s < 32 ? (int)s : -1;
}

__device__ __forceinline__ float3 shfl3(float3 v, int src) {
    const uint32_t F = 0xffffffffu;
    return make_float3(__shfl_sync(F, v.x, src), __shfl_sync(F, v.y, src), __shfl_sync(F, v.z, src));
}

// Copies lane src's walk to this lane (every lane calls it; src: a lane, its own if it has no use).
template <class Stack>
__device__ __forceinline__ void quad_take(RayHit& st, WideWalk& w, const Stack& stk, int src) {
    const uint32_t F = 0xffffffffu;
    st.o = shfl3(st.o, src);
    st.d = shfl3(st.d, src);
    st.inv = shfl3(st.inv, src);
    st.tmin = __shfl_sync(F, st.tmin, src);
    st.tbest = __shfl_sync(F, st.tbest, src);
    st.best = __shfl_sync(F, st.best, src);
    st.slot = __shfl_sync(F, st.slot, src);
    w.cur = __shfl_sync(F, w.cur, src);
    const int old = w.sp;
    w.sp = __shfl_sync(F, old, src);
    const int most = __reduce_max_sync(F, w.sp);
    for (int e = 0; e < most; ++e) {
        const int2 own = e < old ? stk.get(e) : make_int2(0, 0);
        const int2 got = make_int2(__shfl_sync(F, own.x, src), __shfl_sync(F, own.y, src));
        if (e < w.sp) stk.set(e, got);
    }
}

// As wide_steps, for groups of four lanes; `active` is the same in the lanes of a group.
template <int KEEP, bool BEHIND, class Stack>
__device__ __forceinline__ void quad_steps(const float4* __restrict__ wide, const float4* __restrict__ tris, RayHit& st,
                                           WideWalk& w, const Stack& stk, bool active) {
    const uint32_t F = 0xffffffffu;
    const int c = threadIdx.x & 3;
    const int stop = (__popc(__ballot_sync(F, active)) * KEEP) >> 2;
    uint32_t walking;
    do {
        const bool node = active && w.cur >= 0;
        int32_t key = kWideMiss, ref = kWalkDone;
        if (node) {
            const float* q = (const float*)(wide + 8 * (int64_t)w.cur) + c;
            key = wide_key<BEHIND>(st, __ldg(q), __ldg(q + 4), __ldg(q + 8), __ldg(q + 12), __ldg(q + 16), __ldg(q + 20), c);
            ref = __ldg((const int32_t*)q + 24);
        }
        const int32_t k0 = __shfl_sync(F, key, 0, 4), k1 = __shfl_sync(F, key, 1, 4), k2 = __shfl_sync(F, key, 2, 4),
                      k3 = __shfl_sync(F, key, 3, 4);
        const int4 r = make_int4(__shfl_sync(F, ref, 0, 4), __shfl_sync(F, ref, 1, 4), __shfl_sync(F, ref, 2, 4),
                                 __shfl_sync(F, ref, 3, 4));
        if (node) wide_next<BEHIND>(k0, k1, k2, k3, r, st, w, stk);
        const bool leaf = active && w.cur < 0 && w.cur != kWalkDone;
        if (__ballot_sync(F, leaf)) {
            const int32_t word = leaf ? ~w.cur : 0;  // 0: no triangles
            float t = __int_as_float(0x7f800000);    // a hit's t is below the best t, so finite
            int32_t id = 0x7fffffff, slot = -1;
            for (int k = c; k < (word & 7); k += 4) {
                const float4* tp = tris + 3 * (int64_t)((word >> 3) + k);
                const float4 P = __ldg(tp), V1 = __ldg(tp + 1), V2 = __ldg(tp + 2);
                float tt;
                const int32_t ti = __float_as_int(P.w);
                if (tri_hit(st.o, st.d, P, V1, V2, tt) && tt > st.tmin &&
                    (tt < st.tbest || (tt == st.tbest && st.best >= 0 && ti < st.best)) &&
                    (tt < t || (tt == t && ti < id))) {
                    t = tt;
                    id = ti;
                    slot = (word >> 3) + k;
                }
            }
#pragma unroll
            for (int o = 1; o < 4; o <<= 1) {  // the lexicographic (t, index) minimum of the four
                const float t2 = __shfl_xor_sync(F, t, o);
                const int32_t id2 = __shfl_xor_sync(F, id, o), slot2 = __shfl_xor_sync(F, slot, o);
                if (t2 < t || (t2 == t && id2 < id)) {
                    t = t2;
                    id = id2;
                    slot = slot2;
                }
            }
            if (leaf) {
                if (slot >= 0) {
                    st.tbest = t;
                    st.best = id;
                    st.slot = slot;
                }
                w.cur = wide_pop<BEHIND>(st, w, stk);
            }
        }
        walking = __ballot_sync(F, active && w.cur != kWalkDone);
    } while (__popc(walking) > stop);
}

// ---- the last ray of a warp, walked by all 32 lanes ----------------------------------------
// The whole warp takes up to eight nodes off the ray's stack at a time, four lanes to a node and a
// child to a lane, and tests the leaves that were hit eight at a time, a triangle to a lane. More
// boxes are tested than by one lane, in fewer rounds (9 instead of 13 on a bounce ray).
constexpr int kCoopStack = 128;  // entries per warp: at most eight nodes' children are added while 40 fit above
                                 // them (up to kCoopNarrow), then one node's at a time, three more per wide level
constexpr int kCoopNarrow = 40;

struct CoopScratch {
    int2 stk[kCoopStack];
    int32_t leaf[32];
};
static_assert(kCoopNarrow + 24 + 3 * (kWideMaxDepth / 2 + 1) < kCoopStack && kWideStack < kCoopStack - 3, "warp stack");

// Walks lane owner's ray (st, w and stk are that lane's) to its end; every lane calls it and
// receives the ray with its final best hit. Not inlined: the callers' loops keep their registers.
template <bool BEHIND, class Stack>
__device__ __noinline__ RayHit coop_wide(const float4* __restrict__ wide, const float4* __restrict__ tris, RayHit st,
                                         WideWalk w, Stack stk, int owner, CoopScratch* sc) {
    const uint32_t F = 0xffffffffu;
    const int lane = threadIdx.x & 31, slot = lane >> 2, c = lane & 3;
    const uint32_t lt = lanemask_lt();
    st.o = make_float3(__shfl_sync(F, st.o.x, owner), __shfl_sync(F, st.o.y, owner), __shfl_sync(F, st.o.z, owner));
    st.d = make_float3(__shfl_sync(F, st.d.x, owner), __shfl_sync(F, st.d.y, owner), __shfl_sync(F, st.d.z, owner));
    st.inv = make_float3(__shfl_sync(F, st.inv.x, owner), __shfl_sync(F, st.inv.y, owner), __shfl_sync(F, st.inv.z, owner));
    st.tmin = __shfl_sync(F, st.tmin, owner);
    st.tbest = __shfl_sync(F, st.tbest, owner);
    st.best = __shfl_sync(F, st.best, owner);
    st.slot = __shfl_sync(F, st.slot, owner);
    int n = __shfl_sync(F, w.sp, owner) + 1;
    if (lane == owner) {
        for (int i = 0; i < n - 1; ++i) sc->stk[i] = stk.get(i);
        sc->stk[n - 1] = make_int2(INT32_MIN, w.cur);  // the least key: kept
    }
    __syncwarp();
    while (n > 0) {
        const int take = n > kCoopNarrow ? 1 : min(n, 8);
        int2 e = make_int2(0, kWalkDone);
        if (slot < take) e = sc->stk[n - 1 - slot];
        n -= take;
        int32_t key = kWideMiss, ref = kWalkDone;
        if (e.y != kWalkDone && gsp_wide_keep<BEHIND>(e.x, st.tbest)) {
            if (e.y >= 0) {
                const float* q = (const float*)(wide + 8 * (int64_t)e.y) + c;
                key = wide_key<BEHIND>(st, __ldg(q), __ldg(q + 4), __ldg(q + 8), __ldg(q + 12), __ldg(q + 16), __ldg(q + 20), c);
                ref = __ldg((const int32_t*)q + 24);
            } else if (c == 0) {
                key = e.x & ~3;
                ref = e.y;
            }
        }
        const bool hit = key != kWideMiss && ref != kWalkDone;
        const uint32_t nm = __ballot_sync(F, hit && ref >= 0), lm = __ballot_sync(F, hit && ref < 0);
        __syncwarp();  // every lane has read its entry
        if (hit && ref >= 0) sc->stk[n + __popc(nm & lt)] = make_int2(key, ref);
        if (hit && ref < 0) sc->leaf[__popc(lm & lt)] = ~ref;
        n += __popc(nm);
        __syncwarp();
        const int nl = __popc(lm);
        for (int l0 = 0; l0 < nl; l0 += 8) {
            const int32_t word = l0 + slot < nl ? sc->leaf[l0 + slot] : 0;  // 0 triangles
            float t = 0.0f;
            int32_t id = 0, ts = -1;
            bool ok = false;
            for (int k = c; k < (word & 7); k += 4) {  // a lane's second triangle, if any, after its first
                const float4* tp = tris + 3 * (int64_t)((word >> 3) + k);
                const float4 P = __ldg(tp), V1 = __ldg(tp + 1), V2 = __ldg(tp + 2);
                float tt;
                const int32_t ti = __float_as_int(P.w);
                if (tri_hit(st.o, st.d, P, V1, V2, tt) && tt > st.tmin &&
                    (tt < st.tbest || (tt == st.tbest && st.best >= 0 && ti < st.best)) &&
                    (!ok || tt < t || (tt == t && ti < id))) {
                    ok = true;
                    t = tt;
                    id = ti;
                    ts = (word >> 3) + k;
                }
            }
            if (__ballot_sync(F, ok) == 0) continue;
            uint32_t tk = 0xffffffffu;  // t as an unsigned key in float order (-0 and +0 alike)
            if (ok) {
                const uint32_t b = __float_as_uint(t + 0.0f);
                tk = (b & 0x80000000u) ? ~b : (b | 0x80000000u);
            }
            const uint32_t kmin = __reduce_min_sync(F, tk);
            const bool tie = ok && tk == kmin;
            const uint32_t imin = __reduce_min_sync(F, tie ? (uint32_t)id : 0xffffffffu);
            const int win = __ffs(__ballot_sync(F, tie && (uint32_t)id == imin)) - 1;
            st.tbest = __shfl_sync(F, t, win);
            st.best = (int32_t)imin;
            st.slot = __shfl_sync(F, ts, win);
        }
    }
    __syncwarp();  // the scratch may be reused
    return st;
}

}  // namespace gspd
