// path_pool.cuh -- the persistent path kernel of long launches over the four-wide tree: each warp keeps
// more paths than it has lanes. Included by sppm.cu only.
//
// A lane that carries one path from bounce to bounce makes its warp alternate between walking with a
// few lanes left and shading with the few that have finished. Here a warp has a pool of up to kPool
// paths in shared memory: lanes walk the rays of some, the rest wait either with a new ray (ready) or
// for their hit to be shaded (done). A lane whose walk ends puts its hit down and takes the next
// ready ray at once; when nothing is ready, up to 32 done paths are shaded together, and each one that
// ended makes room for the next of the launch's queue. Against a path per lane: eight 512x512 passes
// 7.62 -> 6.57 ms, the Cornell box 480 -> 432 us, a 131x97 pass 301 -> 268 us, shaded 333x217 1.51 -> 1.40
// ms, the batch of 16 scenes 5.78 -> 5.26 ms (128 M instead of 148 M warp instructions for a 256x256
// launch of 262,144 photons, 14.6 instead of 13.4 lanes each). The one-bounce photon pass runs in the
// same launch as the eye paths, whose longest chain it used to wait for: four passes 1.64 -> 1.20 ms.
//
// Not kept: one copy of the shading code for the pool and the last paths (fewer instruction fetches,
// but a longer chain per bounce at the end: 6.95 ms per eight 512x512 passes); the last paths in a
// second launch, spread over all warps (7.30 ms: it starts when the slowest warp has drained its pool).
#pragma once

#include "sppm_paths.cuh"

// Paths a warp keeps. More leave the L1 cache less: 48 against 44: a 131x97 pass 251.5 against 248.0 us, the
// batch 5.18 against 5.13 ms, one bounce per pass 1.186 against 1.172 ms; 36: batch 5.20; 64: 5.39 (of 5.26 then).
#ifndef GSP_POOL
#define GSP_POOL 44
#endif
// Resident blocks per SM: 72 registers, without spills for one scene, 16 bytes for many (8: 1 % slower, 6: 1 %
// faster in the batch, 1 % slower at 512x512); with shading data 96, none for one scene, 36 bytes for many (6 spill
// for one: 1.50 against 1.41 ms).
#ifndef GSP_POOL_MIN_BLOCKS
#define GSP_POOL_MIN_BLOCKS 7
#endif
#ifndef GSP_POOL_SHADE_MIN_BLOCKS
#define GSP_POOL_SHADE_MIN_BLOCKS 5
#endif
#ifndef GSP_POOL_KEEP_READY  // quarters of the walking lanes that walk on while rays are ready / none are
#define GSP_POOL_KEEP_READY 3
#endif
#ifndef GSP_POOL_KEEP_DRY
#define GSP_POOL_KEEP_DRY 2
#endif

namespace gspd {

constexpr int kPool = GSP_POOL;
constexpr int32_t kFreeSlot = 0x40000000;  // meta of a slot without a path

struct PathPool {
    float ray[6][kPool];  // origin, direction
    float t[kPool];       // the finished walk's hit: distance, triangle slot in leaf order (-1: none)
    int32_t hit[kPool];
    float w[3][kPool];    // eye: throughput; photon: flux
    int32_t s[4][kPool];  // PRNG
    int32_t id[kPool];    // pixel or path
    int32_t job[kPool];   // multi-scene launches: the path's job
    int32_t meta[kPool];  // depth | deposits << 8 | eye << 31, or kFreeSlot
    uint8_t ready[kPool], done[kPool];

    __device__ __forceinline__ void put_ray(int k, float3 o, float3 d) {
        ray[0][k] = o.x;
        ray[1][k] = o.y;
        ray[2][k] = o.z;
        ray[3][k] = d.x;
        ray[4][k] = d.y;
        ray[5][k] = d.z;
    }
    __device__ __forceinline__ void get_ray(int k, float3& o, float3& d) const {
        o = make_float3(ray[0][k], ray[1][k], ray[2][k]);
        d = make_float3(ray[3][k], ray[4][k], ray[5][k]);
    }
    __device__ __forceinline__ void put_state(int k, float3 v, const Rng& r, int32_t m) {
        w[0][k] = v.x;
        w[1][k] = v.y;
        w[2][k] = v.z;
#pragma unroll
        for (int j = 0; j < 4; ++j) s[j][k] = r.s[j];
        meta[k] = m;
    }
    __device__ __forceinline__ void get_state(int k, float3& v, Rng& r) const {
        v = make_float3(w[0][k], w[1][k], w[2][k]);
#pragma unroll
        for (int j = 0; j < 4; ++j) r.s[j] = s[j][k];
    }
};

// tmin of a path's ray: primary rays start at the camera.
__device__ __forceinline__ float path_tmin(int32_t meta, float eps) { return meta == (int32_t)0x80000000u ? 0.0f : eps; }

// Shades the hit (triangle slot `hit`, FP32 distance t) of a path's ray. True: the path goes on along
// (o, d), its state updated in v, rng and meta. `lead` as in path_interact.
template <bool SHADE, bool REGEN>
__device__ __forceinline__ bool pool_shade(const PathJob& J, int32_t id, int32_t hit, float t, float3& o, float3& d, float3& v,
                                           Rng& rng, int32_t& meta, bool lead) {
    const DevScene& S = J.S;
    const PassDev& P = J.P;
    const bool eye = meta < 0, one_bounce = REGEN && !eye;
    int32_t depth = meta & 0xff;
    uint32_t ndep = (uint32_t)(meta >> 8) & 0xffu;
    bool more = false;
    if (hit >= 0) {
        Hit h;
        h.slot = hit;
        h.t = t;
        h.u = h.v = 0.0f;
        const float4 v0 = __ldg(S.tris + 3 * (int64_t)hit);
        h.id = __float_as_int(v0.w);
        float tt;
        if (plane_t(f3(v0), f3(__ldg(S.shade + h.id)), f3(__ldg(S.nlo + h.id)), o, d, tt)) h.t = tt;
        const uint32_t base = one_bounce ? (uint32_t)id : (uint32_t)id * kSlotsPerPath;
        more = path_interact<SHADE>(S, P, J.O, J.D, eye, id, h, o, d, v, rng, one_bounce ? base : base + depth,
                                    one_bounce ? base : base + ndep, ndep, lead);
        if (more) {
            ++depth;
            more = eye ? depth <= P.max_eye : depth < P.max_photon;
        }
    }
    if (one_bounce) {  // the path waits for the next pass
        if (lead) {
            J.R.ro[id] = make_float4(o.x, o.y, o.z, __int_as_float(depth));
            J.R.rd[id] = make_float4(d.x, d.y, d.z, __int_as_float(more ? 1 : 0));
            J.R.rphi[id] = make_float4(v.x, v.y, v.z, 0.0f);
        }
        more = false;
    }
    if (!more && !eye && lead) J.D.pcount[id] = ndep;
    meta = depth | (int32_t)(ndep << 8) | (eye ? (int32_t)0x80000000u : 0);
    return more;
}

// The paths of one job (MULTI false: `one`, whose items are its eye-queue entries, then its photon-queue
// entries; a warp takes `chunk` at once) or of many (MULTI: jobs, as k_paths_multi). pool: paths a warp
// keeps (32 .. kPool). REGEN: behind the eye items come the one-bounce photon pass's threads, each of
// which goes on with its stored path or starts a new one, traces one ray and stores the path again.
template <bool MULTI, bool SHADE, bool REGEN>
__global__ void __launch_bounds__(kTraceThreads, SHADE ? GSP_POOL_SHADE_MIN_BLOCKS : GSP_POOL_MIN_BLOCKS)
k_paths_pool(const __grid_constant__ PathJob one, const PathJob* __restrict__ jobs, int32_t njobs, int32_t total_chunks,
             uint32_t* __restrict__ ctr, int32_t chunk, int32_t pool) {
    const uint32_t F = 0xffffffffu;
    __shared__ PathPool pools[kTraceThreads / 32];
    __shared__ CoopScratch scratch[kTraceThreads / 32];
    const int lane = threadIdx.x & 31;
    const uint32_t lt = lanemask_lt();
    PathPool& pl = pools[threadIdx.x >> 5];
    WarpQueue wq;
    MultiQueue mq;
    wait_previous();
    const int32_t ne1 = !MULTI && one.ne_ptr ? (int32_t)*one.ne_ptr : 0;
    if (MULTI)
        mq.init(jobs, njobs, total_chunks);
    else
        wq.init(ne1 + (REGEN ? one.nregen : one.np_ptr ? (int32_t)*one.np_ptr : 0), chunk);
    for (int k = lane; k < pool; k += 32) {
        pl.done[k] = (uint8_t)k;
        pl.meta[k] = kFreeSlot;
    }
    __syncwarp();
    int nready = 0, ndone = pool;
    RayHit st;
    WideWalk w;
    int2 deep[kWideStack];
    const WideStack<0> stk{deep, nullptr};
    uint32_t starts = 0;  // REGEN: paths started by this lane
    int at = -1;          // the slot whose ray this lane walks
    const float4 *wide = one.S.wide, *tris = one.S.tris;  // and the tree it walks (MULTI: its job's)
    st.slot = -1;
    w.cur = kWalkDone;
    w.sp = 0;
    while (true) {
        uint32_t idle = __ballot_sync(F, at < 0);
        if (idle && nready) {  // idle lanes take ready rays
            const int rank = __popc(idle & lt);
            if (at < 0 && rank < nready) {
                at = pl.ready[nready - 1 - rank];
                float3 o, d;
                pl.get_ray(at, o, d);
                const PathJob& J = MULTI ? jobs[pl.job[at]] : one;
                if (MULTI) {
                    wide = J.S.wide;
                    tris = J.S.tris;
                }
                wide_ray(o, d, path_tmin(pl.meta[at], J.P.eps), __int_as_float(0x7f800000), st);
                wide_init(w);
            }
            nready = max(nready - __popc(idle), 0);
            idle = __ballot_sync(F, at < 0);
        }
        const int busy = 32 - __popc(idle);
        if (ndone >= 32 || (ndone && nready == 0 && (ndone >= busy || busy + ndone <= kQuadRays))) {
            const int k = lane < ndone ? pl.done[ndone - 1 - lane] : -1;
            ndone = max(ndone - 32, 0);
            bool vacant = k >= 0, goes_on = false;
            if (k >= 0 && pl.meta[k] != kFreeSlot) {
                float3 o, d, v;
                Rng rng;
                int32_t meta = pl.meta[k];
                pl.get_ray(k, o, d);
                pl.get_state(k, v, rng);
                const PathJob& J = MULTI ? jobs[pl.job[k]] : one;
                goes_on = pool_shade<SHADE, REGEN>(J, pl.id[k], pl.hit[k], pl.t[k], o, d, v, rng, meta, true);
                vacant = !goes_on;
                if (goes_on) {
                    pl.put_ray(k, o, d);
                    pl.put_state(k, v, rng, meta);
                }
            }
            int32_t jb = 0;  // a path that ended makes room for the next item
            const int32_t got = MULTI ? mq.take(vacant, jobs, njobs, ctr, jb) : wq.take(vacant, ctr);
            if (got >= 0) {
                const PathJob& J = MULTI ? jobs[jb] : one;
                const int32_t ne = MULTI ? (J.ne_ptr ? (int32_t)*J.ne_ptr : 0) : ne1;
                const bool eye = got < ne;
                if (MULTI) pl.job[k] = jb;
                if (REGEN && !eye) {
                    const int32_t id = got - ne;
                    Rng rng = rng_seed(J.P.seed, J.P.scene_id, 1u, pass_index(J.P), (uint64_t)id);
                    const float4 a = J.R.ro[id], b = J.R.rd[id];
                    float3 o = f3(a), d = f3(b), phi = f3(J.R.rphi[id]);
                    int32_t depth = __float_as_int(a.w);
                    if (__float_as_int(b.w) == 0) {  // the stored path has ended: start a new one
                        emit_photon(J.E, rng, o, d, phi);
                        depth = 0;
                        ++starts;
                    }
                    pl.put_ray(k, o, d);
                    pl.put_state(k, phi, rng, depth);
                    pl.id[k] = id;
                } else {
                    const PathQ Q = eye ? J.qe : J.qp;
                    const size_t j = (size_t)(eye ? got : got - ne);
                    const float4 a = Q.ray[2 * j], c = Q.ray[2 * j + 1], ww = Q.w[j];
                    pl.put_ray(k, f3(a), f3(c));
                    pl.put_state(k, f3(ww), rng_from(Q.rng[j]), Q.meta[j] | (eye ? (int32_t)0x80000000u : 0));
                    pl.id[k] = __float_as_int(ww.w);
                }
                goes_on = true;
            }
            const uint32_t on = __ballot_sync(F, goes_on);
            if (goes_on) pl.ready[nready + __popc(on & lt)] = (uint8_t)k;
            nready += __popc(on);
            __syncwarp();
            continue;
        }
        if (busy == 0) break;
        if ((MULTI ? mq.done : wq.done) && nready == 0 && ndone == 0 && busy <= kQuadRays) break;
        wide_steps<false>(wide, tris, st, w, stk, at >= 0, nready ? GSP_POOL_KEEP_READY : GSP_POOL_KEEP_DRY);
        const bool fin = at >= 0 && w.cur == kWalkDone;
        const uint32_t fm = __ballot_sync(F, fin);
        if (fin) {
            pl.t[at] = st.tbest;
            pl.hit[at] = st.slot;
            pl.done[ndone + __popc(fm & lt)] = (uint8_t)at;
            at = -1;
        }
        ndone += __popc(fm);
        __syncwarp();
    }
    if (REGEN) {
        const uint32_t sum = __reduce_add_sync(F, starts);
        if (lane == 0 && sum) atomicAdd(one.R.started, (unsigned long long)sum);
    }
    // the last paths: four lanes to a path, which share its slot (the last one walks with all lanes)
    {
        const int from = quad_source(__ballot_sync(F, at >= 0)), src = from < 0 ? lane : from;
        quad_take(st, w, stk, src);
        at = __shfl_sync(F, at, src);
        if (MULTI) {
            wide = (const float4*)__shfl_sync(F, (unsigned long long)wide, src);
            tris = (const float4*)__shfl_sync(F, (unsigned long long)tris, src);
        }
        if (from < 0) at = -1;
    }
    const bool lead = (lane & 3) == 0;
    while (true) {
        const uint32_t act = __ballot_sync(F, at >= 0);
        if (act == 0) return;
        if (__popc(act) == 4) {
            const int owner = __ffs(act) - 1;
            if (MULTI) {
                wide = (const float4*)__shfl_sync(F, (unsigned long long)wide, owner);
                tris = (const float4*)__shfl_sync(F, (unsigned long long)tris, owner);
            }
            st = coop_wide<false>(wide, tris, st, w, stk, owner, &scratch[threadIdx.x >> 5]);
            w.cur = kWalkDone;
        } else {
            quad_steps<GSP_WIDE_KEEP, false>(wide, tris, st, w, stk, at >= 0);
        }
        const bool fin = at >= 0 && w.cur == kWalkDone;
        float3 o = st.o, d = st.d, v = make_float3(0.0f, 0.0f, 0.0f);
        Rng rng;
        int32_t meta = 0, id = 0;
        if (fin) {
            pl.get_state(at, v, rng);
            meta = pl.meta[at];
            id = pl.id[at];
        }
        __syncwarp();  // read by every lane that shares it before one of them writes it back
        if (fin) {
            const PathJob& J = MULTI ? jobs[pl.job[at]] : one;
            if (pool_shade<SHADE, REGEN>(J, id, st.slot, st.tbest, o, d, v, rng, meta, lead)) {
                if (lead) pl.put_state(at, v, rng, meta);
                wide_ray(o, d, J.P.eps, __int_as_float(0x7f800000), st);
                wide_init(w);
            } else {
                at = -1;
            }
        }
        __syncwarp();
    }
}

}  // namespace gspd
