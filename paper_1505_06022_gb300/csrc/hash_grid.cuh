// hash_grid.cuh -- the exact hash grid: points (photon deposits, hit points, a caller's points)
// ordered by (bucket, input order), and the first position of every bucket. Included by sppm.cu only.
//
// Four launches: one most-significant-digit split of the bucket number, then one block per part.
//   k_grid_tiles   a block per tile of the input lists its points and their buckets and counts them
//                  by part (the bucket's high bits);
//   k_grid_scan    per part, the counts of the tiles before each tile;
//   k_grid_split   a block per tile moves its points to their parts, in order;
//   k_grid_parts   a block per part sorts it by the low bits, in order, and writes what is wanted:
//                  the order, copies of the records in that order, the bucket starts of the part.
// A least-significant-digit radix sort (scan_sort.cu) takes five launches per eight bits, a scan for
// the compaction, one for the bucket starts, and an atomic per point for their counts: 17 to 25
// launches of a few microseconds each, on the critical path of a small pass. Here the starts fall out
// of the last step. Measured: 1,000,003 points in 2^21 buckets 152 -> 56 us; a 131x97 pass of 65,536
// photons 387 -> 303 us, four passes of the 64x64 Cornell box 625 -> 470 us, in each the launches saved
// times the few microseconds of a dependent one.
// Every step is ordered by counts and scans alone, so the result does not depend on scheduling.
#pragma once

#include "devcommon.cuh"
#include "persist.cuh"

namespace gspd {

// Teschner et al. 2003 spatial hash of an integer cell, 32-bit wraparound.
__device__ __forceinline__ uint32_t cell_hash(int32_t ix, int32_t iy, int32_t iz, uint32_t mask) {
    return (((uint32_t)ix * 73856093u) ^ ((uint32_t)iy * 19349663u) ^ ((uint32_t)iz * 83492791u)) & mask;
}

// Cell lattice shifted by 0.381966 of a cell so that axis-aligned walls at multiples of the
// cell size (e.g. a floor at 0) do not lie on cell boundaries.
constexpr float kCellOffset = 0.381966f;

__device__ __forceinline__ int32_t cell_of(float x, float inv_h) {
    return (int32_t)floorf(fmaf(x, inv_h, kCellOffset));
}

__device__ __forceinline__ uint32_t bucket_of(float3 x, float inv_h, uint32_t mask) {
    return cell_hash(cell_of(x.x, inv_h), cell_of(x.y, inv_h), cell_of(x.z, inv_h), mask);
}

constexpr int kGridThreads = 256, kGridWarps = kGridThreads / 32;
constexpr int kGridMaxTiles = 480;
constexpr int kGridMaxBits = 21;     // of the bucket number: 11 for the parts, 10 within one
constexpr int kGridMaxParts = 2048, kGridMaxLow = 1024;
constexpr int kGridAux = 8192;       // words: tile counts, part totals, part starts
constexpr int kGridList = 4096;      // points of a tile whose list k_grid_tiles keeps in shared memory
constexpr int kGridItems = 12;       // points per lane that k_grid_split holds in registers
constexpr int kGridSegment = kGridWarps * 32 * kGridItems;  // and so ranks at once (16-bit counters)
constexpr int kPartItems = 4;        // the same for k_grid_parts; larger parts are read again
constexpr int kPartAhead = 8;        // points per lane of a larger part that are fetched at once
constexpr int kScanThreads = 1024;   // of k_grid_scan

// How a grid of `items` inputs and 2^bits buckets is split.
struct GridPlan {
    int32_t low;       // bits of a bucket's number within its part
    int32_t parts;
    int32_t per_tile;  // inputs (points, or photon paths) a tile covers
    int32_t tiles;
};

inline GridPlan grid_plan(int64_t items, int bits) {
    GridPlan p;
    // 256 parts or more keep the chip busy; the rest of the bits, up to ten, stay within a part
    p.low = bits - 8 < 0 ? 0 : bits - 8 < 10 ? bits - 8 : 10;
    if (p.low < bits - 11) p.low = bits - 11;
    p.parts = 1 << (bits - p.low);
    int64_t per = (items + kGridMaxTiles - 1) / kGridMaxTiles;
    per = (per + kGridThreads - 1) / kGridThreads * kGridThreads;
    p.per_tile = (int32_t)(per < kGridThreads ? kGridThreads : per);
    p.tiles = (int32_t)((items + p.per_tile - 1) / p.per_tile);
    return p;
}

// Buffers of one build. keys, vals: (inputs x records per input) words each, the tiles' lists; pairs:
// as many {bucket, value} pairs, the parts' points (one 8-byte store per point: the split scatters
// them, a point or two per part and tile, so the stores are what it costs); counts
// [tiles][parts] (k_grid_parts may overwrite it with the bucket starts); aux: kGridAux words.
struct GridBuf {
    uint32_t *keys0, *vals0;
    uint2* pairs;
    uint32_t *counts, *aux;
    __device__ __forceinline__ uint32_t* tile_count() const { return aux; }
    __device__ __forceinline__ uint32_t* total() const { return aux + 512; }
    __device__ __forceinline__ uint32_t* part_start() const { return aux + 512 + kGridMaxParts; }  // [parts + 1]
};

// What is to be sorted: photon deposits (pcount records of two float4 at slots, `per` slots to a
// path), or points (pcount null, `per` 1; with skip, those whose w holds a negative integer are left out).
struct GridIn {
    const float4* __restrict__ pos;
    const uint32_t* __restrict__ pcount;
    int64_t items;
    int32_t per, skip;
    float inv_h;
    uint32_t mask;
};

// Exclusive sum over the block of one value per thread; total receives the block's sum.
__device__ __forceinline__ uint32_t grid_block_sum(uint32_t v, uint32_t* s_warp, uint32_t& total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    __syncthreads();  // s_warp may still be read from an earlier call
    if (lane == 31) s_warp[warp] = x;
    __syncthreads();
    uint32_t before = 0;
    total = 0;
#pragma unroll
    for (int w = 0; w < kGridWarps; ++w) {
        const uint32_t t = s_warp[w];
        if (w < warp) before += t;
        total += t;
    }
    return before + x - v;
}

// The tile's points, listed in input order at the tile's own range of keys0 / vals0, and their counts
// by part. parts == 0: the list alone (the adjoint's photons need no grid).
__global__ void __launch_bounds__(kGridThreads) k_grid_tiles(GridIn in, GridPlan plan, GridBuf buf) {
    __shared__ uint32_t s_count[kGridMaxParts];
    __shared__ uint32_t s_list[kGridList];
    __shared__ uint32_t s_warp[kGridWarps];
    release_next();
    wait_previous();
    const int64_t first = (int64_t)blockIdx.x * plan.per_tile, end = min(first + plan.per_tile, in.items);
    uint32_t* vals = buf.vals0 + first * in.per;
    uint32_t* keys = buf.keys0 + first * in.per;
    for (int d = threadIdx.x; d < plan.parts; d += kGridThreads) s_count[d] = 0;
    // each thread lists a run of consecutive inputs
    const int run = plan.per_tile / kGridThreads;
    const int64_t a = first + (int64_t)threadIdx.x * run, z = min(a + run, end);
    uint32_t mine = 0;
    for (int64_t k = a; k < z; ++k)
        mine += in.pcount ? in.pcount[k] : (uint32_t)!(in.skip && __float_as_int(in.pos[k].w) < 0);
    uint32_t n;
    uint32_t at = grid_block_sum(mine, s_warp, n);
    const bool listed = plan.parts > 0 && n <= kGridList;  // else the list is read back from memory
    for (int64_t k = a; k < z; ++k) {
        const uint32_t c = in.pcount ? in.pcount[k] : (uint32_t)!(in.skip && __float_as_int(in.pos[k].w) < 0);
        for (uint32_t i = 0; i < c; ++i, ++at) {
            const uint32_t v = (uint32_t)(k * in.per) + i;
            if (listed)
                s_list[at] = v;
            else
                vals[at] = v;
        }
    }
    if (threadIdx.x == 0) buf.tile_count()[blockIdx.x] = n;
    if (plan.parts == 0) return;
    __syncthreads();
    const int stride = in.pcount ? 2 : 1;  // float4 per record
    for (uint32_t e = threadIdx.x; e < n; e += 4 * kGridThreads) {
        uint32_t v[4];
        float4 x[4];
#pragma unroll
        for (int j = 0; j < 4; ++j)
            if (e + j * kGridThreads < n) v[j] = listed ? s_list[e + j * kGridThreads] : vals[e + j * kGridThreads];
#pragma unroll
        for (int j = 0; j < 4; ++j)
            if (e + j * kGridThreads < n) x[j] = __ldg(in.pos + (size_t)stride * v[j]);
#pragma unroll
        for (int j = 0; j < 4; ++j)
            if (e + j * kGridThreads < n) {
                const uint32_t b = bucket_of(f3(x[j]), in.inv_h, in.mask);
                keys[e + j * kGridThreads] = b;
                if (listed) vals[e + j * kGridThreads] = v[j];
                atomicAdd(&s_count[b >> plan.low], 1u);
            }
    }
    __syncthreads();
    for (int d = threadIdx.x; d < plan.parts; d += kGridThreads) buf.counts[(size_t)blockIdx.x * plan.parts + d] = s_count[d];
}

// Per part, counts[t] becomes the sum over the tiles before t; total its sum. A block has 32 parts, each
// of its 32 warps a run of the tiles.
__global__ void __launch_bounds__(kScanThreads) k_grid_scan(GridPlan plan, GridBuf buf) {
    constexpr int kWarps = kScanThreads / 32, kRun = (kGridMaxTiles + kWarps - 1) / kWarps;
    __shared__ uint32_t s_sum[kWarps][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, d = blockIdx.x * 32 + lane;
    const bool live = d < plan.parts;
    uint32_t c[kRun], sum = 0;
    release_next();
    wait_previous();
#pragma unroll
    for (int j = 0; j < kRun; ++j) {
        const int t = warp * kRun + j;
        c[j] = live && t < plan.tiles ? buf.counts[(size_t)t * plan.parts + d] : 0u;
    }
#pragma unroll
    for (int j = 0; j < kRun; ++j) sum += c[j];
    s_sum[warp][lane] = sum;
    __syncthreads();
    if (warp == 0) {  // exclusive sums over the warps
        uint32_t acc = 0;
#pragma unroll
        for (int w = 0; w < kWarps; ++w) {
            const uint32_t x = s_sum[w][lane];
            s_sum[w][lane] = acc;
            acc += x;
        }
        if (live) buf.total()[d] = acc;
    }
    __syncthreads();
    uint32_t acc = s_sum[warp][lane];
#pragma unroll
    for (int j = 0; j < kRun; ++j) {
        const int t = warp * kRun + j;
        if (live && t < plan.tiles) buf.counts[(size_t)t * plan.parts + d] = acc;
        acc += c[j];
    }
}

// The tile's points to their parts, in order: each warp has a contiguous share of the list, counts it
// by part, and after a sum over the warps before it walks it again, 32 points at a time, ranking equal
// parts among the lanes. Block 0 also writes the part starts and clears the word `clear`.
__global__ void __launch_bounds__(kGridThreads)
k_grid_split(GridIn in, GridPlan plan, GridBuf buf, uint32_t* __restrict__ clear) {
    __shared__ uint32_t s_base[kGridMaxParts];
    __shared__ uint16_t s_count[kGridWarps][kGridMaxParts];
    __shared__ uint32_t s_warp[kGridWarps];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t lt = lanemask_lt();
    // where each part starts: an exclusive sum of the totals, then the tiles before this one
    const int run = (plan.parts + kGridThreads - 1) / kGridThreads;
    release_next();
    wait_previous();
    const int a = min((int)threadIdx.x * run, plan.parts), z = min(a + run, plan.parts);
    uint32_t mine = 0, n;
    for (int d = a; d < z; ++d) mine += buf.total()[d];
    uint32_t at = grid_block_sum(mine, s_warp, n);
    for (int d = a; d < z; ++d) {
        if (blockIdx.x == 0) buf.part_start()[d] = at;
        s_base[d] = at;
        at += buf.total()[d];
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        buf.part_start()[plan.parts] = n;
        if (clear) *clear = 0;
    }
    __syncthreads();
    for (int d = threadIdx.x; d < plan.parts; d += kGridThreads) s_base[d] += buf.counts[(size_t)blockIdx.x * plan.parts + d];
    const int64_t first = (int64_t)blockIdx.x * plan.per_tile * in.per;
    const uint32_t m = plan.tiles ? buf.tile_count()[blockIdx.x] : 0u;  // no input: one block, for the starts
    for (uint32_t seg = 0; seg < m; seg += kGridSegment) {
        const uint32_t* keys = buf.keys0 + first + seg;
        const uint32_t* vals = buf.vals0 + first + seg;
        const uint32_t len = min(m - seg, (uint32_t)kGridSegment), share = (len + kGridWarps - 1) / kGridWarps;
        const uint32_t e0 = min(warp * share, len), e1 = min(e0 + share, len);
        uint32_t key[kGridItems];
#pragma unroll
        for (int j = 0; j < kGridItems; ++j) key[j] = e0 + 32 * j + lane < e1 ? keys[e0 + 32 * j + lane] : 0xffffffffu;
        for (int d = lane; d < plan.parts; d += 32) s_count[warp][d] = 0;
        __syncwarp();
#pragma unroll
        for (int j = 0; j < kGridItems; ++j) {
            if (e0 + 32 * j >= e1) break;
            const uint32_t d = key[j] >> plan.low;
            const uint32_t peers = __match_any_sync(0xffffffffu, d);
            if (e0 + 32 * j + lane < e1 && (peers & lt) == 0) s_count[warp][d] += (uint16_t)__popc(peers);
            __syncwarp();
        }
        uint32_t val[kGridItems];
#pragma unroll
        for (int j = 0; j < kGridItems; ++j)
            if (e0 + 32 * j + lane < e1) val[j] = vals[e0 + 32 * j + lane];
        __syncthreads();
        for (int d = threadIdx.x; d < plan.parts; d += kGridThreads) {
            uint32_t acc = 0;
#pragma unroll
            for (int w = 0; w < kGridWarps; ++w) {
                const uint32_t c = s_count[w][d];
                s_count[w][d] = (uint16_t)acc;
                acc += c;
            }
        }
        __syncthreads();
#pragma unroll
        for (int j = 0; j < kGridItems; ++j) {
            if (e0 + 32 * j >= e1) break;
            const bool on = e0 + 32 * j + lane < e1;
            const uint32_t d = key[j] >> plan.low;
            const uint32_t peers = __match_any_sync(0xffffffffu, d), rank = __popc(peers & lt);
            const uint32_t off = on ? s_count[warp][d] : 0u;
            __syncwarp();
            if (on) {
                const uint32_t to = s_base[d] + off + rank;
                buf.pairs[to] = make_uint2(key[j], val[j]);
                if (rank == 0) s_count[warp][d] = (uint16_t)(off + __popc(peers));
            }
            __syncwarp();
        }
        if (seg + kGridSegment >= m) break;
        // more to come: the parts' positions move on by this segment (the last warp's ends are its counts)
        __syncthreads();
        for (int d = threadIdx.x; d < plan.parts; d += kGridThreads) s_base[d] += s_count[kGridWarps - 1][d];
        __syncthreads();
    }
}

// One part: sorted by the low bits of the bucket number as k_grid_split sorts a tile, but with the
// counts turned into bucket starts. A part is one block's work however many points crowd into it, so a larger
// one than the lanes hold is fetched kPartAhead points per lane at once, counted without ranking, and its points
// are placed before any is moved: 1,000,003 points in one bucket 2,220 -> 758 us (745 with radix passes over
// them), spread over some hundred 1,040 -> 362 (410), over 2^21 60.5 -> 56.1. Writes whichever of these is asked for: the order, the records in
// that order (positions and payloads), and the bucket starts (the last part also the end).
__global__ void __launch_bounds__(kGridThreads)
k_grid_parts(GridIn in, GridPlan plan, GridBuf buf, uint32_t* __restrict__ order, float4* __restrict__ spos,
             float4* __restrict__ spay, uint32_t* __restrict__ bstart) {
    __shared__ uint32_t s_count[kGridWarps][kGridMaxLow];
    __shared__ uint32_t s_start[kGridMaxLow];
    __shared__ uint32_t s_warp[kGridWarps];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t lt = lanemask_lt();
    const int nb = 1 << plan.low;
    release_next();
    wait_previous();
    const uint32_t start = buf.part_start()[blockIdx.x], stop = buf.part_start()[blockIdx.x + 1], m = stop - start;
    uint32_t* bs = bstart + (size_t)blockIdx.x * nb;
    if (blockIdx.x == gridDim.x - 1 && threadIdx.x == 0) bstart[(size_t)gridDim.x * nb] = stop;
    if (m == 0) {
        for (int b = threadIdx.x; b < nb; b += kGridThreads) bs[b] = start;
        return;
    }
    const uint2* pairs = buf.pairs + start;
    const uint32_t share = (m + kGridWarps - 1) / kGridWarps, e0 = min(warp * share, m), e1 = min(e0 + share, m);
    const bool held = share <= 32 * kPartItems;  // the lanes hold the warp's points
    const auto point = [&](uint32_t e) {  // its bucket within the part, its value
        const uint2 p = e < e1 ? pairs[e] : make_uint2(0u, 0u);
        return make_uint2(e < e1 ? p.x & (nb - 1) : 0xffffffffu, p.y);
    };
    uint2 own[kPartItems];
    if (held) {
#pragma unroll
        for (int j = 0; j < kPartItems; ++j) own[j] = point(e0 + 32 * j + lane);
    }
    for (int b = lane; b < nb; b += 32) s_count[warp][b] = 0;
    __syncwarp();
    const auto count = [&](uint32_t b) {  // in any order; lanes that add to one counter are combined by the hardware
        if (b != 0xffffffffu) atomicAdd(&s_count[warp][b], 1u);
    };
    if (held) {
#pragma unroll
        for (int j = 0; j < kPartItems; ++j) count(own[j].x);
    } else {
        for (uint32_t e = e0; e < e1; e += 32 * kPartAhead) {
            uint32_t b[kPartAhead];
#pragma unroll
            for (int j = 0; j < kPartAhead; ++j) b[j] = point(e + 32 * j + lane).x;
#pragma unroll
            for (int j = 0; j < kPartAhead; ++j) count(b[j]);
        }
    }
    __syncthreads();
    // bucket starts: sums over the warps, then over the buckets (four consecutive ones per thread)
    for (int b = threadIdx.x; b < nb; b += kGridThreads) {
        uint32_t sum = 0;
#pragma unroll
        for (int w = 0; w < kGridWarps; ++w) sum += s_count[w][b];
        s_start[b] = sum;
    }
    __syncthreads();
    {
        const int a = 4 * threadIdx.x;
        uint32_t c[4], mine = 0, all;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            c[i] = a + i < nb ? s_start[a + i] : 0u;
            mine += c[i];
        }
        uint32_t at = start + grid_block_sum(mine, s_warp, all);
#pragma unroll
        for (int i = 0; i < 4; ++i)
            if (a + i < nb) {
                s_start[a + i] = at;
                at += c[i];
            }
    }
    __syncthreads();
    for (int b = threadIdx.x; b < nb; b += kGridThreads) {
        uint32_t at = s_start[b];
        bs[b] = at;
#pragma unroll
        for (int w = 0; w < kGridWarps; ++w) {
            const uint32_t c = s_count[w][b];
            s_count[w][b] = at;
            at += c;
        }
    }
    __syncthreads();
    // the place of each of 32 lanes' points, in order; then the records move there
    const auto place = [&](const uint32_t b, const uint32_t peers) {
        const bool on = b != 0xffffffffu;
        const uint32_t off = on ? s_count[warp][b] : 0u;
        __syncwarp();
        if (on && (peers & lt) == 0) s_count[warp][b] = off + __popc(peers);
        __syncwarp();
        return off + __popc(peers & lt);
    };
    const auto move = [&](uint2 pt, uint32_t to) {
        if (pt.x == 0xffffffffu) return;
        if (order) order[to] = pt.y;
        if (spos) {
            const float4 x = __ldg(in.pos + 2 * (size_t)pt.y), y = __ldg(in.pos + 2 * (size_t)pt.y + 1);
            spos[to] = x;
            spay[to] = y;
        }
    };
    const auto place_all = [&](const auto& pt) {
        constexpr int K = sizeof pt / sizeof pt[0];
        uint32_t to[K];
#pragma unroll
        for (int j = 0; j < K; ++j) to[j] = __match_any_sync(0xffffffffu, pt[j].x);
#pragma unroll
        for (int j = 0; j < K; ++j) to[j] = place(pt[j].x, to[j]);
#pragma unroll
        for (int j = 0; j < K; ++j) move(pt[j], to[j]);
    };
    if (held) {
        place_all(own);
    } else {
        for (uint32_t e = e0; e < e1; e += 32 * kPartAhead) {
            uint2 pt[kPartAhead];
#pragma unroll
            for (int j = 0; j < kPartAhead; ++j) pt[j] = point(e + 32 * j + lane);
            place_all(pt);
        }
    }
}

}  // namespace gspd
