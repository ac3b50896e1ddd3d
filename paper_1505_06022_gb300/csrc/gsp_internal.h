// gsp_internal.h -- host-side structures shared by the library's translation units.
#pragma once

#include <nvtx3/nvToolsExt.h>
#include <cuda_runtime.h>

#include <cfloat>
#include <cmath>
#include <cstdint>
#include <cstring>
#include <string>
#include <vector>

#include "gsp.h"

// Host copy of the packed BVH (Sec. 3.1): per link set, nodes in that set's preorder.
// Node = 2 float4: {min.xyz, miss link}, {max.xyz, leaf word}; triangle = 3 float4:
// {v0.xyz, triangle index}, {v1.xyz, 0}, {v2.xyz, 0}.
struct HostBVH {
    int64_t nnodes = 0;
    int64_t stride = 0;  // nodes per link set in memory: nnodes + 1 (one padding node)
    int64_t nleaves = 0;
    int32_t depth = 0;
    int32_t link_sets = 0;
    std::vector<float4> nodes;  // link_sets * stride * 2
    std::vector<float4> tris;   // nt * 3, leaf order
    // The same tree as child pairs, for stack-based traversal: per internal node (preorder) four
    // float4 {left.min, left ref}, {left.max, right ref}, {right.min, wide_of}, {right.max, 0}; a ref
    // >= 0 is an internal node, < 0 is ~(leaf word). bin_root: ref of the root.
    std::vector<float4> bin;
    int32_t bin_root = 0;
    // The same tree four-wide (wide.cuh): the entry of each of bin's nodes, -1 for a node of odd depth
    // (gsp_wide_entry makes them). Empty for a tree that is a single leaf or has one link set. The device
    // build keeps none here.
    std::vector<int32_t> wide_of;
    int64_t nwide = 0;  // entries
    double build_ms = 0, thread_ms = 0;
};

#ifdef __CUDACC__
#define GSP_HOST_DEVICE __host__ __device__
#else
#define GSP_HOST_DEVICE
#endif

// The far end x of an interval of box distances, moved out by 2^-19 of its size: what the rounding of a
// box test is covered by (wide.cuh). BEHIND: the slack follows the sign of x, which a factor would not, and is
// relative, so that it is as good behind the origin (a negative tmin) as in front of it; +inf stays, and
// -inf gives a NaN, which no entry distance is at or below. Otherwise only an x that is not negative counts
// (the entry distances compared with it are not), and one product does.
template <bool BEHIND>
GSP_HOST_DEVICE inline float gsp_reach(float x) {
    return BEHIND ? x + fabsf(x) * 0x1p-19f : x * (1.0f + 0x1p-19f);
}

// The bits of an entry distance as an integer in the order of the distances (-0 below +0): as they are, or
// where there can be negative ones (BEHIND) with the order of those turned round.
template <bool BEHIND>
GSP_HOST_DEVICE inline int32_t gsp_wide_order(float t) {
    int32_t i;
    memcpy(&i, &t, sizeof i);
    return BEHIND ? i ^ ((i >> 31) & 0x7fffffff) : i;
}

// Whether a child of the four-wide tree put by with this key (its entry distance in gsp_wide_order, the two
// low bits replaced, which rounds it down) may still hold a closer hit, by the rule it was put by with: where
// surfaces coincide, a triangle's t can be below its box's entry distance by the rounding of either, and
// without the slack the winner of a tie would depend on the order of the walk.
template <bool BEHIND>
GSP_HOST_DEVICE inline bool gsp_wide_keep(int32_t key, float tbest) {
    return (key & ~3) <= gsp_wide_order<BEHIND>(gsp_reach<BEHIND>(tbest) + 0.0f);  // -0 counts as +0
}

// Centre and half extent of an interval of the four-wide tree's boxes: c - h <= lo and hi <= c + h
// with h widened by the factor 1 + 2^-19 (wide.cuh says what that covers). lo <= hi.
GSP_HOST_DEVICE inline void gsp_wide_box(float lo, float hi, float& c, float& h) {
    c = 0.5f * lo + 0.5f * hi;
    const float a = hi - c, b = c - lo;  // each within one rounding (2^-24) of the exact value
    h = (a > b ? a : b) * (1.0f + 0x1p-19f + 0x1p-22f);
}

// The entry of the four-wide tree (layout in wide.cuh) of node i of the child pairs: the boxes of its
// grandchildren, or a child's own where that is a leaf. of(j) is the entry of node j.
template <class Of>
GSP_HOST_DEVICE inline void gsp_wide_entry(const float4* bin, int64_t i, Of of, float4* entry) {
    float* q = (float*)entry;
    int32_t* ref = (int32_t*)entry + 24;
    int m = 0;
    const auto add = [&](const float4& lo, const float4& hi, int32_t r) {
        const float l[3] = {lo.x, lo.y, lo.z}, h[3] = {hi.x, hi.y, hi.z};
        for (int a = 0; a < 3; ++a) gsp_wide_box(l[a], h[a], q[8 * a + m], q[8 * a + 4 + m]);
        ref[m++] = r < 0 ? r : of(r);
    };
    const auto word = [](const float& f) { return *(const int32_t*)&f; };
    for (int c = 0; c < 2; ++c) {
        const float4* b = bin + 4 * i;
        const int32_t r = word(c ? b[1].w : b[0].w);
        if (r < 0) {
            add(b[2 * c], b[2 * c + 1], r);
            continue;
        }
        b = bin + 4 * (int64_t)r;
        add(b[0], b[1], word(b[0].w));
        add(b[2], b[3], word(b[1].w));
    }
    for (; m < 4; ++m) {
        for (int a = 0; a < 3; ++a) q[8 * a + m] = 0.0f, q[8 * a + 4 + m] = -FLT_MAX;  // near beyond far on every ray
        ref[m] = ~0;  // a leaf of no triangles
    }
    for (int k = 28; k < 32; ++k) q[k] = 0.0f;
}

// Which scenes have a four-wide tree: a single link set is there to be walked in its one order (Fig. 4), a
// deeper tree could need more than the walk's stack holds, and in a larger scene (c - o) / d could overflow
// for a tiny d inside a box. Others follow the links, and the tree is not made for them.
constexpr int kWideMaxDepth = 38;
constexpr double kWideMaxExtent = 1e8;
inline bool gsp_wide_usable(int32_t link_sets, int32_t depth, double extent) {
    return link_sets == 6 && depth <= kWideMaxDepth && extent <= kWideMaxExtent;
}

// The entries of all of them on the device: node i has entry index[i] where head[i] is set, or with null head and
// index the one that bin holds (wide_of).
// Where in an allocation of the child pairs the four-wide entries begin (in float4, a whole number of entries).
inline int64_t gsp_wide_at(int64_t bin_size) { return (bin_size + 7) / 8 * 8; }

cudaError_t gsp_wide_build(const float4* bin, int64_t n, const uint32_t* head, const uint32_t* index, float4* wide);

// Builds the binned-SAH tree and writes its hit/miss links (one set per ray direction
// class when link_sets == 6). Returns an empty string on success, else an error message.
std::string bvh_build_host(const float* verts, int64_t nv, const int32_t* tris, int64_t nt,
                           const gsp_bvh_params& p, HostBVH& out);

// Instrumented host walk of a packed BVH (same control flow as the device traversal).
void bvh_host_walk(const HostBVH& bvh, const float* rays, int64_t n, int32_t* tri, float* t,
                   int32_t* visits, int32_t* tests);

struct gsp_context {
    int32_t device = 0;
    int32_t* d_status = nullptr;  // first device-side error (0 = none)
    uint32_t* grid_scratch = nullptr;  // scratch of gsp_hash_grid_build, grown on demand
    int64_t grid_words = 0;
};

struct gsp_scene {
    gsp_context* ctx = nullptr;
    int32_t device = 0;  // the context's: destroying a scene does not read the context, which may be gone
    int64_t nv = 0, nt = 0;
    int32_t nmat = 0;
    std::vector<float> verts;
    std::vector<int32_t> tris, tri_mat;
    std::vector<gsp_material> mats;
    bool has_cam = false;
    gsp_camera cam{};
    double extent = 0;  // diagonal of the vertex bounding box
    // device copies
    float4* d_shade = nullptr;  // per triangle (upload order): unit normal xyz, material (int bits)
    float4* d_nlo = nullptr;    // per triangle (upload order): unit normal - its FP32 rounding (xyz)
    float4* d_mats = nullptr;   // per material: {albedo.rgb, type bits}, {emission.rgb, ior}
    float4* d_nodes = nullptr;
    float4* d_tris = nullptr;
    float4* d_bin = nullptr;  // child-pair layout (HostBVH::bin)
    float4* d_wide = nullptr;  // four-wide layout, behind d_bin in its allocation (gsp_wide_at); null if the tree is
                               // one leaf or not gsp_wide_usable
    unsigned long long* d_counter = nullptr;  // trace kernel: next ray, refine-list length
    int2* d_rlist = nullptr;                  // trace kernel: hits re-evaluated in FP64
    int64_t rlist_cap = 0;
    bool built = false;
    int32_t step_limit = 0;  // gsp_scene_set_step_limit (0 = the default cap)
    // per-vertex shading data (gsp_scene_set_attributes, gsp_scene_set_texture)
    float4* d_attr = nullptr;  // per triangle (upload order): {n0, s0}, {n1, s1}, {n2, s2}, {t0, t1, t2, flags}
    bool has_texcoords = false;
    std::vector<std::vector<float4>> tex;  // per material: texels {r, g, b, 0}, row-major (empty = none)
    std::vector<int2> tex_size;            // per material: width, height
    float4* d_texels = nullptr;            // every texture, one after the other
    int4* d_mtex = nullptr;                // per material: {first texel, width, height, 0}; null if none
    HostBVH bvh;
    int64_t device_bytes = 0;
    // host-buffer tracing (gsp_trace_closest_hit_host): a pipeline of chunks over kHostLanes
    // streams, each with its own device buffers, trace counters, refine list and pinned staging
    static constexpr int kHostLanes = 3;
    struct HostLane {
        cudaStream_t st = nullptr;
        cudaEvent_t done = nullptr;
        float4* d_rays = nullptr;
        int32_t* d_tri = nullptr;
        float* d_t = nullptr;
        float2* d_uv = nullptr;
        unsigned long long* d_ctr = nullptr;
        int2* d_rlist = nullptr;
        void* h_in = nullptr;   // pinned staging for pageable caller buffers
        void* h_out = nullptr;
    } lanes[kHostLanes];
    int64_t lane_cap = 0;  // rays per chunk the lanes were allocated for
    // per-launch timing of the traversal kernel in gsp_trace_closest_hit (gsp_trace_time_launches): event
    // pairs made up front, the first `tev_used` of them recorded
    std::vector<cudaEvent_t> tev;
    int64_t tev_used = 0;
};

// Installs a BVH built elsewhere (host copies + device arrays the scene takes ownership of),
// replacing the scene's current one.
void gsp_scene_adopt_bvh(gsp_scene* s, HostBVH&& bvh, float4* d_nodes, float4* d_tris, float4* d_bin, float4* d_wide);

// A driver entry point through the runtime's query (no link against libcuda); null if the driver does not
// offer it (grid_static.cu).
void* gsp_driver_fn(const char* name);

// NVTX range around a host-side stage (header-only NVTX3: a no-op unless a profiler attaches).
struct NvtxRange {
    explicit NvtxRange(const char* name) { nvtxRangePushA(name); }
    ~NvtxRange() { nvtxRangePop(); }
    NvtxRange(const NvtxRange&) = delete;
    NvtxRange& operator=(const NvtxRange&) = delete;
};

void gsp_set_last_error(const std::string& msg);

// Reports a CUDA failure of the library's own work: sets the message, consumes the runtime's
// last error (so that the next call does not see it as left over by the caller) and maps it to
// GSP_ERR_OOM or GSP_ERR_CUDA.
gsp_status gsp_cuda_fail(cudaError_t e);

// An error that the caller's earlier CUDA work left pending on this thread (the runtime's last
// error, shared with every user of the same CUDA runtime): reported as GSP_ERR_CUDA before the call
// touches anything, rather than discarded or returned later as a failure of the call's own launches.
// The library's failure paths consume the errors they report, so a pending error is never its own.
gsp_status gsp_pending_error(const char* who, cudaError_t e);

#define GSP_CUDA_TRY(expr)                                   \
    do {                                                     \
        cudaError_t e_ = (expr);                             \
        if (e_ != cudaSuccess) return gsp_cuda_fail(e_);     \
    } while (0)

#define GSP_NO_PENDING_ERROR(who)                                        \
    do {                                                                 \
        const cudaError_t p_ = cudaGetLastError();                       \
        if (p_ != cudaSuccess) return gsp_pending_error((who), p_);      \
    } while (0)
