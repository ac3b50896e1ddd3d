// launch.h -- launch configuration and cross-file helpers of the library.
#pragma once

#include "devcommon.cuh"
#include "gsp_internal.h"

constexpr int kTraceThreads = 128;
#ifndef GSP_TRACE_CHUNK
#define GSP_TRACE_CHUNK 64
#endif
#ifndef GSP_TRACE_INNER
#define GSP_TRACE_INNER 8
#endif
#ifndef GSP_TRACE_LEAF_BATCH
#define GSP_TRACE_LEAF_BATCH 12
#endif
#ifndef GSP_TRACE_MIN_BLOCKS
#define GSP_TRACE_MIN_BLOCKS 9
#endif
#ifndef GSP_WIDE_MIN_BLOCKS
#define GSP_WIDE_MIN_BLOCKS 8
#endif
#ifndef GSP_PATH_CHUNK
#define GSP_PATH_CHUNK 32
#endif
#ifndef GSP_PATH_MIN_BLOCKS
#define GSP_PATH_MIN_BLOCKS 8
#endif
constexpr int kTraceChunk = GSP_TRACE_CHUNK;           // rays a warp takes from the global counter at once
constexpr int kTraceInner = GSP_TRACE_INNER;           // traversal steps between refills
constexpr int kTraceLeafBatch = GSP_TRACE_LEAF_BATCH;  // pending leaves that trigger a warp-wide leaf test
constexpr int kWideStack = 64;     // children a walk of the four-wide tree may keep (at most three per wide level)
// most paths a warp of the path kernels takes at once (gsp_chunk); a launch has a block for every four paths (for
// every 128 in a batch) up to what is resident, so that every warp of a short one gets some
constexpr int kPathChunk = GSP_PATH_CHUNK;

// Persistent grid size of the closest-hit kernel: SMs x resident blocks per SM.
int gsp_trace_grid(int device);

// Items a warp of a persistent kernel takes at once when `warps` warps share n of them: an equal
// share while that leaves no warp more than its 32 lanes hold, else a quarter of it, so that warps
// whose items end early take over from others, within 16 and most.
#ifndef GSP_CHUNK_DIV
#define GSP_CHUNK_DIV 4
#endif
inline int gsp_chunk(int64_t n, int64_t warps, int most) {
    if (n <= 32 * warps) return (int)((n + warps - 1) / warps);
    const int64_t c = n / (GSP_CHUNK_DIV * warps);
    return (int)(c < 16 ? 16 : c > most ? most : c);
}

gspd::DevScene gsp_dev_scene(const gsp_scene* s);

// Programmatic dependent launch: a kernel launched with gsp_launch_after is set up while the kernel before
// it in the stream still runs, once every block of that one has called release_next() or ended. It must
// call wait_previous() in every thread before it touches memory, which returns when the kernel before it
// has completed (and so all that came before, as that one waited in the same way). Used in chains of short
// kernels, where the gap between two (1 to 2 us) is a good part of them: emission, paths, hash grid,
// gather, adjoint. A 131x97 pass 267 -> 252 us, four 64x64 passes 399 -> 372, eight replayed 96x96 passes
// 895 -> 740, a hash grid of 1,000,003 points 59.4 -> 58.2. The path kernels do not release the next one:
// its blocks would wait on SMs that another pass's paths could use.
#ifdef __CUDACC__
namespace gspd {
__device__ __forceinline__ void wait_previous() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void release_next() { asm volatile("griddepcontrol.launch_dependents;"); }
}  // namespace gspd

template <class... P, class... A>
inline void gsp_launch_after(void (*kernel)(P...), dim3 grid, int block, cudaStream_t st, A&&... args) {
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t c{};
    c.gridDim = grid;
    c.blockDim = dim3((unsigned)block);
    c.stream = st;
    c.attrs = &at;
    c.numAttrs = 1;
    cudaLaunchKernelEx(&c, kernel, P(args)...);
}
#endif

// Closest hit of rays already on the device (a wavefront queue) whose count is read from d_n.
// With a finite refine_factor, hits whose error factor exceeds it get the FP64 distance (and the
// scene's trace counters are reset first); with refine_factor = INFINITY nothing is re-evaluated
// and the counters are reset only if zero_counters is set (else the caller has reset them).
// out_slot: tri receives the hit's leaf-ordered triangle slot instead of its upload-order index.
// ctr (2 u64: next ray, list length) and rlist (max_n entries) belong to the caller.
cudaError_t gsp_trace_queue(const gsp_scene* s, const float4* rays, int64_t max_n, const uint32_t* d_n, int32_t* tri,
                            float* t, float refine_factor, bool zero_counters, bool out_slot, unsigned long long* ctr,
                            int2* rlist, cudaStream_t st);
