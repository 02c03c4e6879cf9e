// The loop of every vertex of a contour set, for kernels that work on whole
// runs of vertices: a block takes kLoopSpan consecutive vertices (kLoopPer per
// thread). A thread per loop that walks its own vertices touches a 32-byte
// sector for each value; with a thread per vertex every access is coalesced.
#pragma once

#include "common.cuh"

namespace csl {

constexpr int kLoopThreads = 256;
constexpr int kLoopPer = 4;
constexpr int kLoopSpan = kLoopThreads * kLoopPer;

struct LoopSpanSmem {
    int32_t rel[kLoopSpan];   // loop number - the span's first, at the loop's start
    int32_t warp[kLoopThreads / 32];
};

// Loop numbers of this thread's kLoopPer vertices (blockIdx.x * kLoopSpan +
// threadIdx.x * kLoopPer ...): the starts of the loops inside the span go to
// shared memory, a running maximum turns them into loop numbers. first: the
// loop holding each span's first vertex (span_first_loops). All threads of a
// block of kLoopThreads call it.
__device__ __forceinline__ void span_loops(const int64_t* __restrict__ loop_off, int64_t n_loops,
                                           const uint32_t* __restrict__ first, LoopSpanSmem& sm,
                                           uint32_t (&loop)[kLoopPer]) {
    const int64_t v0 = (int64_t)blockIdx.x * kLoopSpan;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int k = 0; k < kLoopPer; ++k) sm.rel[k * kLoopThreads + threadIdx.x] = 0;
    const int64_t L0 = first[blockIdx.x];
    const int64_t L1 = blockIdx.x + 1 < gridDim.x ? (int64_t)first[blockIdx.x + 1] : n_loops - 1;
    __syncthreads();
    // of loops that share a start the last one holds the vertex (the others are empty)
    for (int64_t L = L0 + 1 + threadIdx.x; L <= L1; L += kLoopThreads) {
        const int64_t p = loop_off[L] - v0;
        if (p >= 0 && p < kLoopSpan) atomicMax(&sm.rel[p], (int32_t)(L - L0));
    }
    __syncthreads();
    int32_t r[kLoopPer];
    int32_t m = 0;
#pragma unroll
    for (int k = 0; k < kLoopPer; ++k) {
        m = max(m, sm.rel[threadIdx.x * kLoopPer + k]);
        r[k] = m;
    }
    int32_t inc = m;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int32_t t = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc = max(inc, t);
    }
    if (lane == 31) sm.warp[warp] = inc;
    __syncthreads();
    int32_t before = __shfl_up_sync(0xffffffffu, inc, 1);
    if (lane == 0) before = 0;
    for (int w = 0; w < warp; ++w) before = max(before, sm.warp[w]);
#pragma unroll
    for (int k = 0; k < kLoopPer; ++k) loop[k] = (uint32_t)(L0 + max(r[k], before));
}

inline int64_t loop_spans(int64_t n_verts) { return ceil_div(n_verts, kLoopSpan); }

// first[b] = the loop holding vertex b * kLoopSpan, b < loop_spans(n_verts).
void span_first_loops(const int64_t* loop_off, int64_t n_loops, uint32_t* first, cudaStream_t s);

// vloop[v] = the loop of vertex v.
void loops_of_vertices(const int64_t* loop_off, int64_t n_loops, int64_t n_verts, uint32_t* vloop,
                       cudaStream_t s);

}  // namespace csl
