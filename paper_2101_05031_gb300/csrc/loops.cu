// The loop of every vertex of a contour set (loops.cuh). Bound by the 4 bytes
// written per vertex: 48 us for 28M vertices in loops of about 14 (a thread per
// loop writing its own vertices took 120 us, flags with two scans 200 us).
#include "loops.cuh"

namespace csl {
namespace {

// A thread per loop: the only pass over the offsets outside the spans' own blocks.
__global__ void k_span_first(const int64_t* __restrict__ loop_off, int64_t n_loops,
                             uint32_t* __restrict__ first) {
    for (int64_t L = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; L < n_loops;
         L += (int64_t)gridDim.x * blockDim.x) {
        const int64_t a = loop_off[L], e = loop_off[L + 1];
        for (int64_t b = (a + kLoopSpan - 1) / kLoopSpan; b * kLoopSpan < e; ++b)
            first[b] = (uint32_t)L;
    }
}

__global__ void __launch_bounds__(kLoopThreads) k_loops_of(const int64_t* __restrict__ loop_off,
                                                           int64_t n_loops, int64_t n_verts,
                                                           const uint32_t* __restrict__ first,
                                                           uint32_t* __restrict__ vloop) {
    __shared__ LoopSpanSmem sm;
    uint32_t L[kLoopPer];
    span_loops(loop_off, n_loops, first, sm, L);
    const int64_t v = ((int64_t)blockIdx.x * kLoopThreads + threadIdx.x) * kLoopPer;
    if (v + kLoopPer <= n_verts) {
        *reinterpret_cast<uint4*>(vloop + v) = make_uint4(L[0], L[1], L[2], L[3]);
    } else {
#pragma unroll
        for (int k = 0; k < kLoopPer; ++k)
            if (v + k < n_verts) vloop[v + k] = L[k];
    }
}

}  // namespace

void span_first_loops(const int64_t* loop_off, int64_t n_loops, uint32_t* first, cudaStream_t s) {
    k_span_first<<<grid_for(n_loops, 256), 256, 0, s>>>(loop_off, n_loops, first);
    CSL_LAUNCH_CHECK("first loops of spans");
}

void loops_of_vertices(const int64_t* loop_off, int64_t n_loops, int64_t n_verts, uint32_t* vloop,
                       cudaStream_t s) {
    if (n_verts <= 0 || n_loops <= 0) return;
    DevBuf first((size_t)loop_spans(n_verts) * 4, s);
    span_first_loops(loop_off, n_loops, first.as<uint32_t>(), s);
    k_loops_of<<<(unsigned)loop_spans(n_verts), kLoopThreads, 0, s>>>(
        loop_off, n_loops, n_verts, first.as<uint32_t>(), vloop);
    CSL_LAUNCH_CHECK("loops of vertices");
}

}  // namespace csl
