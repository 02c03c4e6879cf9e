// Topology-preserving simplification of marching-squares contours (the paper
// smooths and simplifies its marching-squares boundaries without creating
// intersections before writing tool paths, Sec. 4).
//
// Every contour vertex lies on a grid edge e and its loop runs from the cell
// on one side of e into the cell on the other. A vertex (loop position q, the
// loop's head at q = 0) is dropped when q is odd in a loop of at least 5
// vertices (its neighbours stay, the loop keeps at least 3), neither cell
// beside e carries a crossing on an edge other than the loop's own two (so
// both cells hold only this loop's segments, and the convex 1 x 2 block they
// form contains the new chord and no other contour piece), and the vertex
// lies within `tol` of the line through its neighbours (decided in FP64).
//
// Device work: each loop's layer, a per-layer bitmap of the grid edges that
// carry a crossing, the keep decisions per vertex, a scan of the kept counts
// and the compaction.
#include <limits.h>
#include <math.h>

#include <algorithm>

#include "loops.cuh"

namespace csl {
namespace {

struct SpGrid {
    int32_t W, H;          // padded sample grid
    int64_t words;         // bitmap words per layer
};

__global__ void k_sp_loop_layer(const int64_t* __restrict__ layer_off, int n_layers,
                                int64_t n_loops, int32_t* __restrict__ loop_layer) {
    for (int64_t L = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; L < n_loops;
         L += (int64_t)gridDim.x * blockDim.x) {
        int lo = 0, hi = n_layers;   // last layer whose first loop is <= L
        while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if (layer_off[mid] <= L) lo = mid; else hi = mid;
        }
        loop_layer[L] = lo;
    }
}

// The crossing bit of every vertex. An edge id outside the padded grid
// (contours of another grid) is skipped and reported through *bad. Bound by
// the bitmap's atomics, which stay in L2 (250 KB per 1000^2 layer).
__global__ void __launch_bounds__(kLoopThreads)
k_sp_mark(const int64_t* __restrict__ loop_off, const int32_t* __restrict__ eid,
          const int32_t* __restrict__ loop_layer, const uint32_t* __restrict__ first,
          int64_t n_loops, int64_t n_verts, SpGrid g, uint32_t* __restrict__ bits,
          uint32_t* bad) {
    __shared__ LoopSpanSmem sm;
    uint32_t L[kLoopPer];
    span_loops(loop_off, n_loops, first, sm, L);
    const int64_t n_ids = 2 * (int64_t)g.W * g.H;
    const int64_t v0 = ((int64_t)blockIdx.x * kLoopThreads + threadIdx.x) * kLoopPer;
#pragma unroll
    for (int k = 0; k < kLoopPer; ++k) {
        if (v0 + k >= n_verts) break;
        const int64_t e = eid[v0 + k];
        if (e < 0 || e >= n_ids)
            atomicOr(bad, 1u);
        else
            atomicOr(bits + (int64_t)loop_layer[L[k]] * g.words + (e >> 5),
                     1u << (uint32_t)(e & 31));
    }
}

__device__ __forceinline__ bool has_edge(const uint32_t* row, int64_t e, const SpGrid& g) {
    if (e < 0 || (e >> 5) >= g.words) return false;
    return (row[e >> 5] >> (e & 31)) & 1u;
}

// Whether cell (I, J) has a crossing on an edge other than the loop's own
// edges a, b, c (its predecessor's, its own and its successor's).
__device__ __forceinline__ bool other_crossing(int I, int J, int64_t a, int64_t b, int64_t c,
                                               const uint32_t* row, const SpGrid& g) {
    if (I < 0 || J < 0 || I > g.W - 2 || J > g.H - 2) return false;
    const int64_t e[4] = {2 * ((int64_t)J * g.W + I), 2 * ((int64_t)(J + 1) * g.W + I),
                          2 * ((int64_t)J * g.W + I) + 1, 2 * ((int64_t)J * g.W + I + 1) + 1};
    for (int k = 0; k < 4; ++k)
        if (e[k] != a && e[k] != b && e[k] != c && has_edge(row, e[k], g)) return true;
    return false;
}

// Whether vertex v lies within tol of the line through p and s (distinct
// points), |cross| <= tol sqrt(L2) in FP64. Decided in FP32 where its rounding
// cannot matter (the differences carry at most 2^-24, every product and sum
// 2^-24 more: 1e-6 of the terms' sizes bounds them all), in FP64 otherwise: the
// FP64 pipe runs at 1/64 of the FP32 rate here.
__device__ __forceinline__ bool on_chord(const float2 p, const float2 v, const float2 s,
                                         double tol) {
    const float fdx = s.x - p.x, fdy = s.y - p.y;
    const float fL2 = fdx * fdx + fdy * fdy;
    const float ftol = (float)tol;
    if (fL2 > 1e-30f && fL2 < 1e30f && ftol >= 1e-30f) {
        const float a = (v.x - p.x) * fdy, b = (v.y - p.y) * fdx;
        const float c = fabsf(a - b), err = 1e-6f * (fabsf(a) + fabsf(b)) + 1e-36f;
        const float rhs = ftol * sqrtf(fL2);
        if (c + err < rhs * (1.0f - 1e-6f)) return true;
        if (c - err > rhs * (1.0f + 1e-6f)) return false;
    }
    const double px = p.x, py = p.y;
    const double dx = (double)s.x - px, dy = (double)s.y - py;
    const double L2 = dx * dx + dy * dy;
    if (L2 == 0.0) return false;
    const double cross = ((double)v.x - px) * dy - ((double)v.y - py) * dx;
    return fabs(cross) <= tol * sqrt(L2);
}

// A thread per kLoopPer vertices: keep bits (32 vertices per word) and the
// words' counts. Bound by the probes of the bitmap and the reads of each
// vertex and its neighbours. Coalesced: for the 49M vertices of a 1000^2 x 250
// part this kernel takes 0.44 ms and the mark kernel 0.17 ms, against 10.1 and
// 0.87 ms with a thread per loop walking its own vertices (a 32-byte sector
// for every 4 or 8 bytes, and the chord test in FP64 throughout).
__global__ void __launch_bounds__(kLoopThreads)
k_sp_keep(const int64_t* __restrict__ loop_off, const int32_t* __restrict__ eid,
          const float2* __restrict__ xy, const int32_t* __restrict__ loop_layer,
          const uint32_t* __restrict__ first, int64_t n_loops, int64_t n_verts, SpGrid g,
          const uint32_t* __restrict__ bits, double tol, uint32_t* __restrict__ keep,
          uint32_t* __restrict__ kept) {
    __shared__ LoopSpanSmem sm;
    uint32_t L[kLoopPer];
    span_loops(loop_off, n_loops, first, sm, L);
    const int64_t v0 = ((int64_t)blockIdx.x * kLoopThreads + threadIdx.x) * kLoopPer;
    uint32_t nib = 0;
#pragma unroll
    for (int k = 0; k < kLoopPer; ++k) {
        const int64_t v = v0 + k;
        if (v >= n_verts) break;
        const int64_t a = loop_off[L[k]], n = loop_off[L[k] + 1] - a;
        const int64_t q = v - a;
        bool drop = false;
        if (n >= 5 && (q & 1)) {
            const int64_t p = v - 1, s = q + 1 == n ? a : v + 1;
            const int64_t ev = eid[v], ep = eid[p], es = eid[s];
            const uint32_t* row = bits + (int64_t)loop_layer[L[k]] * g.words;
            // the two cells beside edge ev
            // a valid ev is below 2 W H < 2^31: a 32-bit division (an
            // invalid one is reported by k_sp_mark; the cell lookups below
            // bound-check whatever I, J it gives)
            const uint32_t base = (uint32_t)ev >> 1;
            const int J = (int)(base / (uint32_t)g.W),
                      I = (int)(base - (uint32_t)J * (uint32_t)g.W);
            const bool vert = ev & 1;
            drop = !other_crossing(vert ? I - 1 : I, vert ? J : J - 1, ep, ev, es, row, g) &&
                   !other_crossing(I, J, ep, ev, es, row, g) && on_chord(xy[p], xy[v], xy[s], tol);
        }
        nib |= (drop ? 0u : 1u) << k;
    }
    // 8 threads make a word
    uint32_t w = nib << (kLoopPer * (threadIdx.x & 7));
#pragma unroll
    for (int o = 1; o < 8; o <<= 1) w |= __shfl_xor_sync(0xffffffffu, w, o);
    if ((threadIdx.x & 7) == 0 && v0 < n_verts) {
        keep[v0 >> 5] = w;
        kept[v0 >> 5] = __popc(w);
    }
}

// Position of vertex v among the kept ones.
__device__ __forceinline__ int64_t kept_before(const uint32_t* __restrict__ keep,
                                               const int64_t* __restrict__ pos, int64_t v) {
    return pos[v >> 5] + __popc(keep[v >> 5] & ((1u << (v & 31)) - 1u));
}

// A thread per vertex: the kept ones to their places (coalesced reads, nearly
// coalesced writes: 0.28 ms for 49M vertices, 1.69 ms with a thread per loop).
__global__ void k_sp_write(const int32_t* __restrict__ eid, const float2* __restrict__ xy,
                           const uint32_t* __restrict__ keep, const int64_t* __restrict__ pos,
                           int64_t n_verts, int32_t* __restrict__ oeid,
                           float2* __restrict__ oxy) {
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n_verts;
         v += (int64_t)gridDim.x * blockDim.x) {
        if (!((keep[v >> 5] >> (v & 31)) & 1u)) continue;
        const int64_t o = kept_before(keep, pos, v);
        oeid[o] = eid[v];
        oxy[o] = xy[v];
    }
}

// The loops' new offsets (the closing one included).
__global__ void k_sp_offsets(const int64_t* __restrict__ loop_off, int64_t n_loops,
                             int64_t n_verts, const uint32_t* __restrict__ keep,
                             const int64_t* __restrict__ pos, const int64_t* __restrict__ total,
                             int64_t* __restrict__ new_off) {
    for (int64_t L = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; L <= n_loops;
         L += (int64_t)gridDim.x * blockDim.x) {
        const int64_t v = loop_off[L];
        new_off[L] = v < n_verts ? kept_before(keep, pos, v) : *total;
    }
}

}  // namespace
}  // namespace csl

using namespace csl;

extern "C" csl_status csl_simplify_contours(const csl_contours* in, int32_t nx, int32_t ny,
                                            double tol, void* stream, csl_contours** out) {
    csl_contours* c = nullptr;
    try {
        if (!in || !out) fail(CSL_ERR_INVALID_ARG, "NULL argument");
        *out = nullptr;
        if (!in->on_device) fail(CSL_ERR_INVALID_ARG, "contours must be on the device");
        if (!in->edge_id) fail(CSL_ERR_INVALID_ARG, "contours need their edge ids");
        if (nx < 1 || ny < 1 || nx > 32000 || ny > 32000)
            fail(CSL_ERR_INVALID_ARG, "nx, ny must be in [1, 32000]");
        if (!(tol >= 0.0) || !isfinite(tol)) fail(CSL_ERR_INVALID_ARG, "tol must be >= 0");
        cudaStream_t s = (cudaStream_t)stream;
        SpGrid g;
        g.W = nx + 2;
        g.H = ny + 2;
        g.words = ceil_div(2 * (int64_t)g.W * g.H, 32);
        const int n_layers = in->n_layers;
        const int64_t n_loops = in->n_loops, n_verts = in->n_verts;
        if ((double)n_layers * (double)g.words * 4.0 > (double)(16ll << 30))
            fail(CSL_ERR_CAPACITY, "edge bitmap above 16 GiB: simplify fewer layers at a time");
        c = new csl_contours();
        c->n_layers = n_layers;
        c->on_device = 1;
        c->n_loops = n_loops;
        auto dst_alloc = [&](void** p, size_t bytes) {
            *p = result_alloc(bytes, s, "device allocation of the contours failed");
        };
        dst_alloc((void**)&c->layer_loop_off, (size_t)(n_layers + 1) * 8);
        dst_alloc((void**)&c->loop_vert_off, (size_t)(n_loops + 1) * 8);
        CSL_CUDA(cudaMemcpyAsync(c->layer_loop_off, in->layer_loop_off, (size_t)(n_layers + 1) * 8,
                                 cudaMemcpyDeviceToDevice, s));
        DevBuf d_layer((size_t)std::max<int64_t>(n_loops, 1) * 4, s);
        DevBuf d_bits((size_t)std::max<int64_t>((int64_t)n_layers * g.words, 1) * 4, s);
        const int64_t n_words = ceil_div(n_verts, 32);   // keep bits, their counts, positions
        DevBuf d_first((size_t)loop_spans(n_verts) * 4, s);
        DevBuf d_keep((size_t)n_words * 4, s), d_kept((size_t)n_words * 4, s);
        DevBuf d_pos((size_t)n_words * 8, s);
        DevBuf d_tot(8, s), d_bad(4, s);
        int64_t n_out = 0;
        if (n_loops > 0) {
            CSL_CUDA(cudaMemsetAsync(d_bad.get(), 0, 4, s));
            CSL_CUDA(cudaMemsetAsync(d_bits.get(), 0, (size_t)n_layers * g.words * 4, s));
            k_sp_loop_layer<<<grid_for(n_loops, 256), 256, 0, s>>>(in->layer_loop_off, n_layers,
                                                                   n_loops, d_layer.as<int32_t>());
            CSL_LAUNCH_CHECK("simplify loop layers");
            if (n_verts > 0) {
                const unsigned spans = (unsigned)loop_spans(n_verts);
                span_first_loops(in->loop_vert_off, n_loops, d_first.as<uint32_t>(), s);
                k_sp_mark<<<spans, kLoopThreads, 0, s>>>(
                    in->loop_vert_off, in->edge_id, d_layer.as<int32_t>(), d_first.as<uint32_t>(),
                    n_loops, n_verts, g, d_bits.as<uint32_t>(), d_bad.as<uint32_t>());
                CSL_LAUNCH_CHECK("simplify edge bitmap");
                k_sp_keep<<<spans, kLoopThreads, 0, s>>>(
                    in->loop_vert_off, in->edge_id, reinterpret_cast<const float2*>(in->xy),
                    d_layer.as<int32_t>(), d_first.as<uint32_t>(), n_loops, n_verts, g,
                    d_bits.as<uint32_t>(), tol, d_keep.as<uint32_t>(), d_kept.as<uint32_t>());
                CSL_LAUNCH_CHECK("simplify decisions");
            }
            exclusive_scan_u32_to_i64(d_kept.as<uint32_t>(), d_pos.as<int64_t>(), n_words,
                                      d_tot.as<int64_t>(), s);
            k_sp_offsets<<<grid_for(n_loops + 1, 256), 256, 0, s>>>(
                in->loop_vert_off, n_loops, n_verts, d_keep.as<uint32_t>(), d_pos.as<int64_t>(),
                d_tot.as<int64_t>(), c->loop_vert_off);
            CSL_LAUNCH_CHECK("simplify offsets");
            n_out = read_i64(d_tot.as<int64_t>(), s);
            uint32_t bad = 0;
            read_to_host(&bad, d_bad.get(), 4, s);
            if (bad) fail(CSL_ERR_INVALID_ARG, "edge ids outside the nx x ny grid");
        } else {
            CSL_CUDA(cudaMemsetAsync(c->loop_vert_off, 0, 8, s));
        }
        c->n_verts = n_out;
        dst_alloc((void**)&c->xy, (size_t)n_out * 8);
        dst_alloc((void**)&c->edge_id, (size_t)n_out * 4);
        if (n_verts > 0 && n_loops > 0) {
            k_sp_write<<<grid_for(n_verts, 256, INT_MAX), 256, 0, s>>>(
                in->edge_id, reinterpret_cast<const float2*>(in->xy), d_keep.as<uint32_t>(),
                d_pos.as<int64_t>(), n_verts, c->edge_id, reinterpret_cast<float2*>(c->xy));
            CSL_LAUNCH_CHECK("simplify write");
        }
        CSL_CUDA(cudaStreamSynchronize(s));
        *out = c;
        return CSL_OK;
    } catch (const Error& e) {
        if (c) csl_contours_free(c);
        set_last_error(e.what());
        return e.code;
    } catch (...) {
        if (c) csl_contours_free(c);
        set_last_error("unknown error");
        return CSL_ERR_CUDA;
    }
}
