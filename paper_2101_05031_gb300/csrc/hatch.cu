// Zigzag infill of every layer's contours (Sec. 6: after the binary image and
// its boundary contours, a zigzag toolpath fills the interior).
//
// Scan lines y_m = y0 + m * spacing (m < n_lines; the same in every layer; y_m
// is y0 + m spacing in double, rounded once to float). An edge a -> b of a
// loop crosses line m when min(a_y, b_y) <= y_m < max(a_y, b_y) (half-open,
// decided in float), at x = a_x + t (b_x - a_x), t = (y_m - a_y) / (b_y - a_y).
// Along each line the crossings, sorted by x, alternate between entering and
// leaving the solid (the loops are closed and do not cross), so consecutive
// pairs are the inside segments. The toolpath of a layer visits the lines in
// increasing m, the segments of even lines from low to high x and those of odd
// lines in the opposite order, each odd-line segment from high to low x.
//
// Device pipeline: loop and layer of every vertex, then a bucket per line (key =
// layer * n_lines + m): crossings counted per line, the counts scanned, the x
// placed in their line's bucket, and a warp per line that sorts its bucket and
// writes its segments. The order inside a line is that of the x alone (equal x
// are the same bits), so the slots that atomics hand out do not show. Where a line
// has more than kLineMost crossings the buckets go to radix sorts by x and then by
// key; so do, without buckets, more lines than vertices (where the lines' counts
// cost more than the crossings).
#include <math.h>
#include <string.h>

#include <algorithm>
#include <functional>
#include <new>

#include "loops.cuh"

namespace csl {
namespace {

// The scan lines' y, computed once in double and rounded to float.
__global__ void k_line_table(double y0, double sp, int n, float* __restrict__ ys) {
    const int m = blockIdx.x * blockDim.x + threadIdx.x;
    if (m < n) ys[m] = (float)(y0 + (double)m * sp);
}

// first m in [0, n] with ys[m] >= v (the table is non-decreasing): a float
// estimate, then exact comparisons against the table
__device__ __forceinline__ int first_line_at_or_above(const float* __restrict__ ys, float y0f,
                                                      float inv_sp, int n, float v) {
    const float e = ceilf((v - y0f) * inv_sp);
    int m = e < 0.0f ? 0 : (e > (float)n ? n : (int)e);
    while (m > 0 && ys[m - 1] >= v) --m;
    while (m < n && ys[m] < v) ++m;
    return m;
}

__global__ void k_mark_i64(const int64_t* __restrict__ off, int64_t n_groups, int64_t n_items,
                           uint32_t* __restrict__ flag) {
    // flag[off[g]] += 1 for every group g >= 1 that starts inside [0, n_items)
    for (int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x + 1; g < n_groups;
         g += (int64_t)gridDim.x * blockDim.x) {
        const int64_t p = off[g];
        if (p >= 0 && p < n_items) atomicAdd(flag + p, 1u);
    }
}

// inclusive scan from the exclusive one: idx[i] = excl[i] + flag[i]
__global__ void k_incl(const uint32_t* __restrict__ flag, uint32_t* __restrict__ idx, int64_t n) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x)
        idx[i] += flag[i];
}

struct HatchConst {
    const float* ys;   // the lines' y (k_line_table)
    float y0f, inv_sp;
    int32_t n_lines;
    int32_t log_copies;   // log2 of a line's counters (count_copies)
    int64_t n_verts;
};

__device__ __forceinline__ void edge_of(const int64_t* __restrict__ loop_off,
                                        const uint32_t* __restrict__ loop_of, int64_t v,
                                        int64_t& w) {
    const uint32_t L = loop_of[v];
    w = v + 1 < loop_off[L + 1] ? v + 1 : loop_off[L];
}

__global__ void k_count(const float2* __restrict__ xy, const int64_t* __restrict__ loop_off,
                        const uint32_t* __restrict__ loop_of, HatchConst c,
                        uint32_t* __restrict__ cnt) {
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < c.n_verts;
         v += (int64_t)gridDim.x * blockDim.x) {
        int64_t w;
        edge_of(loop_off, loop_of, v, w);
        const float ya = xy[v].y, yb = xy[w].y;
        const float lo = fminf(ya, yb), hi = fmaxf(ya, yb);
        uint32_t k = 0;
        if (lo < hi) {
            const int m0 = first_line_at_or_above(c.ys, c.y0f, c.inv_sp, c.n_lines, lo);
            const int m1 = first_line_at_or_above(c.ys, c.y0f, c.inv_sp, c.n_lines, hi);
            k = (uint32_t)(m1 - m0);
        }
        cnt[v] = k;
    }
}

__global__ void k_emit_crossings(const float2* __restrict__ xy, const int64_t* __restrict__ loop_off,
                                 const uint32_t* __restrict__ loop_of,
                                 const uint32_t* __restrict__ layer_of, HatchConst c,
                                 const int64_t* __restrict__ pos, uint32_t* __restrict__ key,
                                 float* __restrict__ xs) {
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < c.n_verts;
         v += (int64_t)gridDim.x * blockDim.x) {
        int64_t w;
        edge_of(loop_off, loop_of, v, w);
        const float2 a = xy[v], b = xy[w];
        const float lo = fminf(a.y, b.y), hi = fmaxf(a.y, b.y);
        if (!(lo < hi)) continue;
        const int m0 = first_line_at_or_above(c.ys, c.y0f, c.inv_sp, c.n_lines, lo);
        const int m1 = first_line_at_or_above(c.ys, c.y0f, c.inv_sp, c.n_lines, hi);
        const uint32_t base = layer_of[loop_of[v]] * (uint32_t)c.n_lines;
        int64_t p = pos[v];
        for (int m = m0; m < m1; ++m, ++p) {
            const float ym = c.ys[m];
            const float t = __fdiv_rn(ym - a.y, b.y - a.y);
            key[p] = base + (uint32_t)m;
            xs[p] = fmaf(t, b.x - a.x, a.x);
        }
    }
}

// float -> uint32 whose unsigned order is the float order, and back
__device__ __forceinline__ uint32_t order_of(float x) {
    const uint32_t b = __float_as_uint(x);
    return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}
__device__ __forceinline__ float float_of(uint32_t k) {
    return __uint_as_float((k & 0x80000000u) ? k & 0x7fffffffu : ~k);
}

// Every crossing of every edge, by whole warps: f(slot, m, a, b, peers), slot = the
// line's key << log_copies | the warp's copy of its counter, peers = the lanes that are
// at a crossing of the same line now. Contours list their loops row by row, so the
// lanes of a warp meet the same few lines: an atomic for each group of them instead of
// one per crossing takes 0.13 ms instead of 1.25 for the counts of 3000 x 1000 squares
// (12 million crossings on 2,000 lines), where atomics on one address took turns. Edges
// of more than kWideEdge lines are taken by all lanes together where that is the
// shorter way, those of more than kLongEdge are only handed to long_edge(v, lines): for
// the whole grid (each_long_crossing). kPerLane edges per lane at a time: the infill of
// 389 million vertices, three in four of whose edges cross no line, takes 11.4 ms with
// 1, 10.4 with 2 (11.0 where k_line_emit has 48 registers, not 40), 12.1 with 3, 11.0
// with an atomic per crossing; 2 from 2^22 vertices on, where the lanes have more edges
// than one.
constexpr int kWideEdge = 32, kLongEdge = 1024;
template <int kPerLane, class F, class G>
__device__ __forceinline__ void each_crossing(const float2* __restrict__ xy,
                                              const int64_t* __restrict__ loop_off,
                                              const uint32_t* __restrict__ loop_of,
                                              const uint32_t* __restrict__ layer_of,
                                              const HatchConst& c, F f, G long_edge) {
    const int lane = threadIdx.x & 31;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x * kPerLane;
    for (int64_t v0 = ((int64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31u)) * kPerLane;
         v0 < c.n_verts; v0 += stride) {
        bool any = false;
        const uint32_t copy =
            (uint32_t)((uint64_t)v0 / (32 * kPerLane)) & ((1u << c.log_copies) - 1u);
        // kPerLane edges per lane: their chains of loads run side by side
        float2 ea[kPerLane], eb[kPerLane];
        int em[kPerLane], en[kPerLane];
        uint32_t ebase[kPerLane];
#pragma unroll
        for (int u = 0; u < kPerLane; ++u) {
            const int64_t v = v0 + 32 * u + lane;
            float2 a = make_float2(0.0f, 0.0f), b = a;
            int m = 0, n = 0;
            ebase[u] = 0;
            if (v < c.n_verts) {
                int64_t w;
                edge_of(loop_off, loop_of, v, w);
                a = xy[v];
                b = xy[w];
                const float lo = fminf(a.y, b.y), hi = fmaxf(a.y, b.y);
                if (lo < hi) {
                    // most edges cross no line or one
                    m = first_line_at_or_above(c.ys, c.y0f, c.inv_sp, c.n_lines, lo);
                    if (m < c.n_lines && c.ys[m] < hi) {
                        n = 1;
                        if (m + 1 < c.n_lines && c.ys[m + 1] < hi)
                            n = first_line_at_or_above(c.ys, c.y0f, c.inv_sp, c.n_lines, hi) - m;
                        ebase[u] = layer_of[loop_of[v]] * (uint32_t)c.n_lines;
                        if (n > kLongEdge) {
                            long_edge(v, n);
                            n = 0;
                        }
                    }
                }
            }
            ea[u] = a;
            eb[u] = b;
            em[u] = m;
            en[u] = n;
            any |= n > 0;
        }
        if (!__any_sync(0xffffffffu, any)) continue;
#pragma unroll
        for (int u = 0; u < kPerLane; ++u) {
            const float2 a = ea[u], b = eb[u];
            const int m = em[u];
            const uint32_t base = ebase[u];
            int n = en[u];
            int most = __reduce_max_sync(0xffffffffu, n);
            uint32_t wide = 0u;
            if (most > kWideEdge) {
                // steps by all lanes together against steps of a lane per edge (which share
                // atomics with their neighbours)
                const int together =
                    __reduce_add_sync(0xffffffffu, n > kWideEdge ? (n + 31) / 32 : 0);
                if (2 * together < most) {
                    wide = __ballot_sync(0xffffffffu, n > kWideEdge);
                    most = kWideEdge;
                }
            }
            for (; wide; wide &= wide - 1u) {
                const int src = __ffs(wide) - 1;
                const float2 p = make_float2(__shfl_sync(0xffffffffu, a.x, src),
                                             __shfl_sync(0xffffffffu, a.y, src));
                const float2 q = make_float2(__shfl_sync(0xffffffffu, b.x, src),
                                             __shfl_sync(0xffffffffu, b.y, src));
                const uint32_t pb = __shfl_sync(0xffffffffu, base, src);
                const int from = __shfl_sync(0xffffffffu, m, src);
                const int pn = __shfl_sync(0xffffffffu, n, src);
                for (int k = lane; k < pn; k += 32)
                    f((pb + (uint32_t)(from + k)) << c.log_copies | copy, from + k, p, q,
                      1u << lane);
                if (lane == src) n = 0;
                __syncwarp();
            }
            for (int k = 0; k < most; ++k) {
                const uint32_t act = __ballot_sync(0xffffffffu, k < n);
                if (k < n) {
                    const uint32_t slot = (base + (uint32_t)(m + k)) << c.log_copies | copy;
                    f(slot, m + k, a, b, __match_any_sync(act, slot));
                }
            }
        }
    }
}

// The crossings of the n listed pieces {vertex, piece of kLongEdge lines}, a block
// each: one side of 100,000 lines in a lane (or a warp) is a chain of as many steps
// (or a 32nd); 200 sides of 40,000 lines beside 30,000 squares: 1.04 ms, 17.4 with a warp
// per side, 10.3 with radix sorts alone and a lane per side. f as above, each lane at a
// line of its own.
constexpr int kLongBlocks = 152 * 8;
template <class F>
__device__ __forceinline__ void each_long_crossing(const float2* __restrict__ xy,
                                                   const int64_t* __restrict__ loop_off,
                                                   const uint32_t* __restrict__ loop_of,
                                                   const uint32_t* __restrict__ layer_of,
                                                   const HatchConst& c,
                                                   const uint2* __restrict__ list, uint32_t n,
                                                   F f) {
    for (uint32_t i = blockIdx.x; i < n; i += gridDim.x) {
        const uint2 e = list[i];
        const int64_t v = e.x;
        int64_t w;
        edge_of(loop_off, loop_of, v, w);
        const float2 a = xy[v], b = xy[w];
        const int m0 = first_line_at_or_above(c.ys, c.y0f, c.inv_sp, c.n_lines, fminf(a.y, b.y));
        const int m1 = first_line_at_or_above(c.ys, c.y0f, c.inv_sp, c.n_lines, fmaxf(a.y, b.y));
        const uint32_t base = layer_of[loop_of[v]] * (uint32_t)c.n_lines;
        const int64_t from = m0 + (int64_t)e.y * kLongEdge;
        const int64_t to = min((int64_t)m1, from + kLongEdge);
        for (int64_t m = from + threadIdx.x; m < to; m += blockDim.x)
            f((base + (uint32_t)m) << c.log_copies | (i & ((1u << c.log_copies) - 1u)), (int)m, a,
              b, 1u << (threadIdx.x & 31));
    }
}

// Crossings per line; the pieces of long edges are listed (n_list[0], room for `cap` of
// them: more have more crossings together than the call takes, n_list[1]).
template <int U>
__global__ void k_line_count(const float2* __restrict__ xy, const int64_t* __restrict__ loop_off,
                             const uint32_t* __restrict__ loop_of,
                             const uint32_t* __restrict__ layer_of, HatchConst c,
                             uint32_t* __restrict__ hist, uint2* __restrict__ list,
                             uint32_t cap, uint32_t* __restrict__ n_list) {
    const uint32_t lane = threadIdx.x & 31;
    each_crossing<U>(
        xy, loop_off, loop_of, layer_of, c,
        [&](uint32_t slot, int, float2, float2, uint32_t peers) {
            if (lane == __ffs(peers) - 1u) atomicAdd(hist + slot, (uint32_t)__popc(peers));
        },
        [&](int64_t v, int lines) {
            const uint32_t n = ((uint32_t)lines + kLongEdge - 1u) / kLongEdge;
            const uint32_t at = atomicAdd(n_list, n);
            if (at >= cap || n > cap - at) atomicOr(n_list + 1, 1u);
            for (uint32_t k = 0; k < n && at + k < cap; ++k) list[at + k] = make_uint2((uint32_t)v, k);
        });
}

__global__ void k_line_count_long(const float2* __restrict__ xy,
                                  const int64_t* __restrict__ loop_off,
                                  const uint32_t* __restrict__ loop_of,
                                  const uint32_t* __restrict__ layer_of, HatchConst c,
                                  uint32_t* __restrict__ hist, const uint2* __restrict__ list,
                                  uint32_t cap, const uint32_t* __restrict__ n_list) {
    each_long_crossing(xy, loop_off, loop_of, layer_of, c, list, min(*n_list, cap),
                       [&](uint32_t slot, int, float2, float2, uint32_t) { atomicAdd(hist + slot, 1u); });
}

// most[0] = the longest line's crossings; a line with an odd count is reported.
__global__ void k_line_most(const uint32_t* __restrict__ hist, int64_t n_keys, int log_copies,
                            uint32_t* __restrict__ status, uint32_t* __restrict__ most) {
    uint32_t m = 0, odd = 0;
    for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < n_keys;
         k += (int64_t)gridDim.x * blockDim.x) {
        uint32_t n = 0;
#pragma unroll 8
        for (int u = 0; u < 1 << log_copies; ++u) n += hist[(k << log_copies) + u];
        m = max(m, n);
        odd |= n & 1u;
    }
    m = __reduce_max_sync(0xffffffffu, m);
    odd = __reduce_or_sync(0xffffffffu, odd);
    if ((threadIdx.x & 31) == 0) {
        if (m) atomicMax(most, m);
        if (odd) atomicOr(status, ST_CAPACITY);
    }
}

// Each crossing's x into its line's bucket: the slots left are counted down in
// hist, which ends at 0. With keys (lines too long for a warp) the crossings' lines
// beside them, and x as it is.
struct LineBuckets {
    const int64_t* __restrict__ start;
    uint32_t* __restrict__ hist;
    uint32_t* __restrict__ xs;
    uint32_t* __restrict__ keys;

    __device__ __forceinline__ void put(const HatchConst& c, uint32_t slot, int m, float2 a,
                                        float2 b, uint32_t peers) const {
        const uint32_t lane = threadIdx.x & 31;
        const float t = __fdiv_rn(c.ys[m] - a.y, b.y - a.y);
        const float x = fmaf(t, b.x - a.x, a.x);
        const int first = __ffs(peers) - 1;
        uint32_t left = 0;
        if (lane == (uint32_t)first) left = atomicSub(hist + slot, (uint32_t)__popc(peers));
        left = __shfl_sync(peers, left, first);
        const int64_t at = start[slot] + left - 1 - __popc(peers & ((1u << lane) - 1u));
        xs[at] = keys ? __float_as_uint(x) : order_of(x);
        if (keys) keys[at] = slot >> c.log_copies;
    }
};

template <int U>
__global__ void __launch_bounds__(256, 6)
k_line_emit(const float2* __restrict__ xy, const int64_t* __restrict__ loop_off,
            const uint32_t* __restrict__ loop_of, const uint32_t* __restrict__ layer_of,
            HatchConst c, LineBuckets to) {
    each_crossing<U>(
        xy, loop_off, loop_of, layer_of, c,
        [&](uint32_t slot, int m, float2 a, float2 b, uint32_t peers) {
            to.put(c, slot, m, a, b, peers);
        },
        [](int64_t, int) {});
}

__global__ void k_line_emit_long(const float2* __restrict__ xy,
                                 const int64_t* __restrict__ loop_off,
                                 const uint32_t* __restrict__ loop_of,
                                 const uint32_t* __restrict__ layer_of, HatchConst c,
                                 LineBuckets to, const uint2* __restrict__ list, uint32_t n) {
    each_long_crossing(xy, loop_off, loop_of, layer_of, c, list, n,
                       [&](uint32_t slot, int m, float2 a, float2 b, uint32_t peers) {
                           to.put(c, slot, m, a, b, peers);
                       });
}

// A warp per line: its crossings sorted in shared memory (a bitonic network over
// the next power of two, at most `room`) and its segments written in toolpath
// order. 250 layers of 500 lines: 0.23 ms, bound by the latency of the loads and
// stages (strides below 32 by shuffles instead: the same); the infill with the
// counts (0.19 ms) and the buckets (0.3 ms) 1.00 ms a call, 1.11 with an atomic per
// crossing in both (0.23 and 0.35; 0.84 ms of kernels, where 7 passes of radix sorts
// made 1.39). 1000 x 1000 squares x 3 layers (2,000 crossings per line): 0.90 ms, 1.68
// with radix sorts alone; 3000 x 1000 (6,000 per line): buckets and radix sorts
// 1.50 ms, 1.67 with radix sorts alone.
constexpr int kLineMost = 2048, kLineWarps = 4;
__global__ void __launch_bounds__(32 * kLineWarps)
k_line_sort(const uint32_t* __restrict__ xs, const int64_t* __restrict__ start, int64_t n_keys,
            int64_t n_rec, int room, HatchConst c, float* __restrict__ out) {
    extern __shared__ uint32_t s_line[];
    const int lane = threadIdx.x & 31;
    uint32_t* q = s_line + (threadIdx.x >> 5) * room;
    const int64_t stride = (int64_t)gridDim.x * kLineWarps;
    for (int64_t k = (int64_t)blockIdx.x * kLineWarps + (threadIdx.x >> 5); k < n_keys;
         k += stride) {
        const int64_t lo = start[k << c.log_copies];
        const int64_t hi = k + 1 < n_keys ? start[(k + 1) << c.log_copies] : n_rec;
        const int n = (int)(hi - lo);
        if (n < 2 || n > room) continue;
        int P = 2;
        while (P < n) P <<= 1;
        __syncwarp();
        for (int i = lane; i < P; i += 32) q[i] = i < n ? xs[lo + i] : 0xffffffffu;
        for (int kk = 2; kk <= P; kk <<= 1)
            for (int j = kk >> 1; j > 0; j >>= 1) {
                __syncwarp();
                for (int t = lane; t < P / 2; t += 32) {
                    const int i = 2 * t - (t & (j - 1));
                    const uint32_t a = q[i], b = q[i + j];
                    if ((a > b) == ((i & kk) == 0)) {
                        q[i] = b;
                        q[i + j] = a;
                    }
                }
            }
        __syncwarp();
        const int m = (int)((uint32_t)k % (uint32_t)c.n_lines);
        const float ym = c.ys[m];
        const bool odd = (m & 1) != 0;
        // floats 3 o + r of the line's segments, in order
        float* o = out + 3 * (lo / 2);
        for (int i = lane; i < 3 * (n / 2); i += 32) {
            const int seg = i / 3, r = i - 3 * seg;
            const int at = odd ? n - 1 - (2 * seg + r) : 2 * seg + r;
            o[i] = r == 2 ? ym : float_of(q[at]);
        }
    }
}

// layer_off[k] = first segment of layer k, from the lines' starts
__global__ void k_line_offsets(const int64_t* __restrict__ start, int64_t n_rec, int n_layers,
                               int n_lines, int log_copies, int64_t* __restrict__ layer_off) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k > n_layers) return;
    layer_off[k] = (k == n_layers ? n_rec : start[((int64_t)k * n_lines) << log_copies]) / 2;
}

__global__ void k_x_keys(const float* __restrict__ xs, int64_t n, uint32_t* __restrict__ k,
                         uint32_t* __restrict__ idx) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        k[i] = order_of(xs[i]);
        idx[i] = (uint32_t)i;
    }
}

__global__ void k_gather_u32(const uint32_t* __restrict__ src, const uint32_t* __restrict__ idx,
                             int64_t n, uint32_t* __restrict__ dst) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x)
        dst[i] = src[idx[i]];
}

// Segment s = sorted crossings (2s, 2s + 1), which must lie on one line.
__global__ void k_pairs(const uint32_t* __restrict__ skey, const uint32_t* __restrict__ sidx,
                        const float* __restrict__ xs, int64_t n_seg,
                        uint32_t* __restrict__ seg_key, float2* __restrict__ seg_x,
                        uint32_t* status) {
    for (int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; s < n_seg;
         s += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t k0 = skey[2 * s], k1 = skey[2 * s + 1];
        if (k0 != k1) atomicOr(status, ST_CAPACITY);   // a line with an odd crossing count
        seg_key[s] = k0;
        seg_x[s] = make_float2(xs[sidx[2 * s]], xs[sidx[2 * s + 1]]);
    }
}

__global__ void k_runs(const uint32_t* __restrict__ seg_key, int64_t n_seg,
                       uint32_t* __restrict__ run_lo, uint32_t* __restrict__ run_hi) {
    for (int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; s < n_seg;
         s += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t k = seg_key[s];
        if (s == 0 || seg_key[s - 1] != k) run_lo[k] = (uint32_t)s;
        if (s == n_seg - 1 || seg_key[s + 1] != k) run_hi[k] = (uint32_t)(s + 1);
    }
}

__global__ void k_zigzag(const uint32_t* __restrict__ seg_key, const float2* __restrict__ seg_x,
                         const uint32_t* __restrict__ run_lo, const uint32_t* __restrict__ run_hi,
                         int64_t n_seg, HatchConst c, float* __restrict__ out) {
    for (int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; s < n_seg;
         s += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t k = seg_key[s];
        const int m = (int)(k % (uint32_t)c.n_lines);
        const float2 x = seg_x[s];
        const bool odd = (m & 1) != 0;
        const int64_t o = odd ? (int64_t)run_lo[k] + run_hi[k] - 1 - s : s;
        out[3 * o] = odd ? x.y : x.x;
        out[3 * o + 1] = odd ? x.x : x.y;
        out[3 * o + 2] = c.ys[m];
    }
}

// layer_off[k] = first segment of layer k (keys k * n_lines ...)
__global__ void k_layer_offsets(const uint32_t* __restrict__ seg_key, int64_t n_seg, int n_layers,
                                int n_lines, int64_t* __restrict__ layer_off) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k > n_layers) return;
    const uint32_t target = (uint32_t)k * (uint32_t)n_lines;
    int64_t lo = 0, hi = n_seg;
    while (lo < hi) {
        const int64_t mid = (lo + hi) >> 1;
        if (seg_key[mid] < target) lo = mid + 1;
        else hi = mid;
    }
    layer_off[k] = k == n_layers ? n_seg : lo;
}

// log2 of the counters of a line: few lines of many vertices lie in a few sectors of
// L2, where atomics take turns whatever their address, so each line gets up to 64
// counters (its bucket is one part per counter) while there are no more than 2^14 in
// all and 128 vertices for each. 100,000 squares, 50 lines: 1.04 ms, 2.4 with one counter, 1.14
// with radix sorts alone; 200,000 x 5 squares, 20 lines: 0.77, 1.12 and 0.89.
int count_copies(int64_t n_keys, int64_t n_verts) {
    const int64_t most = n_verts / 128 < 1 << 14 ? n_verts / 128 : 1 << 14;
    int log = 0;
    while (log < 6 && n_keys << (log + 1) <= most) ++log;
    return log;
}

int bits_for(uint64_t n) {
    int b = 1;
    while (b < 32 && ((uint64_t)1 << b) < n) ++b;
    return b;
}

}  // namespace
}  // namespace csl

using namespace csl;

extern "C" {

csl_status csl_hatch_layers(const csl_contours* ct, double y0, double spacing, int32_t n_lines,
                            int32_t dst_on_device, void* stream, csl_hatches** out) {
    try {
        if (!out) fail(CSL_ERR_INVALID_ARG, "out is NULL");
        *out = nullptr;
        if (!ct) fail(CSL_ERR_INVALID_ARG, "contours is NULL");
        if (!ct->on_device) fail(CSL_ERR_INVALID_ARG, "contours must be on the device");
        if (!(isfinite(y0) && isfinite(spacing) && spacing > 0.0))
            fail(CSL_ERR_INVALID_ARG, "y0 must be finite and spacing > 0");
        if (n_lines < 0) fail(CSL_ERR_INVALID_ARG, "n_lines < 0");
        const int64_t n_layers = ct->n_layers, n_loops = ct->n_loops, n_verts = ct->n_verts;
        if ((uint64_t)n_layers * (uint64_t)(n_lines > 0 ? n_lines : 1) >= 0xffffffffull)
            fail(CSL_ERR_CAPACITY, "n_layers * n_lines must be below 2^32");
        if (n_verts >= 0xffffffffLL || n_loops >= 0xffffffffLL)
            fail(CSL_ERR_CAPACITY, "too many vertices");
        cudaStream_t s = (cudaStream_t)stream;
        DevBuf ys_d((size_t)(n_lines > 0 ? n_lines : 1) * 4, s);
        if (n_lines > 0) {
            k_line_table<<<(unsigned)ceil_div(n_lines, 256), 256, 0, s>>>(y0, spacing, n_lines,
                                                                         ys_d.as<float>());
            CSL_LAUNCH_CHECK("hatch lines");
        }
        HatchConst c{ys_d.as<float>(), (float)y0, (float)(1.0 / spacing), n_lines, 0, n_verts};
        const float2* xy = reinterpret_cast<const float2*>(ct->xy);

        int64_t n_rec = 0;
        const uint64_t n_keys = (uint64_t)n_layers * (uint64_t)(n_lines > 0 ? n_lines : 1);
        // small: [0, 1] crossings, [2] status, [3] the longest line's crossings, [4] pieces of
        // long edges, [5] more than their list holds
        DevBuf key, xs, line_start, small(32, s);
        bool by_line = false;
        int line_most = 0;
        CSL_CUDA(cudaMemsetAsync(small.get(), 0, 32, s));
        if (n_verts > 0 && n_lines > 0) {
            // loop of every vertex, layer of every loop
            DevBuf loop_of((size_t)n_verts * 4, s);
            loops_of_vertices(ct->loop_vert_off, n_loops, n_verts, loop_of.as<uint32_t>(), s);
            DevBuf lflag((size_t)n_loops * 4, s), layer_of((size_t)n_loops * 4, s);
            CSL_CUDA(cudaMemsetAsync(lflag.get(), 0, (size_t)n_loops * 4, s));
            k_mark_i64<<<grid_for(n_layers, 256), 256, 0, s>>>(ct->layer_loop_off, n_layers,
                                                               n_loops, lflag.as<uint32_t>());
            CSL_LAUNCH_CHECK("hatch layer starts");
            exclusive_scan_u32(lflag.as<uint32_t>(), layer_of.as<uint32_t>(), n_loops, nullptr, s);
            k_incl<<<grid_for(n_loops, 256), 256, 0, s>>>(lflag.as<uint32_t>(),
                                                          layer_of.as<uint32_t>(), n_loops);
            CSL_LAUNCH_CHECK("hatch layer of loop");
            // the first loops may precede the first layer start only when layer 0
            // has loops; layer_loop_off[0] is 0, so the counts are the layers
            if (n_keys <= (uint64_t)n_verts) {
                c.log_copies = count_copies((int64_t)n_keys, n_verts);
                const int64_t n_slots = (int64_t)n_keys << c.log_copies;
                DevBuf hist((size_t)n_slots * 4, s);
                CSL_CUDA(cudaMemsetAsync(hist.get(), 0, (size_t)n_slots * 4, s));
                // pieces of long edges: at least half of each is lines that it crosses, so
                // this many hold all the crossings that a call may have
                const int64_t pieces = ceil_div(n_lines, kLongEdge);
                const uint32_t long_cap = n_lines <= kLongEdge ? 0u
                    : (uint32_t)std::min<int64_t>(n_verts * pieces, (2ll << 32) / kLongEdge);
                DevBuf long_edges((size_t)std::max(long_cap, 1u) * 8, s);
                const bool two = n_verts >= (1 << 22);
                auto line_count = two ? k_line_count<2> : k_line_count<1>;
                auto line_emit = two ? k_line_emit<2> : k_line_emit<1>;
                line_count<<<grid_for(n_verts, 256), 256, 0, s>>>(
                    xy, ct->loop_vert_off, loop_of.as<uint32_t>(), layer_of.as<uint32_t>(), c,
                    hist.as<uint32_t>(), long_edges.as<uint2>(), long_cap,
                    small.as<uint32_t>() + 4);
                CSL_LAUNCH_CHECK("hatch line counts");
                if (long_cap) {
                    k_line_count_long<<<kLongBlocks, 256, 0, s>>>(
                        xy, ct->loop_vert_off, loop_of.as<uint32_t>(), layer_of.as<uint32_t>(), c,
                        hist.as<uint32_t>(), long_edges.as<uint2>(), long_cap,
                        small.as<uint32_t>() + 4);
                    CSL_LAUNCH_CHECK("hatch line counts of long edges");
                }
                k_line_most<<<grid_for((int64_t)n_keys, 256), 256, 0, s>>>(
                    hist.as<uint32_t>(), (int64_t)n_keys, c.log_copies, small.as<uint32_t>() + 2,
                    small.as<uint32_t>() + 3);
                CSL_LAUNCH_CHECK("hatch longest line");
                line_start.alloc((size_t)n_slots * 8, s);
                exclusive_scan_u32_to_i64(hist.as<uint32_t>(), line_start.as<int64_t>(), n_slots,
                                          small.as<int64_t>(), s);
                uint32_t h[6];
                read_to_host(h, small.get(), sizeof h, s);
                n_rec = (int64_t)(((uint64_t)h[1] << 32) | h[0]);
                if (n_rec >= 0xffffffffLL || h[5]) fail(CSL_ERR_CAPACITY, "too many crossings");
                if (n_rec % 2) fail(CSL_ERR_CUDA, "hatching: odd number of crossings");
                if (h[2]) fail(CSL_ERR_CUDA, "hatching: a line with an odd number of crossings");
                line_most = (int)std::min<uint32_t>(h[3], kLineMost + 1);
                by_line = line_most <= kLineMost;
                if (n_rec) {
                    xs.alloc((size_t)n_rec * 4, s);
                    if (!by_line) key.alloc((size_t)n_rec * 4, s);
                    const LineBuckets to{line_start.as<int64_t>(), hist.as<uint32_t>(),
                                         xs.as<uint32_t>(), by_line ? nullptr : key.as<uint32_t>()};
                    line_emit<<<grid_for(n_verts, 256), 256, 0, s>>>(
                        xy, ct->loop_vert_off, loop_of.as<uint32_t>(), layer_of.as<uint32_t>(), c,
                        to);
                    CSL_LAUNCH_CHECK("hatch line crossings");
                    if (h[4]) {
                        k_line_emit_long<<<kLongBlocks, 256, 0, s>>>(
                            xy, ct->loop_vert_off, loop_of.as<uint32_t>(), layer_of.as<uint32_t>(),
                            c, to, long_edges.as<uint2>(), h[4]);
                        CSL_LAUNCH_CHECK("hatch line crossings of long edges");
                    }
                }
            } else {
                DevBuf cnt((size_t)n_verts * 4, s), pos((size_t)n_verts * 8, s);
                k_count<<<grid_for(n_verts, 256), 256, 0, s>>>(xy, ct->loop_vert_off,
                                                               loop_of.as<uint32_t>(), c,
                                                               cnt.as<uint32_t>());
                CSL_LAUNCH_CHECK("hatch count");
                exclusive_scan_u32_to_i64(cnt.as<uint32_t>(), pos.as<int64_t>(), n_verts,
                                          small.as<int64_t>(), s);
                n_rec = read_i64(small.as<int64_t>(), s);
                if (n_rec >= 0xffffffffLL) fail(CSL_ERR_CAPACITY, "too many crossings");
                if (n_rec % 2) fail(CSL_ERR_CUDA, "hatching: odd number of crossings");
                key.alloc((size_t)(n_rec ? n_rec : 1) * 4, s);
                xs.alloc((size_t)(n_rec ? n_rec : 1) * 4, s);
                if (n_rec)
                    k_emit_crossings<<<grid_for(n_verts, 256), 256, 0, s>>>(
                        xy, ct->loop_vert_off, loop_of.as<uint32_t>(), layer_of.as<uint32_t>(), c,
                        pos.as<int64_t>(), key.as<uint32_t>(), xs.as<float>());
                CSL_LAUNCH_CHECK("hatch crossings");
            }
        }
        const int64_t n_seg = n_rec / 2;

        csl_hatches* h = new csl_hatches();
        memset(h, 0, sizeof(*h));
        h->n_layers = (int32_t)n_layers;
        h->on_device = dst_on_device ? 1 : 0;
        h->n_segments = n_seg;
        auto alloc = [&](void** p, size_t b) {
            if (dst_on_device) {
                *p = result_alloc(b, s, "device allocation of the hatches failed");
            } else {
                *p = host_block_alloc(b ? b : 16);
            }
        };
        try {
            alloc((void**)&h->layer_seg_off, (size_t)(n_layers + 1) * 8);
            alloc((void**)&h->seg, (size_t)n_seg * 12);
            DevBuf lay((size_t)(n_layers + 1) * 8, s), segs((size_t)(n_seg ? n_seg : 1) * 12, s);
            if (n_seg > 0 && by_line) {
                int room = 32;
                while (room < line_most) room <<= 1;
                const int64_t blocks =
                    std::min<int64_t>(ceil_div((int64_t)n_keys, kLineWarps), (int64_t)1 << 30);
                k_line_sort<<<(unsigned)blocks, 32 * kLineWarps, 4 * kLineWarps * room, s>>>(
                    xs.as<uint32_t>(), line_start.as<int64_t>(), (int64_t)n_keys, n_rec, room,
                    c, segs.as<float>());
                CSL_LAUNCH_CHECK("hatch line sort");
                k_line_offsets<<<(unsigned)ceil_div(n_layers + 1, 128), 128, 0, s>>>(
                    line_start.as<int64_t>(), n_rec, (int)n_layers, n_lines, c.log_copies,
                    lay.as<int64_t>());
                CSL_LAUNCH_CHECK("hatch layer offsets");
            } else if (n_seg > 0) {
                // sort by x, then (stably) by line key
                DevBuf k1((size_t)n_rec * 4, s), idx((size_t)n_rec * 4, s), tk((size_t)n_rec * 4, s),
                    tv((size_t)n_rec * 4, s);
                k_x_keys<<<grid_for(n_rec, 256), 256, 0, s>>>(xs.as<float>(), n_rec,
                                                              k1.as<uint32_t>(), idx.as<uint32_t>());
                CSL_LAUNCH_CHECK("hatch x keys");
                radix_sort_pairs(k1.as<uint32_t>(), idx.as<uint32_t>(), tk.as<uint32_t>(),
                                 tv.as<uint32_t>(), n_rec, 32, s);
                k_gather_u32<<<grid_for(n_rec, 256), 256, 0, s>>>(key.as<uint32_t>(),
                                                                  idx.as<uint32_t>(), n_rec,
                                                                  k1.as<uint32_t>());
                CSL_LAUNCH_CHECK("hatch gather keys");
                radix_sort_pairs(k1.as<uint32_t>(), idx.as<uint32_t>(), tk.as<uint32_t>(),
                                 tv.as<uint32_t>(), n_rec, bits_for(n_keys), s);
                DevBuf seg_key((size_t)n_seg * 4, s), seg_x((size_t)n_seg * 8, s);
                k_pairs<<<grid_for(n_seg, 256), 256, 0, s>>>(k1.as<uint32_t>(), idx.as<uint32_t>(),
                                                             xs.as<float>(), n_seg,
                                                             seg_key.as<uint32_t>(),
                                                             seg_x.as<float2>(),
                                                             small.as<uint32_t>() + 2);
                CSL_LAUNCH_CHECK("hatch pairs");
                DevBuf run_lo((size_t)n_keys * 4, s), run_hi((size_t)n_keys * 4, s);
                k_runs<<<grid_for(n_seg, 256), 256, 0, s>>>(seg_key.as<uint32_t>(), n_seg,
                                                            run_lo.as<uint32_t>(),
                                                            run_hi.as<uint32_t>());
                CSL_LAUNCH_CHECK("hatch runs");
                k_zigzag<<<grid_for(n_seg, 256), 256, 0, s>>>(seg_key.as<uint32_t>(),
                                                              seg_x.as<float2>(),
                                                              run_lo.as<uint32_t>(),
                                                              run_hi.as<uint32_t>(), n_seg, c,
                                                              segs.as<float>());
                CSL_LAUNCH_CHECK("hatch zigzag");
                k_layer_offsets<<<(unsigned)ceil_div(n_layers + 1, 128), 128, 0, s>>>(
                    seg_key.as<uint32_t>(), n_seg, (int)n_layers, n_lines, lay.as<int64_t>());
                CSL_LAUNCH_CHECK("hatch layer offsets");
                uint32_t st = 0;
                read_to_host(&st, small.as<uint32_t>() + 2, 4, s);
                if (st) fail(CSL_ERR_CUDA, "hatching: a line with an odd number of crossings");
            } else {
                CSL_CUDA(cudaMemsetAsync(lay.get(), 0, (size_t)(n_layers + 1) * 8, s));
            }
            const cudaMemcpyKind kind =
                dst_on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost;
            CSL_CUDA(cudaMemcpyAsync(h->layer_seg_off, lay.get(), (size_t)(n_layers + 1) * 8,
                                     kind, s));
            if (n_seg)
                CSL_CUDA(cudaMemcpyAsync(h->seg, segs.get(), (size_t)n_seg * 12, kind, s));
            CSL_CUDA(cudaStreamSynchronize(s));
        } catch (...) {
            csl_hatches_free(h);
            throw;
        }
        *out = h;
        return CSL_OK;
    } catch (const Error& e) {
        set_last_error(e.what());
        return e.code;
    } catch (const std::bad_alloc&) {
        set_last_error("host allocation failed");
        return CSL_ERR_OOM;
    } catch (...) {
        set_last_error("unknown error");
        return CSL_ERR_CUDA;
    }
}

void csl_hatches_free(csl_hatches* h) {
    if (!h) return;
    if (h->on_device) {
        result_free(h->layer_seg_off);
        result_free(h->seg);
    } else {
        host_block_free(h->layer_seg_off);
        host_block_free(h->seg);
    }
    delete h;
}

}  // extern "C"
