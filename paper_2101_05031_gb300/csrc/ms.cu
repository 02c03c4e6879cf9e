// Marching squares on each layer's binary image and assembly of closed loops
// (Sec. 4, last paragraph: the binary image is traced by marching squares).
//
// Grid: pixel samples padded by one ring of outside samples (padded sample
// (I, J) is pixel (I-1, J-1)), so every contour closes. Grid-edge ids are
// 2 (J W + I) for the edge to (I+1, J) and 2 (J W + I) + 1 for the edge to
// (I, J+1), W = nx + 2. The field kernel leaves the inside mask (one bit per
// padded sample, rows of 32-bit words).
//   1. k_edge_words: per mask word (32 samples of one row), the crossing bits
//      of their two grid edges by shift and xor, interleaved (h, v) into two
//      32-bit edge words per mask word;
//   2. a prefix sum of the edge words' popcounts numbers the crossings in
//      (layer, edge id) order: id = prefix[word] + popc(lower bits);
//   3. k_emit: per crossing, its vertex (the zero of the linear interpolant of
//      Sigma - C) and its successor, the other crossing side of the one of the
//      two cells sharing the edge that the contour enters there. Walking a
//      cell's sides counter-clockwise, a side from an inside to an outside
//      corner is an entry, from outside to inside an exit; a saddle (two
//      inside corners on a diagonal) joins its inside corners when the mean of
//      the 4 corner values is >= C, i.e. each entry turns to the next side,
//      else to the previous one. Inside lies on the left.
//   4. the head of a loop is its smallest id, which is a local minimum
//      (pred > id < succ). Splitters = all local minima plus a hashed sample
//      of crossings; each splitter walks its segment to the next
//      splitter, so no thread walks a whole long loop;
//   5. on the graph of splitters (one cycle per loop), a cycle of at most 16
//      splitters (32 in small chunks; every small loop) is resolved by walking
//      it; on the rest, pointer jumping (by one block in shared memory up to
//      kLongBlock splitters, by the grid above) gives every splitter its cycle's minimum (the head)
//      and, with the cycles cut before their heads, weighted list ranking
//      gives every segment its distance from the head;
//   6. a prefix sum over the heads (loop length) numbers the loops in head
//      order and places them; every splitter writes its segment there.
// Vertices, edge ids (where asked for) and successors lie in arrays of their
// own: a walk follows the 4-byte successors alone.
#include <math.h>

#include <algorithm>

#include "slice.cuh"

namespace csl {
namespace {

struct MsConst {
    int32_t nx, ny, W, H;
    int32_t mwr;          // mask words per row
    int32_t ewr;          // edge words per row (2 per mask word)
    int64_t mask_wpl;     // mask words per layer
    int64_t edge_wpl;     // edge words per layer
    int32_t n_layers;
    float C, fx0, fy0, fpx;
};

__device__ __forceinline__ uint32_t spread16(uint32_t x) {
    x &= 0xffffu;
    x = (x | (x << 8)) & 0x00ff00ffu;
    x = (x | (x << 4)) & 0x0f0f0f0fu;
    x = (x | (x << 2)) & 0x33333333u;
    x = (x | (x << 1)) & 0x55555555u;
    return x;
}

// grid: x over (row J, mask word k), y = layer. cnt: the crossings of each
// edge word (the input of the numbering scan).
__global__ void k_edge_words(const uint32_t* __restrict__ mask, MsConst c,
                             uint32_t* __restrict__ ew, uint32_t* __restrict__ cnt) {
    const int layer = blockIdx.y;
    const uint32_t idx = blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= (uint32_t)c.H * (uint32_t)c.mwr) return;
    const int J = (int)(idx / (uint32_t)c.mwr), k = (int)(idx - (uint32_t)J * c.mwr);
    const uint32_t* m = mask + (int64_t)layer * c.mask_wpl;
    const uint32_t in0 = m[(int64_t)J * c.mwr + k];
    const uint32_t in1 = k + 1 < c.mwr ? m[(int64_t)J * c.mwr + k + 1] : 0u;
    const uint32_t up = J + 1 < c.H ? m[(int64_t)(J + 1) * c.mwr + k] : 0u;
    const uint32_t h = in0 ^ ((in0 >> 1) | (in1 << 31));   // edge to (I+1, J)
    const uint32_t v = in0 ^ up;                           // edge to (I, J+1)
    uint2 out;
    out.x = spread16(h) | (spread16(v) << 1);
    out.y = spread16(h >> 16) | (spread16(v >> 16) << 1);
    const int64_t row = (int64_t)layer * c.edge_wpl + (int64_t)J * c.ewr;
    reinterpret_cast<uint2*>(ew + row)[k] = out;
    reinterpret_cast<uint2*>(cnt + row)[k] = make_uint2(__popc(out.x), __popc(out.y));
}

// Crossing numbering: the crossing on the edge with bit `bit` of edge word w
// has id prefix[w] + popc(ew[w] & ((1 << bit) - 1)).
struct Dense {
    const uint32_t* ew;
    const uint32_t* prefix;
    int64_t edge_wpl;
    int32_t ewr;
};

// The fused pass's vertex lists (FusedVerts, as the field kernel leaves them).
struct FusedIn {
    const uint32_t* tbase;
    const uint16_t* roff;
    const float2* verts;
    const uint32_t* saddle;
    int32_t T, ntx, n_tiles;
};

// Vertex of the crossing on the edge from padded sample (I, J) in direction
// dir (0: x, 1: y): the tile owning the sample lists its crossings in edge-id
// order, so its place is the tile's base + the row's offset + the number of
// crossing edges of row J from the row's first owned sample up to this edge
// (the interleaved edge words hold exactly those bits).
__device__ __forceinline__ float2 fused_vertex(const FusedIn& F, const Dense& D, int layer, int I,
                                               int J, int dir) {
    const int tx = I == 0 ? 0 : (I - 1) / F.T, ty = J == 0 ? 0 : (J - 1) / F.T;
    const int b = J - 1 - ty * F.T;                 // tile-local row, -1 .. T - 1
    const int Ia = tx == 0 ? 0 : tx * F.T + 1;      // first sample of the row the tile owns
    const uint32_t* row = D.ew + (int64_t)layer * D.edge_wpl + (int64_t)J * D.ewr;
    const int lo = 2 * Ia, hi = 2 * I + dir;
    uint32_t rank = 0;
    for (int w = lo >> 5; w <= ((hi - 1) >> 5) && hi > lo; ++w) {
        uint32_t m = row[w];
        if (w == (lo >> 5)) m &= 0xffffffffu << (lo & 31);
        if (w == (hi >> 5)) m &= (1u << (hi & 31)) - 1u;
        rank += __popc(m);
    }
    const int64_t tl = (int64_t)layer * F.n_tiles + (int64_t)ty * F.ntx + tx;
    return F.verts[(int64_t)F.tbase[tl] + F.roff[tl * (F.T + 1) + b + 1] + rank];
}

// A block of k_emit covers a band of kEmitRows sample rows and kEmitWords mask
// words (32 samples each) of one layer, a warp per row at a time. A lane takes a
// crossing: it computes the vertex and, from the two cells that share the
// edge, the crossing after it on the contour and whether it is a local minimum,
// so that vertices and successors are written in order and the splitters are
// known here.
// The crossings of a warp's row are listed in shared memory first (ids are
// consecutive along a row), which keeps every lane busy; edge words and their
// prefix sums of the band and of one row and one word around it are staged as
// pairs {word, prefix}. Sigma is read where a crossing needs it (through L1):
// a tile of it in shared memory costs a barrier and half the warps.
constexpr int kEmitRows = 8, kEmitWords = 32, kEmitWarps = 4;
constexpr int kEmitList = 512;                     // crossings listed at a time per warp
constexpr int kEmitPitch = 2 * kEmitWords + 2;     // edge words 2 k0 - 1 .. 2 (k0 + kEmitWords)

// Splitters cut every loop into short segments: every local minimum
// (pred > id < succ; the loop's smallest id is one) and a hashed sample of one
// in 2^bits, so that a smooth loop with a single local minimum is cut too:
// 1 in 32; in small chunks 1 in 8 or 16, because there the longest walk is what
// the segment kernels take (one 2000^2 layer: 15 + 24 us at 1 in 32, 5 + 9 us at
// 1 in 8; 200^2 x 50: 35 + 33 us and, at 1 in 16, 10 + 13 us), and the splitters
// more are few enough for the block that resolves long cycles.
int splitter_bits(int64_t n_cross) {
    return n_cross <= ((int64_t)1 << 16) ? 3 : (n_cross <= ((int64_t)1 << 18) ? 4 : 5);
}

// grid: x over (band of kEmitRows rows J <= ny, segment of kEmitWords mask
// words), y = layer. FUSED: vertices and saddle decisions from the fused pass
// (F) instead of Sigma. nxt[i] = succ(i) | (i is a splitter) << 31, the only
// array the segment walks read and the one whose top bits number the
// splitters. 389 million crossings of 500 layers of 2000^2: 3.55 ms, bound by
// issue (about 200 instructions per crossing); a thread per mask word stepping
// through its cells, with a Sigma tile in shared memory and 16-byte records
// written in parts, took 6.9 ms and the splitters 1.5 ms more (19 of 32 lanes
// active). 8 warps per block 4.3 ms, 16 rows per block 4.3, 4 rows 3.9.
template <bool FUSED>
__global__ void __launch_bounds__(32 * kEmitWarps, 12) k_emit(
    const float* __restrict__ sigma, const uint32_t* __restrict__ mask, MsConst c, Dense D,
    FusedIn F, int bits, float2* __restrict__ oxy, int32_t* __restrict__ oeid,
    uint32_t* __restrict__ nxt, uint32_t n_cap, uint32_t* flag) {
    __shared__ uint2 s_e[(kEmitRows + 2) * kEmitPitch];   // row J0 - 1 + r, word 2 k0 - 1 + x
    __shared__ uint32_t s_in[kEmitRows * kEmitWords];
    __shared__ uint16_t s_list[kEmitWarps * kEmitList];   // edge word << 5 | bit
    const int layer = blockIdx.y;
    const int n_segs = (c.mwr + kEmitWords - 1) / kEmitWords;
    const int band = blockIdx.x / n_segs, seg = blockIdx.x - band * n_segs;
    const int J0 = band * kEmitRows, k0 = seg * kEmitWords;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t* m = mask + (int64_t)layer * c.mask_wpl;
    const float* sg = FUSED ? nullptr : sigma + (int64_t)layer * c.nx * c.ny;
    const int64_t ebase = layer * D.edge_wpl;
#pragma unroll
    for (int x = threadIdx.x; x < (kEmitRows + 2) * kEmitPitch; x += 32 * kEmitWarps) {
        const int r = x / kEmitPitch, w = 2 * k0 - 1 + (x - r * kEmitPitch), Jr = J0 - 1 + r;
        uint2 v = make_uint2(0u, 0u);
        if (Jr >= 0 && Jr < c.H && w >= 0 && w < D.ewr) {
            const int64_t at = ebase + (int64_t)Jr * D.ewr + w;
            v = make_uint2(D.ew[at], D.prefix[at]);
        }
        s_e[x] = v;
    }
#pragma unroll
    for (int r = warp; r < kEmitRows; r += kEmitWarps)
        s_in[r * kEmitWords + lane] = J0 + r < c.H && k0 + lane < c.mwr
                                          ? m[(int64_t)(J0 + r) * c.mwr + k0 + lane]
                                          : 0u;
    __syncthreads();

    // Sigma at padded sample (I, J) (0 outside the grid, like the ring)
    auto value = [&](int I, int J) -> float {
        return (uint32_t)(I - 1) < (uint32_t)c.nx && (uint32_t)(J - 1) < (uint32_t)c.ny
                   ? __ldg(sg + (int64_t)(J - 1) * c.nx + (I - 1))
                   : 0.0f;
    };
    // saddle cell (I, J): its inside corners are joined
    auto joined = [&](int I, int J) -> bool {
        if (FUSED) {
            const uint32_t sw =
                F.saddle[(int64_t)layer * c.mask_wpl + (int64_t)J * c.mwr + (I >> 5)];
            return (sw >> (I & 31)) & 1u;
        }
        const float w0 = value(I, J), w1 = value(I + 1, J);
        const float w2 = value(I + 1, J + 1), w3 = value(I, J + 1);
        return 0.25f * (w0 + w1 + w2 + w3) >= c.C;
    };

    uint16_t* list = s_list + warp * kEmitList;
    for (int wr = warp; wr < kEmitRows; wr += kEmitWarps) {
        const int J = J0 + wr;
        const uint2* er = s_e + (wr + 1) * kEmitPitch + 1;   // row J from word 2 k0
        const uint2 ea = er[2 * lane], eb = er[2 * lane + 1];
        // the row's crossings in this segment: ids first .. first + n - 1 (words past
        // the end of the row hold no crossings)
        const uint32_t first = er[0].y;
        const int n = (int)__reduce_add_sync(0xffffffffu, __popc(ea.x) + __popc(eb.x));
        // Sigma of row J where it is inside the grid, and of the row after it
        const bool row0 = (uint32_t)(J - 1) < (uint32_t)c.ny, row1 = (uint32_t)J < (uint32_t)c.ny;
        const float* srow = FUSED ? nullptr : sg + ((int64_t)(J - 1) * c.nx + 32 * k0 - 1);
        const int eid0 = (int)(2 * ((int64_t)J * c.W + 32 * k0));
        for (int base = 0; base < n; base += kEmitList) {
            __syncwarp();
#pragma unroll
            for (int half = 0; half < 2; ++half) {
                uint32_t bitsw = half ? eb.x : ea.x;
                int at = (int)((half ? eb.y : ea.y) - first) - base;
                const int code = (2 * lane + half) << 5;
                for (; bitsw; bitsw &= bitsw - 1u, ++at)
                    if ((uint32_t)at < (uint32_t)kEmitList)
                        list[at] = (uint16_t)(code | (__ffs(bitsw) - 1));
            }
            __syncwarp();
            const int room = min(kEmitList, n - base);
            for (int t = lane; t < room; t += 32) {
                const int e = list[t], dir = e & 1, il = e >> 1, I = 32 * k0 + il;
                const uint32_t id = first + (uint32_t)(base + t);
                const bool in0 = (s_in[wr * kEmitWords + (il >> 5)] >> (il & 31)) & 1u;
                // The contour enters cell (I, J) where inside lies on its left, else the
                // cell on the other side of the edge, through side `own` (0 bottom, 1
                // right, 2 top, 3 left). Its successor is the other crossing side; in a
                // saddle cell the side after `own` if joined, else the one before.
                const bool here = in0 != (dir != 0);
                const int cl = il - (here ? 0 : dir), down = here ? 0 : 1 - dir;
                const int own = here ? 3 * dir : 2 - dir;
                const uint2* cw = er - down * kEmitPitch + (cl >> 4);
                const uint2 lo = cw[0], up = cw[kEmitPitch];
                const uint2 ri = er[((cl + 1) >> 4) - down * kEmitPitch];
                const int sh = 2 * cl & 31, sr = (2 * cl + 2 & 31) + 1;
                const uint32_t hv = lo.x >> sh;
                const uint32_t others = ((hv & 1u) | (((ri.x >> sr) & 1u) << 1) |
                                         (((up.x >> sh) & 1u) << 2) | ((hv & 2u) << 2)) &
                                        ~(1u << own);
                int side = 31 - __clz(others);
                if (others & (others - 1u))
                    side = (own + (joined(32 * k0 + cl, J - down) ? 1 : 3)) & 3;
                const uint2 sw = side == 2 ? up : (side == 1 ? ri : lo);
                const int sbit = side == 1 ? sr : sh + (side == 3);
                const uint32_t succ = sw.y + __popc(sw.x & ((1u << sbit) - 1u));
                // Ids order edges by row and, in a row, by column, so a local minimum is
                // an edge (I, J) -> (I, J+1) (of the cell below an edge (I, J) -> (I+1, J)
                // every other side comes first) that is joined to the top side of the
                // cell on its left and not to the bottom side of the one on its right.
                const uint2* lw = er + ((il - 1) >> 4);
                const int sl = 2 * il - 2 & 31;
                bool lowest = dir && ((lw[kEmitPitch].x >> sl) & 1u);
                if (lowest) {
                    if (((lw[0].x >> sl) & 3u) == 3u) lowest = joined(I - 1, J) != here;
                    if ((er[il >> 4].x >> (2 * il & 31)) & 1u) {   // bottom, or a saddle
                        const uint32_t rv = er[(il + 1) >> 4].x >> ((2 * il + 2 & 31) + 1);
                        const uint32_t rt = er[kEmitPitch + (il >> 4)].x >> (2 * il & 31);
                        lowest = lowest && (rv & rt & 1u) && joined(I, J) != here;
                    }
                }
                if (max(id, succ) >= n_cap) {
                    atomicOr(flag, 1u);
                    continue;
                }
                float2 xy;
                if (FUSED) {
                    xy = fused_vertex(F, D, layer, I, J, dir);
                } else {
                    const bool in_x = (uint32_t)(I - 1) < (uint32_t)c.nx;
                    const bool nx_x = dir ? in_x : (uint32_t)I < (uint32_t)c.nx;
                    const float v0 = in_x && row0 ? __ldg(srow + il) : 0.0f;
                    const float v1 = nx_x && (dir ? row1 : row0)
                                         ? __ldg(srow + (il + (dir ? c.nx : 1)))
                                         : 0.0f;
                    const float sa = in0 ? v0 : v1, sb = in0 ? v1 : v0;
                    const float tt = __fdividef(sa - c.C, sa - sb);   // in [0, 1]; sa > C > sb
                    const float p0 = (float)(dir ? J : I);
                    const float p = in0 ? (p0 - 0.5f + tt) : (p0 + 0.5f - tt);
                    xy = dir ? make_float2(c.fx0 + ((float)I - 0.5f) * c.fpx, c.fy0 + p * c.fpx)
                             : make_float2(c.fx0 + p * c.fpx, c.fy0 + ((float)J - 0.5f) * c.fpx);
                }
                oxy[id] = xy;
                if (oeid) oeid[id] = eid0 + e;
                const bool sampled = ((id * 2654435761u) >> (32 - bits)) == 0u;
                nxt[id] = succ | (lowest || sampled ? 0x80000000u : 0u);
            }
        }
    }
}

// Each splitter walks its segment up to the next splitter (nxt: successor |
// splitter bit, one 4-byte load per step), a thread per splitter: several walks in
// lockstep per thread were no faster, the walks of the other warps hide the loads.
__global__ void k_segments(const uint32_t* __restrict__ nxt,
                           const uint32_t* __restrict__ spos, const uint32_t* __restrict__ split_id,
                           int64_t ns, int64_t n, uint32_t* __restrict__ seg_next,
                           uint32_t* __restrict__ seg_len, uint32_t* status) {
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < ns;
         t += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t s0 = split_id[t];
        // (beyond n: a replay whose sizes changed, flagged: no walk)
        uint32_t j = (int64_t)s0 < n ? nxt[s0] & 0x7fffffffu : 0xffffffffu, sn = 0;
        int64_t len = 1;
        bool bad = true;
        while ((int64_t)j < n && len <= n) {   // else corrupt links
            const uint32_t v = nxt[j];
            if (v >> 31) {   // the next splitter
                sn = spos[j];
                bad = (int64_t)sn >= ns;   // more splitters than planned (flagged)
                break;
            }
            j = v & 0x7fffffffu;
            ++len;
        }
        if (bad) {   // report, never loop forever
            atomicOr(status, ST_CAPACITY);
            sn = (uint32_t)t;
            len = 1;
        }
        seg_next[t] = sn;
        seg_len[t] = (uint32_t)len;
    }
}

// One doubling step of the cycle minimum over the splitter graph:
// (cm, nx) -> (min(cm, cm[nx]), nx[nx]); sets done[it] when it changes cm.
// Once a step changed nothing, the later steps only copy cm forward, so the
// result is always in the buffer of the last step.
__global__ void k_jump_min(const uint32_t* __restrict__ cm, const uint32_t* __restrict__ nx,
                           uint32_t* __restrict__ cm2, uint32_t* __restrict__ nx2, int64_t ns,
                           uint32_t* done, int it) {
    if (it > 0 && done[it - 1] == 0) {   // converged: carry the result forward
        for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < ns;
             t += (int64_t)gridDim.x * blockDim.x)
            cm2[t] = cm[t];
        return;
    }
    bool changed = false;
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < ns;
         t += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t a = cm[t];
        uint32_t nt = nx[t];
        if ((int64_t)nt >= ns) nt = (uint32_t)t;   // only in a flagged replay
        const uint32_t b = cm[nt];
        const uint32_t m = b < a ? b : a;
        changed |= m != a;
        cm2[t] = m;
        nx2[t] = nx[nt];
    }
    if (__syncthreads_or(changed) && threadIdx.x == 0) done[it] = 1u;
}

// One doubling step of weighted list ranking: dist += dist[nx], nx = nx[nx].
__global__ void k_jump_rank(const uint32_t* __restrict__ dist, const uint32_t* __restrict__ nx,
                            uint32_t* __restrict__ dist2, uint32_t* __restrict__ nx2, int64_t ns,
                            uint32_t* done, int it) {
    if (it > 0 && done[it - 1] == 0) {   // every list ended: carry the result forward
        for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < ns;
             t += (int64_t)gridDim.x * blockDim.x)
            dist2[t] = dist[t];
        return;
    }
    bool live = false;
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < ns;
         t += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t nt = nx[t];
        if ((int64_t)nt >= ns) {   // list end (or, in a flagged replay, a bad link)
            dist2[t] = dist[t];
            nx2[t] = nt;
        } else {
            dist2[t] = dist[t] + dist[nt];
            const uint32_t nn = nx[nt];
            nx2[t] = nn;
            live |= (int64_t)nn < ns;
        }
    }
    if (__syncthreads_or(live) && threadIdx.x == 0) done[it] = 1u;
}

// Chunks of at most this many splitters resolve their long cycles before the
// host knows how many there are.
constexpr int64_t kAheadSplitters = (int64_t)1 << 17;

// Splitter cycles of at most short_cycle splitters (all the small loops) are
// resolved by walking them; the rest go to pointer jumping on a compact list.
// 16, or 32 where splitter_bits samples more densely.
int short_cycle_of(int64_t n_cross) { return splitter_bits(n_cross) < 5 ? 32 : 16; }
constexpr uint32_t kNil = 0xffffffffu;

// cm[t] = the cycle's smallest splitter id when t's cycle closes within
// short_cycle steps; otherwise t is appended to the long list. The head of a
// short cycle (the splitter holding its smallest id) then walks it once more:
// rank_start = crossings of the loop before each segment, loop_len at the head.
__global__ void k_short_cycles(const uint32_t* __restrict__ split_id,
                               const uint32_t* __restrict__ seg_next,
                               const uint32_t* __restrict__ seg_len, int64_t ns, int short_cycle,
                               uint32_t* __restrict__ cm, uint32_t* __restrict__ long_list,
                               uint32_t* __restrict__ long_pos, uint32_t* __restrict__ n_long,
                               uint32_t* __restrict__ rank_start,
                               uint32_t* __restrict__ loop_len) {
    const int lane = threadIdx.x & 31;
    for (int64_t base = (int64_t)blockIdx.x * blockDim.x; base < ns;
         base += (int64_t)gridDim.x * blockDim.x) {
        const int64_t t = base + threadIdx.x;
        bool is_long = false;
        if (t < ns) {
            uint32_t v = seg_next[t], mn = split_id[t];
            int n = 1;
            while (v != (uint32_t)t && n < short_cycle) {
                const uint32_t id = split_id[v];
                mn = id < mn ? id : mn;
                v = seg_next[v];
                ++n;
            }
            is_long = v != (uint32_t)t;
            cm[t] = is_long ? kNil : mn;
            long_pos[t] = kNil;
            if (!is_long && mn == split_id[t]) {   // the head: rank the cycle's segments
                uint32_t acc = 0, w = (uint32_t)t;
                int m = 0;
                do {
                    rank_start[w] = acc;
                    acc += seg_len[w];
                    w = seg_next[w];
                } while (w != (uint32_t)t && ++m < short_cycle);
                loop_len[t] = acc;
            }
        }
        const uint32_t ball = __ballot_sync(0xffffffffu, is_long);
        uint32_t pos = 0;
        if (lane == 0 && ball) pos = atomicAdd(n_long, (uint32_t)__popc(ball));
        pos = __shfl_sync(0xffffffffu, pos, 0);
        if (is_long) {
            const uint32_t q = pos + __popc(ball & ((1u << lane) - 1u));
            long_list[q] = (uint32_t)t;
            long_pos[t] = q;
        }
    }
}

// Compact long-cycle graph: node u = long_list[u]; next in compact indices.
__global__ void k_long_setup(const uint32_t* __restrict__ long_list,
                             const uint32_t* __restrict__ long_pos,
                             const uint32_t* __restrict__ split_id,
                             const uint32_t* __restrict__ seg_next, int64_t nl,
                             uint32_t* __restrict__ lcm, uint32_t* __restrict__ lnx) {
    for (int64_t u = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; u < nl;
         u += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t t = long_list[u];
        const uint32_t nt = seg_next[t];   // < ns by construction of k_segments
        lcm[u] = split_id[t];
        lnx[u] = long_pos[nt];
    }
}

// Break each long cycle before its head (nx = NIL there); dist = segment length.
__global__ void k_long_break(const uint32_t* __restrict__ lcm, const uint32_t* __restrict__ long_list,
                             const uint32_t* __restrict__ long_pos,
                             const uint32_t* __restrict__ split_id,
                             const uint32_t* __restrict__ seg_next,
                             const uint32_t* __restrict__ seg_len, int64_t nl,
                             uint32_t* __restrict__ nx, uint32_t* __restrict__ dist) {
    for (int64_t u = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; u < nl;
         u += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t t = long_list[u];
        const uint32_t nt = seg_next[t];
        const uint32_t nu = long_pos[nt];
        nx[u] = ((int64_t)nu >= nl || lcm[nu] == split_id[nt]) ? kNil : nu;
        dist[u] = seg_len[t];
    }
}

// Back to splitter order: cm, rank_start = loop length - dist, loop_len at heads.
__global__ void k_long_ranks(const uint32_t* __restrict__ lcm, const uint32_t* __restrict__ dist,
                             const uint32_t* __restrict__ long_list,
                             const uint32_t* __restrict__ long_pos,
                             const uint32_t* __restrict__ spos, int64_t nl, int64_t ns,
                             uint32_t* __restrict__ cm, uint32_t* __restrict__ rank_start,
                             uint32_t* __restrict__ loop_len) {
    for (int64_t u = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; u < nl;
         u += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t t = long_list[u];
        const uint32_t sp = spos[lcm[u]];
        uint32_t hu = (int64_t)sp < ns ? long_pos[sp] : kNil;
        if ((int64_t)hu >= nl) hu = (uint32_t)u;   // only in a flagged replay
        cm[t] = lcm[u];
        rank_start[t] = dist[hu] - dist[u];
        if (hu == (uint32_t)u) loop_len[t] = dist[u];
    }
}

// The whole resolution of the long cycles by one block, for at most kLongBlock
// of their splitters: the cycle minima by doubling, the break before each head,
// the ranks by doubling, back to splitter order, as the kernels above do it
// over the grid, with the links in shared memory. One launch instead of 2 log2
// + 4 (each step then costs a launch of about 3 us whatever the count: 22 of
// them for the 2,000 long-cycle splitters of a 200^2 x 50 slice). Does nothing
// where there are more.
constexpr int kLongBlock = 12288;
constexpr int kLongThreads = 1024;

__global__ void __launch_bounds__(kLongThreads)
k_long_block(const uint32_t* __restrict__ n_long, const uint32_t* __restrict__ long_list,
             const uint32_t* __restrict__ long_pos, const uint32_t* __restrict__ split_id,
             const uint32_t* __restrict__ seg_next, const uint32_t* __restrict__ seg_len,
             const uint32_t* __restrict__ spos, int64_t ns, int64_t cap,
             uint32_t* __restrict__ cm, uint32_t* __restrict__ rank_start,
             uint32_t* __restrict__ loop_len) {
    extern __shared__ uint32_t s_link[];
    const uint32_t count = *n_long;
    if (count == 0u || count > (uint32_t)kLongBlock) return;
    // (a replay whose sizes changed, flagged, may count more than its list holds)
    const uint32_t nl = (uint32_t)min((int64_t)count, cap);
    uint32_t *a = s_link, *an = a + nl, *b = an + nl, *bn = b + nl;
    for (uint32_t u = threadIdx.x; u < nl; u += kLongThreads) {
        const uint32_t t = long_list[u];
        const uint32_t nu = long_pos[seg_next[t]];
        a[u] = split_id[t];
        an[u] = nu < nl ? nu : u;   // out of range only in a flagged replay
    }
    __syncthreads();
    for (int it = 0; it < 32; ++it) {   // cycle minimum; done when a step changes nothing
        bool changed = false;
        for (uint32_t u = threadIdx.x; u < nl; u += kLongThreads) {
            const uint32_t x = a[u], nt = an[u];
            const uint32_t m = min(x, a[nt]);
            changed |= m != x;
            b[u] = m;
            bn[u] = an[nt];
        }
        const bool more = __syncthreads_or(changed);
        uint32_t* t = a; a = b; b = t;
        t = an; an = bn; bn = t;
        if (!more) break;
    }
    // a: the minima. The cycles broken before their heads: an = next, b = distance
    for (uint32_t u = threadIdx.x; u < nl; u += kLongThreads) {
        const uint32_t t = long_list[u];
        const uint32_t nt = seg_next[t];
        const uint32_t nu = long_pos[nt];
        an[u] = (nu >= nl || a[nu] == split_id[nt]) ? kNil : nu;
        b[u] = seg_len[t];
        cm[t] = a[u];
    }
    __syncthreads();
    uint32_t *d = b, *d2 = a;   // the minima are in cm from here on
    for (int it = 0; it < 32; ++it) {   // distance to the end of the broken cycle
        bool live = false;
        for (uint32_t u = threadIdx.x; u < nl; u += kLongThreads) {
            const uint32_t nt = an[u];
            if (nt >= nl) {
                d2[u] = d[u];
                bn[u] = nt;
            } else {
                d2[u] = d[u] + d[nt];
                bn[u] = an[nt];
                live |= an[nt] < nl;
            }
        }
        const bool more = __syncthreads_or(live);
        uint32_t* t = d; d = d2; d2 = t;
        t = an; an = bn; bn = t;
        if (!more) break;
    }
    for (uint32_t u = threadIdx.x; u < nl; u += kLongThreads) {
        const uint32_t t = long_list[u];
        const uint32_t sp = spos[cm[t]];
        uint32_t hu = (int64_t)sp < ns ? long_pos[sp] : kNil;
        if (hu >= nl) hu = u;   // only in a flagged replay
        rank_start[t] = d[hu] - d[u];
        if (hu == u) loop_len[t] = d[u];
    }
}

// packed[t] = (1 << 32) | loop length for heads, else 0 (splitter order).
__global__ void k_head_flags(const uint32_t* __restrict__ cm, const uint32_t* __restrict__ split_id,
                             const uint32_t* __restrict__ loop_len, int64_t ns,
                             int64_t* __restrict__ packed) {
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < ns;
         t += (int64_t)gridDim.x * blockDim.x)
        packed[t] = cm[t] == split_id[t] ? (((int64_t)1 << 32) | loop_len[t]) : 0;
}

// Replay checks: a device count against the planned one, and the status word.
__global__ void k_check_u32(const uint32_t* __restrict__ v, uint32_t expect, uint32_t* flag) {
    if (threadIdx.x == 0 && blockIdx.x == 0 && *v != expect) atomicOr(flag, 1u);
}
__global__ void k_check_packed(const int64_t* __restrict__ total, int64_t n_loops, int64_t n_cross,
                               const uint32_t* __restrict__ status, uint32_t* flag) {
    if (threadIdx.x != 0 || blockIdx.x != 0) return;
    if ((*total >> 32) != n_loops || (*total & 0xffffffffLL) != n_cross) atomicOr(flag, 1u);
    if (*status) atomicOr(flag, 2u);
}

// Each splitter writes its segment at its loop's offset + rank_start. Lanes walk
// up to kWriteSteps steps of their segments (the 4-byte successors only) and list
// the crossings with their places in shared memory; the warp then moves the
// listed vertices, all lanes busy and their loads independent of the walk and of
// one another. 389 million vertices: 2.65 ms (8 steps 3.0, 16 steps 3.8, 2 steps
// 3.2; 3.95 with each lane moving its own 16-byte records, a chain of loads).
constexpr int kWriteSteps = 4;
__global__ void __launch_bounds__(256)
k_write_segments(const uint32_t* __restrict__ nxt, const float2* __restrict__ xy,
                 const int32_t* __restrict__ eid, const uint32_t* __restrict__ cm,
                 const uint32_t* __restrict__ spos, const uint32_t* __restrict__ split_id,
                 const uint32_t* __restrict__ seg_len, const uint32_t* __restrict__ rank_start,
                 const int64_t* __restrict__ scan, int64_t ns, int64_t n, int64_t n_loops,
                 int64_t vofs, int64_t* __restrict__ loop_off, float2* __restrict__ oxy,
                 int32_t* __restrict__ oeid) {
    __shared__ uint2 s_move[256 * kWriteSteps];   // {crossing, place}
    uint2* move = s_move + (threadIdx.x & ~31u) * kWriteSteps;
    const int lane = threadIdx.x & 31;
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    uint32_t j = 0, place = 0, left = 0;
    if (t < ns) {
        const uint32_t ht = cm[t];
        const uint32_t h = (int64_t)ht < n ? spos[ht] : 0xffffffffu;   // the loop's head splitter
        if ((int64_t)h < ns) {                       // else the links were inconsistent
            const int64_t sc = scan[h], voff = sc & 0xffffffffLL;
            if (h == (uint32_t)t && (sc >> 32) < n_loops) loop_off[sc >> 32] = vofs + voff;
            const int64_t b = voff + (int64_t)rank_start[t];
            const int64_t l = seg_len[t];
            if (b >= 0 && b + l <= n) {              // else the links were inconsistent
                place = (uint32_t)b;
                left = (uint32_t)l;
                j = split_id[t];
            }
        }
    }
    while (__any_sync(0xffffffffu, left > 0)) {
        const uint32_t steps = min(left, (uint32_t)kWriteSteps);
        uint32_t at = steps;                         // inclusive prefix sum over the lanes
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const uint32_t v = __shfl_up_sync(0xffffffffu, at, d);
            if (lane >= d) at += v;
        }
        const uint32_t total = __shfl_sync(0xffffffffu, at, 31);
        at -= steps;
        for (uint32_t r = 0; r < steps; ++r) {
            move[at + r] = make_uint2(j, place + r);
            j = (int64_t)j < n ? nxt[j] & 0x7fffffffu : j;
        }
        left -= steps;
        place += steps;
        __syncwarp();
        for (uint32_t q = lane; q < total; q += 32) {
            const uint2 m = move[q];
            if ((int64_t)m.x < n) {
                oxy[m.y] = xy[m.x];
                if (oeid) oeid[m.y] = eid[m.x];
            }
        }
        __syncwarp();
    }
}

// layer_loops[l] = loops whose head lies before the first crossing of layer l
// (+ lofs); the chunk's closing vertex offset (+ vofs)
__global__ void k_layer_loops(const uint32_t* __restrict__ prefix, int64_t edge_wpl, int n_layers,
                              const uint32_t* __restrict__ spos, const int64_t* __restrict__ scan,
                              int64_t n_cross, int64_t ns, int64_t n_loops, int64_t lofs,
                              int64_t vofs, int64_t* __restrict__ layer_loops,
                              int64_t* __restrict__ loop_off) {
    int l = blockIdx.x * blockDim.x + threadIdx.x;
    if (l > n_layers) return;
    const int64_t first = l < n_layers ? (int64_t)prefix[(int64_t)l * edge_wpl] : n_cross;
    const int64_t sp = first < n_cross ? (int64_t)spos[first] : ns;
    layer_loops[l] = lofs + (sp < ns ? (scan[sp] >> 32) : n_loops);
    if (l == 0) loop_off[n_loops] = vofs + n_cross;
}

__global__ void k_fill_i64(int64_t* __restrict__ a, int64_t n, int64_t v) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x)
        a[i] = v;
}

}  // namespace

void contours_chunk(const ChunkGeom& g, double C, const float* sigma, const uint32_t* mask,
                    bool want_eid, ChunkContours& out, cudaStream_t s, const Replay* rp,
                    const FusedVerts* fv, const ChunkDest* dest) {
    const bool replay = rp && rp->replay;
    MsConst c;
    c.nx = g.nx;
    c.ny = g.ny;
    c.W = g.nx + 2;
    c.H = g.ny + 2;
    c.mwr = (int32_t)mask_words_per_row(g.nx);
    c.ewr = 2 * c.mwr;
    c.mask_wpl = mask_words_per_layer(g.nx, g.ny);
    c.edge_wpl = 2 * c.mask_wpl;
    c.n_layers = g.n_layers;
    c.C = (float)C;
    c.fx0 = (float)g.x0;
    c.fy0 = (float)g.y0;
    c.fpx = (float)g.px;
    const int64_t n_words = c.edge_wpl * g.n_layers;
    // 32-bit crossing ids: fewer than 2^27 edge words keeps every count below 2^32
    if (n_words >= ((int64_t)1 << 27)) fail(CSL_ERR_CAPACITY, "marching squares: chunk too large");

    // small: [0] status, [1] crossings, [2] splitters, [3..66] done, [67] long
    // count, [68, 69] loops << 32 | crossings they cover
    DevBuf small(4 * 80, s);
    CSL_CUDA(cudaMemsetAsync(small.get(), 0, 4 * 80, s));
    uint32_t* status = small.as<uint32_t>();
    uint32_t* done = small.as<uint32_t>() + 3;
    uint32_t* n_long = small.as<uint32_t>() + 67;
    int64_t* tot = reinterpret_cast<int64_t*>(small.as<uint32_t>() + 68);
    uint32_t* flag = rp ? rp->flag : status;   // where replay mismatches go

    DevBuf ew((size_t)n_words * 4, s), prefix((size_t)n_words * 4, s);
    {
        const int64_t n_thr = (int64_t)c.H * c.mwr;
        dim3 grid((unsigned)ceil_div(n_thr, 256), (unsigned)g.n_layers);
        k_edge_words<<<grid, 256, 0, s>>>(mask, c, ew.as<uint32_t>(), prefix.as<uint32_t>());
        CSL_LAUNCH_CHECK("ms edge words");
    }
    exclusive_scan_u32(prefix.as<uint32_t>(), prefix.as<uint32_t>(), n_words, status + 1, s);
    int64_t n_cross;
    if (replay) {
        n_cross = rp->plan->n_cross;
        k_check_u32<<<1, 32, 0, s>>>(status + 1, (uint32_t)n_cross, flag);
        CSL_LAUNCH_CHECK("check crossings");
    } else {
        uint32_t v = 0;
        read_to_host(&v, status + 1, 4, s);
        n_cross = v;
        if (rp) rp->plan->n_cross = n_cross;
    }
    out.n_verts = n_cross;
    out.layer_loops.ensure((size_t)(g.n_layers + 1) * 8, s);
    if (n_cross == 0) {
        out.n_loops = 0;
        if (dest) {   // no loops: every layer starts at the running loop count
            dest->make_room(dest->v_base, dest->l_base + 1);
            k_fill_i64<<<1, 128, 0, s>>>(out.layer_loops.as<int64_t>(), g.n_layers + 1,
                                         dest->l_base);
            CSL_LAUNCH_CHECK("ms empty layers");
            k_fill_i64<<<1, 32, 0, s>>>(dest->loop_off + dest->l_base, 1, dest->v_base);
            CSL_LAUNCH_CHECK("ms empty chunk");
        } else {
            CSL_CUDA(cudaMemsetAsync(out.layer_loops.get(), 0, (size_t)(g.n_layers + 1) * 8, s));
            out.loop_off.ensure(8, s);
            CSL_CUDA(cudaMemsetAsync(out.loop_off.get(), 0, 8, s));
        }
        if (rp && !replay) rp->plan->ns = rp->plan->nl = rp->plan->n_loops = 0;
        return;
    }
    // the splitter bit in k_emit's successors needs ids below 2^31
    if (n_cross >= ((int64_t)1 << 31)) fail(CSL_ERR_CAPACITY, "marching squares: too many crossings");
    DevBuf vxy((size_t)n_cross * 8, s), veid(want_eid ? (size_t)n_cross * 4 : 4, s);
    int32_t* ve = want_eid ? veid.as<int32_t>() : nullptr;
    // The lane of k_emit that takes a crossing writes its vertex and successor.
    // A replay (planned sizes) may leave some unwritten when its sizes changed:
    // there successors start as 0 (no splitter).
    DevBuf spos((size_t)n_cross * 4, s), nxt((size_t)n_cross * 4, s);
    if (rp) CSL_CUDA(cudaMemsetAsync(nxt.get(), 0, (size_t)n_cross * 4, s));

    Dense D{ew.as<uint32_t>(), prefix.as<uint32_t>(), c.edge_wpl, c.ewr};
    {
        const int64_t n_bands = ceil_div((int64_t)c.ny + 1, kEmitRows);
        const int64_t n_segs = ceil_div((int64_t)c.mwr, kEmitWords);
        dim3 grid((unsigned)(n_bands * n_segs), (unsigned)g.n_layers);
        const int bits = splitter_bits(n_cross);
        FusedIn F{};
        if (fv) {
            F.tbase = fv->tbase.as<uint32_t>();
            F.roff = fv->roff.as<uint16_t>();
            F.verts = fv->verts.as<float2>();
            F.saddle = fv->saddle.as<uint32_t>();
            F.T = g.T;
            F.ntx = g.ntx;
            F.n_tiles = g.ntx * g.nty;
            k_emit<true><<<grid, 32 * kEmitWarps, 0, s>>>(sigma, mask, c, D, F, bits,
                                                         vxy.as<float2>(), ve, nxt.as<uint32_t>(),
                                                         (uint32_t)n_cross, flag);
        } else {
            k_emit<false><<<grid, 32 * kEmitWarps, 0, s>>>(sigma, mask, c, D, F, bits,
                                                          vxy.as<float2>(), ve, nxt.as<uint32_t>(),
                                                          (uint32_t)n_cross, flag);
        }
        CSL_LAUNCH_CHECK("ms emit");
    }
    // ---- loops: splitters, segments, pointer jumping on the splitter graph
    // one scan over nxt's top bits numbers the splitters (spos, for every
    // crossing) and lists them (split_id) in the same pass
    // the list's room: every crossing, or a replay's planned count
    const int64_t ns_cap = replay ? rp->plan->ns : n_cross;
    DevBuf split_id((size_t)std::max<int64_t>(ns_cap, 1) * 4, s);
    // a replay whose sizes changed leaves entries unwritten: make them valid ids
    if (replay) CSL_CUDA(cudaMemsetAsync(split_id.get(), 0, (size_t)ns_cap * 4, s));
    scan_flags_list(nxt.as<uint32_t>(), n_cross, spos.as<uint32_t>(), split_id.as<uint32_t>(),
                    ns_cap, status + 2, status, s);
    int64_t ns;
    if (replay) {
        ns = rp->plan->ns;
        k_check_u32<<<1, 32, 0, s>>>(status + 2, (uint32_t)ns, flag);
        CSL_LAUNCH_CHECK("check splitters");
    } else {
        uint32_t head2[3];
        read_to_host(head2, small.get(), 12, s);
        if (head2[0]) fail(CSL_ERR_CUDA, "marching squares: a crossing has no successor");
        ns = head2[2];
        if (rp) rp->plan->ns = ns;
    }
    DevBuf seg_next((size_t)ns * 4, s), seg_len((size_t)ns * 4, s);
    const unsigned gs = grid_for(ns, 256);
    k_segments<<<gs, 256, 0, s>>>(nxt.as<uint32_t>(), spos.as<uint32_t>(),
                                  split_id.as<uint32_t>(), ns, n_cross, seg_next.as<uint32_t>(),
                                  seg_len.as<uint32_t>(), status);
    CSL_LAUNCH_CHECK("ms segments");
    // short splitter cycles by walking them; long ones by pointer jumping
    DevBuf cm((size_t)ns * 4, s), long_list((size_t)ns * 4, s), long_pos((size_t)ns * 4, s);
    DevBuf rank_start((size_t)ns * 4, s), loop_len((size_t)ns * 4, s);
    if (replay) CSL_CUDA(cudaMemsetAsync(long_list.get(), 0, (size_t)ns * 4, s));
    k_short_cycles<<<gs, 256, 0, s>>>(split_id.as<uint32_t>(), seg_next.as<uint32_t>(),
                                      seg_len.as<uint32_t>(), ns, short_cycle_of(n_cross),
                                      cm.as<uint32_t>(), long_list.as<uint32_t>(), long_pos.as<uint32_t>(), n_long,
                                      rank_start.as<uint32_t>(), loop_len.as<uint32_t>());
    CSL_LAUNCH_CHECK("ms short cycles");
    // Long cycles: by one block where they fit. A small chunk does not read
    // their count first (a read-back takes as long as the block): it is read
    // with the loop count below, and only if the block could not take them do
    // the grid's kernels run, and the numbering of the loops again.
    const bool ahead = !replay && ns <= kAheadSplitters;
    auto long_block = [&] {
        const int smem = 4 * 4 * (int)std::min<int64_t>(ns, kLongBlock);
        CSL_CUDA(cudaFuncSetAttribute(k_long_block, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      4 * 4 * kLongBlock));
        k_long_block<<<1, kLongThreads, smem, s>>>(
            n_long, long_list.as<uint32_t>(), long_pos.as<uint32_t>(), split_id.as<uint32_t>(),
            seg_next.as<uint32_t>(), seg_len.as<uint32_t>(), spos.as<uint32_t>(), ns, ns,
            cm.as<uint32_t>(), rank_start.as<uint32_t>(), loop_len.as<uint32_t>());
        CSL_LAUNCH_CHECK("ms long cycles");
    };
    int64_t nl = 0;
    if (replay) {
        nl = rp->plan->nl;
        k_check_u32<<<1, 32, 0, s>>>(n_long, (uint32_t)nl, flag);
        CSL_LAUNCH_CHECK("check long cycles");
    } else if (!ahead) {
        uint32_t v = 0;
        read_to_host(&v, n_long, 4, s);
        nl = v;
        if (rp) rp->plan->nl = nl;
    }
    if (ahead || (nl > 0 && nl <= kLongBlock)) long_block();
    auto long_grid = [&] {
        // cycle minimum by doubling (later steps copy the converged result forward)
        int max_it = 1;
        while (((int64_t)1 << max_it) < nl + 1) ++max_it;
        max_it += 1;
        if (max_it > 60) fail(CSL_ERR_CAPACITY, "marching squares: too many splitters");
        DevBuf cmA((size_t)nl * 4, s), cmB((size_t)nl * 4, s), nxA((size_t)nl * 4, s),
            nxB((size_t)nl * 4, s);
        const unsigned gl = grid_for(nl, 256);
        k_long_setup<<<gl, 256, 0, s>>>(long_list.as<uint32_t>(), long_pos.as<uint32_t>(),
                                        split_id.as<uint32_t>(), seg_next.as<uint32_t>(), nl,
                                        cmA.as<uint32_t>(), nxA.as<uint32_t>());
        CSL_LAUNCH_CHECK("ms long setup");
        uint32_t *a_cm = cmA.as<uint32_t>(), *a_nx = nxA.as<uint32_t>();
        uint32_t *b_cm = cmB.as<uint32_t>(), *b_nx = nxB.as<uint32_t>();
        for (int it = 0; it < max_it; ++it) {
            k_jump_min<<<gl, 256, 0, s>>>(a_cm, a_nx, b_cm, b_nx, nl, done, it);
            CSL_LAUNCH_CHECK("ms cycle minimum");
            std::swap(a_cm, b_cm);
            std::swap(a_nx, b_nx);
        }
        uint32_t* lcm = a_cm;   // the buffer the last step wrote
        DevBuf dA((size_t)nl * 4, s), dB((size_t)nl * 4, s), nxr_buf((size_t)nl * 4, s);
        uint32_t *nxr = nxr_buf.as<uint32_t>(), *nxr2 = (lcm == cmA.as<uint32_t>())
                                                            ? cmB.as<uint32_t>()
                                                            : cmA.as<uint32_t>();
        k_long_break<<<gl, 256, 0, s>>>(lcm, long_list.as<uint32_t>(), long_pos.as<uint32_t>(),
                                        split_id.as<uint32_t>(), seg_next.as<uint32_t>(),
                                        seg_len.as<uint32_t>(), nl, nxr, dA.as<uint32_t>());
        CSL_LAUNCH_CHECK("ms break cycles");
        CSL_CUDA(cudaMemsetAsync(done, 0, 4 * 64, s));
        uint32_t *dist = dA.as<uint32_t>(), *dist2 = dB.as<uint32_t>();
        for (int it = 0; it < max_it; ++it) {
            k_jump_rank<<<gl, 256, 0, s>>>(dist, nxr, dist2, nxr2, nl, done, it);
            CSL_LAUNCH_CHECK("ms list ranking");
            std::swap(dist, dist2);
            std::swap(nxr, nxr2);
        }
        k_long_ranks<<<gl, 256, 0, s>>>(lcm, dist, long_list.as<uint32_t>(),
                                        long_pos.as<uint32_t>(), spos.as<uint32_t>(), nl, ns,
                                        cm.as<uint32_t>(), rank_start.as<uint32_t>(),
                                        loop_len.as<uint32_t>());
        CSL_LAUNCH_CHECK("ms long ranks");
    };
    if (nl > kLongBlock) long_grid();
    DevBuf packed((size_t)ns * 8, s), scan((size_t)ns * 8, s);
    auto number_loops = [&] {
        k_head_flags<<<gs, 256, 0, s>>>(cm.as<uint32_t>(), split_id.as<uint32_t>(),
                                        loop_len.as<uint32_t>(), ns, packed.as<int64_t>());
        CSL_LAUNCH_CHECK("ms heads");
        exclusive_scan_i64(packed.as<int64_t>(), scan.as<int64_t>(), ns, tot, s);
    };
    number_loops();
    int64_t n_loops;
    if (replay) {
        n_loops = rp->plan->n_loops;
        k_check_packed<<<1, 32, 0, s>>>(tot, n_loops, n_cross, status, flag);
        CSL_LAUNCH_CHECK("check loops");
    } else {
        uint32_t h[70];
        read_to_host(h, small.get(), sizeof h, s);
        if (ahead) {
            nl = h[67];
            if (rp) rp->plan->nl = nl;
            if (nl > kLongBlock) {
                long_grid();
                number_loops();
                read_to_host(h, small.get(), sizeof h, s);
            }
        }
        if (h[0]) fail(CSL_ERR_CUDA, "marching squares: inconsistent successor links");
        const int64_t packed_total = (int64_t)(((uint64_t)h[69] << 32) | h[68]);
        n_loops = packed_total >> 32;
        if ((packed_total & 0xffffffffLL) != n_cross)
            fail(CSL_ERR_CUDA, "marching squares: loops do not cover every crossing");
        if (rp) rp->plan->n_loops = n_loops;
    }
    out.n_loops = n_loops;
    // where the vertices and loop offsets go: the chunk's own arrays, or the
    // caller's growing result at its running bases
    int64_t* o_loop;
    float2* o_xy;
    int32_t* o_eid;
    int64_t vofs = 0, lofs = 0;
    if (dest) {
        dest->make_room(dest->v_base + n_cross, dest->l_base + n_loops + 1);
        vofs = dest->v_base;
        lofs = dest->l_base;
        o_loop = dest->loop_off + lofs;
        o_xy = dest->xy + vofs;
        o_eid = want_eid ? dest->eid + vofs : nullptr;
    } else {
        out.loop_off.ensure((size_t)(n_loops + 1) * 8, s);
        out.xy.ensure((size_t)n_cross * 8, s);
        if (want_eid) out.eid.ensure((size_t)n_cross * 4, s);
        o_loop = out.loop_off.as<int64_t>();
        o_xy = out.xy.as<float2>();
        o_eid = want_eid ? out.eid.as<int32_t>() : nullptr;
    }
    // one thread per splitter, not a grid-stride loop over a capped grid: a
    // CTA retires as soon as its 256 walks are done (walk lengths vary), and
    // the walks in flight are those of consecutive splitters (100M workload:
    // contour stage 141 -> 132 ms against 64 CTAs per SM)
    const unsigned gw = (unsigned)std::max<int64_t>(ceil_div(ns, (int64_t)256), (int64_t)1);
    k_write_segments<<<gw, 256, 0, s>>>(nxt.as<uint32_t>(), vxy.as<float2>(), ve,
                                        cm.as<uint32_t>(), spos.as<uint32_t>(),
                                        split_id.as<uint32_t>(), seg_len.as<uint32_t>(),
                                        rank_start.as<uint32_t>(), scan.as<int64_t>(), ns, n_cross,
                                        n_loops, vofs, o_loop, o_xy, o_eid);
    CSL_LAUNCH_CHECK("ms write");
    k_layer_loops<<<(unsigned)ceil_div(g.n_layers + 1, 128), 128, 0, s>>>(
        prefix.as<uint32_t>(), c.edge_wpl, g.n_layers, spos.as<uint32_t>(), scan.as<int64_t>(),
        n_cross, ns, n_loops, lofs, vofs, out.layer_loops.as<int64_t>(), o_loop);
    CSL_LAUNCH_CHECK("ms layer loops");
}

}  // namespace csl
