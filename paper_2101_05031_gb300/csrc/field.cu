// Field kernel: Sigma(p) = sum_j w_j I_j(p) (Eq. 6) on every pixel of a slab
// of S layers, one CTA per (slab, 16x16-pixel tile).
//
// I_j(p) is the integral of the quartic kernel (Eq. 5) along edge j by arc
// length (Eq. 7 with its Jacobian). In the frame of the edge, with
// p - v_s = t0 u + e (e orthogonal to u) and w^2 = R^2 - |e|^2, the kernel is
// (w^2 - tau^2)^2 / R^4 at tau = t - t0, and the edge covers
// tau in [tau1, tau2] = [max(-t0, -w), min(L - t0, w)]. The integrand is a
// polynomial of degree 4 in tau, so 3-point Gauss-Legendre on [tau1, tau2] is
// exact (it integrates degree <= 5 exactly); its terms are all >= 0, so FP32
// keeps a few-ulp relative error instead of the cancellation of the printed
// difference of quintics. With m = (tau1 + tau2)/2, h = (tau2 - tau1)/2,
// c = w^2 - m^2, A = c - 0.6 h^2 and B = 2 m h sqrt(0.6):
//   I R^4 = h [ (10/9)(A^2 + B^2) + (8/9) c^2 ].
//
// Coordinates are taken relative to the tile's corner (a double split into
// two floats), so no absolute pixel position ever rounds at the magnitude of
// the part (an ulp at 200 mm is 1.5e-5 mm, far above the 1e-5 relative field
// tolerance at strut surfaces).
//
// Work per CTA: the tile's edge list, which the binner stores contiguously (the
// records themselves, in list order), is staged into shared memory in chunks of
// 256 records by one bulk copy (TMA, cp.async.bulk) completed on an mbarrier;
// each thread converts its record to tile-local coordinates, then computes for
// every (record, layer) item whether the edge's support can reach each warp's block
// of 8x4 or 8x8 pixels (xy box of the edge clipped to |z - z_layer| <= R, grown by
// R, and the block centre's distance to the line). Warps then walk only the
// records whose bit is set (ballot + ffs); the per-pixel evaluation is
// branch-free.
#include <math.h>

#include <algorithm>
#include <vector>

#include "field_tile.cuh"
#include "slice.cuh"

namespace csl {
namespace {

struct FieldConst {
    int32_t nx, ny, ntx, n_tiles;
    int32_t n_layers;      // layers in this chunk
    float R2, fpx, fdz;
    TileCull tc;
    float C;            // iso-value (inside mask)
    const float2* org_x;   // per tile column: x of its first pixel edge, (hi, lo)
    const float2* org_y;   // per tile row
    const float2* org_z;   // per slab: z of its first layer
    int32_t mwr;        // mask words per row
    int64_t mask_wpl;   // mask words per layer
    uint32_t* err;      // device status word: ST_TIMEOUT when a wait gave up
};

// One (tile, slab) of the field: called by the grid kernel (one CTA per
// (tile, slab)) and by the persistent batch kernel (one item at a time).
//
// The tile's records are contiguous (the binner copies them in list order), so
// each chunk of up to 256 records is staged by one bulk copy (TMA) issued by
// thread 0 and completed on an mbarrier; every thread then converts its record
// to tile-local coordinates in place. bar: the CTA's mbarrier (initialised
// with one arrival), phase: its parity, kept by the caller across tiles.
// Returns false (after setting ST_TIMEOUT in *c.err) when a copy never
// completed; the caller must then stop using the barrier.
//
// PX: pixel rows per thread (1, or 2: a warp then owns 8 x 8 pixels and the CTA
// has 4 warps; rows j and j + 4 of a thread share x, so dx and dz, the walk
// over the records and the layer tests).
template <int S, int PX, bool COUNT>
__device__ __forceinline__ bool field_tile(const csl_rec* __restrict__ recs,
                                           const uint32_t* __restrict__ tstart,
                                           const uint32_t* __restrict__ tend, const FieldConst& c,
                                           float* __restrict__ sigma, uint32_t* __restrict__ mask,
                                           unsigned long long* __restrict__ n_pairs, int tile,
                                           int slab, uint64_t* bar, uint32_t& phase) {
    __shared__ __align__(16) float4 s_rec[kFieldThreads][2];   // raw, then tile-local
    __shared__ uint64_t s_mask[kFieldThreads];   // byte l: warps reached at layer l

    const int tx = tile % c.ntx, ty = tile / c.ntx;
    const uint32_t key = (uint32_t)slab * (uint32_t)c.n_tiles + (uint32_t)tile;
    const uint32_t beg = tstart[key], end = tend[key];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int wx = warp & 1, wy = warp >> 1;
    constexpr int kThreads = kFieldThreads / PX;
    const int il = wx * 8 + (lane & 7), jl = wy * 4 * PX + (lane >> 3);
    const int l0 = slab * S;
    const int nl = min(S, c.n_layers - l0);

    float acc[S][PX];
#pragma unroll
    for (int l = 0; l < S; ++l)
#pragma unroll
        for (int k = 0; k < PX; ++k) acc[l][k] = 0.0f;
    uint32_t n_nonzero = 0, n_eval = 0;

    if (end > beg) {
        // the tile's corner and the slab's first plane, each a (hi, lo) float pair
        const float2 ox = c.org_x[tx], oy = c.org_y[ty], oz = c.org_z[slab];
        const float oxh = ox.x, oxl = ox.y, oyh = oy.x, oyl = oy.y, ozh = oz.x, ozl = oz.y;
        const float pxl = ((float)il + 0.5f) * c.fpx;
        float pyl[PX];
#pragma unroll
        for (int k = 0; k < PX; ++k) pyl[k] = ((float)(jl + 4 * k) + 0.5f) * c.fpx;
        const TileCull cull = c.tc;

        for (uint32_t c0 = beg; c0 < end; c0 += kFieldThreads) {
            const int cnt = (int)min((uint32_t)kFieldThreads, end - c0);
            if (threadIdx.x == 0) {
                fence_proxy_async_smem();   // the block's earlier reads of s_rec come first
                bulk_load(s_rec, recs + c0, (uint32_t)cnt * (uint32_t)sizeof(csl_rec), bar);
            }
            // a copy that never completes: report it, wait once more (bounded)
            // for the copy still in flight, and give the tile up
            if (__syncthreads_or(!mbar_wait(bar, phase))) {
                if (threadIdx.x == 0) atomicOr(c.err, ST_TIMEOUT);
                mbar_wait(bar, phase);
                return false;
            }
            phase ^= 1u;
#pragma unroll 1
            for (int r = threadIdx.x; r < cnt; r += kThreads) {
                const float4 r0 = s_rec[r][0], r1 = s_rec[r][1];
                s_rec[r][0] =
                    make_float4((r0.x - oxh) - oxl, (r0.y - oyh) - oyl, (r0.z - ozh) - ozl, r0.w);
                s_rec[r][1] = make_float4(r1.x, r1.y, r1.z, r1.w * cull.inv_R4);
                s_mask[r] = 0;
            }
            __syncthreads();
            // cull masks: one (record, layer) item per thread; byte l of s_mask[r]
            // holds the warps of layer l
#pragma unroll 1
            for (int item = threadIdx.x; item < cnt * S; item += kThreads) {
                const int r = item / S, l = item % S;
                if (l < nl)
                    reinterpret_cast<uint8_t*>(s_mask)[8 * r + l] =
                        (uint8_t)cull_layer<PX>(s_rec[r][0], s_rec[r][1], l, cull);
            }
            __syncthreads();
#pragma unroll 1
            for (int i0 = 0; i0 < cnt; i0 += 32) {
                const int i = i0 + lane;
                const uint32_t wm = i < cnt ? warp_layers(s_mask[i], warp) : 0u;
                uint32_t ball = __ballot_sync(0xffffffffu, wm != 0u);
#pragma unroll 1
                while (ball) {
                    const int b = __ffs(ball) - 1;
                    ball &= ball - 1u;
                    const uint32_t lm = __shfl_sync(0xffffffffu, wm, b);
                    const float4 A = s_rec[i0 + b][0], B = s_rec[i0 + b][1];
                    const float dx = pxl - A.x;
                    float dy[PX], txy[PX];
#pragma unroll
                    for (int k = 0; k < PX; ++k) {
                        dy[k] = pyl[k] - A.y;
                        txy[k] = fmaf(dy[k], B.x, dx * A.w);
                    }
#pragma unroll
                    for (int l = 0; l < S; ++l) {
                        if (lm & (1u << l)) {
                            const float dz = (float)l * c.fdz - A.z;
                            float t0[PX], h2[PX];
                            bool near = PX == 2;
#pragma unroll
                            for (int k = 0; k < PX; ++k) {
                                t0[k] = fmaf(dz, B.y, txy[k]);
                                const float ex = fmaf(-t0[k], A.w, dx);
                                const float ey = fmaf(-t0[k], B.x, dy[k]);
                                const float ez = fmaf(-t0[k], B.y, dz);
                                const float d2 = fmaf(ez, ez, fmaf(ey, ey, ex * ex));
                                h2[k] = fmaxf(c.R2 - d2, 0.0f);
                                near |= h2[k] > 0.0f;
                            }
                            // the rest only when some pixel of the warp is within R (with
                            // two rows per thread, for wide supports, nearly always)
                            if (PX == 2 || __any_sync(0xffffffffu, near)) {
#pragma unroll
                                for (int k = 0; k < PX; ++k) {
                                    const float I = segment_term_R4(t0[k], h2[k], B.z);
                                    acc[l][k] = fmaf(B.w, I, acc[l][k]);
                                    if (COUNT) {
                                        n_nonzero += I > 0.0f;
                                        ++n_eval;
                                    }
                                }
                            }
                        }
                    }
                }
            }
            // the next chunk reuses s_rec and s_mask; after the last one each warp
            // goes on to its own pixels without waiting (a persistent caller
            // synchronises before the next item)
            if (c0 + (uint32_t)kFieldThreads < end) __syncthreads();
        }
    }
    if (COUNT) {   // n_pairs[0]: nonzero terms, n_pairs[1]: evaluated terms
        unsigned long long t = n_nonzero, e = n_eval;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            t += __shfl_down_sync(0xffffffffu, t, o);
            e += __shfl_down_sync(0xffffffffu, e, o);
        }
        if (lane == 0 && t) atomicAdd(n_pairs, t);
        if (lane == 0 && e) atomicAdd(n_pairs + 1, e);
    }
    const int gi = tx * kTile + il;
#pragma unroll
    for (int k = 0; k < PX; ++k) {
        const int gj = ty * kTile + jl + 4 * k;
        const bool in_grid = gi < c.nx && gj < c.ny;
        if (in_grid && sigma) {   // no Sigma plane when only the mask is wanted
#pragma unroll
            for (int l = 0; l < S; ++l)
                if (l < nl) sigma[((int64_t)(l0 + l) * c.ny + gj) * c.nx + gi] = acc[l][k];
        }
        if (mask) {
            // inside bits of 8 x 4 pixels: one byte per pixel row, OR-ed into the
            // padded row (pixel i is padded sample i + 1)
            const int I0 = tx * kTile + wx * 8 + 1;
            const int sh = I0 & 31;
#pragma unroll
            for (int l = 0; l < S; ++l) {
                if (l >= nl) break;
                const uint32_t ball = __ballot_sync(0xffffffffu, in_grid && acc[l][k] >= c.C);
                if (lane < 4) {
                    const uint32_t byte = (ball >> (8 * lane)) & 0xffu;
                    if (byte) {
                        const int J = ty * kTile + wy * 4 * PX + 4 * k + lane + 1;
                        uint32_t* row = mask + (int64_t)(l0 + l) * c.mask_wpl + (int64_t)J * c.mwr;
                        atomicOr(row + (I0 >> 5), byte << sh);
                        const uint32_t hi = sh > 24 ? byte >> (32 - sh) : 0u;
                        if (hi) atomicOr(row + (I0 >> 5) + 1, hi);
                    }
                }
            }
        }
    }
    return true;
}

template <int S, int PX, bool COUNT>
__global__ void __launch_bounds__(kFieldThreads / PX, PX == 2 ? 10 : 8)
k_field(const csl_rec* __restrict__ recs, const uint32_t* __restrict__ tstart,
        const uint32_t* __restrict__ tend, FieldConst c, float* __restrict__ sigma,
        uint32_t* __restrict__ mask, unsigned long long* __restrict__ n_pairs) {
    __shared__ __align__(8) uint64_t bar;
    if (threadIdx.x == 0) {
        mbar_init(&bar, 1);
        fence_mbar_init();
    }
    __syncthreads();
    uint32_t phase = 0;
    field_tile<S, PX, COUNT>(recs, tstart, tend, c, sigma, mask, n_pairs, blockIdx.x, blockIdx.y,
                         &bar, phase);
}

// One job of a batch, as the persistent kernel reads it.
struct FieldJob {
    FieldConst c;
    const csl_rec* recs;   // the binned records, in list order
    const uint32_t* tstart;
    const uint32_t* tend;
    float* sigma;
    uint32_t* mask;
};
static_assert(sizeof(FieldJob) % 4 == 0, "FieldJob is copied as 32-bit words");

// Persistent field kernel over the (job, slab, tile) items of a batch: each
// CTA takes the next item from a shared counter, in the order `order` gives
// (longest tile lists first, so the short ones fill the tail). CTAS: how many of
// them an SM must hold (field_batch_run).
template <int S, int PX, int CTAS>
__global__ void __launch_bounds__(kFieldThreads / PX, CTAS)
k_field_batch(const FieldJob* __restrict__ jobs, const uint2* __restrict__ items,
              const uint32_t* __restrict__ order, uint32_t n_items, uint32_t* counter) {
    __shared__ uint32_t s_item;
    __shared__ FieldJob s_job;
    __shared__ __align__(8) uint64_t bar;
    if (threadIdx.x == 0) {
        mbar_init(&bar, 1);
        fence_mbar_init();
    }
    __syncthreads();
    uint32_t phase = 0;
    uint32_t cur_job = 0xffffffffu;
    for (;;) {
        if (threadIdx.x == 0) s_item = atomicAdd(counter, 1u);
        __syncthreads();
        const uint32_t it = s_item;
        if (it >= n_items) break;
        const uint2 item = items[order[it]];
        if (item.x != cur_job) {   // consecutive items often belong to the same job
            cur_job = item.x;
            const uint32_t* src = reinterpret_cast<const uint32_t*>(jobs + item.x);
            for (int i = threadIdx.x; i < (int)(sizeof(FieldJob) / 4); i += kFieldThreads / PX)
                reinterpret_cast<uint32_t*>(&s_job)[i] = src[i];
            __syncthreads();
        }
        const uint32_t n_tiles = (uint32_t)s_job.c.n_tiles;
        if (!field_tile<S, PX, false>(s_job.recs, s_job.tstart, s_job.tend, s_job.c, s_job.sigma,
                                  s_job.mask, nullptr, (int)(item.y % n_tiles),
                                  (int)(item.y / n_tiles), &bar, phase))
            break;   // a bulk copy gave up (reported): this CTA takes no more items
        __syncthreads();   // shared memory is reused by the next item
    }
}

// The field kernel's bounded mbarrier wait on a barrier that nothing arms: it
// must give up after `polls` polls and report ST_TIMEOUT (test of the path).
__global__ void k_wait_nothing(uint32_t polls, uint32_t* err) {
    __shared__ __align__(8) uint64_t bar;
    if (threadIdx.x == 0) {
        mbar_init(&bar, 1);
        fence_mbar_init();
    }
    __syncthreads();
    if (__syncthreads_or(!mbar_wait(&bar, 0, polls)) && threadIdx.x == 0) atomicOr(err, ST_TIMEOUT);
}

// items[i] = (job, slab * n_tiles + tile) for the jobs' item ranges off[j]..off[j+1].
__global__ void k_make_items(const int64_t* __restrict__ off, int n_jobs, uint2* __restrict__ items) {
    const int64_t n = off[n_jobs];
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        int lo = 0, hi = n_jobs - 1;   // the last job with off[j] <= i
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (off[mid] <= i) lo = mid;
            else hi = mid - 1;
        }
        items[i] = make_uint2((uint32_t)lo, (uint32_t)(i - off[lo]));
    }
}

// Sort keys for the item queue: longest tile list first (16-bit key).
__global__ void k_item_keys(const FieldJob* __restrict__ jobs, const uint2* __restrict__ items,
                            uint32_t n, uint32_t* __restrict__ keys, uint32_t* __restrict__ vals) {
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const uint2 it = items[i];
        const FieldJob& J = jobs[it.x];
        const uint32_t len = J.tend[it.y] - J.tstart[it.y];
        keys[i] = 0xffffu - min(len, 0xffffu);
        vals[i] = i;
    }
}

// Corner of each tile column / row and first plane of each slab, computed in
// double (non-fused) and split into a (hi, lo) float pair.
__global__ void k_origins(float2* __restrict__ org, int ntx, int nty, int n_slabs, double x0,
                          double y0, double z0, double px, double dz, int first_layer, int S,
                          int T) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    double v;
    if (i < ntx) v = __dadd_rn(x0, __dmul_rn((double)(i * T), px));
    else if (i < ntx + nty) v = __dadd_rn(y0, __dmul_rn((double)((i - ntx) * T), px));
    else if (i < ntx + nty + n_slabs)
        v = __dadd_rn(z0, __dmul_rn((double)(first_layer + (i - ntx - nty) * S), dz));
    else return;
    const float hi = (float)v;
    org[i] = make_float2(hi, (float)__dsub_rn(v, (double)hi));
}

}  // namespace

namespace {

// Kernel constants of a chunk; org = the chunk's origin tables (ntx + nty +
// n_slabs float2, as k_origins writes them).
FieldConst make_field_const(const ChunkGeom& g, float C, const float2* org, int rows) {
    FieldConst c;
    c.C = C;
    c.org_x = org;
    c.org_y = org + g.ntx;
    c.org_z = org + g.ntx + g.nty;
    c.mwr = (int32_t)mask_words_per_row(g.nx);
    c.mask_wpl = mask_words_per_layer(g.nx, g.ny);
    c.nx = g.nx;
    c.ny = g.ny;
    c.ntx = g.ntx;
    c.n_tiles = g.ntx * g.nty;
    c.n_layers = g.n_layers;
    c.R2 = (float)(g.R * g.R);
    c.fpx = (float)g.px;
    c.fdz = (float)g.dz;
    c.tc.cull = (float)(g.R * (1.0 + 1e-5) + 1e-6);
    {
        // pixel centres of a warp's block of 8 x 4 rows pixels lie within 3.5 x
        // (2 rows - 1/2) pixels of its centre
        const double hy = 2.0 * rows - 0.5;
        double hd = g.px * sqrt(3.5 * 3.5 + hy * hy) * (1.0 + 1e-5);
        double r = (double)c.tc.cull + hd;
        c.tc.cull_line2 = (float)(r * r);
    }
    c.tc.fpx = c.fpx;
    c.tc.fdz = c.fdz;
    c.tc.inv_R4 = (float)(1.0 / (g.R * g.R * g.R * g.R));
    return c;
}

// Pixel rows per thread of the block kernel. Two halve the visits of records and
// their layer tests, and cost lanes where a support covers few pixels (1,332
// against 1,151 million evaluated terms for 818 million nonzero ones at R = 26
// px, with 17 % fewer instructions in all). Field of 2000^2 px x 200 layers at R
// = 26 px: 20.4 ms with one row, 17.5 with two (90 % issue); at 15 px (12 batched
// lattices) 8.0 and 6.6 ms, at 10.5 px (780^2 x 190) 4.11 and 3.91 ms. Below, one
// row: there the automatic choice takes the footprint kernel, and the volume
// fraction's samples (R = 5 px) keep 8 x 4 blocks.
int rows_per_thread(const ChunkGeom& g) { return g.R >= 10.0 * g.px ? 2 : 1; }

void launch_origins(const ChunkGeom& g, float2* org, cudaStream_t s) {
    k_origins<<<(unsigned)ceil_div(g.ntx + g.nty + g.n_slabs, 128), 128, 0, s>>>(
        org, g.ntx, g.nty, g.n_slabs, g.x0, g.y0, g.z0, g.px, g.dz, g.first_layer, g.S, g.T);
    CSL_LAUNCH_CHECK("origins");
}

}  // namespace

void field_chunk(const csl_lattice* L, const ChunkGeom& g, const SlabBins& bins, float C,
                 float* sigma, uint32_t* mask, unsigned long long* count_pairs, cudaStream_t s,
                 FusedVerts* fv) {
    // tile and slab origins in double, each split into a (hi, lo) float pair
    DevBuf org_d(((size_t)g.ntx + g.nty + g.n_slabs) * sizeof(float2), s);
    launch_origins(g, org_d.as<float2>(), s);
    if (g.kernel == kFieldFootprint) {
        field_chunk_fp(g, bins, C, org_d.as<float2>(), L->status.as<uint32_t>(), sigma, mask,
                       count_pairs, s, fv);
        return;
    }
    if (g.fused || fv) fail(CSL_ERR_INVALID_ARG, "the fused pass needs the footprint kernel");
    if (g.T != kTile) fail(CSL_ERR_INVALID_ARG, "the block field kernel takes 16-pixel tiles");
    const int rows = rows_per_thread(g);
    FieldConst c = make_field_const(g, C, org_d.as<float2>(), rows);
    c.err = L->status.as<uint32_t>();
    dim3 grid((unsigned)c.n_tiles, (unsigned)g.n_slabs);
    const csl_rec* recs = bins.recs.as<csl_rec>();
    const uint32_t* ts = bins.tile_start.as<uint32_t>();
    const uint32_t* te = bins.tile_end.as<uint32_t>();
#define CSL_FIELD_LAUNCH(SV, PXV, CNT)                                                       \
    k_field<SV, PXV, CNT><<<grid, kFieldThreads / PXV, 0, s>>>(recs, ts, te, c, sigma, mask,  \
                                                               count_pairs)
#define CSL_FIELD_CASE(SV)                                                                    \
    case SV:                                                                                  \
        if (rows == 2 && count_pairs) CSL_FIELD_LAUNCH(SV, 2, true);                          \
        else if (rows == 2) CSL_FIELD_LAUNCH(SV, 2, false);                                   \
        else if (count_pairs) CSL_FIELD_LAUNCH(SV, 1, true);                                  \
        else CSL_FIELD_LAUNCH(SV, 1, false);                                                  \
        break;
    switch (g.S) {
        CSL_FIELD_CASE(1)
        CSL_FIELD_CASE(2)
        CSL_FIELD_CASE(4)
        CSL_FIELD_CASE(8)
        default: fail(CSL_ERR_INVALID_ARG, "slab depth must be 1, 2, 4 or 8");
    }
#undef CSL_FIELD_CASE
#undef CSL_FIELD_LAUNCH
    CSL_LAUNCH_CHECK("field");
}

void field_batch_prepare(const std::vector<FieldBatchJob>& jobs, FieldBatch& fb, cudaStream_t s) {
    const int n_jobs = (int)jobs.size();
    if (n_jobs == 0) fail(CSL_ERR_INVALID_ARG, "empty batch");
    const int S = jobs[0].g.S;
    const int kern = jobs[0].g.kernel, T = jobs[0].g.T, K = jobs[0].g.K;
    size_t n_org = 0;
    std::vector<int64_t> off(n_jobs + 1, 0);
    for (int j = 0; j < n_jobs; ++j) {
        const ChunkGeom& g = jobs[j].g;
        if (g.S != S) fail(CSL_ERR_INVALID_ARG, "batch: one slab depth for every job");
        if (g.kernel != kern || g.T != T || g.K != K || g.fused)
            fail(CSL_ERR_INVALID_ARG, "batch: one field kernel, tile and staging chunk");
        if (kern == kFieldBlock && T != kTile)
            fail(CSL_ERR_INVALID_ARG, "batch: the block field kernel takes 16-pixel tiles");
        n_org += (size_t)g.ntx + g.nty + g.n_slabs;
        off[j + 1] = off[j] + (int64_t)g.n_slabs * g.ntx * g.nty;
    }
    if (off[n_jobs] >= 0xffffffffLL) fail(CSL_ERR_CAPACITY, "batch: more than 2^32 - 1 tiles");
    fb.S = S;
    fb.kernel = kern;
    fb.T = T;
    fb.K = K;
    fb.n_items = off[n_jobs];
    fb.rows = 2;   // one kernel for all jobs
    for (const FieldBatchJob& J : jobs) fb.rows = std::min(fb.rows, rows_per_thread(J.g));
    fb.origins.alloc_persistent(n_org * sizeof(float2));
    std::vector<FieldJob> hj(n_jobs);
    std::vector<const float2*> orgs(n_jobs);
    size_t o = 0;
    for (int j = 0; j < n_jobs; ++j) {
        const FieldBatchJob& J = jobs[j];
        float2* org = fb.origins.as<float2>() + o;
        orgs[j] = org;
        launch_origins(J.g, org, s);
        o += (size_t)J.g.ntx + J.g.nty + J.g.n_slabs;
        hj[j].c = make_field_const(J.g, (float)J.L->C, org, fb.rows);
        hj[j].c.err = J.err;
        hj[j].recs = J.bins->recs.as<csl_rec>();
        hj[j].tstart = J.bins->tile_start.as<uint32_t>();
        hj[j].tend = J.bins->tile_end.as<uint32_t>();
        hj[j].sigma = J.sigma;
        hj[j].mask = J.mask;
    }
    fb.jobs.alloc_persistent(sizeof(FieldJob) * n_jobs);
    DevBuf off_d((size_t)(n_jobs + 1) * 8, s);
    CSL_CUDA(cudaMemcpyAsync(fb.jobs.get(), hj.data(), sizeof(FieldJob) * n_jobs,
                             cudaMemcpyHostToDevice, s));
    std::vector<unsigned char> hfp;
    if (kern == kFieldFootprint) {
        fp_batch_jobs(jobs, orgs.data(), hfp);
        fb.fp_jobs.alloc_persistent(hfp.size());
        CSL_CUDA(cudaMemcpyAsync(fb.fp_jobs.get(), hfp.data(), hfp.size(),
                                 cudaMemcpyHostToDevice, s));
    }
    CSL_CUDA(cudaMemcpyAsync(off_d.get(), off.data(), (size_t)(n_jobs + 1) * 8,
                             cudaMemcpyHostToDevice, s));
    const size_t n = (size_t)fb.n_items;
    fb.items.alloc_persistent(n * sizeof(uint2));
    fb.keys.alloc_persistent(n * 4);
    fb.vals.alloc_persistent(n * 4);
    fb.tmp_keys.alloc_persistent(n * 4);
    fb.tmp_vals.alloc_persistent(n * 4);
    fb.counter.alloc_persistent(4);
    k_make_items<<<grid_for(fb.n_items, 256), 256, 0, s>>>(off_d.as<int64_t>(), n_jobs,
                                                          fb.items.as<uint2>());
    CSL_LAUNCH_CHECK("batch items");
    CSL_CUDA(cudaStreamSynchronize(s));   // the host tables above go out of scope
}

int field_batch_most_ctas(const FieldBatch& fb) {
    return fb.kernel == kFieldBlock && fb.rows == 2 ? 4 : 6;
}

void field_batch_run(FieldBatch& fb, int n_sm, int ctas, cudaStream_t s) {
    ctas = std::min(ctas, field_batch_most_ctas(fb));
    const int n_ctas = n_sm * ctas;
    if (fb.n_items == 0) return;
    const uint32_t n = (uint32_t)fb.n_items;
    k_item_keys<<<grid_for(fb.n_items, 256), 256, 0, s>>>(
        fb.jobs.as<FieldJob>(), fb.items.as<uint2>(), n, fb.keys.as<uint32_t>(),
        fb.vals.as<uint32_t>());
    CSL_LAUNCH_CHECK("batch item keys");
    radix_sort_pairs(fb.keys.as<uint32_t>(), fb.vals.as<uint32_t>(), fb.tmp_keys.as<uint32_t>(),
                     fb.tmp_vals.as<uint32_t>(), fb.n_items, 16, s);
    CSL_CUDA(cudaMemsetAsync(fb.counter.get(), 0, 4, s));
    const FieldJob* jobs = fb.jobs.as<FieldJob>();
    const uint2* items = fb.items.as<uint2>();
    const uint32_t* order = fb.vals.as<uint32_t>();
    uint32_t* counter = fb.counter.as<uint32_t>();
    if (fb.kernel == kFieldFootprint) {
        fp_batch_launch(fb.fp_jobs.get(), items, order, n, counter, fb.T, fb.S, fb.K, n_ctas, s);
        return;
    }
    // With two pixel rows per thread a CTA has half the threads: twice as many CTAs, 8
    // per SM at most, so 4 in the units of `ctas`. Registers for 8 of them (64 each)
    // where they are wanted, else for 6 (79), which are a little faster while they are
    // all there are: 12 batched lattices, S = 8, with 2, 3 and 4 per SM: 9.72, 8.45
    // and 8.45 ms for 6 (the fourth did not fit), 9.86, 8.60 and 8.23 for 8. Room for 10
    // or 12 costs spills: 8.46 and 8.61 ms at 6 per SM.
#define CSL_FIELD_LAUNCH(SV, PXV, CT)                                                          \
    k_field_batch<SV, PXV, CT><<<PXV * n_ctas, kFieldThreads / PXV, 0, s>>>(jobs, items, order, \
                                                                            n, counter)
#define CSL_FIELD_CASE(SV)                                                                     \
    case SV:                                                                                   \
        if (fb.rows == 2 && ctas > 3) CSL_FIELD_LAUNCH(SV, 2, 8);                              \
        else if (fb.rows == 2) CSL_FIELD_LAUNCH(SV, 2, 6);                                     \
        else CSL_FIELD_LAUNCH(SV, 1, 6);                                                       \
        break;
    switch (fb.S) {
        CSL_FIELD_CASE(1)
        CSL_FIELD_CASE(2)
        CSL_FIELD_CASE(4)
        CSL_FIELD_CASE(8)
        default: fail(CSL_ERR_INVALID_ARG, "slab depth must be 1, 2, 4 or 8");
    }
#undef CSL_FIELD_CASE
#undef CSL_FIELD_LAUNCH
    CSL_LAUNCH_CHECK("batch field");
}

}  // namespace csl

namespace {

csl_status wait_nothing(uint32_t polls, cudaStream_t s, uint32_t* err, bool report) {
    try {
        if (polls == 0 || polls > csl::kWaitLimit) csl::fail(CSL_ERR_INVALID_ARG, "polls in [1, 2^22]");
        csl::DevBuf own;
        if (!err) {
            own.alloc(4, s);
            err = own.as<uint32_t>();
            CSL_CUDA(cudaMemsetAsync(err, 0, 4, s));
        }
        csl::k_wait_nothing<<<1, 64, 0, s>>>(polls, err);
        CSL_LAUNCH_CHECK("wait test");
        uint32_t st = 0;
        csl::read_to_host(&st, err, 4, s);
        if (report && (st & csl::ST_TIMEOUT))
            csl::fail(CSL_ERR_TIMEOUT, "the wait gave up as it should");
        return CSL_OK;
    } catch (const csl::Error& e) {
        csl::set_last_error(e.what());
        return e.code;
    } catch (...) {
        csl::set_last_error("unknown error");
        return CSL_ERR_CUDA;
    }
}

}  // namespace

extern "C" csl_status csl_debug_wait_timeout(uint32_t polls, void* stream) {
    return wait_nothing(polls, (cudaStream_t)stream, nullptr, true);
}

extern "C" csl_status csl_debug_lattice_timeout(csl_lattice* L, uint32_t polls, void* stream) {
    if (!L) {
        csl::set_last_error("lattice is NULL");
        return CSL_ERR_INVALID_ARG;
    }
    return wait_nothing(polls, (cudaStream_t)stream, L->status.as<uint32_t>(), false);
}
