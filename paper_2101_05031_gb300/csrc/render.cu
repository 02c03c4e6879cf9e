// Ray casting of the implicit solid {Sigma >= C} into a headless depth image
// (the paper renders its lattices by ray tracing the implicit function,
// without a mesh; the field is that of Eq. 5-7).
//
// The struts are binned into a uniform 3D grid (each strut into every cell
// that its support can meet: count, scan, emit, radix sort by cell). A ray is
// sampled at t_in + k * step from where it enters the lattice's box grown by
// R; Sigma at a sample sums the struts listed for the sample's cell (every
// strut whose support reaches the point is listed there, in the order of the
// records); the first sample with Sigma >= C is refined by `refine` halvings
// of the last step. A cell with no strut has Sigma = 0 everywhere, so the ray
// jumps over it. A strut that cannot reach a sample adds nothing, so neither
// the cell size nor the culling below changes any sum.
#include <math.h>

#include <algorithm>
#include <vector>

#include "common.cuh"
#include "field_tile.cuh"
#include "slice.cuh"

namespace csl {
namespace {

struct RvGrid {
    float lox, loy, loz, h, inv_h;   // grid corner and cell edge
    float reach;   // R plus a slack far above the rounding of a sample's position and cell
    float near;    // reach plus that slack again, for the ranges of cells along a strut
    int32_t nx, ny, nz;
};

struct RvConst {
    float ex, ey, ez;          // eye
    float fx, fy, fz;          // forward
    float rx, ry, rz;          // right
    float ux, uy, uz;          // up
    float half_w, half_h;      // image-plane half extents at distance 1
    int32_t width, height, tiles_x;   // tiles of 128 pixels, one per block
    int32_t log_wx, log_bx;           // log2 of a warp's pixels and a block's warps along x
    float step;
    int32_t refine;
    float blo[3], bhi[3];      // the lattice's box grown by R
    float R2, inv_R4, C;
};

// Narrows [t0, t1] to the part of a strut whose coordinate s + t u lies in
// [lo, hi] (inv = 1 / u, 0 where the strut runs across the axis).
__device__ __forceinline__ void clip_strut(float lo, float hi, float s, float inv, float& t0,
                                           float& t1) {
    if (inv == 0.0f) return;
    const float a = (lo - s) * inv, b = (hi - s) * inv;
    t0 = fmaxf(t0, fminf(a, b));
    t1 = fminf(t1, fmaxf(a, b));
}

// Calls f(cell) for every cell that the strut's support (radius R with its
// slack) can meet: the cells of its box, without those that the strut's line
// passes farther than R from (the separating axis from the line to the
// centre; a cell reaches at most h/2 |e|_1 / |e| along it). Of a layer of cells
// only the rows beside the part of the strut that comes near the layer are
// looked at, of a row only the cells beside the part that comes near the row, so
// that a strut costs as many tests as it lists cells, about: a depth image of one
// strut of 140 mm, R = 0.5 mm, across its box takes 1.7 ms, 203 ms with the whole
// box tested by the strut's thread, of 500 of them 2.8 and 332 ms (429,039 struts of
// about 1 mm: the same 4.1 ms either way).
template <class F>
__device__ __forceinline__ void strut_cells(const csl_rec& r, const RvGrid& g, F f) {
    const float R = g.reach;
    const float end[3] = {r.ax + r.len * r.ux, r.ay + r.len * r.uy, r.az + r.len * r.uz};
    const float beg[3] = {r.ax, r.ay, r.az};
    const float o[3] = {g.lox, g.loy, g.loz};
    const int n[3] = {g.nx, g.ny, g.nz};
    int a[3], b[3];
    for (int k = 0; k < 3; ++k) {
        const float lo = fminf(beg[k], end[k]) - R, hi = fmaxf(beg[k], end[k]) + R;
        a[k] = max(0, min(n[k] - 1, (int)floorf((lo - o[k]) * g.inv_h)));
        b[k] = max(0, min(n[k] - 1, (int)floorf((hi - o[k]) * g.inv_h)));
    }
    const float W = g.near;
    const float inv_y = fabsf(r.uy) > 1e-12f ? 1.0f / r.uy : 0.0f;
    const float inv_z = fabsf(r.uz) > 1e-12f ? 1.0f / r.uz : 0.0f;
    for (int k = a[2]; k <= b[2]; ++k) {
        const float z = g.loz + g.h * (float)k, qz = g.loz + g.h * ((float)k + 0.5f) - r.az;
        float t0 = 0.0f, t1 = r.len;
        clip_strut(z - W, z + g.h + W, r.az, inv_z, t0, t1);
        if (t0 > t1) continue;
        const float ya = r.ay + t0 * r.uy, yb = r.ay + t1 * r.uy;
        const int j0 = max(a[1], (int)floorf((fminf(ya, yb) - W - g.loy) * g.inv_h));
        const int j1 = min(b[1], (int)floorf((fmaxf(ya, yb) + W - g.loy) * g.inv_h));
        for (int j = j0; j <= j1; ++j) {
            const float y = g.loy + g.h * (float)j, qy = g.loy + g.h * ((float)j + 0.5f) - r.ay;
            float s0 = t0, s1 = t1;
            clip_strut(y - W, y + g.h + W, r.ay, inv_y, s0, s1);
            if (s0 > s1) continue;
            const float xa = r.ax + s0 * r.ux, xb = r.ax + s1 * r.ux;
            const int i0 = max(a[0], (int)floorf((fminf(xa, xb) - W - g.lox) * g.inv_h));
            const int i1 = min(b[0], (int)floorf((fmaxf(xa, xb) + W - g.lox) * g.inv_h));
            for (int i = i0; i <= i1; ++i) {
                const float qx = g.lox + g.h * ((float)i + 0.5f) - r.ax;
                const float t = qx * r.ux + qy * r.uy + qz * r.uz;
                const float ex = qx - t * r.ux, ey = qy - t * r.uy, ez = qz - t * r.uz;
                const float e2 = ex * ex + ey * ey + ez * ez;
                const float l1 = fabsf(ex) + fabsf(ey) + fabsf(ez);
                // |e| - h/2 l1 / |e| > R, i.e. e2 - h/2 l1 > R |e|
                const float gap = e2 - 0.5f * g.h * l1;
                if (gap > 0.0f && gap * gap > R * R * e2) continue;
                f((uint32_t)(((int64_t)k * g.ny + j) * g.nx + i));
            }
        }
    }
}

__global__ void k_rv_count(const csl_rec* __restrict__ rec, int64_t n, RvGrid g,
                           uint32_t* __restrict__ cnt) {
    for (int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; s < n;
         s += (int64_t)gridDim.x * blockDim.x) {
        uint32_t c = 0;
        strut_cells(rec[s], g, [&](uint32_t) { ++c; });
        cnt[s] = c;
    }
}

__global__ void k_rv_emit(const csl_rec* __restrict__ rec, int64_t n, RvGrid g,
                          const int64_t* __restrict__ off, uint32_t* __restrict__ keys,
                          uint32_t* __restrict__ vals) {
    for (int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; s < n;
         s += (int64_t)gridDim.x * blockDim.x) {
        int64_t o = off[s];
        strut_cells(rec[s], g, [&](uint32_t cell) {
            keys[o] = cell;
            vals[o] = (uint32_t)s;
            ++o;
        });
    }
}

__global__ void k_rv_bounds(const uint32_t* __restrict__ keys, int64_t n,
                            uint32_t* __restrict__ beg, uint32_t* __restrict__ end) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t k = keys[i];
        if (i == 0 || keys[i - 1] != k) beg[k] = (uint32_t)i;
        if (i == n - 1 || keys[i + 1] != k) end[k] = (uint32_t)(i + 1);
    }
}

// Cell of a point, or -1 outside the grid.
__device__ __forceinline__ int64_t cell_of(float px, float py, float pz, const RvGrid& g,
                                           int& ci, int& cj, int& ck) {
    ci = (int)floorf((px - g.lox) * g.inv_h);
    cj = (int)floorf((py - g.loy) * g.inv_h);
    ck = (int)floorf((pz - g.loz) * g.inv_h);
    if (ci < 0 || cj < 0 || ck < 0 || ci >= g.nx || cj >= g.ny || ck >= g.nz) return -1;
    return ((int64_t)ck * g.ny + cj) * g.nx + ci;
}

// Sigma >= C at a point, from its cell's list (cell < 0: outside the grid,
// Sigma = 0). The terms are not negative, so the sum only grows (rounding
// included) and is left once it has reached C. kRvBatch records are loaded
// before the first is used: a list is a chain of loads (index, record) and the
// march has little else to hide them behind.
constexpr int kRvBatch = 4;
__device__ __forceinline__ bool inside(float px, float py, float pz, int64_t cell,
                                       const csl_rec* __restrict__ rec,
                                       const uint32_t* __restrict__ vals,
                                       const uint32_t* __restrict__ cbeg,
                                       const uint32_t* __restrict__ cend, const RvConst& c) {
    if (cell < 0) return 0.0f >= c.C;
    float sig = 0.0f;
    const uint32_t e = cend[cell];
    for (uint32_t q = cbeg[cell]; q < e && !(sig >= c.C); q += kRvBatch) {
        csl_rec r[kRvBatch];
#pragma unroll
        for (int u = 0; u < kRvBatch; ++u) r[u] = rec[vals[min(q + u, e - 1)]];
#pragma unroll
        for (int u = 0; u < kRvBatch; ++u) {
            const float qx = px - r[u].ax, qy = py - r[u].ay, qz = pz - r[u].az;
            const float t0 = qx * r[u].ux + qy * r[u].uy + qz * r[u].uz;
            const float ex = qx - t0 * r[u].ux, ey = qy - t0 * r[u].uy, ez = qz - t0 * r[u].uz;
            const float h2 = c.R2 - (ex * ex + ey * ey + ez * ez);
            if (q + u < e && h2 > 0.0f && r[u].len > 0.0f)
                sig += (r[u].w * c.inv_R4) * segment_term_R4(t0, h2, r[u].len);
        }
    }
    return sig >= c.C;
}

// One thread per pixel, a warp per 8 x 4 block of pixels (its rays meet the
// same cells, so their loads of a list coincide; image_tiles for narrow images): depth along the pixel's unit
// ray, +inf for a miss. Bound by the instructions of the sums. All rays of a
// warp first march to their hit, then all halve their last step together:
// halving at once in the march would run the warp through the halvings once
// for every sample index at which one of its rays hits (1920 x 1080 rays into
// 429,039 struts: 10.3 ms with that and cells of 2 R by bounding boxes, 3.3 ms
// now).
__global__ void __launch_bounds__(128)
k_rv_render(const csl_rec* __restrict__ rec, const uint32_t* __restrict__ vals,
            const uint32_t* __restrict__ cbeg, const uint32_t* __restrict__ cend, RvGrid g,
            RvConst c, float* __restrict__ depth) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int wx = c.log_wx, bx = c.log_bx;
    const int i = (((int)(blockIdx.x % (uint32_t)c.tiles_x) << bx | (warp & ((1 << bx) - 1))) << wx) +
                  (lane & ((1 << wx) - 1));
    const int j = (((int)(blockIdx.x / (uint32_t)c.tiles_x) << (2 - bx) | warp >> bx) << (5 - wx)) +
                  (lane >> wx);
    if (i >= c.width || j >= c.height) return;
    const float x = (((float)i + 0.5f) / (float)c.width * 2.0f - 1.0f) * c.half_w;
    const float y = (1.0f - ((float)j + 0.5f) / (float)c.height * 2.0f) * c.half_h;
    float dx = c.fx + x * c.rx + y * c.ux, dy = c.fy + x * c.ry + y * c.uy,
          dz = c.fz + x * c.rz + y * c.uz;
    const float inv = 1.0f / sqrtf(dx * dx + dy * dy + dz * dz);
    dx *= inv;
    dy *= inv;
    dz *= inv;
    const float o[3] = {c.ex, c.ey, c.ez}, d[3] = {dx, dy, dz};
    // the ray's interval in the box grown by R
    float t_in = 0.0f, t_out = INFINITY;
    bool miss = false;
    for (int k = 0; k < 3 && !miss; ++k) {
        if (d[k] == 0.0f) {
            miss = o[k] < c.blo[k] || o[k] > c.bhi[k];
            continue;
        }
        float a = (c.blo[k] - o[k]) / d[k], b = (c.bhi[k] - o[k]) / d[k];
        if (a > b) {
            const float t = a;
            a = b;
            b = t;
        }
        t_in = fmaxf(t_in, a);
        t_out = fminf(t_out, b);
        miss = t_in > t_out;
    }
    float result = INFINITY;
    const uint32_t live = __ballot_sync(__activemask(), !miss);
    if (!miss) {
        const int64_t k_max = (int64_t)floorf((t_out - t_in) / c.step);
        const float lo3[3] = {g.lox, g.loy, g.loz};
        int64_t k = 0;
        bool hit = false;
        while (k <= k_max) {
            const float t = t_in + c.step * (float)k;
            const float px = o[0] + t * d[0], py = o[1] + t * d[1], pz = o[2] + t * d[2];
            int cc[3];
            const int64_t cell = cell_of(px, py, pz, g, cc[0], cc[1], cc[2]);
            if (cell >= 0 && cbeg[cell] == cend[cell]) {
                // an empty cell: jump to the first sample past it
                float t_exit = INFINITY;
                for (int a = 0; a < 3; ++a) {
                    if (d[a] == 0.0f) continue;
                    const float bound = lo3[a] + g.h * (float)(d[a] > 0.0f ? cc[a] + 1 : cc[a]);
                    t_exit = fminf(t_exit, (bound - o[a]) / d[a]);
                }
                const int64_t kn = (int64_t)floorf((t_exit - t_in) / c.step) + 1;
                k = kn > k ? kn : k + 1;
                continue;
            }
            hit = inside(px, py, pz, cell, rec, vals, cbeg, cend, c);
            if (hit) break;
            ++k;
        }
        __syncwarp(live);
        if (hit) {
            if (k == 0) {
                result = t_in;
            } else {
                float lo = t_in + c.step * (float)(k - 1), hi = t_in + c.step * (float)k;
                for (int it = 0; it < c.refine; ++it) {
                    const float m = 0.5f * (lo + hi);
                    const float px = o[0] + m * d[0], py = o[1] + m * d[1], pz = o[2] + m * d[2];
                    int cc[3];
                    const int64_t cell = cell_of(px, py, pz, g, cc[0], cc[1], cc[2]);
                    if (inside(px, py, pz, cell, rec, vals, cbeg, cend, c))
                        hi = m;
                    else
                        lo = m;
                }
                result = 0.5f * (lo + hi);
            }
        }
    }
    depth[(int64_t)j * c.width + i] = result;
}

// The pixels of a warp and a block: 8 x 4 and 2 x 2 of them; in an image narrower
// or lower than that as many as it has, so that lanes are not spent outside it
// (1 x 200,000 rays into 429,039 struts: 2.63 ms with 8 x 4 throughout, 1.03 so;
// 200,000 x 1: 1.43 and 1.03). Returns the number of blocks.
int64_t image_tiles(RvConst& c) {
    c.log_wx = 3;
    while (c.log_wx > 0 && c.width <= 1 << (c.log_wx - 1)) --c.log_wx;
    while (c.log_wx < 5 && c.width > 1 << c.log_wx && c.height <= 1 << (4 - c.log_wx)) ++c.log_wx;
    c.log_bx = c.width <= 1 << c.log_wx ? 0 : (c.height <= 1 << (5 - c.log_wx) ? 2 : 1);
    const int log_x = c.log_wx + c.log_bx;   // of 128 pixels
    c.tiles_x = ((c.width - 1) >> log_x) + 1;   // (up to 2^31 - 1 pixels)
    return (int64_t)c.tiles_x * (((c.height - 1) >> (7 - log_x)) + 1);
}

}  // namespace
}  // namespace csl

using namespace csl;

extern "C" csl_status csl_render_depth(const csl_lattice* L, const csl_camera* cam, float* depth,
                                       void* stream) {
    try {
        if (!L || !cam || !depth) fail(CSL_ERR_INVALID_ARG, "NULL argument");
        require_device_resident(L);
        if (cam->width < 1 || cam->height < 1 || (int64_t)cam->width * cam->height >= (1ll << 31))
            fail(CSL_ERR_INVALID_ARG, "width and height must be >= 1");
        if (!(cam->fov_y > 0.0 && cam->fov_y < M_PI)) fail(CSL_ERR_INVALID_ARG, "fov_y in (0, pi)");
        if (!(cam->step > 0.0) || !isfinite(cam->step)) fail(CSL_ERR_INVALID_ARG, "step must be > 0");
        if (cam->refine < 0 || cam->refine > 60) fail(CSL_ERR_INVALID_ARG, "refine in [0, 60]");
        double f[3], up[3], r[3], u[3];
        for (int k = 0; k < 3; ++k) {
            if (!isfinite(cam->eye[k]) || !isfinite(cam->target[k]) || !isfinite(cam->up[k]))
                fail(CSL_ERR_INVALID_ARG, "non-finite camera");
            f[k] = cam->target[k] - cam->eye[k];
            up[k] = cam->up[k];
        }
        const double fn = sqrt(f[0] * f[0] + f[1] * f[1] + f[2] * f[2]);
        if (!(fn > 0.0)) fail(CSL_ERR_INVALID_ARG, "target equals eye");
        for (int k = 0; k < 3; ++k) f[k] /= fn;
        r[0] = f[1] * up[2] - f[2] * up[1];
        r[1] = f[2] * up[0] - f[0] * up[2];
        r[2] = f[0] * up[1] - f[1] * up[0];
        const double rn = sqrt(r[0] * r[0] + r[1] * r[1] + r[2] * r[2]);
        if (!(rn > 0.0)) fail(CSL_ERR_INVALID_ARG, "up is parallel to the view direction");
        for (int k = 0; k < 3; ++k) r[k] /= rn;
        u[0] = r[1] * f[2] - r[2] * f[1];
        u[1] = r[2] * f[0] - r[0] * f[2];
        u[2] = r[0] * f[1] - r[1] * f[0];
        cudaStream_t s = (cudaStream_t)stream;
        const int64_t n_px = (int64_t)cam->width * cam->height;
        const int64_t ne = L->n_edges;
        const double R = L->R;
        RvConst c;
        c.ex = (float)cam->eye[0];
        c.ey = (float)cam->eye[1];
        c.ez = (float)cam->eye[2];
        c.fx = (float)f[0]; c.fy = (float)f[1]; c.fz = (float)f[2];
        c.rx = (float)r[0]; c.ry = (float)r[1]; c.rz = (float)r[2];
        c.ux = (float)u[0]; c.uy = (float)u[1]; c.uz = (float)u[2];
        c.half_h = (float)tan(0.5 * cam->fov_y);
        c.half_w = (float)(tan(0.5 * cam->fov_y) * cam->width / cam->height);
        c.width = cam->width;
        c.height = cam->height;
        const int64_t n_blocks = image_tiles(c);
        c.step = (float)cam->step;
        c.refine = cam->refine;
        for (int k = 0; k < 3; ++k) {
            c.blo[k] = (float)((double)L->bbox_lo[k] - R);
            c.bhi[k] = (float)((double)L->bbox_hi[k] + R);
        }
        c.R2 = (float)(R * R);
        c.inv_R4 = (float)(1.0 / (R * R * R * R));
        c.C = (float)L->C;
        if (ne == 0) {
            // no struts: every ray misses
            std::vector<float> inf(n_px, INFINITY);
            CSL_CUDA(cudaMemcpyAsync(depth, inf.data(), n_px * 4, cudaMemcpyHostToDevice, s));
            CSL_CUDA(cudaStreamSynchronize(s));
            return CSL_OK;
        }
        // at most 2^24 samples along any ray through the box, so that the
        // sample index k is exact in float and every march ends in bounded time
        {
            double diag2 = 0.0;
            for (int k = 0; k < 3; ++k) {
                const double e = (double)c.bhi[k] - (double)c.blo[k];
                diag2 += e * e;
            }
            if (sqrt(diag2) / cam->step > (double)(1 << 24))
                fail(CSL_ERR_INVALID_ARG, "step too small: more than 2^24 samples across the box");
        }
        // The grid: cells of edge >= 1.3 R, at most 2^24 of them. Smaller cells
        // shorten the lists that a sample sums and make more pairs to sort
        // (429,039 struts of about 1 mm, R = 0.525 mm, 1920 x 1080 rays: cells of
        // 0.75, 1, 1.3 and 1.6 R take 5.3, 4.5, 4.2 and 4.3 ms, of which the rays
        // 2.7, 3.1, 3.3 and 3.7 ms). Where that makes many pairs for the pixels the
        // sort costs more than the rays, and the cells are of 2 R: above 2^23 pairs and 64
        // for each pixel, where no lattice timed lost by it (3.5 million struts, 64 x 48
        // rays: 3.6 ms, 5.9 with cells of 1.3 R, 5.0 with cells of 2 R by bounding
        // boxes; 1280 x 720: 5.6, 7.4 and 10.0; 1 million short struts, 320 x 240: 2.0, 2.2
        // and 2.9, but 640 x 480: 3.3 and 3.1 ms). Where that makes
        // more than 2^27 strut-cell pairs (2 GB of lists) the edge is doubled, and
        // again while there are 2^31 pairs.
        RvGrid g;
        double scale = 1.0;
        for (int k = 0; k < 3; ++k)
            scale = std::max({scale, fabs((double)c.blo[k]), fabs((double)c.bhi[k])});
        g.reach = (float)(R + 1e-3 * R + 4e-6 * scale);
        g.near = (float)(R + 1e-3 * R + 8e-6 * scale);
        const csl_rec* rec = L->rec.as<csl_rec>();
        DevBuf d_cnt((size_t)ne * 4, s), d_off((size_t)ne * 8, s), d_tot(8, s);
        int64_t n_cells = 0, n_pairs = 0;
        double base = 1.3 * R;
        for (int grow = 0;; ++grow) {
            double h = std::max(ldexp(base, grow), 1e-6);
            const double want = h;
            int dims[3];
            auto dims_of = [&](double hh) {
                double tot = 1;
                for (int k = 0; k < 3; ++k) {
                    const double n =
                        std::max<double>(1.0, ceil((double)(c.bhi[k] - c.blo[k]) / hh) + 1.0);
                    dims[k] = (int)std::min(n, 2e9);
                    tot *= n;
                }
                return tot;
            };
            while (dims_of(h) > (double)(1ll << 24)) h *= 1.25;
            g.lox = c.blo[0];
            g.loy = c.blo[1];
            g.loz = c.blo[2];
            g.h = (float)h;
            g.inv_h = (float)(1.0 / h);
            g.nx = dims[0];
            g.ny = dims[1];
            g.nz = dims[2];
            n_cells = (int64_t)g.nx * g.ny * g.nz;
            k_rv_count<<<grid_for(ne, 256), 256, 0, s>>>(rec, ne, g, d_cnt.as<uint32_t>());
            CSL_LAUNCH_CHECK("render cell counts");
            exclusive_scan_u32_to_i64(d_cnt.as<uint32_t>(), d_off.as<int64_t>(), ne,
                                      d_tot.as<int64_t>(), s);
            n_pairs = read_i64(d_tot.as<int64_t>(), s);
            if (grow == 0 && n_pairs <= (1ll << 27) && h == want && base < 2.0 * R &&
                n_pairs > (1ll << 23) + 64 * n_px) {
                base = 2.0 * R;
                grow = -1;
                continue;
            }
            if (n_pairs <= (1ll << 27) || (grow > 0 && n_pairs < (1ll << 31))) break;
            if (n_cells == 8) fail(CSL_ERR_CAPACITY, "more than 2^31 strut-cell pairs");
        }
        const size_t pb = (size_t)std::max<int64_t>(n_pairs, 1) * 4;
        DevBuf d_k(pb, s), d_v(pb, s), d_k2(pb, s), d_v2(pb, s);
        DevBuf d_cb((size_t)n_cells * 4, s), d_ce((size_t)n_cells * 4, s);
        CSL_CUDA(cudaMemsetAsync(d_cb.get(), 0, (size_t)n_cells * 4, s));
        CSL_CUDA(cudaMemsetAsync(d_ce.get(), 0, (size_t)n_cells * 4, s));
        k_rv_emit<<<grid_for(ne, 256), 256, 0, s>>>(rec, ne, g, d_off.as<int64_t>(),
                                                    d_k.as<uint32_t>(), d_v.as<uint32_t>());
        CSL_LAUNCH_CHECK("render cell pairs");
        int bits = 1;
        while (bits < 32 && (1ll << bits) < n_cells) ++bits;
        radix_sort_pairs(d_k.as<uint32_t>(), d_v.as<uint32_t>(), d_k2.as<uint32_t>(),
                         d_v2.as<uint32_t>(), n_pairs, bits, s);
        k_rv_bounds<<<grid_for(n_pairs, 256), 256, 0, s>>>(d_k.as<uint32_t>(), n_pairs,
                                                           d_cb.as<uint32_t>(), d_ce.as<uint32_t>());
        CSL_LAUNCH_CHECK("render cell bounds");
        k_rv_render<<<(unsigned)n_blocks, 128, 0, s>>>(rec, d_v.as<uint32_t>(), d_cb.as<uint32_t>(),
                                                       d_ce.as<uint32_t>(), g, c, depth);
        CSL_LAUNCH_CHECK("render rays");
        CSL_CUDA(cudaStreamSynchronize(s));
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
