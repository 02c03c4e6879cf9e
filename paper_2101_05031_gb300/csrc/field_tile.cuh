// Device helpers shared by the field kernels, the volume-fraction adjoint and the
// ray caster: bulk copies, one edge record in a tile's frame, the per-warp cull
// mask of the block kernel, and the closed-form segment integral (Eq. 7) by 3-point
// Gauss-Legendre on the clipped interval.
#pragma once

#include "lattice.cuh"

namespace csl {

constexpr int kTileWarps = 8;   // blocks of 8 x 4 pixels in a tile, a warp each (or for two)

struct TileCull {
    float fpx, fdz;      // pixel size, layer spacing (float)
    float cull;          // R plus rounding slack
    float cull_line2;    // (cull + half-diagonal of a warp's pixel block)^2
    float inv_R4;
};

// ---- bulk copy (TMA) into shared memory, completion on an mbarrier ----
__device__ __forceinline__ uint32_t smem_addr(const void* p) {
    return (uint32_t)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(bar)), "r"(count)
                 : "memory");
}
// makes the initialised barrier visible to the asynchronous (bulk copy) proxy
__device__ __forceinline__ void fence_mbar_init() {
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
// orders this thread's (and, after a barrier, the block's) ordinary shared
// memory accesses before the bulk copy's writes
__device__ __forceinline__ void fence_proxy_async_smem() {
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}
// one arrival that also expects `bytes` of transactions, then the copy of
// `bytes` (a multiple of 16, both addresses 16-byte aligned) from global memory
__device__ __forceinline__ void bulk_load(void* dst, const void* src, uint32_t bytes,
                                          uint64_t* bar) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(bar)),
                 "r"(bytes)
                 : "memory");
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::
            "r"(smem_addr(dst)),
        "l"(src), "r"(bytes), "r"(smem_addr(bar))
        : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
    uint32_t done;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
        " selp.u32 %0, 1, 0, p;\n}" : "=r"(done) : "r"(smem_addr(bar)), "r"(parity) : "memory");
    return done != 0;
}
// Waits for the barrier's phase `parity` to complete, at most kWaitLimit polls
// (each may suspend the thread for a while); false when it gave up.
constexpr uint32_t kWaitLimit = 1u << 22;
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity,
                                          uint32_t limit = kWaitLimit) {
    for (uint32_t i = 0; i < limit; ++i)
        if (mbar_try_wait(bar, parity)) return true;
    return false;
}

__device__ __forceinline__ float sqrt_approx(float x) {
    float r;
    asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// Loads record rp in coordinates relative to the tile's corner and the slab's
// first layer plane (each given as a (hi, lo) float pair): A = (ax, ay, az, ux),
// B = (uy, uz, len, w / R^4).
__device__ __forceinline__ void load_record(const csl_rec* rp_rec, float oxh, float oxl, float oyh,
                                            float oyl, float ozh, float ozl, float inv_R4,
                                            float4& A, float4& B) {
    const float4* rp = reinterpret_cast<const float4*>(rp_rec);
    const float4 r0 = __ldg(rp), r1 = __ldg(rp + 1);
    A = make_float4((r0.x - oxh) - oxl, (r0.y - oyh) - oyl, (r0.z - ozh) - ozl, r0.w);
    B = make_float4(r1.x, r1.y, r1.z, r1.w * inv_R4);
}

// The warps of one layer l whose block of 8 x 4 PX pixels the staged edge (A, B)
// may reach, i.e. the block meets the xy box of the edge clipped to |z - z_l| <=
// cull grown by cull, and its centre lies within cull + half its diagonal of the
// edge's line (c.cull_line2): bit w set for warp w of the tile's 8 / PX.
template <int PX>
__device__ __forceinline__ uint32_t cull_layer(const float4 A, const float4 B, int l,
                                               const TileCull& c) {
    const float ax = A.x, ay = A.y, az = A.z, ux = A.w, uy = B.x, uz = B.y, len = B.z;
    const float zl = (float)l * c.fdz;
    float t_lo = 0.0f, t_hi = len;
    if (uz > 1e-12f) {
        const float inv_uz = 1.0f / uz;
        t_lo = fmaxf((zl - c.cull - az) * inv_uz, 0.0f);
        t_hi = fminf((zl + c.cull - az) * inv_uz, len);
    } else if (fabsf(az - zl) > c.cull) {
        return 0u;
    }
    if (t_lo > t_hi) return 0u;
    const float xa = fmaf(t_lo, ux, ax), xb = fmaf(t_hi, ux, ax);
    const float ya = fmaf(t_lo, uy, ay), yb = fmaf(t_hi, uy, ay);
    const float xmin = fminf(xa, xb) - c.cull, xmax = fmaxf(xa, xb) + c.cull;
    const float ymin = fminf(ya, yb) - c.cull, ymax = fmaxf(ya, yb) + c.cull;
    const float qz = zl - az;
    uint32_t m = 0;
#pragma unroll
    for (int w = 0; w < kTileWarps / PX; ++w) {
        const float rx0 = ((float)((w & 1) * 8) + 0.5f) * c.fpx;
        const float rx1 = ((float)((w & 1) * 8) + 7.5f) * c.fpx;
        const float ry0 = ((float)((w >> 1) * 4 * PX) + 0.5f) * c.fpx;
        const float ry1 = ((float)((w >> 1) * 4 * PX) + (4 * PX - 0.5f)) * c.fpx;
        if (xmax >= rx0 && xmin <= rx1 && ymax >= ry0 && ymin <= ry1) {
            const float qx = 0.5f * (rx0 + rx1) - ax;
            const float qy = 0.5f * (ry0 + ry1) - ay;
            const float t = fmaf(qz, uz, fmaf(qy, uy, qx * ux));
            const float ex = fmaf(-t, ux, qx), ey = fmaf(-t, uy, qy);
            const float ez = fmaf(-t, uz, qz);
            if (fmaf(ez, ez, fmaf(ey, ey, ex * ex)) <= c.cull_line2) m |= 1u << w;
        }
    }
    return m;
}

// Byte l of `bytes` holds the warp bits of layer l; returns warp w's layer
// bits (bit l = layer l).
__device__ __forceinline__ uint32_t warp_layers(uint64_t bytes, int w) {
    const uint64_t b = (bytes >> w) & 0x0101010101010101ull;
    return (uint32_t)((b * 0x0102040810204080ull) >> 56);
}

// In the frame of the edge: p - v_s = t0 u + e, h2 = max(R^2 - |e|^2, 0),
// w = sqrt(h2); the edge covers tau = t - t0 in [tau1, tau2] =
// [max(-t0, -w), min(L - t0, w)] and the kernel there is (h2 - tau^2)^2 / R^4.
// Returns R^4 I = integral of (h2 - tau^2)^2 over [tau1, tau2], by 3-point
// Gauss-Legendre (exact for this degree-4 polynomial, all terms >= 0). With
// m = (tau1 + tau2)/2, h = (tau2 - tau1)/2, c = h2 - m^2, A = c - 0.6 h^2 and
// B = 2 m h sqrt(0.6): R^4 I = h [(10/9)(A^2 + B^2) + (8/9) c^2].
__device__ __forceinline__ float segment_term_R4(float t0, float h2, float len) {
    const float w = sqrt_approx(h2);
    const float tau1 = fmaxf(-t0, -w);
    const float tau2 = fminf(len - t0, w);
    const float d = fmaxf(tau2 - tau1, 0.0f);   // 2 h
    const float s = tau2 + tau1;                 // 2 m
    const float cc = fmaf(-0.25f * s, s, h2);    // h2 - m^2
    const float d15 = 0.15f * d;
    const float Av = fmaf(-d15, d, cc);          // h2 - m^2 - 0.6 h^2
    const float ds = d15 * s;
    const float B2 = ds * (d * s);               // (2 m h sqrt(0.6))^2 = 0.15 d^2 s^2
    return d * fmaf(5.0f / 9.0f, fmaf(Av, Av, B2), (4.0f / 9.0f) * (cc * cc));
}

}  // namespace csl
