// Vertex position optimisation for self-support (Sec. 5.3.2, Eq. 16-17).
//
// Every interior vertex of a tetrahedral mesh moves to lower
//   J(v) = sum_{e at v} r_e L_e g(theta_e) / sum_{e at v} r_e L_e     (Eq. 16)
// (theta_e = arccos |u_e . t_P|, Eq. 11; g of Eq. 12, 0 for theta <= alpha)
// inside the inscribed sphere of its star (Eq. 17). The paper visits the
// vertices one by one; here a greedy colouring (vertex order, smallest colour
// free among the neighbours) orders them colour by colour. Vertices of one
// colour share no edge, so each colour is one kernel launch with half a warp or a
// warp per vertex, and the result equals the sequential sweep in that order.
//
// A move goes along -grad J by step * tau0 (tau0: the smallest distance from
// the vertex's initial position o to the faces opposite it), halved up to
// `backtracks` times until the position lies in the ball |p - o| <= ball *
// tau0, every incident tetrahedron keeps its orientation and min_volume of its
// initial volume, and J decreases. Rounds repeat until nothing moves. Positions,
// gradients and sums are FP64 in one fixed order (the build compiles device code
// with --fmad=false); a trial's tests are screened in FP32 with error bounds and
// decided in FP64 where those leave them open, so that the moves are those of FP64.
#include <limits.h>
#include <math.h>

#include <algorithm>
#include <array>
#include <chrono>
#include <vector>

#include "common.cuh"

namespace csl {
namespace {

constexpr int kPoThreads = 128;
// k_po_move: one warp per block, so that the warps of a colour spread evenly
// over the SMs (864 warps of the FP64 pipe's work on 152 SMs: 42 us of the
// busiest SM's pipe with 6 warps, 57 us with two blocks of 4)
constexpr int kPoMoveThreads = 32;

struct PoConst {
    double tx, ty, tz, alpha;
    double a[6];
    double step, ball, min_volume;
    int32_t backtracks;
    float g2_max;   // bound of |g''| on [0, pi / 2], for the FP32 screening
};

// g(theta) of Eq. 12 and its derivative, by Horner (0, 0 for theta <= alpha).
__device__ __forceinline__ void g_dg(double th, const PoConst& c, double& g, double& dg) {
    g = 0.0;
    dg = 0.0;
    if (th <= c.alpha) return;
    for (int i = 5; i >= 0; --i) {
        dg = dg * th + g;
        g = g * th + c.a[i];
    }
}

// The G lanes (16 or 32) of a warp that work on one vertex.
template <int G>
struct Group {
    int lane;        // in the group
    unsigned mask;   // its lanes in the warp
    __device__ __forceinline__ Group() {
        const int l = threadIdx.x & 31;
        lane = l & (G - 1);
        mask = (G == 32 ? 0xffffffffu : 0xffffu) << (l & ~(G - 1));
    }
    __device__ __forceinline__ bool any(bool p) const { return (__ballot_sync(mask, p) & mask) != 0; }
    template <class T>
    __device__ __forceinline__ T from(T v, int src) const {
        return __shfl_sync(mask, v, src, G);
    }
    __device__ __forceinline__ float sum(float v) const {
#pragma unroll
        for (int o = G / 2; o > 0; o >>= 1) v += __shfl_xor_sync(mask, v, o, G);
        return v;
    }
};

// A group evaluates J(v) at (vx, vy, vz) over the vertex's edges [b, e) of the
// CSR: each lane computes the terms of its edges; then lane k takes component
// k of the sums (N, D and, with GRAD, the gradients of N and D) through shared
// memory, in edge order, the order of the sequential definition: one FP64
// addition per edge for all components together (the pipe takes 32 lanes as
// long as one). Every lane returns the same values. sm: G * (GRAD ? 8 : 2)
// doubles of the group's own.
template <int G, bool GRAD>
__device__ double group_J(const Group<G>& gr, double vx, double vy, double vz,
                          const int32_t* __restrict__ nbr, const double* __restrict__ rad,
                          int64_t b, int64_t e, const double* __restrict__ pos, const PoConst& c,
                          double* sm, double* grad) {
    constexpr int K = GRAD ? 8 : 2;
    const double tk[3] = {c.tx, c.ty, c.tz};
    double acc = 0.0;
    for (int64_t base = b; base < e; base += G) {
        const int64_t i = base + gr.lane;
        double t[8] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0};   // N, D, dN, dD
        bool live = false;
        if (i < e) {
            const int32_t w = nbr[i];
            const double r = rad[i];
            const double d[3] = {vx - pos[3 * (int64_t)w], vy - pos[3 * (int64_t)w + 1],
                                 vz - pos[3 * (int64_t)w + 2]};
            const double L = sqrt(d[0] * d[0] + d[1] * d[1] + d[2] * d[2]);
            if (L != 0.0) {
                live = true;
                const double s = d[0] * c.tx + d[1] * c.ty + d[2] * c.tz;
                const double cs = fmin(fabs(s) / L, 1.0);
                const double th = acos(cs);
                double g, dg;
                g_dg(th, c, g, dg);
                t[0] = r * L * g;
                t[1] = r * L;
                if (GRAD) {
                    const double dL[3] = {d[0] / L, d[1] / L, d[2] / L};
                    for (int k = 0; k < 3; ++k) t[5 + k] = r * dL[k];
                    if (g != 0.0 || dg != 0.0) {
                        const double sg = copysign(1.0, s);
                        const double s2 = sqrt(fmax(1.0 - cs * cs, 1e-300));
                        for (int k = 0; k < 3; ++k) {
                            const double dc = (sg * tk[k] - cs * dL[k]) / L;
                            const double dth = -dc / s2;
                            t[2 + k] = r * (dL[k] * g + L * dg * dth);
                        }
                    }
                }
            }
        }
        const int n = (int)min((int64_t)G, e - base);
        const unsigned live_mask =
            __ballot_sync(gr.mask, live) >> (G == 32 ? 0 : (threadIdx.x & 16));
#pragma unroll
        for (int k = 0; k < K; ++k) sm[k * G + gr.lane] = t[k];
        __syncwarp(gr.mask);
        if (gr.lane < K)
            for (int j = 0; j < n; ++j)   // edge order; a zero-length edge adds nothing
                if ((live_mask >> j) & 1u) acc += sm[gr.lane * G + j];
        __syncwarp(gr.mask);
    }
    const double N = gr.from(acc, 0), D = gr.from(acc, 1);
    if (GRAD) {
        for (int k = 0; k < 3; ++k) {
            const double dN = gr.from(acc, 2 + k), dD = gr.from(acc, 5 + k);
            grad[k] = D == 0.0 ? 0.0 : (dN * D - N * dD) / (D * D);
        }
    }
    return D == 0.0 ? 0.0 : N / D;
}

__device__ __forceinline__ double orient(const double* a, const double* b, const double* c,
                                         const double* d) {
    const double ax = b[0] - a[0], ay = b[1] - a[1], az = b[2] - a[2];
    const double bx = c[0] - a[0], by = c[1] - a[1], bz = c[2] - a[2];
    const double cx = d[0] - a[0], cy = d[1] - a[1], cz = d[2] - a[2];
    return ax * (by * cz - bz * cy) - ay * (bx * cz - bz * cx) + az * (bx * cy - by * cx);
}

__device__ __forceinline__ double plane_distance(const double* p, const double* a,
                                                 const double* b, const double* c) {
    const double ux = b[0] - a[0], uy = b[1] - a[1], uz = b[2] - a[2];
    const double wx = c[0] - a[0], wy = c[1] - a[1], wz = c[2] - a[2];
    const double nx = uy * wz - uz * wy, ny = uz * wx - ux * wz, nz = ux * wy - uy * wx;
    const double nn = sqrt(nx * nx + ny * ny + nz * nz);
    if (nn == 0.0) return 0.0;
    const double px = p[0] - a[0], py = p[1] - a[1], pz = p[2] - a[2];
    return fabs(px * nx + py * ny + pz * nz) / nn;
}

__constant__ int kFace[4][3] = {{1, 2, 3}, {0, 2, 3}, {0, 1, 3}, {0, 1, 2}};

// tau0 of every listed vertex (smallest distance to the faces opposite it)
// and vol0 of every tetrahedron, on the initial mesh.
__global__ void k_po_tau0(const int32_t* __restrict__ list, int64_t n, const double* __restrict__ pos,
                          const int4* __restrict__ tets, const int64_t* __restrict__ vt_off,
                          const int32_t* __restrict__ vt, double* __restrict__ tau0) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        const int32_t v = list[i];
        double best = INFINITY;
        for (int64_t q = vt_off[v]; q < vt_off[v + 1]; ++q) {
            const int32_t ti = vt[q] >> 2, k = vt[q] & 3;
            const int4 t = tets[ti];
            const int32_t id[4] = {t.x, t.y, t.z, t.w};
            const double d = plane_distance(pos + 3 * (int64_t)v, pos + 3 * (int64_t)id[kFace[k][0]],
                                            pos + 3 * (int64_t)id[kFace[k][1]],
                                            pos + 3 * (int64_t)id[kFace[k][2]]);
            best = fmin(best, d);
        }
        tau0[v] = best;
    }
}

__global__ void k_po_vol0(const int4* __restrict__ tets, int64_t n, const double* __restrict__ pos,
                          double* __restrict__ vol0) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        const int4 t = tets[i];
        vol0[i] = orient(pos + 3 * (int64_t)t.x, pos + 3 * (int64_t)t.y, pos + 3 * (int64_t)t.z,
                         pos + 3 * (int64_t)t.w);
    }
}

// A trial's tests in FP32, on offsets from the vertex's position p0 taken in
// FP64 and rounded once (relative error 2^-24; the step's offset 2^-23).
// Each returns +1 / -1 where the FP64 test must come out true / false whatever
// the rounding of this evaluation, 0 where it might not: then the FP64 test
// decides. FP64 runs at 1/64 of the FP32 rate here, and most trials are far
// from every bound.
struct Screen {
    // this lane's edge: offset p0 - neighbour and radius (r = 0: none)
    float ex, ey, ez, r;
    // this lane's tetrahedra (up to 2): the three other corners' offsets from
    // p0, the sign that turns their determinant into the oriented volume times
    // sign(vol0), and |vol0| min_volume
    float q[2][9], sign[2], least[2];
    int n_tets;
};

// |cand - o| <= rb?
__device__ __forceinline__ int screen_ball(const float (&w)[3], const float (&dl)[3], float rb) {
    const float x = w[0] + dl[0], y = w[1] + dl[1], z = w[2] + dl[2];
    const float dist = sqrtf(x * x + y * y + z * z);
    const float size = fabsf(w[0]) + fabsf(w[1]) + fabsf(w[2]) + fabsf(dl[0]) + fabsf(dl[1]) +
                       fabsf(dl[2]);
    if (!(size > 1e-15f && size < 1e15f)) return 0;   // squares in range
    const float m = 1e-6f * (size + rb);
    return dist + m < rb ? 1 : (dist - m > rb ? -1 : 0);
}

// Does tetrahedron k keep its orientation and its least volume? A product of
// three offsets errs by less than 3e-6 of the product of their sizes.
__device__ __forceinline__ int screen_volume(const Screen& S, int k, const float (&dl)[3]) {
    float e[9], size = 1.0f;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        float a = 0.0f;
#pragma unroll
        for (int x = 0; x < 3; ++x) {
            e[3 * i + x] = S.q[k][3 * i + x] - dl[x];
            a += fabsf(S.q[k][3 * i + x]) + fabsf(dl[x]);
        }
        size *= a;
    }
    const float det = e[0] * (e[4] * e[8] - e[5] * e[7]) - e[1] * (e[3] * e[8] - e[5] * e[6]) +
                      e[2] * (e[3] * e[7] - e[4] * e[6]);
    if (!(size > 1e-30f && size < 1e30f)) return 0;
    const float y = S.sign[k] * det, m = 3e-6f * size;
    return y - m > S.least[k] * (1.0f + 1e-6f) ? 1
                                                : (y + m < S.least[k] * (1.0f - 1e-6f) ? -1 : 0);
}

// J(cand) < J0? The angle's error follows from the offset's (acos moves by at
// most 1.5 e / sin near its argument, g by |g'| e + g'' e^2); an angle within
// its error of alpha, or an error above 1e-4, leaves the question open.
template <int G>
__device__ __forceinline__ int screen_J(const Group<G>& gr, const Screen& S, const float (&dl)[3],
                                        float J0, const PoConst& c) {
    float N = 0.0f, D = 0.0f, eN = 0.0f, eD = 0.0f;
    bool open = false;
    if (S.r > 0.0f) {
        const float x = S.ex + dl[0], y = S.ey + dl[1], z = S.ez + dl[2];
        const float L2 = x * x + y * y + z * z;
        const float L = sqrtf(L2);
        const float size = fabsf(S.ex) + fabsf(S.ey) + fabsf(S.ez) + fabsf(dl[0]) + fabsf(dl[1]) +
                           fabsf(dl[2]);
        const float ed = __fdividef(4e-7f * size, L);
        const float cs = fminf(
            __fdividef(fabsf(x * (float)c.tx + y * (float)c.ty + z * (float)c.tz), L), 1.0f);
        const float sin2 = fmaxf(1.0f - cs * cs, 0.0f);
        const float ecs = 2.0f * ed + 6e-7f;
        const float eth = (ecs < 0.25f * sin2 ? 1.5f * ecs * rsqrtf(sin2) : 1.6f * sqrtf(ecs)) +
                          1e-6f;
        const float th = acosf(cs), over = th - (float)c.alpha;
        const float rL = S.r * L;
        open = !(L2 > 1e-30f && L2 < 1e30f && rL > 1e-30f && rL < 1e30f && eth <= 1e-4f &&
                 fabsf(over) > eth);
        float g = 0.0f, dg = 0.0f, eg = 0.0f;
        if (over > 0.0f) {
            float size_g = 0.0f;   // sum |a_i| th^i: Horner rounds by less than 11 2^-24 of it
#pragma unroll
            for (int i = 5; i >= 0; --i) {
                dg = dg * th + g;
                g = g * th + (float)c.a[i];
                size_g = size_g * th + fabsf((float)c.a[i]);
            }
            eg = eth * (fabsf(dg) + eth * c.g2_max) + 1.5e-6f * size_g;
        }
        N = rL * g;
        D = rL;
        eN = rL * eg + fabsf(N) * (ed + 6e-6f);
        eD = rL * (ed + 6e-6f);
    }
    open = gr.any(open);
    N = gr.sum(N);
    D = gr.sum(D);
    eN = gr.sum(eN);
    eD = gr.sum(eD);
    if (open || !(eD < 0.1f * D)) return 0;
    const float J = N / D;
    const float m = 2.0f * (eN + fabsf(J) * eD) / D + 1e-6f * (fabsf(J) + fabsf(J0));
    return J + m < J0 ? 1 : (J - m > J0 ? -1 : 0);
}

// One colour: G lanes per vertex of the list (no two share an edge). The lanes
// share the edge terms and the incident tetrahedra's checks; the trials of the
// backtracking run in order. Bound by the FP64 pipe and its latency: the
// gradient and J at the vertex's position are FP64 (two vertices per warp where
// degrees allow), the trials' tests are screened in FP32 (of 373,000 values of
// J in a call on 93,750 tetrahedra 21,000 stay open). That call's 136 launches:
// 17.0 ms with a warp per vertex in FP64 throughout, 7.5 ms now.
//
// A vertex's move depends only on its own position and its neighbours' (all
// the vertices of its tetrahedra) besides constants; so a vertex that did not
// move at its last visit (calm_at: that colour step) and whose star has not
// moved since (moved_at of it and of its neighbours older than that step)
// would not move now either, and is skipped: the result of the sequential
// sweep exactly, without re-evaluating the calm part of the mesh.
template <int G>
__global__ void __launch_bounds__(kPoMoveThreads)
k_po_move(const int32_t* __restrict__ list, int64_t n, double* __restrict__ pos,
          const double* __restrict__ o, const double* __restrict__ tau0,
          const int64_t* __restrict__ e_off, const int32_t* __restrict__ nbr,
          const double* __restrict__ rad, const int64_t* __restrict__ vt_off,
          const int32_t* __restrict__ vt, const int4* __restrict__ tets,
          const double* __restrict__ vol0, PoConst c, int32_t step,
          int32_t* __restrict__ moved_at, int32_t* __restrict__ calm_at, unsigned int* moves) {
    __shared__ double s_terms[kPoMoveThreads / G][8 * G];
    const Group<G> gr;
    double* sm = s_terms[threadIdx.x / G];
    const int64_t groups = (int64_t)gridDim.x * (kPoMoveThreads / G);
    for (int64_t i = ((int64_t)blockIdx.x * kPoMoveThreads + threadIdx.x) / G; i < n; i += groups) {
        const int32_t v = list[i];
        const int64_t eb = e_off[v], ee = e_off[v + 1];
        const int32_t ca = calm_at[v];
        if (ca >= 0 && moved_at[v] < ca) {   // calm before: has the star moved since?
            bool moved = false;
            for (int64_t q = eb + gr.lane; q < ee; q += G) moved |= moved_at[nbr[q]] > ca;
            if (!gr.any(moved)) continue;
        }
        double* pv = pos + 3 * (int64_t)v;
        const double p0 = pv[0], p1 = pv[1], p2 = pv[2];
        double grad[3];
        const double J0 = group_J<G, true>(gr, p0, p1, p2, nbr, rad, eb, ee, pos, c, sm, grad);
        const double gn = sqrt(grad[0] * grad[0] + grad[1] * grad[1] + grad[2] * grad[2]);
        if (gn == 0.0) {
            if (gr.lane == 0) calm_at[v] = step;
            continue;
        }
        const double u[3] = {grad[0] / gn, grad[1] / gn, grad[2] / gn};
        const double* ov = o + 3 * (int64_t)v;
        const double rb = c.ball * tau0[v];
        const int64_t tb = vt_off[v], te = vt_off[v + 1];
        // the screening's data: an edge and up to two tetrahedra per lane
        const bool screened = ee - eb <= G && te - tb <= 2 * G;
        Screen S;
        S.r = 0.0f;
        S.n_tets = 0;
        if (screened) {
            if (eb + gr.lane < ee) {
                const double* pw = pos + 3 * (int64_t)nbr[eb + gr.lane];
                S.ex = (float)(p0 - pw[0]);
                S.ey = (float)(p1 - pw[1]);
                S.ez = (float)(p2 - pw[2]);
                S.r = (float)rad[eb + gr.lane];
            }
#pragma unroll
            for (int m = 0; m < 2; ++m) {
                const int64_t q = tb + gr.lane + m * G;
                if (q >= te) continue;
                S.n_tets = m + 1;
                const int32_t ti = vt[q] >> 2, k = vt[q] & 3;
                const int4 t = tets[ti];
                const int32_t id[4] = {t.x, t.y, t.z, t.w};
#pragma unroll
                for (int j = 0; j < 3; ++j) {
                    const double* pw = pos + 3 * (int64_t)id[kFace[k][j]];
                    S.q[m][3 * j] = (float)(pw[0] - p0);
                    S.q[m][3 * j + 1] = (float)(pw[1] - p1);
                    S.q[m][3 * j + 2] = (float)(pw[2] - p2);
                }
                // moving corner k to the front is an odd permutation for odd k
                const double v0 = vol0[ti];
                S.sign[m] = v0 == 0.0 ? NAN : (((k & 1) != 0) != (v0 < 0.0) ? -1.0f : 1.0f);
                S.least[m] = (float)(c.min_volume * fabs(v0));
            }
        }
        const float w[3] = {(float)(p0 - ov[0]), (float)(p1 - ov[1]), (float)(p2 - ov[2])};
        const float uf[3] = {(float)u[0], (float)u[1], (float)u[2]};
        bool went = false;
        const double s0 = c.step * tau0[v];
        float sf = (float)s0;
        for (int it = 0; it <= c.backtracks; ++it, sf *= 0.5f) {
            const float dl[3] = {-sf * uf[0], -sf * uf[1], -sf * uf[2]};
            // the FP64 candidate, where it is needed: s0 halved `it` times (exact)
            auto candidate = [&](double (&cand)[3]) {
                const double s = s0 * __hiloint2double((1023 - it) << 20, 0);
                cand[0] = p0 - s * u[0];
                cand[1] = p1 - s * u[1];
                cand[2] = p2 - s * u[2];
            };
            double cand[3];
            int in = screened ? screen_ball(w, dl, (float)rb) : 0;
            if (in == 0) {
                candidate(cand);
                const double dx = cand[0] - ov[0], dy = cand[1] - ov[1], dz = cand[2] - ov[2];
                in = sqrt(dx * dx + dy * dy + dz * dz) > rb ? -1 : 1;
            }
            if (in < 0) continue;
            int vol[2] = {1, 1};
            bool bad = false, open = !screened;
            if (screened) {
#pragma unroll
                for (int m = 0; m < 2; ++m)
                    if (m < S.n_tets) vol[m] = screen_volume(S, m, dl);
                bad = gr.any(vol[0] < 0 || vol[1] < 0);
                open = gr.any(vol[0] == 0 || vol[1] == 0);
            }
            if (bad) continue;
            if (open) {
                candidate(cand);
                bool ok = true;
                for (int64_t q = tb + gr.lane, m = 0; q < te; q += G, ++m) {
                    if (screened && vol[m] > 0) continue;
                    const int32_t ti = vt[q] >> 2, k = vt[q] & 3;
                    const int4 t = tets[ti];
                    const int32_t id[4] = {t.x, t.y, t.z, t.w};
                    const double* P[4];
                    for (int j = 0; j < 4; ++j) P[j] = j == k ? cand : pos + 3 * (int64_t)id[j];
                    const double vc = orient(P[0], P[1], P[2], P[3]);
                    ok = ok && vc * vol0[ti] > 0.0 && fabs(vc) >= c.min_volume * fabs(vol0[ti]);
                }
                if (gr.any(!ok)) continue;
            }
            int less = screened ? screen_J(gr, S, dl, (float)J0, c) : 0;
            if (less == 0) {
                candidate(cand);
                const double J1 = group_J<G, false>(gr, cand[0], cand[1], cand[2], nbr, rad, eb, ee,
                                                    pos, c, sm, nullptr);
                less = J1 < J0 ? 1 : -1;
            }
            if (less > 0) {
                __syncwarp(gr.mask);   // every lane has read pv before lane 0 writes it
                if (gr.lane == 0) {
                    candidate(cand);
                    pv[0] = cand[0];
                    pv[1] = cand[1];
                    pv[2] = cand[2];
                    moved_at[v] = step;
                    atomicAdd(moves, 1u);
                }
                went = true;
                break;
            }
        }
        if (!went && gr.lane == 0) calm_at[v] = step;
    }
}

// Gamma / Psi sums of Eq. 13-14 over the mesh's edges: per block in a fixed
// tree order, then the blocks in order (deterministic).
__global__ void k_po_metrics(const int2* __restrict__ edges, const double* __restrict__ er,
                             int64_t n, const double* __restrict__ pos, PoConst c,
                             double* __restrict__ partial) {
    __shared__ double s[4][kPoThreads];
    double acc[4] = {0.0, 0.0, 0.0, 0.0};   // r L g (unsupported), r L, L (supported), L
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        const int2 e = edges[i];
        const double* a = pos + 3 * (int64_t)e.x;
        const double* b = pos + 3 * (int64_t)e.y;
        const double d0 = b[0] - a[0], d1 = b[1] - a[1], d2 = b[2] - a[2];
        const double L = sqrt(d0 * d0 + d1 * d1 + d2 * d2);
        const double cs = L > 0.0 ? fmin(fabs(d0 * c.tx + d1 * c.ty + d2 * c.tz) / L, 1.0) : 0.0;
        const double th = acos(cs);
        double g, dg;
        g_dg(th, c, g, dg);
        if (th <= c.alpha)
            acc[2] += L;
        else
            acc[0] += er[i] * L * g;
        acc[1] += er[i] * L;
        acc[3] += L;
    }
    for (int k = 0; k < 4; ++k) s[k][threadIdx.x] = acc[k];
    __syncthreads();
    for (int w = kPoThreads / 2; w > 0; w >>= 1) {
        if ((int)threadIdx.x < w)
            for (int k = 0; k < 4; ++k) s[k][threadIdx.x] += s[k][threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0)
        for (int k = 0; k < 4; ++k) partial[4 * blockIdx.x + k] = s[k][0];
}

__global__ void k_po_metrics_total(const double* __restrict__ partial, int nb, double* out) {
    if (threadIdx.x != 0 || blockIdx.x != 0) return;
    double t[4] = {0.0, 0.0, 0.0, 0.0};
    for (int b = 0; b < nb; ++b)
        for (int k = 0; k < 4; ++k) t[k] += partial[4 * b + k];
    for (int k = 0; k < 4; ++k) out[k] = t[k];
}

void metrics(const DevBuf& edges, const DevBuf& er, int64_t n_e, const DevBuf& pos,
             const PoConst& c, DevBuf& partial, DevBuf& tot, cudaStream_t s, double* gamma,
             double* psi) {
    const int nb = 152 * 2;
    k_po_metrics<<<nb, kPoThreads, 0, s>>>(edges.as<int2>(), er.as<double>(), n_e, pos.as<double>(),
                                           c, partial.as<double>());
    CSL_LAUNCH_CHECK("support metrics partials");
    k_po_metrics_total<<<1, 32, 0, s>>>(partial.as<double>(), nb, tot.as<double>());
    CSL_LAUNCH_CHECK("support metrics total");
    double h[4];
    read_to_host(h, tot.get(), sizeof(h), s);
    *gamma = h[1] > 0.0 ? h[0] / h[1] : 0.0;
    *psi = h[3] > 0.0 ? 100.0 * h[2] / h[3] : 0.0;
}

template <class T>
void upload(DevBuf& d, const std::vector<T>& h, cudaStream_t s) {
    d.ensure(std::max<size_t>(h.size() * sizeof(T), 16), s);
    if (!h.empty())
        CSL_CUDA(cudaMemcpyAsync(d.get(), h.data(), h.size() * sizeof(T), cudaMemcpyHostToDevice, s));
}

}  // namespace
}  // namespace csl

using namespace csl;

extern "C" csl_status csl_support_optimize(float* nodes, int64_t n_nodes, const int32_t* tets,
                                           int64_t n_tets, const float* radius,
                                           const csl_po_params* p, void* stream,
                                           csl_po_result* out, int32_t* moves_per_round) {
    try {
        using clk = std::chrono::steady_clock;
        const auto t_start = clk::now();
        if (!p || !out) fail(CSL_ERR_INVALID_ARG, "NULL argument");
        if (n_nodes < 0 || n_tets < 0) fail(CSL_ERR_INVALID_ARG, "negative count");
        if ((n_nodes && !nodes) || (n_tets && !tets)) fail(CSL_ERR_INVALID_ARG, "NULL array");
        if (n_nodes >= (1ll << 30) || n_tets >= (1ll << 29))
            fail(CSL_ERR_CAPACITY, "too many nodes or tetrahedra");
        const double tn = sqrt(p->t_p[0] * p->t_p[0] + p->t_p[1] * p->t_p[1] + p->t_p[2] * p->t_p[2]);
        if (!(tn > 0.0) || !isfinite(tn)) fail(CSL_ERR_INVALID_ARG, "t_p must be a nonzero vector");
        if (!(p->alpha >= 0.0 && p->alpha <= M_PI / 2)) fail(CSL_ERR_INVALID_ARG, "alpha in [0, pi/2]");
        if (!(p->step > 0.0) || !(p->ball > 0.0) || !isfinite(p->step) || !isfinite(p->ball))
            fail(CSL_ERR_INVALID_ARG, "step and ball must be > 0");
        if (!(p->min_volume >= 0.0 && p->min_volume < 1.0))
            fail(CSL_ERR_INVALID_ARG, "min_volume in [0, 1)");
        if (p->backtracks < 0 || p->backtracks > 60) fail(CSL_ERR_INVALID_ARG, "backtracks in [0, 60]");
        if (p->max_rounds < 0 || p->max_rounds > 100000) fail(CSL_ERR_INVALID_ARG, "max_rounds in [0, 1e5]");
        for (int i = 0; i < 6; ++i)
            if (!isfinite(p->a[i])) fail(CSL_ERR_INVALID_ARG, "non-finite coefficient");
        for (int64_t i = 0; i < 3 * n_nodes; ++i)
            if (!isfinite(nodes[i])) fail(CSL_ERR_INVALID_ARG, "non-finite node coordinate");
        for (int64_t i = 0; i < 4 * n_tets; ++i)
            if (tets[i] < 0 || tets[i] >= n_nodes) fail(CSL_ERR_INVALID_ARG, "node index out of range");

        PoConst c;
        c.tx = p->t_p[0] / tn;
        c.ty = p->t_p[1] / tn;
        c.tz = p->t_p[2] / tn;
        c.alpha = p->alpha;
        for (int i = 0; i < 6; ++i) c.a[i] = p->a[i];
        c.step = p->step;
        c.ball = p->ball;
        c.min_volume = p->min_volume;
        c.backtracks = p->backtracks;
        double g2_max = 0.0;
        for (int i = 2; i < 6; ++i) g2_max += i * (i - 1) * fabs(p->a[i]) * pow(1.6, i - 2);
        c.g2_max = (float)g2_max;
        cudaStream_t s = (cudaStream_t)stream;

        // vertex -> (tetrahedron, corner)
        std::vector<int64_t> vt_off(n_nodes + 1, 0);
        for (int64_t i = 0; i < 4 * n_tets; ++i) ++vt_off[tets[i] + 1];
        for (int64_t v = 0; v < n_nodes; ++v) vt_off[v + 1] += vt_off[v];
        std::vector<int32_t> vt(vt_off[n_nodes]);
        {
            std::vector<int64_t> fill(vt_off.begin(), vt_off.end() - 1);
            for (int64_t t = 0; t < n_tets; ++t)
                for (int k = 0; k < 4; ++k) vt[fill[tets[4 * t + k]]++] = (int32_t)(t * 4 + k);
        }
        // per vertex, its distinct neighbours in ascending order (the edges are
        // then the pairs (v, w > v) in (v, w) order), and its boundary faces:
        // a face (v < b < c) is on the boundary when one tetrahedron has it
        std::vector<int64_t> e_off(n_nodes + 1, 0);
        std::vector<int32_t> nbr;
        nbr.reserve((size_t)n_tets * 4);
        std::vector<uint8_t> fixed(n_nodes, 0);
        std::vector<int64_t> up_off(n_nodes + 1, 0);   // edges (v, w > v) start at up_off[v]
        {
            std::vector<int32_t> tmp;
            std::vector<uint64_t> faces;
            std::vector<int64_t> stamp(n_nodes, -1);   // stamp[w] == v: w already listed for v
            for (int64_t v = 0; v < n_nodes; ++v) {
                tmp.clear();
                faces.clear();
                for (int64_t q = vt_off[v]; q < vt_off[v + 1]; ++q) {
                    const int32_t* tv = tets + 4 * (int64_t)(vt[q] >> 2);
                    const int k = vt[q] & 3;
                    for (int j = 0; j < 4; ++j)
                        if (j != k && tv[j] != v && stamp[tv[j]] != v) {
                            stamp[tv[j]] = v;
                            tmp.push_back(tv[j]);
                        }
                    for (int f = 0; f < 4; ++f) {   // faces containing v as their smallest id
                        if (f == k) continue;
                        int32_t o[2];
                        int m = 0;
                        bool smallest = true;
                        for (int j = 0; j < 4; ++j) {
                            if (j == f || j == k) continue;
                            o[m++] = tv[j];
                            smallest = smallest && tv[j] > v;
                        }
                        if (smallest)
                            faces.push_back(((uint64_t)(uint32_t)std::min(o[0], o[1]) << 32) |
                                            (uint32_t)std::max(o[0], o[1]));
                    }
                }
                std::sort(tmp.begin(), tmp.end());
                nbr.insert(nbr.end(), tmp.begin(), tmp.end());
                e_off[v + 1] = (int64_t)nbr.size();
                up_off[v + 1] = up_off[v] + (int64_t)(tmp.end() - std::upper_bound(tmp.begin(), tmp.end(), (int32_t)v));
                std::sort(faces.begin(), faces.end());
                for (size_t i = 0; i < faces.size();) {
                    size_t j = i;
                    while (j < faces.size() && faces[j] == faces[i]) ++j;
                    if (j - i == 1) {
                        fixed[v] = 1;
                        fixed[(int32_t)(faces[i] >> 32)] = 1;
                        fixed[(int32_t)(faces[i] & 0xffffffffu)] = 1;
                    }
                    i = j;
                }
            }
        }
        const int64_t n_e = up_off[n_nodes];
        std::vector<int2> h_edges(n_e);
        std::vector<double> h_er(n_e);
        for (int64_t v = 0; v < n_nodes; ++v) {
            int64_t id = up_off[v];
            for (int64_t q = e_off[v]; q < e_off[v + 1]; ++q)
                if (nbr[q] > v) {
                    h_edges[id] = make_int2((int32_t)v, nbr[q]);
                    h_er[id] = radius ? (double)radius[id] : 1.0;
                    if (!(h_er[id] > 0.0) || !isfinite(h_er[id]))
                        fail(CSL_ERR_INVALID_ARG, "radius must be > 0");
                    ++id;
                }
        }
        // the radius of every (vertex, neighbour) entry: its edge is (min, max)
        std::vector<double> rad(nbr.size());
        for (int64_t v = 0; v < n_nodes; ++v)
            for (int64_t q = e_off[v]; q < e_off[v + 1]; ++q) {
                const int32_t w = nbr[q];
                const int32_t a = std::min((int32_t)v, w), b = std::max((int32_t)v, w);
                const int32_t* lo = nbr.data() + e_off[a];
                const int32_t* hi = nbr.data() + e_off[a + 1];
                const int32_t* first_up = std::upper_bound(lo, hi, a);
                const int64_t rank = std::lower_bound(first_up, hi, b) - first_up;
                rad[q] = h_er[up_off[a] + rank];
            }
        // greedy colouring in vertex order
        std::vector<int32_t> col(n_nodes, -1);
        int32_t n_col = 0;
        {
            std::vector<int64_t> seen;   // seen[c] == v: colour c taken by a neighbour of v
            for (int64_t v = 0; v < n_nodes; ++v) {
                for (int64_t q = e_off[v]; q < e_off[v + 1]; ++q) {
                    const int32_t cw = col[nbr[q]];
                    if (cw >= 0) {
                        if ((size_t)cw >= seen.size()) seen.resize(cw + 1, -1);
                        seen[cw] = v;
                    }
                }
                int32_t cc = 0;
                while ((size_t)cc < seen.size() && seen[cc] == v) ++cc;
                col[v] = cc;
                n_col = std::max(n_col, cc + 1);
            }
        }
        std::vector<int64_t> col_off(n_col + 1, 0);
        for (int64_t v = 0; v < n_nodes; ++v)
            if (!fixed[v]) ++col_off[col[v] + 1];
        for (int32_t k = 0; k < n_col; ++k) col_off[k + 1] += col_off[k];
        std::vector<int32_t> list(col_off[n_col]);
        {
            std::vector<int64_t> fill(col_off.begin(), col_off.end() - 1);
            for (int64_t v = 0; v < n_nodes; ++v)
                if (!fixed[v]) list[fill[col[v]]++] = (int32_t)v;
        }

        const double host_ms =
            std::chrono::duration<double, std::milli>(clk::now() - t_start).count();
        std::vector<double> h_pos(3 * n_nodes);
        for (int64_t i = 0; i < 3 * n_nodes; ++i) h_pos[i] = (double)nodes[i];
        std::vector<int4> h_tets(n_tets);
        for (int64_t t = 0; t < n_tets; ++t)
            h_tets[t] = make_int4(tets[4 * t], tets[4 * t + 1], tets[4 * t + 2], tets[4 * t + 3]);
        DevBuf d_pos, d_o, d_tau, d_eoff, d_nbr, d_rad, d_vtoff, d_vt, d_tets, d_vol0, d_list;
        DevBuf d_edges, d_er, d_part((size_t)152 * 2 * 4 * sizeof(double), s), d_tot(64, s);
        DevBuf d_moves(16, s);
        // colour step of each vertex's last move and of its last visit without one
        DevBuf d_moved_at(std::max<size_t>((size_t)n_nodes * 4, 16), s),
            d_calm_at(std::max<size_t>((size_t)n_nodes * 4, 16), s);
        CSL_CUDA(cudaMemsetAsync(d_moved_at.get(), 0xff, d_moved_at.size(), s));
        CSL_CUDA(cudaMemsetAsync(d_calm_at.get(), 0xff, d_calm_at.size(), s));
        upload(d_pos, h_pos, s);
        upload(d_o, h_pos, s);
        upload(d_eoff, e_off, s);
        upload(d_nbr, nbr, s);
        upload(d_rad, rad, s);
        upload(d_vtoff, vt_off, s);
        upload(d_vt, vt, s);
        upload(d_tets, h_tets, s);
        upload(d_list, list, s);
        upload(d_edges, h_edges, s);
        upload(d_er, h_er, s);
        d_tau.ensure(std::max<size_t>((size_t)n_nodes * 8, 16), s);
        d_vol0.ensure(std::max<size_t>((size_t)n_tets * 8, 16), s);
        const int64_t n_list = (int64_t)list.size();
        if (n_list) {
            k_po_tau0<<<grid_for(n_list, kPoThreads), kPoThreads, 0, s>>>(
                d_list.as<int32_t>(), n_list, d_pos.as<double>(), d_tets.as<int4>(),
                d_vtoff.as<int64_t>(), d_vt.as<int32_t>(), d_tau.as<double>());
            CSL_LAUNCH_CHECK("inscribed radii");
        }
        if (n_tets) {
            k_po_vol0<<<grid_for(n_tets, kPoThreads), kPoThreads, 0, s>>>(
                d_tets.as<int4>(), n_tets, d_pos.as<double>(), d_vol0.as<double>());
            CSL_LAUNCH_CHECK("initial volumes");
        }
        // two vertices per warp where every vertex's edges fit 16 lanes and its
        // tetrahedra two per lane (the interior of a Kuhn mesh: 14 and 24)
        bool half_warps = true;
        for (int64_t i = 0; i < n_list && half_warps; ++i) {
            const int32_t v = list[i];
            half_warps = e_off[v + 1] - e_off[v] <= 16 && vt_off[v + 1] - vt_off[v] <= 32;
        }
        csl_po_result r = {};
        r.n_colours = n_col;
        metrics(d_edges, d_er, n_e, d_pos, c, d_part, d_tot, s, &r.gamma_before, &r.psi_before);
        for (int32_t round = 0; round < p->max_rounds && n_list; ++round) {
            CSL_CUDA(cudaMemsetAsync(d_moves.get(), 0, 4, s));
            for (int32_t k = 0; k < n_col; ++k) {
                const int64_t b = col_off[k], n = col_off[k + 1] - b;
                if (!n) continue;
                auto move = half_warps ? k_po_move<16> : k_po_move<32>;
                move<<<grid_for(n * (half_warps ? 16 : 32), kPoMoveThreads, INT_MAX), kPoMoveThreads, 0, s>>>(
                    d_list.as<int32_t>() + b, n, d_pos.as<double>(), d_o.as<double>(),
                    d_tau.as<double>(), d_eoff.as<int64_t>(), d_nbr.as<int32_t>(),
                    d_rad.as<double>(), d_vtoff.as<int64_t>(), d_vt.as<int32_t>(),
                    d_tets.as<int4>(), d_vol0.as<double>(), c, round * n_col + k,
                    d_moved_at.as<int32_t>(), d_calm_at.as<int32_t>(), d_moves.as<unsigned int>());
                CSL_LAUNCH_CHECK("vertex moves");
            }
            unsigned int moved = 0;
            read_to_host(&moved, d_moves.get(), 4, s);
            if (moves_per_round) moves_per_round[round] = (int32_t)moved;
            r.moves += moved;
            ++r.rounds;
            if (moved == 0) break;
        }
        metrics(d_edges, d_er, n_e, d_pos, c, d_part, d_tot, s, &r.gamma_after, &r.psi_after);
        if (n_nodes) read_to_host(h_pos.data(), d_pos.get(), h_pos.size() * 8, s);
        for (int64_t i = 0; i < 3 * n_nodes; ++i) nodes[i] = (float)h_pos[i];
        r.host_ms = host_ms;
        r.wall_ms = std::chrono::duration<double, std::milli>(clk::now() - t_start).count();
        *out = r;
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
