// Stable least-significant-digit radix sort of (uint32 key, uint32 value)
// pairs, 8 bits per pass. Each pass: a per-tile digit histogram, a
// device-wide scan of the digit-major histogram table, then a scatter in
// which every tile is put into digit order in shared memory first, equal digits
// in input order, so equal keys keep their input order (the sort is
// deterministic).
#include "common.cuh"

namespace csl {
namespace {

constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;
constexpr int kItems = 16;
constexpr int kTile = kThreads * kItems;
constexpr int kRadix = 256;

__global__ void __launch_bounds__(kThreads) k_hist(const uint32_t* __restrict__ keys, int64_t n,
                                                   int shift, uint32_t* __restrict__ hist,
                                                   int64_t n_tiles) {
    __shared__ uint32_t h[kRadix];
    h[threadIdx.x] = 0;
    __syncthreads();
    int64_t base = (int64_t)blockIdx.x * kTile;
#pragma unroll 4
    for (int i = 0; i < kItems; ++i) {
        int64_t idx = base + (int64_t)i * kThreads + threadIdx.x;
        if (idx < n) atomicAdd(&h[(keys[idx] >> shift) & 0xffu], 1u);
    }
    __syncthreads();
    // digit-major: all tiles of digit 0, then digit 1, ...
    hist[(int64_t)threadIdx.x * n_tiles + blockIdx.x] = h[threadIdx.x];
}

// A tile in shared memory: the pairs in digit order and the counters.
struct TileSmem {
    uint32_t cnt[kWarps][kRadix];   // per warp: items of each digit, then their offsets
    uint32_t start[kRadix];         // first place of each digit in the tile
    uint32_t warp_tot[kWarps];
    uint32_t key[kTile], val[kTile];
};

// Puts a tile's pairs into digit order in shared memory, equal digits in input
// order: thread t of warp w holds items w * 32 kItems + 32 i + lane (key[i],
// val[i]; those from `count` on do not exist). Every warp ranks its own items
// round by round against its own counters, so the block meets only for the
// offsets of the warps and digits. All threads; ends synchronised.
__device__ __forceinline__ void sort_tile(TileSmem& sm, const uint32_t (&key)[kItems],
                                          const uint32_t (&val)[kItems], int count, int shift) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned lt_mask = (1u << lane) - 1u;
    const int first = warp * 32 * kItems + lane;
#pragma unroll
    for (int w = 0; w < kWarps; ++w) sm.cnt[w][threadIdx.x] = 0;
    __syncthreads();
    uint32_t rank[kItems];
    uint32_t* cnt = sm.cnt[warp];
#pragma unroll
    for (int i = 0; i < kItems; ++i) {
        const bool valid = first + 32 * i < count;
        // invalid lanes get a digit of their own (256) that matches no real one
        const uint32_t digit = valid ? ((key[i] >> shift) & 0xffu) : 256u;
        const unsigned peers = __match_any_sync(0xffffffffu, digit);
        const uint32_t old = valid ? cnt[digit] : 0u;
        rank[i] = old + __popc(peers & lt_mask);
        __syncwarp();
        if (valid && (peers & lt_mask) == 0) cnt[digit] = old + __popc(peers);
        __syncwarp();
    }
    __syncthreads();
    {   // digit threadIdx.x: exclusive offsets over the warps, then over the digits
        uint32_t acc = 0;
#pragma unroll
        for (int w = 0; w < kWarps; ++w) {
            const uint32_t c = sm.cnt[w][threadIdx.x];
            sm.cnt[w][threadIdx.x] = acc;
            acc += c;
        }
        uint32_t inc = acc;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t t = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += t;
        }
        if (lane == 31) sm.warp_tot[warp] = inc;
        __syncthreads();
        uint32_t before = inc - acc;
        for (int w = 0; w < warp; ++w) before += sm.warp_tot[w];
        sm.start[threadIdx.x] = before;
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < kItems; ++i)
        if (first + 32 * i < count) {
            const uint32_t d = (key[i] >> shift) & 0xffu;
            const uint32_t p = sm.start[d] + cnt[d] + rank[i];
            sm.key[p] = key[i];
            sm.val[p] = val[i];
        }
    __syncthreads();
}

// One tile per block: into digit order in shared memory, then out to the
// digits' places, neighbouring threads writing neighbouring items of a digit.
// Bound by the ranking's chain through shared memory: the binner's 32 passes for
// 103 million struts take 3.9 ms, 5.0 with items written straight from their
// ranks and a barrier of the block for every 256 of them; 3 passes over the
// 7 million pairs of a depth image 0.26 ms, 0.36 before.
__global__ void __launch_bounds__(kThreads) k_scatter(const uint32_t* __restrict__ keys_in,
                                                      const uint32_t* __restrict__ vals_in,
                                                      uint32_t* __restrict__ keys_out,
                                                      uint32_t* __restrict__ vals_out, int64_t n,
                                                      int shift,
                                                      const uint32_t* __restrict__ hist_scan,
                                                      int64_t n_tiles) {
    __shared__ TileSmem sm;
    __shared__ uint32_t gbase[kRadix];
    const int64_t base = (int64_t)blockIdx.x * kTile;
    const int count = (int)min((int64_t)kTile, n - base);
    const int first = (threadIdx.x >> 5) * 32 * kItems + (threadIdx.x & 31);
    uint32_t key[kItems], val[kItems];
#pragma unroll
    for (int i = 0; i < kItems; ++i) {
        const bool valid = first + 32 * i < count;
        key[i] = valid ? keys_in[base + first + 32 * i] : 0u;
        val[i] = valid ? vals_in[base + first + 32 * i] : 0u;
    }
    const uint32_t g = hist_scan[(int64_t)threadIdx.x * n_tiles + blockIdx.x];
    sort_tile(sm, key, val, count, shift);
    gbase[threadIdx.x] = g - sm.start[threadIdx.x];
    __syncthreads();
    for (int t = threadIdx.x; t < count; t += kThreads) {
        const uint32_t k = sm.key[t];
        const uint32_t o = gbase[(k >> shift) & 0xffu] + (uint32_t)t;
        keys_out[o] = k;
        vals_out[o] = sm.val[t];
    }
}

// At most one tile of pairs: every pass in one launch, in place (a pass over the
// grid is three launches of 2 to 3 us whatever the count).
__global__ void __launch_bounds__(kThreads) k_sort_one(uint32_t* __restrict__ keys,
                                                       uint32_t* __restrict__ vals, int count,
                                                       int passes) {
    __shared__ TileSmem sm;
    const int first = (threadIdx.x >> 5) * 32 * kItems + (threadIdx.x & 31);
    uint32_t key[kItems], val[kItems];
    for (int p = 0; p < passes; ++p) {
#pragma unroll
        for (int i = 0; i < kItems; ++i) {
            const int t = first + 32 * i;
            const bool valid = t < count;
            key[i] = valid ? (p ? sm.key[t] : keys[t]) : 0u;
            val[i] = valid ? (p ? sm.val[t] : vals[t]) : 0u;
        }
        __syncthreads();
        sort_tile(sm, key, val, count, 8 * p);
    }
    for (int t = threadIdx.x; t < count; t += kThreads) {
        keys[t] = sm.key[t];
        vals[t] = sm.val[t];
    }
}

}  // namespace

void radix_sort_pairs(uint32_t* keys, uint32_t* vals, uint32_t* tmp_keys, uint32_t* tmp_vals,
                      int64_t n, int key_bits, cudaStream_t s) {
    if (n <= 1 || key_bits <= 0) return;
    if (n > (int64_t)0xffffffffLL) fail(CSL_ERR_CAPACITY, "radix sort: more than 2^32 elements");
    if (n <= kTile) {
        k_sort_one<<<1, kThreads, 0, s>>>(keys, vals, (int)n, (key_bits + 7) / 8);
        CSL_LAUNCH_CHECK("radix one tile");
        return;
    }
    int64_t n_tiles = ceil_div(n, kTile);
    DevBuf hist((size_t)kRadix * n_tiles * sizeof(uint32_t), s);
    int passes = (key_bits + 7) / 8;
    uint32_t *ki = keys, *vi = vals, *ko = tmp_keys, *vo = tmp_vals;
    for (int p = 0; p < passes; ++p) {
        int shift = 8 * p;
        k_hist<<<(unsigned)n_tiles, kThreads, 0, s>>>(ki, n, shift, hist.as<uint32_t>(), n_tiles);
        CSL_LAUNCH_CHECK("radix hist");
        exclusive_scan_u32(hist.as<uint32_t>(), hist.as<uint32_t>(), kRadix * n_tiles, nullptr, s);
        k_scatter<<<(unsigned)n_tiles, kThreads, 0, s>>>(ki, vi, ko, vo, n, shift,
                                                         hist.as<uint32_t>(), n_tiles);
        CSL_LAUNCH_CHECK("radix scatter");
        uint32_t* t;
        t = ki; ki = ko; ko = t;
        t = vi; vi = vo; vo = t;
    }
    if (ki != keys) {   // odd number of passes: copy back
        CSL_CUDA(cudaMemcpyAsync(keys, ki, n * sizeof(uint32_t), cudaMemcpyDeviceToDevice, s));
        CSL_CUDA(cudaMemcpyAsync(vals, vi, n * sizeof(uint32_t), cudaMemcpyDeviceToDevice, s));
    }
}

}  // namespace csl

extern "C" csl_status csl_debug_sort_pairs(uint32_t* keys, uint32_t* vals, int64_t n,
                                           int32_t key_bits, void* stream) {
    try {
        if (!keys || !vals || n < 0 || key_bits < 1 || key_bits > 32)
            csl::fail(CSL_ERR_INVALID_ARG, "device arrays, n >= 0 and key_bits in [1, 32]");
        cudaStream_t s = (cudaStream_t)stream;
        const size_t bytes = (size_t)(n > 0 ? n : 1) * 4;
        csl::DevBuf tk(bytes, s), tv(bytes, s);
        csl::radix_sort_pairs(keys, vals, tk.as<uint32_t>(), tv.as<uint32_t>(), n, key_bits, s);
        CSL_CUDA(cudaStreamSynchronize(s));
        return CSL_OK;
    } catch (const csl::Error& e) {
        csl::set_last_error(e.what());
        return e.code;
    } catch (const std::exception& e) {
        csl::set_last_error(e.what());
        return CSL_ERR_CUDA;
    }
}
