// Device arrays handed to the caller. Host code only.
#include <mutex>
#include <unordered_map>

#include "common.cuh"

namespace csl {
namespace {

struct Pooled {
    int dev;   // the device whose pool holds the array
    size_t bytes;
};
std::mutex g_result_mu;
std::unordered_map<void*, Pooled> g_result_pooled;   // arrays that came from a pool
size_t g_result_bytes = 0;                           // their sum

}  // namespace

void* result_alloc(size_t bytes, cudaStream_t s, const char* what) {
    if (bytes == 0) bytes = 16;
    void* p = nullptr;
    int dev = 0;
    bool pool = bytes <= kResultPoolBytes && cudaGetDevice(&dev) == cudaSuccess;
    if (pool) {
        std::lock_guard<std::mutex> lk(g_result_mu);
        pool = g_result_bytes + bytes <= kResultPoolTotal;
        if (pool) g_result_bytes += bytes;
    }
    if (pool) {
        keep_pool_memory();
        if (cudaMallocAsync(&p, bytes, s) == cudaSuccess) {
            std::lock_guard<std::mutex> lk(g_result_mu);
            try {
                g_result_pooled[p] = Pooled{dev, bytes};
            } catch (...) {
                g_result_bytes -= bytes;
                cudaFreeAsync(p, s);
                throw;
            }
            return p;
        }
        cudaGetLastError();
        std::lock_guard<std::mutex> lk(g_result_mu);
        g_result_bytes -= bytes;
    }
    if (cudaMalloc(&p, bytes) != cudaSuccess) {
        cudaGetLastError();
        fail(CSL_ERR_OOM, what);
    }
    return p;
}

void result_free(void* p) {
    if (!p) return;
    Pooled a{-1, 0};
    {
        std::lock_guard<std::mutex> lk(g_result_mu);
        const auto it = g_result_pooled.find(p);
        if (it != g_result_pooled.end()) {
            a = it->second;
            g_result_pooled.erase(it);
            g_result_bytes -= a.bytes;
        }
    }
    if (a.dev < 0) {
        cudaFree(p);
        return;
    }
    // The caller may have made another device current since: wait for the one
    // that holds the array (any of its streams may still use it) and free the
    // array on that one's default stream.
    int cur = a.dev;
    cudaGetDevice(&cur);
    if (cur != a.dev) cudaSetDevice(a.dev);
    cudaDeviceSynchronize();
    cudaFreeAsync(p, 0);
    if (cur != a.dev) cudaSetDevice(cur);
}

}  // namespace csl
