// scratch.cu -- device and page-locked host blocks of the stateless calls.
#include "scratch.h"

#include <mutex>
#include <vector>

namespace nb {

namespace {

constexpr int kMaxDevices = 64;
constexpr unsigned long long kKeepDevice = 32ull << 20;
constexpr size_t kKeepHost = 4, kKeepHostBytes = 8u << 20;

struct HostBlock {
    char *p;
    size_t bytes;
};

std::mutex g_lock;
cudaMemPool_t g_pool[kMaxDevices];
std::vector<HostBlock> *g_host = nullptr;  // leaked: no order of destruction at exit to mind

cudaError_t pool_of(int dev, cudaMemPool_t *out) {
    std::lock_guard<std::mutex> hold(g_lock);
    if (!g_pool[dev]) {
        cudaMemPoolProps props{};
        props.allocType = cudaMemAllocationTypePinned;
        props.location.type = cudaMemLocationTypeDevice;
        props.location.id = dev;
        cudaError_t e = cudaMemPoolCreate(&g_pool[dev], &props);
        if (e != cudaSuccess) {
            g_pool[dev] = nullptr;
            return e;
        }
        unsigned long long keep = kKeepDevice;
        e = cudaMemPoolSetAttribute(g_pool[dev], cudaMemPoolAttrReleaseThreshold, &keep);
        if (e != cudaSuccess) return e;
    }
    *out = g_pool[dev];
    return cudaSuccess;
}

}  // namespace

cudaError_t Scratch::take(size_t dev_bytes, size_t host_bytes) {
    if (dev_bytes) {
        int d = 0;
        cudaError_t e = cudaGetDevice(&d);
        if (e != cudaSuccess) return e;
        if (d < 0 || d >= kMaxDevices) return cudaErrorInvalidDevice;
        cudaMemPool_t pool = nullptr;
        e = pool_of(d, &pool);
        void *p = nullptr;
        if (e == cudaSuccess) e = cudaMallocFromPoolAsync(&p, dev_bytes, pool, stream_);
        if (e != cudaSuccess) return e;
        dev = static_cast<char *>(p);
    }
    if (host_bytes) {
        {
            std::lock_guard<std::mutex> hold(g_lock);
            if (g_host)
                for (size_t k = 0; k < g_host->size(); k++)
                    if ((*g_host)[k].bytes >= host_bytes) {
                        host = (*g_host)[k].p;
                        host_bytes_ = (*g_host)[k].bytes;
                        (*g_host)[k] = g_host->back();
                        g_host->pop_back();
                        break;
                    }
        }
        if (!host) {
            void *p = nullptr;
            const cudaError_t e = cudaHostAlloc(&p, host_bytes, cudaHostAllocPortable | cudaHostAllocMapped);
            if (e != cudaSuccess) return e;
            host = static_cast<char *>(p);
            host_bytes_ = host_bytes;
        }
    }
    return cudaSuccess;
}

cudaError_t Scratch::finish() {
    finished_ = true;
    return cudaStreamSynchronize(stream_);
}

Scratch::~Scratch() {
    if (!finished_) cudaStreamSynchronize(stream_);
    if (dev) cudaFreeAsync(dev, stream_);
    if (!host) return;
    {
        std::lock_guard<std::mutex> hold(g_lock);
        if (!g_host) g_host = new std::vector<HostBlock>();
        if (g_host->size() < kKeepHost && host_bytes_ <= kKeepHostBytes) {
            g_host->push_back({host, host_bytes_});
            host = nullptr;
        }
    }
    if (host) cudaFreeHost(host);
}

void Scratch::give_back() {
    std::vector<HostBlock> blocks;
    {
        std::lock_guard<std::mutex> hold(g_lock);
        for (cudaMemPool_t p : g_pool)
            if (p) cudaMemPoolTrimTo(p, 0);
        if (g_host) blocks.swap(*g_host);
    }
    for (const HostBlock &b : blocks) cudaFreeHost(b.p);
}

}  // namespace nb
