// buffers.h -- device buffers that grow, and the capacities they stand for.
#pragma once

#include <cuda_runtime.h>
#include <stddef.h>

#include <initializer_list>

namespace nb {

struct DevBuf {
    void *p = nullptr;
    size_t bytes = 0;
};

inline cudaError_t ensure(DevBuf &b, size_t bytes) {
    if (b.bytes >= bytes && b.p) return cudaSuccess;
    if (b.p) {
        cudaError_t e = cudaFree(b.p);
        b.p = nullptr;
        b.bytes = 0;
        if (e != cudaSuccess) return e;
    }
    size_t want = bytes ? bytes : 16;
    cudaError_t e = cudaMalloc(&b.p, want);
    if (e != cudaSuccess) {
        b.p = nullptr;
        return e;
    }
    b.bytes = want;
    return cudaSuccess;
}

struct BufSize {
    DevBuf *buf;
    size_t bytes;
};

// Grows the buffers of one capacity.  The capacity is zero while they grow, so
// after a failure (some buffers new, one freed, the rest as they were) the next
// call, however small, takes them all again and initialises what is new.
template <typename T>
cudaError_t grow(T &cap, T want, std::initializer_list<BufSize> bufs) {
    cap = 0;
    for (const BufSize &b : bufs) {
        const cudaError_t e = ensure(*b.buf, b.bytes);
        if (e != cudaSuccess) return e;
    }
    cap = want;
    return cudaSuccess;
}

}  // namespace nb
