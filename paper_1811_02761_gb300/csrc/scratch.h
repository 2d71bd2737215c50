// scratch.h -- device and page-locked host blocks of the stateless calls.
//
// A call's device block comes from a memory pool of its own per device
// (stream-ordered: taken and returned on the call's stream, so calls on
// several streams and threads never share one in flight), which keeps at most
// kKeepDevice bytes between calls; its host block from a list of at most
// kKeepHost blocks.  finish() waits for the call's stream; a call that ends
// before it (a failed step after others were queued) waits in the destructor,
// so that no kernel or copy in flight still uses the host block, or the
// caller's arrays, when they are given back.  Both kinds are given back when a
// context is destroyed.
#pragma once

#include <cuda_runtime.h>
#include <stddef.h>

namespace nb {

class Scratch {
public:
    explicit Scratch(cudaStream_t s) : stream_(s) {}
    ~Scratch();
    Scratch(const Scratch &) = delete;
    Scratch &operator=(const Scratch &) = delete;
    cudaError_t take(size_t dev_bytes, size_t host_bytes);
    cudaError_t finish();     // the call's work is done: waits for it
    static void give_back();  // the memory no call is using
    char *dev = nullptr, *host = nullptr;

private:
    cudaStream_t stream_;
    size_t host_bytes_ = 0;
    bool finished_ = false;
};

}  // namespace nb
