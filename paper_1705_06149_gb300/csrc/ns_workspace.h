// Device buffers of one call, given back however the call ends.
#pragma once

#include <cuda_runtime.h>

#include <algorithm>
#include <cstddef>
#include <vector>

// The destructor waits for the stream, whose work may still use the buffers,
// and frees them, so a return from the middle of a call leaves none behind.
class Workspace {
public:
    explicit Workspace(cudaStream_t stream) : stream_(stream) {}
    Workspace(const Workspace&) = delete;
    Workspace& operator=(const Workspace&) = delete;
    ~Workspace() {
        if (mine_.empty()) return;
        cudaStreamSynchronize(stream_);
        for (void* p : mine_) cudaFree(p);
    }
    // n elements; null, and ok() false from then on, when there is no memory.
    template <typename T>
    T* get(size_t n) {
        void* p = nullptr;
        if (cudaMalloc(&p, std::max<size_t>(n * sizeof(T), 16)) != cudaSuccess) {
            cudaGetLastError();
            ok_ = false;
            return nullptr;
        }
        mine_.push_back(p);
        return static_cast<T*>(p);
    }
    bool ok() const { return ok_; }

private:
    cudaStream_t stream_;
    std::vector<void*> mine_;
    bool ok_ = true;
};
