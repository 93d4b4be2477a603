// dp_pinned.h -- pinned host memory that a handle keeps for its calls.
#pragma once

#include <cuda_runtime.h>

#include <cstddef>

namespace dpk {

// Page-locked doubles, grown on demand and kept until release().  Only as good
// as the host's page-locked memory: where there is none, reserve() gives NULL,
// keeps what it had, leaves no CUDA error behind, and the caller goes without.
class PinnedDoubles {
public:
    // At least `count` doubles, or NULL; a larger buffer is allocated with room
    // for twice as many, at most `most` (count <= most).  No call that uses the
    // old one may be in flight.
    double* reserve(size_t count, size_t most)
    {
        if (count <= cap_) return p_;
        const size_t cap = 2 * count < most ? 2 * count : most;
        double* p = nullptr;
        if (cudaMallocHost((void**)&p, cap * sizeof(double)) != cudaSuccess) {
            cudaGetLastError();
            return nullptr;
        }
        release();
        p_ = p;
        cap_ = cap;
        return p_;
    }
    void release()
    {
        if (p_) cudaFreeHost(p_);
        p_ = nullptr;
        cap_ = 0;
    }

private:
    double* p_ = nullptr;
    size_t cap_ = 0;
};

}  // namespace dpk
