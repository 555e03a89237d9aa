// Host tables gathered into one device allocation.
#pragma once

#include <algorithm>
#include <cstring>
#include <vector>

#include <cuda_runtime.h>

namespace sg {

// Several tables in one device allocation and one copy: add() each, then put().
struct Arena {
    std::vector<unsigned char> host;
    template <typename T>
    size_t add(const T *v, size_t k)
    {
        const size_t o = (host.size() + 255) & ~(size_t)255;
        host.resize(o + std::max<size_t>(1, k) * sizeof(T));
        if (k) std::memcpy(host.data() + o, v, k * sizeof(T));
        return o;
    }
    template <typename T>
    size_t add(const std::vector<T> &v) { return add(v.data(), v.size()); }
    // *base: the allocation, `more` bytes longer than the tables (from more_at on)
    cudaError_t put(unsigned char **base, size_t more = 0, size_t *more_at = nullptr)
    {
        const size_t end = (host.size() + 255) & ~(size_t)255;
        if (more_at) *more_at = end;
        *base = nullptr;
        cudaError_t e = cudaMalloc(reinterpret_cast<void **>(base), std::max<size_t>(1, end + more));
        if (e == cudaSuccess && !host.empty()) e = cudaMemcpy(*base, host.data(), host.size(), cudaMemcpyHostToDevice);
        return e;
    }
};

}  // namespace sg
