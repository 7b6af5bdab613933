// devbuf.h -- owning device buffer (cudaMalloc / cudaFree), host side.
#pragma once
#include <cuda_runtime.h>

#include <cstddef>

namespace dg {

template <typename T>
struct DevBuf {
    T *ptr = nullptr;
    size_t n = 0;
    DevBuf() = default;
    DevBuf(const DevBuf &) = delete;
    DevBuf &operator=(const DevBuf &) = delete;
    DevBuf(DevBuf &&o) noexcept : ptr(o.ptr), n(o.n)
    {
        o.ptr = nullptr;
        o.n = 0;
    }
    DevBuf &operator=(DevBuf &&o) noexcept
    {
        if (this != &o) {
            release();
            ptr = o.ptr;
            n = o.n;
            o.ptr = nullptr;
            o.n = 0;
        }
        return *this;
    }
    ~DevBuf() { release(); }
    cudaError_t alloc(size_t count)
    {
        release();
        if (count == 0) return cudaSuccess;
        const cudaError_t e = cudaMalloc(reinterpret_cast<void **>(&ptr), count * sizeof(T));
        if (e == cudaSuccess) n = count;
        else ptr = nullptr;
        return e;
    }
    void release()
    {
        if (ptr) cudaFree(ptr);
        ptr = nullptr;
        n = 0;
    }
};

}  // namespace dg
