// Device and pinned host buffers that grow on demand and are freed with their owner.  Host code over the CUDA runtime's C
// interface.
#pragma once

#include <cuda_runtime_api.h>

#include <algorithm>
#include <cstddef>

struct DevBuf {
    void *p = nullptr;
    size_t cap = 0;
    bool pooled = false;  // from the stream-ordered pool (cudaMallocAsync): freed with cudaFreeAsync
    bool view = false;    // a part of another buffer: nothing to free
    bool writing = false;             // pooled: work on `writer` may still be writing it
    cudaStream_t writer = nullptr;    // pooled: the stream it was allocated on
    void set_view(void *q, size_t bytes) {
        release();
        p = q, cap = bytes, view = true;
    }
    // allocates exactly `bytes` from the device's stream-ordered pool on stream s (no device-wide synchronisation,
    // unlike cudaMalloc / cudaFree); for buffers that are written once, such as a new version of the graph store, by work
    // on s, until settle()
    cudaError_t alloc_pooled(size_t bytes, cudaStream_t s) {
        release();
        cudaError_t e = cudaMallocAsync(&p, std::max<size_t>(256, bytes), s);
        if (e != cudaSuccess) {
            cudaGetLastError();
            p = nullptr;
            return e;
        }
        cap = std::max<size_t>(256, bytes);
        pooled = writing = true;
        writer = s;
        return cudaSuccess;
    }
    void settle() { writing = false; }  // the work on `writer` is complete
    cudaError_t ensure(size_t bytes) { return bytes <= cap && p ? cudaSuccess : ensure_exact(bytes + bytes / 8); }
    // the same; *fresh tells whether the memory is newly allocated, and so holds anything.  The address does not tell: an
    // allocation that replaces a smaller one may come back at the same place.
    cudaError_t ensure(size_t bytes, bool *fresh) {
        *fresh = !(bytes <= cap && p);
        return ensure(bytes);
    }
    cudaError_t ensure_exact(size_t bytes) {
        if (bytes <= cap && p) return cudaSuccess;
        if (p) cudaFree(p);
        p = nullptr;
        cap = 0;
        const size_t nb = std::max<size_t>(256, bytes);
        cudaError_t e = cudaMalloc(&p, nb);
        if (e == cudaSuccess) cap = nb; else cudaGetLastError();
        return e;
    }
    // grows to at least `bytes`, keeping the first `keep` bytes (copied on stream s)
    cudaError_t grow(size_t bytes, size_t keep, cudaStream_t s) {
        if (bytes <= cap && p) return cudaSuccess;
        void *q = nullptr;
        const size_t nb = std::max<size_t>(256, bytes + bytes / 4);
        cudaError_t e = cudaMalloc(&q, nb);
        if (e != cudaSuccess) {
            cudaGetLastError();
            return e;
        }
        if (p && keep > 0) e = cudaMemcpyAsync(q, p, std::min(keep, cap), cudaMemcpyDeviceToDevice, s);
        if (e == cudaSuccess && p) e = cudaStreamSynchronize(s);
        if (p) cudaFree(p);
        p = q;
        cap = nb;
        return e;
    }
    // A pooled buffer returns to the pool on the calling thread's default stream, without waiting: its readers
    // have synchronised their own streams before they let go of it.  Before it has settled (an update that fails half-way)
    // it returns in the order of the stream whose kernels may still be writing it.
    void release() {
        if (p && !view) {
            if (pooled) cudaFreeAsync(p, writing ? writer : cudaStreamPerThread);
            else cudaFree(p);
        }
        p = nullptr;
        cap = 0;
        pooled = view = writing = false;
    }
    template <class T>
    T *as() const { return static_cast<T *>(p); }
};

struct PinnedBuf {
    void *p = nullptr;
    size_t cap = 0;
    cudaError_t ensure(size_t bytes) {
        if (bytes <= cap && p) return cudaSuccess;
        if (p) cudaFreeHost(p);
        p = nullptr;
        cap = 0;
        const size_t nb = std::max<size_t>(256, bytes + bytes / 8);
        cudaError_t e = cudaMallocHost(&p, nb);
        if (e == cudaSuccess) cap = nb; else cudaGetLastError();
        return e;
    }
    void release() {
        if (p) cudaFreeHost(p);
        p = nullptr;
        cap = 0;
    }
    template <class T>
    T *as() const { return static_cast<T *>(p); }
};
