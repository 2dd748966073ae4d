// staging.h -- read-backs of small results through page-locked host memory.
//
// A device-to-host copy into pageable memory returns only when it is done, some
// 8 us for a few bytes, and a read-back takes several (a field's four arrays and
// the error word).  Copies into page-locked memory are queued: they go down
// together, the caller waits once, and the bytes are moved to where the caller
// wants them.  What does not fit is copied straight to its place.  A run of 100 steps
// with its rows, field and error word took 851 us a call with pageable copies and 807 so.
//
// Page-locked memory is dear to make and to free (105 and 160 us, as much as 30
// copies save), so a handle copies directly until it has made that many, and
// slabs go from a closed handle to the next: at most kSlabs are kept, of kSlabBytes
// each.  A slab belongs to one handle at a time, and nothing is in flight in it
// between calls.
#pragma once

#include <cstddef>
#include <cstring>
#include <cuda_runtime.h>
#include <mutex>

namespace pic {

// Page-locked memory is made and freed while another stream may be captured into a
// graph, which either call would end in the default capture mode.
class RelaxedCapture {
public:
    RelaxedCapture() { ok_ = cudaThreadExchangeStreamCaptureMode(&mode_) == cudaSuccess; }
    ~RelaxedCapture() {
        if (ok_) (void)cudaThreadExchangeStreamCaptureMode(&mode_);
    }
    bool ok() const { return ok_; }

private:
    cudaStreamCaptureMode mode_ = cudaStreamCaptureModeRelaxed;
    bool ok_;
};

class Slabs {
public:
    static constexpr int kSlabs = 8;
    static constexpr size_t kSlabBytes = 384 * 1024;     // 512 history rows, four fields of 8192 nodes

    // A kept slab, or a new one if `make`; nullptr: none.
    static void *take(bool make) {
        State &s = state();
        {
            std::lock_guard<std::mutex> lock(s.mutex);
            while (s.n > 0) {
                void *p = s.slab[--s.n];
                cudaPointerAttributes at;                // (gone after a device reset)
                if (cudaPointerGetAttributes(&at, p) == cudaSuccess && at.type == cudaMemoryTypeHost) return p;
                (void)cudaGetLastError();
            }
        }
        void *p = nullptr;
        if (!make) return p;
        RelaxedCapture relaxed;
        if (!relaxed.ok()) return p;
        if (cudaMallocHost(&p, kSlabBytes) != cudaSuccess) {
            p = nullptr;
            (void)cudaGetLastError();
        }
        return p;
    }

    static void give(void *p) {
        State &s = state();
        {
            std::lock_guard<std::mutex> lock(s.mutex);
            if (s.n < kSlabs) {
                s.slab[s.n++] = p;
                return;
            }
        }
        RelaxedCapture relaxed;
        (void)cudaFreeHost(p);
    }

private:
    struct State {
        std::mutex mutex;
        void *slab[kSlabs];
        int n = 0;
    };
    static State &state() {
        static State *s = new State;                     // outlives every handle
        return *s;
    }
};

class Staging {
public:
    std::mutex mutex;            // held by a read-back from its first add to finish

    Staging() = default;
    Staging(const Staging &) = delete;
    Staging &operator=(const Staging &) = delete;
    ~Staging() {
        if (mem_) Slabs::give(mem_);
    }

    // Queue a copy of `bytes` at device address src to host address dst.
    cudaError_t add(void *dst, const void *src, size_t bytes, cudaStream_t s) {
        if (!mem_ && !none_) {
            const bool make = ++copies_ > kDirect;
            mem_ = Slabs::take(make);
            none_ = make && !mem_;
        }
        const size_t off = used_;
        if (!mem_ || n_ == kItems || bytes > Slabs::kSlabBytes - off)
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

    // Start afresh after an error, when what was queued before it has arrived.
    void abandon(cudaStream_t s) {
        (void)cudaStreamSynchronize(s);
        drop();
    }

private:
    void drop() { n_ = 0, used_ = 0; }

    static constexpr int kItems = 8, kDirect = 32;
    struct Item {
        void *dst;
        size_t off, bytes;
    };
    void *mem_ = nullptr;
    bool none_ = false;          // no page-locked memory to be had
    int copies_ = 0;             // made without a slab
    size_t used_ = 0;
    int n_ = 0;
    Item items_[kItems];
};

}  // namespace pic
