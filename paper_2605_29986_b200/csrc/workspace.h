// Device scratch of the calls that are not per-step (grouping, loading a partition): such a call waits for its stream
// before it returns, so the memory it used is free for the next call on any stream. Allocating and releasing a few
// megabytes costs more than the kernels of these calls (cudaMalloc and cudaFree: 0.3 ms together), so one block per
// device is kept between calls, up to kMost bytes and only while the process holds a context or a grammar of the
// library; the last of those to go gives it back. A call that finds the block in use by another thread allocates its own.
#pragma once

#include <cuda_runtime.h>

#include <cstddef>
#include <mutex>

namespace cfgzip {

class Workspace {
  public:
    static constexpr size_t kMost = size_t(64) << 20;

    explicit Workspace(size_t bytes) {
        int dev = -1;
        if (cudaGetDevice(&dev) != cudaSuccess) {
            cudaGetLastError();
            return;
        }
        if (bytes <= kMost && dev >= 0 && dev < kDevices) {
            std::lock_guard<std::mutex> lock(shared().mutex);
            Kept& k = shared().kept[dev];
            if (!k.busy) {
                if (k.bytes < bytes) {
                    if (k.ptr) cudaFree(k.ptr);
                    k.ptr = allocate(bytes);
                    k.bytes = k.ptr ? bytes : 0;
                }
                if (k.ptr) {
                    k.busy = true;
                    ptr = k.ptr;
                    kept_ = &k;
                }
                return;
            }
        }
        ptr = allocate(bytes);
    }
    ~Workspace() {
        if (!kept_) {
            if (ptr) cudaFree(ptr);
            return;
        }
        std::lock_guard<std::mutex> lock(shared().mutex);
        kept_->busy = false;
        if (shared().holders == 0) kept_->release();
    }
    Workspace(const Workspace&) = delete;
    Workspace& operator=(const Workspace&) = delete;

    // A context or grammar comes to life / goes.
    static void hold() {
        std::lock_guard<std::mutex> lock(shared().mutex);
        ++shared().holders;
    }
    static void drop() {
        std::lock_guard<std::mutex> lock(shared().mutex);
        if (--shared().holders > 0) return;
        for (Kept& k : shared().kept)
            if (!k.busy) k.release();
    }

    void* ptr = nullptr;  // null: no memory

  private:
    static constexpr int kDevices = 64;
    struct Kept {
        void* ptr = nullptr;
        size_t bytes = 0;
        bool busy = false;
        void release() {
            if (ptr && cudaFree(ptr) != cudaSuccess) cudaGetLastError();
            ptr = nullptr;
            bytes = 0;
        }
    };
    struct Shared {
        std::mutex mutex;
        Kept kept[kDevices];
        long holders = 0;
    };
    static Shared& shared() {
        static Shared* s = new Shared();  // never destroyed: the driver may be gone when static objects are
        return *s;
    }
    static void* allocate(size_t bytes) {
        void* p = nullptr;
        if (cudaMalloc(&p, bytes) != cudaSuccess) {
            cudaGetLastError();
            return nullptr;
        }
        return p;
    }
    Kept* kept_ = nullptr;
};

}  // namespace cfgzip
