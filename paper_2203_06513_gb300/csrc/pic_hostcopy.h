// pic_hostcopy.h -- device to pageable host copies by several threads (private to libpic).
//
// A copy into freshly allocated pageable memory is bound by the destination's page faults,
// which the driver's copy takes on one thread (64 MB: 28 to 56 ms).  Here a few threads each
// bring a piece into page-locked memory of their own and copy it on, so the faults are
// taken in parallel while other pieces cross the link.
#pragma once

#include <algorithm>
#include <atomic>
#include <cstring>
#include <thread>
#include <vector>

#include <cuda_runtime.h>

namespace pic {

class HostCopy {
public:
    ~HostCopy() { release(); }

    // Copies `bytes` to pageable host memory; the data must be complete on the device (the
    // caller has synchronised its stream).  False: not done (small copies, or no memory or
    // threads for it); the caller copies plainly.
    bool run(void *dst, const void *src, size_t bytes, int device)
    {
        if (bytes < kLeast || !setup(device)) return false;
        std::atomic<size_t> next{0};
        std::atomic<bool> ok{true};
        auto work = [&](int t) {
            if (cudaSetDevice(device) != cudaSuccess) { ok = false; return; }
            for (size_t off; ok && (off = next.fetch_add(kPiece)) < bytes;) {
                const size_t n = std::min(kPiece, bytes - off);
                if (cudaMemcpyAsync(pin_ + t * kPiece, static_cast<const char *>(src) + off, n, cudaMemcpyDeviceToHost,
                                    streams_[t]) != cudaSuccess ||
                    cudaStreamSynchronize(streams_[t]) != cudaSuccess) {
                    ok = false;
                    return;
                }
                std::memcpy(static_cast<char *>(dst) + off, pin_ + t * kPiece, n);
            }
        };
        std::vector<std::thread> pool;
        try {
            pool.reserve(kThreads - 1);
            for (int t = 1; t < kThreads; ++t) pool.emplace_back(work, t);
        } catch (...) {
            // fewer threads share the pieces
        }
        work(0);
        for (std::thread &t : pool) t.join();
        return ok;
    }

    void release()
    {
        for (cudaStream_t &s : streams_)
            if (s) { cudaStreamDestroy(s); s = nullptr; }
        if (pin_) cudaFreeHost(pin_);
        pin_ = nullptr;
    }

private:
    static constexpr int kThreads = 8;
    static constexpr size_t kPiece = 1u << 20, kLeast = 8u << 20;
    char *pin_ = nullptr;
    cudaStream_t streams_[kThreads] = {};

    bool setup(int device)
    {
        if (pin_) return true;
        if (cudaSetDevice(device) != cudaSuccess) return false;
        if (cudaMallocHost(reinterpret_cast<void **>(&pin_), kThreads * kPiece) != cudaSuccess) {
            cudaGetLastError();
            pin_ = nullptr;
            return false;
        }
        for (cudaStream_t &s : streams_)
            if (cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking) != cudaSuccess) {
                cudaGetLastError();
                release();
                return false;
            }
        return true;
    }
};

}  // namespace pic
