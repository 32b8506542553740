// pic_hostcopy.h -- device to pageable host copies by several threads (private to libpic).
//
// A copy into freshly allocated pageable memory is bound by the destination's page faults,
// which the driver's copy takes on one thread (64 MB: 28 to 56 ms).  Here a few threads each
// bring a piece into page-locked memory of their own and copy it on, so the faults are
// taken in parallel while other pieces cross the link.
//
// The page-locked pieces (8 MB) and the streams belong to the device, not to a handle: the
// handles that have copied share one set, one copy at a time, and the last of them to be
// destroyed gives it back.
#pragma once

#include <algorithm>
#include <atomic>
#include <cstring>
#include <mutex>
#include <thread>
#include <vector>

#include <cuda_runtime.h>

namespace pic {

class HostCopy {
public:
    HostCopy() = default;
    HostCopy(const HostCopy &) = delete;
    HostCopy &operator=(const HostCopy &) = delete;
    ~HostCopy()
    {
        if (device_ < 0) return;
        Set &s = set(device_);
        std::lock_guard<std::mutex> lock(s.mu);
        if (--s.users == 0) s.release();
    }

    // Copies `bytes` to pageable host memory; the data must be complete on the device (the
    // caller has synchronised its stream).  False: not done (small copies, another copy under
    // way, or no memory or threads for it); the caller copies plainly.
    bool run(void *dst, const void *src, size_t bytes, int device)
    {
        if (bytes < kLeast || device < 0 || device >= kDevices || (device_ >= 0 && device_ != device)) return false;
        Set &s = set(device);
        std::unique_lock<std::mutex> lock(s.mu, std::try_to_lock);
        if (!lock.owns_lock()) return false;
        int before = device;
        if (cudaGetDevice(&before) != cudaSuccess || !s.setup(device)) return false;
        if (device_ < 0) {
            device_ = device;
            ++s.users;
        }
        std::atomic<size_t> next{0};
        std::atomic<bool> ok{true};
        auto work = [&](int t) {
            if (cudaSetDevice(device) != cudaSuccess) { ok = false; return; }
            for (size_t off; ok && (off = next.fetch_add(kPiece)) < bytes;) {
                const size_t n = std::min(kPiece, bytes - off);
                if (cudaMemcpyAsync(s.pin + t * kPiece, static_cast<const char *>(src) + off, n, cudaMemcpyDeviceToHost,
                                    s.streams[t]) != cudaSuccess ||
                    cudaStreamSynchronize(s.streams[t]) != cudaSuccess) {
                    ok = false;
                    return;
                }
                std::memcpy(static_cast<char *>(dst) + off, s.pin + t * kPiece, n);
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
        cudaSetDevice(before);
        return ok;
    }

private:
    static constexpr int kThreads = 8, kDevices = 64;
    static constexpr size_t kPiece = 1u << 20, kLeast = 8u << 20;

    struct Set {
        std::mutex mu;
        int users = 0;                  // handles that have copied
        char *pin = nullptr;
        cudaStream_t streams[kThreads] = {};

        void release()
        {
            for (cudaStream_t &s : streams)
                if (s) { cudaStreamDestroy(s); s = nullptr; }
            if (pin) cudaFreeHost(pin);
            pin = nullptr;
        }

        bool setup(int device)
        {
            if (pin) return true;
            int before = device;
            cudaGetDevice(&before);
            if (cudaSetDevice(device) != cudaSuccess) return false;
            bool good = cudaMallocHost(reinterpret_cast<void **>(&pin), kThreads * kPiece) == cudaSuccess;
            if (!good) pin = nullptr;
            for (cudaStream_t &s : streams)
                if (good && cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking) != cudaSuccess) {
                    s = nullptr;
                    good = false;
                }
            if (!good) {
                cudaGetLastError();
                release();
            }
            cudaSetDevice(before);
            return good;
        }
    };

    // (nothing is given back at the process's exit: a handle may still be there)
    static Set &set(int device)
    {
        static Set sets[kDevices];
        return sets[device];
    }

    int device_ = -1;                   // where this handle counts as a user
};

}  // namespace pic
