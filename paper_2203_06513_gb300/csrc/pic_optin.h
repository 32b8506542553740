// pic_optin.h -- shared-memory limits of kernels, kept by device (private to libpic).
#pragma once

#include <mutex>

#include <cuda_runtime.h>

namespace pic {

// The dynamic shared memory a kernel (or a group of kernels) has been allowed beyond the
// default 48 KB.  The limit belongs to a device, so it is kept by device; it is never
// lowered.
class SmemOptin {
public:
    // whether `bytes` are allowed on the current device
    bool allowed(size_t bytes)
    {
        std::lock_guard<std::mutex> lock(mu_);
        int d;
        return bytes <= kDefault || (device(d) && bytes <= bytes_[d]);
    }
    // allows `bytes` for the kernels on the current device; false: refused
    template <size_t N>
    bool raise(const void *const (&fn)[N], size_t bytes)
    {
        std::lock_guard<std::mutex> lock(mu_);
        int d;
        const bool known = device(d);
        if (bytes <= kDefault || (known && bytes <= bytes_[d])) return true;
        for (const void *f : fn)
            if (cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes) != cudaSuccess) return false;
        if (known) bytes_[d] = bytes;
        return true;
    }
    bool raise(const void *fn, size_t bytes)
    {
        const void *const one[] = {fn};
        return raise(one, bytes);
    }

private:
    static constexpr size_t kDefault = 47 * 1024;      // what kernels use statically comes on top
    static constexpr int kDevices = 64;
    static bool device(int &d) { return cudaGetDevice(&d) == cudaSuccess && d >= 0 && d < kDevices; }
    std::mutex mu_;
    size_t bytes_[kDevices] = {};
};

}  // namespace pic
