// What the kernels of one device have been opted in to, in bytes of dynamic shared memory.  Plain C++ (no CUDA header), so
// that it can be tested without a device.
#pragma once

#include <stddef.h>

#include <mutex>
#include <unordered_map>

namespace fq {

class SmemOptIn {
public:
    // `set(bytes)` opts the kernel in and returns 0 for success.  Look-up, call and record are one critical section and the
    // value only rises: a kernel's size varies with the shape, and of two host threads that met here the one with the smaller
    // size could otherwise leave the attribute lower than the record, after which every larger launch fails.
    template <typename Set>
    auto raise(const void* kernel, size_t bytes, Set set) -> decltype(set(bytes)) {
        std::lock_guard<std::mutex> lock(mutex_);
        size_t& have = bytes_[kernel];
        if (have >= bytes) return decltype(set(bytes))();
        const auto e = set(bytes);
        if (e == decltype(set(bytes))()) have = bytes;
        return e;
    }

private:
    std::mutex mutex_;
    std::unordered_map<const void*, size_t> bytes_;
};

}  // namespace fq
