// Whether a kernel may access a caller's buffer directly (host code only).
#pragma once

#include <cstddef>
#include <cstdint>

namespace fsl {

struct BufferInfo {
    bool device_memory;      // device memory, not host or managed memory
    int device;
    std::uintptr_t base;     // the allocation that holds the address
    std::size_t size;
};

// [p, p + bytes) is aligned and lies inside one allocation of device memory of
// device dev. lookup(p, info) describes the allocation at an address, false
// where there is none. (Both ends being device memory is not enough: the
// range could leave its allocation and reach over a gap into another.)
template <class Lookup>
bool kernel_may_access(const void* p, std::size_t bytes, std::size_t align, int dev, Lookup lookup) {
    const std::uintptr_t a = reinterpret_cast<std::uintptr_t>(p);
    if (a % align) return false;
    BufferInfo b = {};
    if (!lookup(p, b) || !b.device_memory || b.device != dev) return false;
    return a >= b.base && a - b.base <= b.size && bytes <= b.size - (a - b.base);
}

}  // namespace fsl
