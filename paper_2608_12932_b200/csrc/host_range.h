// Whether a kernel may use a host buffer where it is (plain C++: the decision is tested on the CPU).
#pragma once
#include <cstddef>
#include <cstdint>

namespace w4a8 {

// What the driver reports for the address of a buffer's first byte.
struct HostMemory {
    bool pinned;           // page-locked host memory that the device can address
    void* device;          // its address on the device
    uint64_t start, size;  // the one allocation or registration that holds the byte
};

// The buffer's address for the device, or null where the bytes have to be copied: the buffer must lie within one pinned
// range as a whole (a range may have been registered for a part of an allocation only; a kernel that ran past its end
// would fault where a copy returns an error), 16-byte aligned.
inline void* in_place_address(const HostMemory& m, const void* p, size_t bytes) {
    const uint64_t at = reinterpret_cast<uintptr_t>(p);
    if (!m.pinned || !m.device || (reinterpret_cast<uintptr_t>(m.device) & 15) != 0) return nullptr;
    if (at < m.start || bytes > m.size || at - m.start > m.size - bytes) return nullptr;
    return m.device;
}

}  // namespace w4a8
