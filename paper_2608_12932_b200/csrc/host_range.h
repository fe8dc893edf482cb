// Whether kernels use host buffers where they are (plain C++: the decision is tested on the CPU).
#pragma once
#include <cstddef>
#include <cstdint>

namespace w4a8 {

// Requests whose buffers are worth using in place.  Up to 512 KiB each way; and rows of up to 32768 channels, because one CTA
// reads a row, a longer one twice and at the latency of the bus (measured on B200, copies against in place: 1 x 32768 -> 1024
// 37.4 and 33.5 us a request; 1 x 65536 -> 512 61.9 and 65.0; 1 x 131072 -> 256 97 and 117; 1 x 262144 -> 128 179 and 226).
constexpr size_t HOST_IN_PLACE_MAX_BYTES = 512 * 1024;
constexpr int HOST_IN_PLACE_MAX_K = 32768;
inline bool reads_in_place(int M, int K) { return K <= HOST_IN_PLACE_MAX_K && (size_t)M * K * 2 <= HOST_IN_PLACE_MAX_BYTES; }
inline bool writes_in_place(int M, int N, int K) { return reads_in_place(M, K) && (size_t)M * N * 2 <= HOST_IN_PLACE_MAX_BYTES; }

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
