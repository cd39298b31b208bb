// Which host buffers a kernel may read and write in place.  Plain C++ (no CUDA), so that it is testable by itself.
#pragma once

#include <cstddef>
#include <cstdint>

namespace lopro {

// What the driver says about the first byte of a buffer: its address on the device and the one allocation or registration
// that holds it.  Zeros where it knows nothing of it.
struct HostRange {
    uint64_t device, start;
    size_t size;
};

// True if that one piece holds all of the buffer.  The last byte's being pinned too says nothing of what lies between: two
// ranges registered on their own, with pages between them that are not, look alike from both ends.
inline bool holds_whole_buffer(const HostRange& r, size_t bytes) {
    if (r.device == 0 || r.size == 0 || bytes == 0 || r.device < r.start) return false;
    const uint64_t before = r.device - r.start;
    return before < r.size && bytes <= r.size - before;
}

}  // namespace lopro
