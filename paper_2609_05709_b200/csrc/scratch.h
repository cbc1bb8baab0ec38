// Growth of a handle's scratch: buffers that share one capacity are replaced together.
#pragma once
#include <cstddef>
#include <cstdint>
#include <initializer_list>

namespace soap {

struct ScratchBuffer { void** ptr; size_t bytes; };

// Replaces all buffers of a group, through `allocate(void**, size_t) -> bool` and `release(void*)`.  Only when every one of
// them is there does `capacity` become `want`; else none is left and the capacity is zero, so that whoever looks at it
// next allocates again and nobody works in a buffer that is gone.
template <class Allocate, class Release>
bool regrow_group(int64_t& capacity, int64_t want, std::initializer_list<ScratchBuffer> buffers, Allocate allocate, Release release) {
    capacity = 0;
    auto drop = [&]() {
        for (const ScratchBuffer& b : buffers)
            if (*b.ptr) { release(*b.ptr); *b.ptr = nullptr; }
    };
    drop();
    for (const ScratchBuffer& b : buffers)
        if (!allocate(b.ptr, b.bytes)) {
            *b.ptr = nullptr;
            drop();
            return false;
        }
    capacity = want;
    return true;
}

}  // namespace soap
