// mrlt_input.h -- the way of a caller's initial data to the device.
#pragma once
#include <cstddef>
#include <cstdint>

namespace mrlt {

// Data of this size and more are read in place by the kernel that stores them
// (see load_finest).
constexpr size_t kReadInPlace = 16u << 20;

// May a kernel read the `bytes` of doubles at q0 in place?  host_tables: the GPU
// reads any host memory through the host's page tables; short_lived: the memory
// is released right after.  The kernel loads whole doubles, so they must lie on
// their boundary: a caller's array need not (a view into a file or a message
// behind an odd header), and a copy takes it at any address.
inline bool read_in_place(const void* q0, size_t bytes, bool short_lived, bool host_tables)
{
    return host_tables && !short_lived && bytes >= kReadInPlace &&
           reinterpret_cast<uintptr_t>(q0) % alignof(double) == 0;
}

} // namespace mrlt
