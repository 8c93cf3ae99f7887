// Which arrays in host memory a kernel may access itself, as facts and a rule (host code only; no CUDA headers, so that
// the rule can be checked without a GPU).
#pragma once
#include <stdint.h>

namespace lce {

// What the CUDA driver says of a host address.
struct HostMemory {
    bool pinned;
    uintptr_t view;  // the device's address of it
};

// The address at which a kernel may access a host array, 0 where only the copy engine may.  The kernels go by words of 4
// bytes (16 where the address allows), the copy engine by bytes: an array that does not start on 4 is left to it.
inline uintptr_t kernel_view(uintptr_t array, const HostMemory &m)
{
    return m.pinned && ((array | m.view) & 3) == 0 ? m.view : 0;
}

}  // namespace lce
