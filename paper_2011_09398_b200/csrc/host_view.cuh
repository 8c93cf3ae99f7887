// Which arrays in host memory a kernel may access itself, as facts and a rule (host code only; no CUDA headers, so that
// the rule can be checked without a GPU).
#pragma once
#include <stddef.h>
#include <stdint.h>

namespace lce {

// What the CUDA driver says of a host address.
struct HostMemory {
    bool pinned;
    uintptr_t view;         // the device's address of it
    uintptr_t first;        // where the pinned range that holds it begins, in the device's addresses, and its bytes: one
    size_t bytes;           //   allocation (cudaHostAlloc) or one registration (cudaHostRegister)
    bool writable;          // by the device: not so if registered read-only
};

// The address at which a kernel may access a host array (`write`: store to it), 0 where only the copy engine may.
//   - The kernels go by words of 4 bytes (16 where the address allows), the copy engine by bytes: an array that does not
//     start on 4 is left to it.
//   - An array that reaches past the pinned range its first byte lies in (only its front registered, or front and back
//     but not the middle) is an access outside the mapping in a kernel; the copy engine's call looks at the whole array.
inline uintptr_t kernel_view(uintptr_t array, size_t bytes, bool write, const HostMemory &m)
{
    if (!m.pinned || !m.view || ((array | m.view) & 3) != 0 || (write && !m.writable)) return 0;
    if (m.view < m.first || m.view - m.first > m.bytes || bytes > m.bytes - (m.view - m.first)) return 0;
    return m.view;
}

}  // namespace lce
