// The copies of lce_bconv2d_host in one kernel each way.  What bounds the call for a small layer is the number of stream
// operations: each cudaMemcpyAsync costs about 4 us of the stream whatever its size, more where the stream changes between
// copy engine and SMs, and a layer brings weights and one or two per-channel arrays beside its input.  Pinned host memory
// is visible to the device, so one kernel fetches them all over PCIe (its latency once, about 4 us together), and one
// brings the output back.  The copy engine is a little faster per byte (0.8 MB: 18.0 against 20.6 us): large arrays stay
// with it.
#include <cuda.h>

#include "common.cuh"
#include "host_view.cuh"

namespace lce {
namespace {

constexpr int kCopyThreads = 256;

struct CopyParams {
    const uint32_t *src[kHostCopies];
    uint32_t *dst[kHostCopies];
    int32_t first[kHostCopies + 1];  // piece at which an array begins; a piece is 4 words, the last one of an array may be short
    int32_t words[kHostCopies];
};

__global__ void __launch_bounds__(kCopyThreads) host_copy_kernel(const CopyParams p)
{
    asm volatile("griddepcontrol.wait;" ::: "memory");
    for (int i = blockIdx.x * kCopyThreads + threadIdx.x; i < p.first[kHostCopies]; i += gridDim.x * kCopyThreads) {
        const uint32_t *src = p.src[0];
        uint32_t *dst = p.dst[0];
        int at = i * 4, words = p.words[0];
#pragma unroll
        for (int k = 1; k < kHostCopies; ++k) {
            if (i >= p.first[k]) {
                src = p.src[k];
                dst = p.dst[k];
                at = (i - p.first[k]) * 4;
                words = p.words[k];
            }
        }
        if (at + 4 <= words && ((reinterpret_cast<uintptr_t>(src) | reinterpret_cast<uintptr_t>(dst)) & 15) == 0) {
            *reinterpret_cast<uint4 *>(dst + at) = *reinterpret_cast<const uint4 *>(src + at);
        } else {
            for (int k = at; k < min(at + 4, words); ++k) dst[k] = src[k];
        }
    }
}

// cuPointerGetAttributes, which tells all of HostMemory in one call (0.6 us); null if the driver has none.
using PointerAttributes = CUresult (*)(unsigned int, CUpointer_attribute *, void **, CUdeviceptr);
PointerAttributes pointer_attributes()
{
    static const PointerAttributes found = [] {
        void *entry = nullptr;
        cudaDriverEntryPointQueryResult result = cudaDriverEntryPointSymbolNotFound;
        if (cudaGetDriverEntryPointByVersion("cuPointerGetAttributes", &entry, 7000, cudaEnableDefault, &result) != cudaSuccess) cudaGetLastError();
        return result == cudaDriverEntryPointSuccess ? reinterpret_cast<PointerAttributes>(entry) : nullptr;
    }();
    return found;
}

}  // namespace

void *pinned_host_view(const void *host, size_t bytes, bool write)
{
    const PointerAttributes query = pointer_attributes();
    uint64_t type = 0, managed = 0, view = 0, first = 0, size = 0, access = 0;  // as wide as the widest value the driver writes
    CUpointer_attribute names[] = {CU_POINTER_ATTRIBUTE_MEMORY_TYPE, CU_POINTER_ATTRIBUTE_IS_MANAGED, CU_POINTER_ATTRIBUTE_DEVICE_POINTER,
                                   CU_POINTER_ATTRIBUTE_RANGE_START_ADDR, CU_POINTER_ATTRIBUTE_RANGE_SIZE, CU_POINTER_ATTRIBUTE_ACCESS_FLAGS};
    void *values[] = {&type, &managed, &view, &first, &size, &access};
    constexpr unsigned kNames = sizeof(names) / sizeof(names[0]);
    const CUdeviceptr address = reinterpret_cast<CUdeviceptr>(host);
    if (!query) return nullptr;
    if (query(kNames, names, values, address) != CUDA_SUCCESS) {
        // a host thread's first CUDA call: the runtime makes the device's context current
        cudaPointerAttributes a{};
        if (cudaPointerGetAttributes(&a, host) != cudaSuccess) cudaGetLastError();
        if (query(kNames, names, values, address) != CUDA_SUCCESS) return nullptr;
    }
    const HostMemory m{type == CU_MEMORYTYPE_HOST && !managed, (uintptr_t)view, (uintptr_t)first, (size_t)size, access == CU_POINTER_ATTRIBUTE_ACCESS_FLAG_READWRITE};
    return reinterpret_cast<void *>(kernel_view(reinterpret_cast<uintptr_t>(host), bytes, write, m));
}

lce_status launch_host_copies(const HostCopy (&copies)[kHostCopies], cudaStream_t s)
{
    CopyParams p{};
    int32_t pieces = 0;
    for (int k = 0; k < kHostCopies; ++k) {
        p.src[k] = static_cast<const uint32_t *>(copies[k].src);
        p.dst[k] = static_cast<uint32_t *>(copies[k].dst);
        p.first[k] = pieces;
        p.words[k] = (int32_t)(copies[k].bytes / 4);
        pieces += (p.words[k] + 3) / 4;
    }
    p.first[kHostCopies] = pieces;
    if (pieces == 0) return LCE_OK;
    const int blocks = (pieces + kCopyThreads - 1) / kCopyThreads;
    return launch_dependent(host_copy_kernel, dim3((unsigned)(blocks < 148 * 8 ? blocks : 148 * 8)), kCopyThreads, 0, s, p);
}

}  // namespace lce
