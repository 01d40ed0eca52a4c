// Which host memory a kernel may read where it is.
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace impact {

// Do `bytes` bytes from p lie inside [start, start + size)?
inline bool range_holds(unsigned long long start, size_t size, const void* p, size_t bytes) {
    const unsigned long long at = (unsigned long long)reinterpret_cast<uintptr_t>(p);
    return bytes <= size && at >= start && at - start <= size - bytes;
}

// Are `bytes` bytes from p one range of pinned host memory -- one allocation or one registration, from the first byte to the
// last -- that the device reads at the host's own addresses?  The first byte's range settles it: two ranges with a hole
// between them, which a look at the first and the last byte cannot tell from one, are not one range.  (cuPointerGetAttributes
// answers for memory that CUDA does not know with zeros; no error of a call, and none is left behind.)
inline bool pinned_in_one_range(const void* p, size_t bytes) {
    using GetAttributes = CUresult (*)(unsigned int, CUpointer_attribute*, void**, CUdeviceptr);
    static const GetAttributes get_attributes = [] {
        void* f = nullptr;
        cudaDriverEntryPointQueryResult found = cudaDriverEntryPointSymbolNotFound;
        if (cudaGetDriverEntryPointByVersion("cuPointerGetAttributes", &f, 12000, cudaEnableDefault, &found) != cudaSuccess) {
            cudaGetLastError();
            f = nullptr;
        }
        return found == cudaDriverEntryPointSuccess ? reinterpret_cast<GetAttributes>(f) : nullptr;
    }();
    if (!get_attributes) return false;
    unsigned int type = 0;
    int managed = 0;
    CUdeviceptr on_device = 0, start = 0;
    size_t size = 0;
    CUpointer_attribute which[] = {CU_POINTER_ATTRIBUTE_MEMORY_TYPE, CU_POINTER_ATTRIBUTE_IS_MANAGED,
                                   CU_POINTER_ATTRIBUTE_DEVICE_POINTER, CU_POINTER_ATTRIBUTE_RANGE_START_ADDR,
                                   CU_POINTER_ATTRIBUTE_RANGE_SIZE};
    void* out[] = {&type, &managed, &on_device, &start, &size};
    const CUdeviceptr at = (CUdeviceptr)reinterpret_cast<uintptr_t>(p);
    return get_attributes(5, which, out, at) == CUDA_SUCCESS && type == CU_MEMORYTYPE_HOST && !managed && on_device == at &&
           range_holds(start, size, p, bytes);
}

}  // namespace impact
