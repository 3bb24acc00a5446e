// Page-locked host memory that kernels write to.  Host code; it compiles as plain C++, too.
#pragma once
#include <cuda.h>
#include <cuda_runtime_api.h>
#include <stddef.h>
#include <stdint.h>

// Device address of `bytes` of page-locked host memory, or null if the device cannot write to all of it.  Memory may be
// page-locked in pieces (cudaHostRegister), so its ranges are gone through one after the other: a buffer whose first and last
// byte are page-locked can have a gap, and a kernel that writes there faults.  (The runtime does not tell where a range ends, the
// driver does; 0.5 us a range.)
template <typename T>
T* pinned_address(T* host, size_t bytes) {
    typedef CUresult (*Attribute)(void*, CUpointer_attribute, CUdeviceptr);
    static const Attribute attribute = [] {
        void* fn = nullptr;
        cudaDriverEntryPointQueryResult found;
        const bool ok = cudaGetDriverEntryPoint("cuPointerGetAttribute", &fn, cudaEnableDefault, &found) == cudaSuccess;
        return ok && found == cudaDriverEntryPointSuccess ? (Attribute)fn : (Attribute)nullptr;
    }();
    if (!host || !bytes || !attribute) return nullptr;
    const uintptr_t first = (uintptr_t)host, end = first + bytes;
    uintptr_t device = 0;
    for (uintptr_t at = first; at < end;) {
        cudaPointerAttributes a;
        if (cudaPointerGetAttributes(&a, (const void*)at) != cudaSuccess) {
            cudaGetLastError();
            return nullptr;
        }
        if (a.type != cudaMemoryTypeHost || !a.devicePointer) return nullptr;
        const uintptr_t here = (uintptr_t)a.devicePointer;
        if (at == first) device = here;
        else if (here - device != at - first) return nullptr;
        CUdeviceptr start = 0;
        size_t size = 0;
        if (attribute(&start, CU_POINTER_ATTRIBUTE_RANGE_START_ADDR, here) != CUDA_SUCCESS ||
            attribute(&size, CU_POINTER_ATTRIBUTE_RANGE_SIZE, here) != CUDA_SUCCESS || here < start || here - start >= size)
            return nullptr;
        at += size - (here - start);
    }
    return (T*)device;
}
