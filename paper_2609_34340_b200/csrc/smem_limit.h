// The limit of dynamic shared memory of a kernel.  Host code; it compiles as plain C++ too.
#pragma once
#include <cuda_runtime_api.h>

#include "variopath.h"

// Dynamic shared memory that a launch may use on a device whose opt-in maximum is `optin`: the rest is for static variables (at
// most 288 bytes in the kernels launched so).
inline int dynamic_smem_limit(int optin) { return optin - 2048; }

// Sets a kernel's limit on the current device to that.  The limit belongs to the function, not to a launch: launches are planned
// once and replayed from a memo, several catalogs and threads share the kernels, and one kernel is launched with different
// sizes.  So it is one constant, whoever sets it, and not what a plan needs: a table of the largest size so far, kept instead,
// was full after 64 pairs of kernel and device, and a later plan then lowered the limit under launches planned before.
inline int set_dynamic_smem_limit(const void* fn, int optin) {
    return cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, dynamic_smem_limit(optin)) == cudaSuccess ? VP_OK : VP_E_CUDA;
}
