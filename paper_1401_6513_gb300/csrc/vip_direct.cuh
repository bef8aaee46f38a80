// Calls that take a caller's arrays: when a kernel may use them where they lie.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace vip {

// Can a kernel on the device read x and write y, n entries each, in place of the caller's
// arrays?  Both lie in this device's memory from the first to the last entry, are aligned as
// doubles, and do not overlap.  Host arrays and other devices' are staged by the caller of this.
inline bool direct_vectors(int device, const double* x, const double* y, int64_t n) {
    if (n <= 0 || (reinterpret_cast<uintptr_t>(x) | reinterpret_cast<uintptr_t>(y)) % sizeof(double)) return false;
    if (x < y + n && y < x + n) return false;
    for (const double* p : {x, x + n - 1, y, y + n - 1}) {
        cudaPointerAttributes a;
        if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
            cudaGetLastError();
            return false;
        }
        if (a.type != cudaMemoryTypeDevice || a.device != device) return false;
    }
    return true;
}

}  // namespace vip
