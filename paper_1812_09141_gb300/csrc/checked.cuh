// Index checks of the checked build (SSJ_CHECKED, see kChecked), shared by the
// kernels.
#pragma once

#include <cstdint>

#include "ssj_internal.h"

namespace ssj {

// Checked build: false, and ERR_BOUNDS set, when idx is not below n.
__device__ __forceinline__ bool in_bounds(uint64_t idx, uint64_t n, uint32_t* err) {
    if (kChecked && idx >= n) {
        atomicOr(err, ERR_BOUNDS);
        return false;
    }
    return true;
}

// Element idx of a read-only array of n (checked build: zero past its end).
template <class T>
__device__ __forceinline__ T ld_at(const T* p, uint64_t idx, uint64_t n, uint32_t* err) {
    if (!in_bounds(idx, n, err)) return T();
    return __ldg(p + idx);
}

}  // namespace ssj
