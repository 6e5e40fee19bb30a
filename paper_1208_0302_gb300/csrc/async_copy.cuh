// Element copies from global to shared memory that hold no registers while
// they are in flight (cp.async).
#pragma once

#include <cuda_runtime.h>

namespace genesis {

template <class R> __device__ __forceinline__ void copy_async(R *dst, const R *src)
{
    static_assert(sizeof(R) == 4 || sizeof(R) == 8, "cp.async moves 4, 8 or 16 bytes");
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    if (sizeof(R) == 4) asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(d), "l"(src) : "memory");
    else asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(d), "l"(src) : "memory");
}

// All of the warp's copies have landed and every lane sees them.
__device__ __forceinline__ void copy_wait()
{
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncwarp();
}

}  // namespace genesis
