// f32_split.cuh - what the FP32 tensor-core kernels (f32_tc.cu, student_x3.cu) share: the exact split of
// an FP32 value in three BF16 parts, bounded waits, and the error word's protocol.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/membrane.h"
#include "tc_ptx.cuh"

namespace mb {

constexpr uint64_t kXWaitNs = 4000000000ull;  // limit of every device-side wait

__device__ __forceinline__ uint64_t x_gtime() {
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// False (and the CTA-wide abort flag raised, the error word set) when the phase did not complete within
// the limit, or at once while the CTA is aborting.
__device__ __forceinline__ bool x_wait(uint64_t* bar, uint32_t parity, volatile int* abort_flag, int* err,
                                       uint64_t limit_ns) {
    if (ptx::mbar_test(bar, parity)) return true;  // a completed phase costs one poll
    if (*abort_flag) return false;
    const uint64_t t0 = x_gtime();
    uint32_t n = 0;
    while (!ptx::mbar_test(bar, parity)) {
        if ((++n & 255u) == 0) {
            if (*abort_flag) return false;
            if (x_gtime() - t0 > limit_ns) {
                *abort_flag = 1;
                *(volatile int*)err = MB_ERR_TIMEOUT;
                return false;
            }
        }
    }
    return true;
}

// Waits (bounded) for this thread's own tcgen05 operations before TMEM is released.
__device__ __forceinline__ void x_drain(uint64_t* fin, int* err, uint64_t limit_ns) {
    ptx::mma_commit(fin);
    const uint64_t t0 = x_gtime();
    while (!ptx::mbar_test(fin, 0)) {
        if (x_gtime() - t0 > limit_ns) {
            *(volatile int*)err = MB_ERR_TIMEOUT;
            break;
        }
    }
}

// The leading 8 significant bits of two floats as a BF16 pair; the floats keep what is left (exact).
__device__ __forceinline__ uint32_t take_part(float& a, float& b) {
    const uint32_t ua = __float_as_uint(a), ub = __float_as_uint(b);
    a -= __uint_as_float(ua & 0xffff0000u);
    b -= __uint_as_float(ub & 0xffff0000u);
    return __byte_perm(ua, ub, 0x7632);
}

}  // namespace mb
