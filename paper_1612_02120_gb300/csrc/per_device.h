// per_device.h - things that are set once per device. A kernel's shared-memory attribute belongs to the
// device that was current when it was set, and a process may hold nets on several.
#pragma once
#include <stdint.h>

#include <atomic>

#include "../../include/membrane.h"

namespace mb {

// Calls set() unless it has succeeded for this device before. Two threads may both call it: setting it
// twice does no harm. Devices beyond 63 are set on every call.
template <class Set>
mb_status once_per_device(std::atomic<uint64_t>& done, int device, Set set) {
    const uint64_t bit = device >= 0 && device < 64 ? (uint64_t)1 << device : 0;
    if (done.load(std::memory_order_acquire) & bit) return MB_OK;
    const mb_status s = set();
    if (s == MB_OK) done.fetch_or(bit, std::memory_order_release);
    return s;
}

}  // namespace mb
