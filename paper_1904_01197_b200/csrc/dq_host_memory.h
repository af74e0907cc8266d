// Which host buffers the kernels of the *_host calls may work on without a copy: page-locked ones, from the first byte
// to the last.  (No CUDA here: the decision is tested with made-up ranges.)
#pragma once

#include <stdint.h>

namespace dq {

// The page-locked range (one allocation or one registration) that an address lies in.
struct PinnedRange {
    uint64_t device;      // device address of the byte that was asked about
    uint64_t start, size; // the range
};

// Device address of `bytes` bytes of host memory that one page-locked range holds completely; 0 for anything else, also
// for a buffer that begins in such a range and ends outside (part of an allocation may be registered: the kernels would
// run into unmapped memory), and for a device address that is not 16-byte aligned.
// look(address, &range): the range that an address lies in, false when it is not page-locked.
template <typename Look>
uint64_t pinned_device_address(const void* host, uint64_t bytes, Look look)
{
    PinnedRange r = {0u, 0u, 0u};
    if (host == nullptr || !look(host, &r)) return 0u;
    const uint64_t p = static_cast<uint64_t>(reinterpret_cast<uintptr_t>(host));
    if (p < r.start || bytes > r.size || p - r.start > r.size - bytes) return 0u;
    return (r.device & 15u) == 0u ? r.device : 0u;
}

}  // namespace dq
