// host_view.h -- the device address of a page-locked host array (plain C++, no CUDA headers).
#pragma once

#include <algorithm>
#include <cstdint>

namespace fdllm {

// device_of(p): the device address through which the GPU reaches the host byte p, null for memory
// that is not page-locked.  Host memory is locked by pages, so one byte of each page speaks for it:
// the address of the first byte where every page of the array is mapped in one piece, else null.
template <typename DeviceOf>
uint8_t *whole_view(uint8_t *host, int64_t bytes, int64_t page, DeviceOf device_of)
{
    uint8_t *const first = device_of(host);
    if (first == nullptr)
        return nullptr;
    for (int64_t at = 0; at < bytes - 1;) {
        at = std::min(at + page, bytes - 1);
        if (device_of(host + at) != first + at)
            return nullptr;
    }
    return first;
}

}  // namespace fdllm
