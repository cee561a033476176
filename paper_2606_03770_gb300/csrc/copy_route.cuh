// copy_route.cuh -- which of the copies between a context's arrays and the
// caller's may be made by one kernel.  Plain C++, so that it is tested on the host.
#pragma once

#include <stddef.h>

namespace e2 {

// A kernel on the context's stream may read or write an array of the caller's
// when the array is device memory of the context's own device (`owner` and
// `context` are device ids) and that device is current, as a launch on its
// stream needs.  With another device current, or for another device's array, a
// copy call works and a kernel does not: its launch is refused, or, on the
// default stream, it runs on the wrong device.
constexpr bool copied_by_kernel(bool device_memory, int owner, int context, int current)
{
    return device_memory && owner == context && current == context;
}

// Whether two arrays share a byte.  The blocks of one kernel write in no order,
// so outputs that do must not be written by the same one.
inline bool overlap(const unsigned char *a, size_t na, const unsigned char *b, size_t nb)
{
    return a < b + nb && b < a + na;
}

}  // namespace e2
