// host_view.h -- which host arrays a kernel may read where they are.  Plain
// code, so that a host program can run it on ranges of its own.
#pragma once

#include <cstddef>

namespace dspg {

// The device address of the bytes at p, or null when a kernel may not read
// them all: view(q) is the device address of byte q, null when q is not in
// page-locked memory that the GPU reaches.  An array can start in such memory
// and end past it (cudaHostRegister takes any range), so the last byte has to
// be there too, as far from the first as on the host.
template <class V>
inline void *range_view(V view, void *p, size_t bytes) {
    char *first = (char *)view(p);
    if (!first || bytes <= 1) return first;
    const char *last = (const char *)view((char *)p + (bytes - 1));
    return last == first + (bytes - 1) ? first : nullptr;
}

}  // namespace dspg
