// host_view.h -- which host arrays a kernel may read where they are.  Plain
// code, so that a host program can run it on ranges of its own.
#pragma once

#include <cstddef>
#include <cstdint>

namespace dspg {

// The device address of the bytes at p, or null when a kernel may not access
// them all: view(q) is the device address of byte q, null when q is not in
// page-locked memory that the GPU reaches.  An array can start in such memory
// and end past it (cudaHostRegister takes any range), so the last byte has to
// be there too, as far from the first as on the host.  Memory is locked by
// the page: inside the first byte's page there is nothing more to ask.
template <class V>
inline void *range_view(V view, void *p, size_t bytes) {
    char *first = (char *)view(p);
    if (!first || ((uintptr_t)p ^ ((uintptr_t)p + (bytes ? bytes - 1 : 0))) < 4096) return first;
    const char *last = (const char *)view((char *)p + (bytes - 1));
    return last == first + (bytes - 1) ? first : nullptr;
}

// The same for an array of n values of `size` bytes each; null also when it
// is not aligned to them.
template <class V>
inline void *array_view(V view, void *p, int64_t n, size_t size) {
    if (!p || (uintptr_t)p % size != 0 || n < 0 || n > (int64_t)1 << 56) return nullptr;
    return range_view(view, p, (size_t)n * size);
}

}  // namespace dspg
