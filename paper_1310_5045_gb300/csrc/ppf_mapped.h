// ppf_mapped.h -- which caller buffers a kernel may store to directly.
#pragma once

#include <cstddef>
#include <cstdint>

namespace ppf {

// The device address of the caller's page-locked p[0, bytes) when a kernel may
// store 8-byte words there, else nullptr: the words must be aligned, and the
// last byte must be mapped where the first one's mapping puts it (a registered
// range can end inside the buffer).  Memory is mapped in whole pages of at
// least 4096 bytes, so a last byte on the first one's page is not asked for (a
// question costs about 0.2 us of the 2.7 us a queued estimate takes the host).
// bytes <= 4096.  map(p) is the device address of one mapped host byte, nullptr
// where there is none.
template <typename Map>
inline void *mapped_words(void *p, size_t bytes, Map map)
{
    if (reinterpret_cast<uintptr_t>(p) % 8 != 0)
        return nullptr;
    char *first = static_cast<char *>(map(p));
    if (!first || reinterpret_cast<uintptr_t>(first) % 8 != 0)
        return nullptr;
    char *end = static_cast<char *>(p) + bytes - 1;
    if (reinterpret_cast<uintptr_t>(end) / 4096 == reinterpret_cast<uintptr_t>(p) / 4096)
        return first;
    return map(end) == first + bytes - 1 ? first : nullptr;
}

}  // namespace ppf
