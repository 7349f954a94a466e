// ppf_mapped.h -- which caller buffers a kernel may store to directly.
#pragma once

#include <cstddef>
#include <cstdint>

namespace ppf {

// The device address of the caller's page-locked p[0, bytes) when a kernel may
// store 8-byte words there, else nullptr: the words must be aligned, and the
// last byte must be mapped where the first one's mapping puts it (a registered
// range can end inside the buffer).  map(p) is the device address of one
// mapped host byte, nullptr where there is none.
template <typename Map>
inline void *mapped_words(void *p, size_t bytes, Map map)
{
    if (reinterpret_cast<uintptr_t>(p) % 8 != 0)
        return nullptr;
    char *first = static_cast<char *>(map(p));
    if (!first || reinterpret_cast<uintptr_t>(first) % 8 != 0)
        return nullptr;
    const void *last = map(static_cast<char *>(p) + bytes - 1);
    return last == first + bytes - 1 ? first : nullptr;
}

}  // namespace ppf
