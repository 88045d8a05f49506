// Two buffers that are used together: allocated both or neither, so that a caller that
// looks at one of them knows about the other.  No CUDA in here: `alloc(void**, size_t)`
// returns whether it succeeded, `release(void*)` frees.
#pragma once

#include <cstddef>

namespace jdft {

template <typename Alloc, typename Release>
bool alloc_pair(void** a, size_t bytes_a, void** b, size_t bytes_b, Alloc alloc, Release release) {
    if (*a && *b) return true;
    if (!alloc(a, bytes_a)) {
        *a = nullptr;
        return false;
    }
    if (!alloc(b, bytes_b)) {
        release(*a);
        *a = *b = nullptr;
        return false;
    }
    return true;
}

}  // namespace jdft
