// pinned_range.cuh -- whether a batch of host rasters lies in pinned memory as
// a whole.  A pointer into pinned memory says nothing about the bytes that
// follow it: a program may have registered the first part of a larger array.
// A copy call checks the range that it is given; a kernel that reads the
// device mapping would go on past its end.
#pragma once

#include <stddef.h>
#include <stdint.h>

namespace cpt {

// Whether the `bytes` bytes from p lie in the one allocation or registration
// that query(p, &start, &size) reports for p (false: it knows none).
template <typename Query>
bool in_one_range(const void *p, int64_t bytes, Query query) {
    uintptr_t start = 0;
    size_t size = 0;
    if (bytes < 0 || !query(p, &start, &size)) return false;
    const uintptr_t at = reinterpret_cast<uintptr_t>(p);
    return at >= start && at - start <= size && (uint64_t)bytes <= size - (at - start);
}

}  // namespace cpt
