// pfc_alloc.h -- one allocation for memory that is needed and a work space that
// is not.
#pragma once

#include <stddef.h>

namespace pfc {

// Allocates `need` bytes and, in the same block, `work` more at a multiple of
// 256; where that much is not to be had, `need` alone and *work_at = null.
// alloc(bytes) returns null where it fails.  One block: memory of 2 MB or more
// is mapped for itself, which takes 100 us.
template <class Alloc>
bool alloc_with_work(Alloc alloc, size_t need, size_t work, void** block, void** work_at)
{
    const size_t at = (need + 255) / 256 * 256;
    *work_at = nullptr;
    *block = work ? alloc(at + work) : nullptr;
    if (*block) *work_at = (char*)*block + at;
    else *block = alloc(need);
    return *block != nullptr;
}

}  // namespace pfc
