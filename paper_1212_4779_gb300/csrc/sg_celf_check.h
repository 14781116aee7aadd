// sg_celf_check.h -- lazy evaluation's check of itself: what each seed newly
// covered against the gain it was chosen for (host code, no CUDA).
#pragma once

#include <stdint.h>

namespace sgi {

// First of k seeds whose newly covered (node, snapshot) pairs are not its gain,
// -1 if there is none.  before[i]: pairs covered when seed i was chosen, after:
// pairs covered at the end.  Comparing the two sums alone would let errors that
// cancel pass.
inline int32_t celf_first_mismatch(const long long *before, long long after, const int64_t *gains, int32_t k)
{
    for (int32_t i = 0; i < k; ++i)
        if ((i + 1 < k ? before[i + 1] : after) - before[i] != (long long)gains[i]) return i;
    return -1;
}

}  // namespace sgi
