// The order-preserving key of a block's score: what block selection (select_core.cuh) compares.  Plain C++, so that the host can be asked
// as well.
#pragma once
#include <stdint.h>

#ifdef __CUDACC__
#define SV_KEY_FN __host__ __device__ inline
#else
#define SV_KEY_FN inline
#endif

namespace svsel {

constexpr uint32_t kForcedKey = 0xFFFFFFFFu;   // key of a block that is kept whatever its score (sink / local)

// The key of a score with these bits: larger score, larger key.  The NaN that arithmetic gives has all bits below its sign set, and would get
// kForcedKey: every block of a list whose query or representatives hold one would count as kept without eviction, more than the list has
// room for.  It ranks just below instead, above every number, equal NaNs by their index.
SV_KEY_FN uint32_t key_of_bits(uint32_t bits)
{
    const uint32_t k = (bits & 0x80000000u) ? ~bits : (bits | 0x80000000u);
    return k < kForcedKey ? k : kForcedKey - 1u;
}

}  // namespace svsel
