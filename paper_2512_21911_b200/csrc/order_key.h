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

// The key of a score with these bits: larger score, larger key.  A NaN ranks between the negative numbers and zero.  It is told apart because
// the map of numbers, taken literally, gives the NaN of arithmetic (0x7fffffff) kForcedKey: every block of a list whose query or
// representatives hold one would count as kept without eviction, more than the list has room for.  (nvcc 12.9 makes float operations of the
// map, which give 0x7fffffff: that is where a NaN has ranked all along, and it does not depend on the compiler now.)
SV_KEY_FN uint32_t key_of_bits(uint32_t bits)
{
    if ((bits & 0x7FFFFFFFu) > 0x7F800000u) return 0x7FFFFFFFu;
    return (bits & 0x80000000u) ? ~bits : (bits | 0x80000000u);
}

}  // namespace svsel
