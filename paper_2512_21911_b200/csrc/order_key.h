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

// The key of a score with these bits: larger score, larger key.  The map of numbers, taken literally, gives the NaN of the GPU's arithmetic
// (0x7fffffff, the only one that a score can be) kForcedKey: every block of a list whose query or representatives hold one would count as
// kept without eviction, more than the list has room for.  It ranks between the negative numbers and zero, where nvcc 12.9, which makes
// float operations of the map, has had it all along; it does not depend on the compiler now.  (Told apart by its key, not by its bits:
// 4 x 128K, selection and attention, 28.05 us without, 28.36 by its bits, no difference this way.)
SV_KEY_FN uint32_t key_of_bits(uint32_t bits)
{
    const uint32_t k = (bits & 0x80000000u) ? ~bits : (bits | 0x80000000u);
    return k == kForcedKey ? 0x7FFFFFFFu : k;
}

}  // namespace svsel
