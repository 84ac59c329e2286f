// Which stages of a TMA ring were last filled by a copy of their CTA's own, and at which parity of the stage's barrier that copy
// completes.  A CTA in which a role has given up waits for the stages that this names before it leaves: shared memory may not be
// given up under a copy.  (Host code may include this file.)
#pragma once
#include <stdint.h>

#ifdef __CUDACC__
#define SV_RING_FN __device__ __forceinline__
#else
#define SV_RING_FN inline
#endif

namespace svk {

struct RingCopies {
    uint32_t stages = 0, odd = 0;
    // the stage's round `it` (its it-th use, from 0 on) is a copy
    SV_RING_FN void copied(int stage, int it)
    {
        stages |= 1u << stage;
        odd = (odd & ~(1u << stage)) | ((uint32_t)(it & 1) << stage);
    }
    // ... is filled by somebody else (the copy before it has been read, so it is through)
    SV_RING_FN void filled_otherwise(int stage) { stages &= ~(1u << stage); }
    SV_RING_FN bool waits_for(int stage) const { return (stages >> stage) & 1u; }
    SV_RING_FN uint32_t parity(int stage) const { return (odd >> stage) & 1u; }
};

// Of a ring whose units first .. end - 1 are copies (a unit before them is not).
SV_RING_FN RingCopies copies_of_units(int first, int end, int n_stages)
{
    RingCopies ring;
    for (int u = end - n_stages > first ? end - n_stages : first; u < end; ++u) ring.copied(u % n_stages, u / n_stages);
    return ring;
}

// Whether threads that take every step-th unit of a ring each may wait for the units' full barriers.  A wait names a parity and passes
// while the barrier is in a phase of the other one, so it tells a unit only from the one before it on the same stage.  A thread that
// has waited for that one itself cannot be early; where it was another thread's, it may not have landed yet, and the
// wait for the unit a round later passes: the tile is read while it is being written, and the stage handed back with its copy in
// flight, so that its barrier is armed twice in a phase.
#ifdef __CUDACC__
__host__ __device__
#endif
constexpr bool stages_keep_their_thread(int n_stages, int step) { return n_stages % step == 0; }

}  // namespace svk
