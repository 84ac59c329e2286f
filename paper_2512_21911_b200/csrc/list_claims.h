// How the lists of a launch are handed out to its CTAs through two words in global memory, zero before and after a launch:
// word 0 counts the claims, word 1 the CTAs that have left.  CTA i starts with list i; a claim gives it the list of that number
// behind those first ones, or refuses it (-1) when there are none left.  A CTA that gives up just leaves: the lists it
// has not claimed go to the others, and the words still come back to zero, because the last CTA to leave -- by then every claim
// has been made -- clears both.  (Host code may include this file: Words stands for the two atomics.)
#pragma once
#include <stdint.h>

#ifdef __CUDACC__
#define SV_CLAIMS_FN __host__ __device__ inline
#else
#define SV_CLAIMS_FN inline
#endif

namespace svk {

// The list of the claim that found `before` claims made (n_lists >= n_ctas).
SV_CLAIMS_FN int claimed_list(uint32_t before, int n_lists, int n_ctas)
{
    return before < (uint32_t)(n_lists - n_ctas) ? (int)before + n_ctas : -1;
}

// Behind a CTA's last claim, once per CTA.
template <class Words>
SV_CLAIMS_FN void leave_claims(Words words, int n_ctas)
{
    if (words.add(1, 1u) == (uint32_t)n_ctas - 1u) {
        words.set(0, 0u);
        words.set(1, 0u);
    }
}

}  // namespace svk
