// How a row of the acceptance (accept.cu) is shared out: 16-byte words per thread and batch, and batches.  Plain C++, so that
// the host can be asked as well.
#pragma once

namespace svk {

constexpr int kAcceptThreads = 512;   // threads of a CTA
constexpr int kAcceptHeld = 8;        // words of either distribution that a thread can hold (64 registers)

struct AcceptShare {
    int words;     // words per thread and batch
    int batches;   // 1: a thread holds its whole share of a row in registers
};

// A vocabulary over `ctas` CTAs.  Every CTA has the same number of words a thread, so what is rounded up is left out by the
// last ones: the batches are no larger than they have to be, less than one word per thread and batch stays unused.  (151936
// entries on 8 CTAs are 10 words a thread: two batches of five.  Two of eight filled five CTAs and left three without any: 12
// sequences 38.9 -> 28.7 us with nothing in L2, 32 with four rejections in a row 92 -> 68; 262148 entries, 8 sequences 49 -> 39;
// 128256, one batch, the same.)
constexpr AcceptShare accept_share(int vocab, int ctas)
{
    const int threads = ctas * kAcceptThreads, need = (vocab / 4 + threads - 1) / threads;
    const int batches = need > kAcceptHeld ? (need + kAcceptHeld - 1) / kAcceptHeld : 1;
    return {need > 0 ? (need + batches - 1) / batches : 1, batches};
}

}  // namespace svk
