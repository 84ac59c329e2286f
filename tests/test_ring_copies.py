"""Which copies a CTA has to wait for before it leaves (csrc/ring_copies.h), driven on the host against a model of the ring's barriers:
units that are copies and units that are filled otherwise in random order, stopped anywhere.  The stages named are those
whose latest use is a copy, and the parity named is one that the barrier passes exactly when that copy has landed."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

DRIVER = r"""
#include <cstdio>
#include <random>
#include "ring_copies.h"
int main()
{
    std::mt19937 rng(1);
    for (int trial = 0; trial < 20000; ++trial) {
        const int n_stages = 1 + rng() % 6, units = rng() % 40, filled = rng() % 5;
        svk::RingCopies ring;
        int last_is_copy[6] = {}, uses[6] = {};
        for (int u = 0; u < units; ++u) {
            const int stage = u % n_stages, it = u / n_stages;
            const bool copy = (int)(rng() % 5) >= filled;
            copy ? ring.copied(stage, it) : ring.filled_otherwise(stage);
            last_is_copy[stage] = copy, uses[stage] = it + 1;
        }
        for (int s = 0; s < n_stages; ++s) {
            if (ring.waits_for(s) != (last_is_copy[s] != 0)) return printf("stage %d of %d, %d units\n", s, n_stages, units), 1;
            if (!ring.waits_for(s)) continue;
            // a parity wait passes while the barrier's current phase has the other parity; every earlier use has completed
            const auto passes = [&](int phases_done) { return (uint32_t)(phases_done & 1) != ring.parity(s); };
            if (passes(uses[s] - 1) || !passes(uses[s])) return printf("parity of stage %d, use %d\n", s, uses[s]), 1;
        }
    }
    // one unit that is no copy, or none, then copies: the same as noting each of them
    for (int n_stages = 1; n_stages <= 6; ++n_stages)
        for (int first = 0; first <= 1; ++first)
            for (int end = 0; end <= 20; ++end) {
                svk::RingCopies want;
                for (int u = first; u < end; ++u) want.copied(u % n_stages, u / n_stages);
                const svk::RingCopies got = svk::copies_of_units(first, end, n_stages);
                for (int s = 0; s < n_stages; ++s)
                    if (got.waits_for(s) != want.waits_for(s) || (got.waits_for(s) && got.parity(s) != want.parity(s)))
                        return printf("%d stages, units %d..%d, stage %d\n", n_stages, first, end, s), 1;
            }
    return 0;
}
"""


def test_stages_to_wait_for(tmp_path):
    src = tmp_path / "ring.cpp"
    src.write_text(DRIVER)
    exe = tmp_path / "ring"
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", os.path.join(ROOT, "paper_2512_21911_b200", "csrc"), str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout
