"""How lists are handed out to the CTAs of a launch (csrc/list_claims.h), driven on the host: CTAs in random interleavings, some of which
give up after a random number of lists.  No list is taken twice, a launch with a healthy CTA left takes all lists but those the
others held or had just claimed, and the words are zero again, so that the launch behind is complete."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

DRIVER = r"""
#include <cstdio>
#include <cstdlib>
#include <random>
#include <vector>
#include "list_claims.h"
struct Words {
    uint32_t *at;
    uint32_t add(int i, uint32_t v) const { const uint32_t b = at[i]; at[i] += v; return b; }
    void set(int i, uint32_t v) const { at[i] = v; }
};
struct Cta { int list, until; bool left; };   // gives up once it has worked on `until` lists
int main()
{
    std::mt19937 rng(1);
    for (int trial = 0; trial < 20000; ++trial) {
        uint32_t words[2] = {0, 0};
        for (int launch = 0; launch < 2; ++launch) {
            const int n_ctas = 1 + rng() % 12, n_lists = n_ctas + rng() % 60;
            const bool faults = launch == 0;
            std::vector<Cta> ctas(n_ctas);
            std::vector<int> taken(n_lists, 0), lost(n_lists, 0);
            for (int i = 0; i < n_ctas; ++i) ctas[i] = {i, faults && rng() % 3 == 0 ? (int)(rng() % 6) : 1 << 30, false};
            int here = n_ctas;
            bool healthy = false;
            for (auto &c : ctas) healthy = healthy || c.until == 1 << 30;
            while (here) {
                Cta &c = ctas[rng() % n_ctas];
                if (c.left) continue;
                // the claim for the list behind this one is made before this one is worked on
                const int next = svk::claimed_list(Words{words}.add(0, 1u), n_lists, n_ctas);
                const bool gives_up = c.until == 0;
                taken[c.list]++;
                if (gives_up) { lost[c.list] = 1; if (next >= 0) { taken[next]++; lost[next] = 1; } }
                if (gives_up || next < 0) {
                    c.left = true, --here;
                    svk::leave_claims(Words{words}, n_ctas);
                } else {
                    c.list = next, --c.until;
                }
            }
            if (words[0] || words[1]) return printf("words %u %u\n", words[0], words[1]), 1;
            for (int l = 0; l < n_lists; ++l) {
                if (taken[l] > 1) return printf("list %d taken %d times\n", l, taken[l]), 1;
                if (healthy && !taken[l]) return printf("list %d never taken\n", l), 1;
                if (!faults && lost[l]) return printf("list %d lost\n", l), 1;
            }
        }
    }
    // refused, however far the count is
    for (uint32_t before : {852u, 0x7fffffffu, 0xf0000000u, 0xffffffffu})
        if (svk::claimed_list(before, 1000, 148) != -1) return printf("count %u\n", before), 1;
    return svk::claimed_list(851, 1000, 148) != 999 || svk::claimed_list(0, 1000, 148) != 148;
}
"""


def test_claims_with_ctas_that_give_up(tmp_path):
    src = tmp_path / "claims.cpp"
    src.write_text(DRIVER)
    exe = tmp_path / "claims"
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", os.path.join(ROOT, "paper_2512_21911_b200", "csrc"), str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout
