"""How a row of the acceptance is shared out (csrc/accept_share.h), driven on the host: every word of every vocabulary is somebody's, a
thread never holds more than it can, a share that fits is one batch, and what the shares have room for beyond the vocabulary is less
than a word per thread and batch.  On the GPU: every kernel for several batches at the edges of its range, against the oracle."""
import os
import subprocess

import pytest

import sv_inputs as si

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

DRIVER = r"""
#include <cstdio>
#include "accept_share.h"
int main()
{
    for (int ctas = 1; ctas <= 16; ctas *= 2)
        for (int vocab = 4; vocab <= 2000000; vocab += vocab < 40000 ? 4 : 4 * 97) {
            const svk::AcceptShare s = svk::accept_share(vocab, ctas);
            const long long words = vocab / 4, threads = ctas * svk::kAcceptThreads, room = threads * s.words * s.batches;
            const long long need = (words + threads - 1) / threads;
            const bool fits = need <= svk::kAcceptHeld;
            if (s.words < 1 || s.words > svk::kAcceptHeld || room < words || (s.batches == 1) != fits || (fits && s.words != need) ||
                (!fits && 2 * s.words <= svk::kAcceptHeld) || room - words >= threads * s.batches)
                return printf("vocabulary %d on %d CTAs: %d batches of %d words\n", vocab, ctas, s.batches, s.words), 1;
            // (so of n CTAs fewer than n / words have none: three of eight had, with eight words where five do)
            const long long idle = ctas - (words + room / ctas - 1) / (room / ctas);
            if (s.batches > 1 && idle * s.words >= ctas) return printf("vocabulary %d: %lld of %d CTAs idle\n", vocab, idle, ctas), 1;
        }
    const svk::AcceptShare s = svk::accept_share(151936, 8);
    return s.words == 5 && s.batches == 2 ? 0 : 1;
}
"""


def test_shares(tmp_path):
    src = tmp_path / "share.cpp"
    src.write_text(DRIVER)
    exe = tmp_path / "share"
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", os.path.join(ROOT, "paper_2512_21911_b200", "csrc"), str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout


@pytest.mark.gpu
@pytest.mark.parametrize("words", [9, 10, 11, 12, 13, 14, 15, 16])
def test_accept_of_several_batches(words):
    from test_accept_ranges import _check
    for V in (16384 * (words - 1) + 4, 16384 * words):   # on eight CTAs: more sequences than clusters of 16 fit
        c = si.make_accept_case(10, 4, V, seed=V, tree=True)
        c["parent"][:] = [-1, 0, 0, 0]
        c["u_accept"][::2] = 0.9995   # two rejections in a row, and the draw from a residual
        _check(c)
