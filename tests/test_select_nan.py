"""Scores that are not numbers: the key of a score (csrc/order_key.h), driven on the host, is never that of a block kept without eviction; on the
GPU a NaN query or NaN representatives leave every list at its length, with the NaN blocks between the negative scores and zero, and nothing behind it written."""
import math
import os
import subprocess

import pytest
import torch

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

DRIVER = r"""
#include <cmath>
#include <cstdio>
#include <cstring>
#include "order_key.h"
static float number(uint32_t bits) { float x; memcpy(&x, &bits, 4); return x; }
int main()
{
    using svsel::key_of_bits;
    for (uint64_t b = 0; b < 1ull << 32; b += (b & 0x7FFFFF) < 3 || (b & 0x7FFFFF) > 0x7FFFF0 ? 1 : 61)
        if (key_of_bits((uint32_t)b) == svsel::kForcedKey) return printf("%08x has the key of a forced block\n", (unsigned)b), 1;
    // neighbouring numbers, from -inf to +inf, in their order; arithmetic's NaN between the largest negative one and zero
    for (uint32_t b = 0x807FFFFFu; b < 0xFF800000u; b += 4099)
        if (!(number(b + 1) < number(b) && key_of_bits(b + 1) < key_of_bits(b))) return printf("order at %08x\n", b), 1;
    for (uint32_t b = 0; b < 0x7F800000u; b += 4099)
        if (!(number(b) < number(b + 1) && key_of_bits(b) < key_of_bits(b + 1))) return printf("order at %08x\n", b), 1;
    if (!(key_of_bits(0xFF800000u) < key_of_bits(0x80800000u) && key_of_bits(0x80000001u) < key_of_bits(0u))) return printf("signs\n"), 1;
    const uint32_t nan = 0x7FFFFFFFu;
    if (!std::isnan(number(nan)) || key_of_bits(nan) <= key_of_bits(0x80000001u) || key_of_bits(nan) >= key_of_bits(0u)) return printf("NaN\n"), 1;
    return 0;
}
"""


def test_no_score_has_the_key_of_a_forced_block(tmp_path):
    src, exe = tmp_path / "key.cpp", tmp_path / "key"
    src.write_text(DRIVER)
    subprocess.run(["g++", "-std=c++17", "-O2", "-I", os.path.join(ROOT, "paper_2512_21911_b200", "csrc"), str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout


@pytest.mark.gpu
@pytest.mark.parametrize("seqs", [24, 320])   # CTAs of 512 threads, of 256
@pytest.mark.parametrize("nb", [20, 47, 48, 64, 65, 96, 97, 300, 700, 1100, 2500, 4300])   # every way a list is selected
def test_lists_of_nan_scores_keep_their_length(seqs, nb):
    import paper_2512_21911_b200 as sv
    g = torch.Generator().manual_seed(nb)
    keep, n_sink, n_local = 11, 1, 2
    scores = torch.randn((seqs, nb), generator=g)
    nan = float("nan")
    for s in range(seqs):
        n_nan = (0, 1, 2, 5, 9, nb // 2, nb)[s % 7]   # none, fewer than are kept, more, all
        scores[s, torch.randperm(nb, generator=g)[:n_nan]] = nan if s % 2 else -nan
        if s % 5 == 1:
            scores[s, nb // 3] = float("inf")
    reps = torch.zeros((seqs, 1, nb, 128))
    reps[:, 0, :, 0] = scores
    q = torch.zeros((seqs, 1, 1, 128))
    q[..., 0] = 1.0
    q[3::7, ..., 0] = nan    # (every score of these)
    scores[3::7] = nan
    room = torch.full((seqs * keep + 2 * nb,), -7, dtype=torch.int32, device="cuda")   # room for all that could be written behind the lists
    idx, cnt = room[:seqs * keep].view(seqs, 1, keep), torch.zeros((seqs, 1), dtype=torch.int32, device="cuda")
    lens, budget = torch.full((seqs,), nb * 64, dtype=torch.int32), torch.full((seqs,), keep, dtype=torch.int32)
    sv.sv_select_blocks(sv.make_geom(seqs, 1, 1, 128, 64, nb, 1), q.bfloat16().cuda(), reps.cuda(), lens.cuda(), budget.cuda(), n_sink, n_local,
                        idx, cnt)
    assert bool((room[seqs * keep:] == -7).all()) and bool((cnt == keep).all())
    forced = [0, nb - 2, nb - 1]
    got = idx.cpu()
    for s, of in enumerate(scores.tolist()):
        rest = sorted(range(1, nb - 2), key=lambda b: (-of[b], b) if not math.isnan(of[b]) else (1e-40, b))
        assert got[s, 0].tolist() == sorted(forced + rest[:keep - 3]), (s, nb)


@pytest.mark.gpu
@pytest.mark.parametrize("n_sink, n_local", [(1 << 30, 1 << 30), (2 ** 31 - 1, 1), (2 ** 31 - 1, 2 ** 31 - 1), (12, 0)])
def test_forced_blocks_beyond_the_list_are_refused(n_sink, n_local):
    import paper_2512_21911_b200 as sv
    q, reps = torch.ones((1, 1, 1, 128), device="cuda").bfloat16(), torch.zeros((1, 1, 64, 128), device="cuda")
    idx, cnt = torch.full((1, 1, 11), -7, dtype=torch.int32, device="cuda"), torch.full((1, 1), -7, dtype=torch.int32, device="cuda")
    i32 = lambda x: torch.tensor([x], dtype=torch.int32, device="cuda")
    with pytest.raises(sv.SvError) as e:
        sv.sv_select_blocks(sv.make_geom(1, 1, 1, 128, 64, 64, 1), q, reps, i32(64 * 64), i32(11), n_sink, n_local, idx, cnt)
    assert e.value.status == 4 and bool((idx == -7).all()) and int(cnt) == -7
