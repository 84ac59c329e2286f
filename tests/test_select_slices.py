"""Selection over tables whose length is at, just above and just below what the CTAs of a cluster take in whole passes: every block
is scored once (fp32 sums of 128 products: a relative error of 128 ulp of the largest partial sum at most) and the list is the
one these scores give."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("seqs, heads", [(1, 2), (9, 8), (40, 8)])   # clusters of 8 or 16, of 4 or 2, single CTAs
@pytest.mark.parametrize("blocks", [1, 3, 4, 33, 63, 64, 65, 127, 129, 157, 256, 257, 258, 287, 512, 513, 515, 516, 517, 577, 1025, 2047, 2049, 2065, 4097])
def test_every_block_is_scored_once(seqs, heads, blocks):
    import paper_2512_21911_b200 as sv
    if seqs * heads * blocks > 400_000:
        pytest.skip("large")
    g = torch.Generator(device="cuda").manual_seed(blocks)
    reps = torch.randn((seqs, heads, blocks, 128), generator=g, device="cuda")
    q = torch.randn((seqs, 1, heads * 3, 128), generator=g, device="cuda").to(torch.bfloat16)
    lens = torch.randint(1, blocks * 64 + 1, (seqs,), generator=torch.Generator().manual_seed(blocks), dtype=torch.int32)
    lens[0] = blocks * 64
    keep = max(2, blocks // 3)
    geom = sv.make_geom(seqs, heads * 3, heads, 128, 64, blocks, 1)
    idx = torch.full((seqs, heads, keep), -1, dtype=torch.int32, device="cuda")
    cnt = torch.zeros((seqs, heads), dtype=torch.int32, device="cuda")
    scores = torch.full((seqs, heads, blocks), float("nan"), device="cuda")
    budget = torch.full((seqs,), keep, dtype=torch.int32, device="cuda")
    sv.sv_select_blocks(geom, q, reps, lens.cuda(), budget, 1, 1, idx, cnt, out_scores=scores)
    want = torch.einsum("shbd,shd->shb", reps.double(), q.double().view(seqs, heads, 3, 128).mean(2))
    for s in range(seqs):
        nb = -(-int(lens[s]) // 64)
        assert torch.isnan(scores[s, :, nb:]).all()
        got = scores[s, :, :nb]
        assert float((got.double() - want[s, :, :nb]).abs().max()) < 128 * 2.0 ** -24 * 128 * 4
        n = min(keep, nb)
        assert (cnt[s] == n).all()
        key = got.clone()
        key[:, 0] = key[:, nb - 1] = torch.inf
        order = torch.sort(key, dim=-1, descending=True, stable=True).indices[:, :n].sort(-1).values
        assert torch.equal(idx[s, :, :n].long(), order)
