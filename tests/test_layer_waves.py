"""A layer of more lists than SMs: handed out by turns, or whole lists in a first launch and the rest in clusters in a second one.  The rest's
pointers are the batch's moved on, so every sequence is compared with plain fp32 attention over its own list (bounds of test_wide_tiles)."""
import pytest
import torch

from test_wide_tiles import _reference

pytestmark = pytest.mark.gpu

SHAPES = [  # seqs, heads, kv_heads, block, draft, tree, kept blocks
    (19, 32, 8, 64, 5, True, 15),    # 144 lists whole, 8 in clusters
    (20, 64, 8, 64, 16, False, 16),  # ... of 128 rows
    (39, 8, 4, 128, 7, True, 8),     # 148 and 8, blocks of 128
    (149, 3, 1, 64, 3, True, 14),    # 148 and one
    (31, 32, 8, 64, 8, False, 5),    # 248 lists by turns
    (40, 16, 8, 64, 30, True, 4),    # 320, 60 rows
    (19, 8, 8, 64, 40, True, 6),     # 152, 40 rows of 40 draft tokens
    (40, 8, 8, 64, 40, True, 6),     # 320 of them by turns
]


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("entry", ["sv_verify_attn", "sv_verify_attn_reused"])
def test_waves_of_lists_against_plain_attention(shape, entry):
    import paper_2512_21911_b200 as sv
    S, Hq, Hkv, B, T, tree, keep = shape
    g = torch.Generator().manual_seed(S * T)
    gg = torch.Generator(device="cuda").manual_seed(T)
    NB = keep + 3
    lens = torch.tensor([NB * B - (s * 13) % B if s % 5 else 1 + (s * 29) % (NB * B) for s in range(S)], dtype=torch.int32)
    rnd = lambda *s: (torch.randn(s, generator=gg, device="cuda") * 1.5).to(torch.bfloat16)
    k, v, q = rnd(S * NB, Hkv, B, 128), rnd(S * NB, Hkv, B, 128), rnd(S, T, Hq, 128)
    dk, dv = rnd(S, T, Hkv, 128), rnd(S, T, Hkv, 128)
    table = torch.randperm(S * NB, generator=g, dtype=torch.int32).view(S, NB)
    parent = torch.arange(-1, T - 1, dtype=torch.int32).repeat(S, 1)
    if tree:
        for i in range(1, T):
            parent[:, i] = torch.randint(0, i, (S,), generator=g, dtype=torch.int32)
    # the same list for all heads of a sequence, so that the reference can cut the sequence to it
    idx, cnt, kept_table, kept_lens = torch.zeros((S, Hkv, keep), dtype=torch.int32), torch.zeros((S, Hkv), dtype=torch.int32), [], []
    for s in range(S):
        nb = -(-int(lens[s]) // B)
        n = min(nb, keep)
        chosen = torch.cat([torch.randperm(nb - 1, generator=g)[:n - 1].sort().values, torch.tensor([nb - 1])])   # the last one too
        idx[s, :, :n], cnt[s] = chosen.int(), n
        kept_table.append(torch.cat([table[s, chosen], torch.zeros(keep - n, dtype=torch.int32)]))
        kept_lens.append((n - 1) * B + int(lens[s]) - (nb - 1) * B)
    geom = sv.make_geom(S, Hq, Hkv, 128, B, NB, T)
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    out, lse = torch.full_like(q, float("nan")), torch.full((S, T, Hq), float("nan"), device="cuda")
    tables = table.cuda(), lens.cuda()
    getattr(sv, entry)(geom, q, sv.make_kv(k, v, *tables), dk, dv, parent.cuda() if tree else None, idx.cuda(), cnt.cuda(), out, lse=lse,
                       status_word=status)
    want = _reference(q, k, v, dk, dv, torch.stack(kept_table).cuda(), torch.tensor(kept_lens), parent, B)
    assert int(status) == 0 and bool(torch.isfinite(lse).all())
    assert float((out.float() - want).norm() / want.norm()) < 2.8e-3
    for s in range(S):
        err = (out[s].float() - want[s]).norm(dim=-1) / want[s].norm(dim=-1)
        assert float(err.max()) < 8.5e-3, (s, int(lens[s]), float(err.max()))
