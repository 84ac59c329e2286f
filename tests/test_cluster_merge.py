"""Splits that are merged inside a thread-block cluster: cluster sizes of two to eight, fewer rows than CTAs, shares that do not divide the
rows, lists so short that CTAs have no unit, one, or only the draft's.  Against plain fp32 attention, with the bounds of test_wide_tiles."""
import pytest
import torch

from test_wide_tiles import _reference

pytestmark = pytest.mark.gpu

SHAPES = [  # seqs, heads, kv_heads, block, draft, tree
    (1, 8, 1, 64, 8, True),       # 64 rows, eight CTAs
    (1, 4, 1, 64, 1, False),      # four rows: CTAs without rows
    (1, 8, 2, 64, 4, False),      # 16 rows
    (2, 32, 8, 64, 5, True),      # 20 rows over six CTAs
    (1, 16, 16, 64, 32, True),    # 32 draft tokens
    (4, 32, 8, 64, 8, False),     # four CTAs
    (4, 32, 8, 128, 3, True),     # blocks of 128
    (5, 28, 4, 64, 9, True),      # 63 rows
    (6, 32, 8, 64, 7, False),     # three splits, clusters of two
    (9, 32, 8, 64, 16, True),     # 64 rows, two CTAs
    (9, 64, 8, 64, 16, True),     # 128 rows, two CTAs
    (18, 28, 4, 128, 10, False),  # 70 rows, blocks of 128
    (4, 64, 8, 64, 16, False),    # 128 rows, four CTAs
    (4, 64, 8, 128, 16, True),    # ... cut at units
    (8, 28, 4, 64, 11, True),     # 77 rows over four CTAs
    (9, 40, 5, 64, 14, False),    # 112 rows over three CTAs
    (3, 8, 4, 64, 60, True),      # 120 rows of 60 draft tokens
    (2, 32, 8, 64, 60, True),     # two tiles, 128 and 112 rows, clusters of four
    (1, 28, 4, 128, 58, True),    # four tiles, the last one of 28 rows, cut at units
    (4, 32, 8, 64, 33, False),    # two tiles, the second one of four rows, clusters of two
]


@pytest.mark.parametrize("shape", SHAPES)
def test_cluster_merge_against_plain_attention(shape):
    import paper_2512_21911_b200 as sv
    S, Hq, Hkv, B, T, tree = shape
    g = torch.Generator().manual_seed(S * T)
    gg = torch.Generator(device="cuda").manual_seed(T)
    NB = 16 * 64 // B
    lengths = (1024, 0, 1, 64, 65, 1000, 128, 191, 300, 449, 640, 700, 1023)
    rnd = lambda *s: (torch.randn(s, generator=gg, device="cuda") * 1.5).to(torch.bfloat16)
    k, v, q = rnd(S * NB, Hkv, B, 128), rnd(S * NB, Hkv, B, 128), rnd(S, T, Hq, 128)
    dk, dv = rnd(S, T, Hkv, 128), rnd(S, T, Hkv, 128)
    table = torch.randperm(S * NB, generator=g, dtype=torch.int32).view(S, NB)
    parent = torch.arange(-1, T - 1, dtype=torch.int32).repeat(S, 1)
    if tree:
        for i in range(1, T):
            parent[:, i] = torch.randint(0, i, (S,), generator=g, dtype=torch.int32)
    geom = sv.make_geom(S, Hq, Hkv, 128, B, NB, T)
    assert sv.sv_verify_attn_splits(geom, NB) > 1
    table_d, parent_d = table.cuda(), parent.cuda() if tree else None
    workspace = torch.empty(sv.sv_workspace_bytes(geom, NB), dtype=torch.uint8, device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    for turn in range(len(lengths) if S == 1 else 1):   # a single sequence meets all lengths
        lens = torch.tensor([lengths[(s + turn) % len(lengths)] for s in range(S)], dtype=torch.int32)
        lens_d = lens.cuda()
        out, lse = torch.full_like(q, float("nan")), torch.full((S, T, Hq), float("nan"), device="cuda")
        sv.sv_verify_attn(geom, q, sv.make_kv(k, v, table_d, lens_d), dk, dv, parent_d, None, None, out, lse=lse, workspace=workspace,
                          status_word=status)
        want = _reference(q, k, v, dk, dv, table_d, lens, parent, B)
        assert int(status) == 0 and bool(torch.isfinite(lse).all())
        assert float((out.float() - want).norm() / want.norm()) < 2.8e-3
        for s in range(S):
            err = (out[s].float() - want[s]).norm(dim=-1) / want[s].norm(dim=-1)
            assert float(err.max()) < 8.5e-3, (s, int(lens[s]), float(err.max()))
