"""A stack's attention launch with its lists handed out to one CTA per SM, against the layers one by one, which the other
tests compare with the oracle.  Sizes where it can go wrong: lists of one block and of many, lengths that end inside a
block, blocks of 128, every row layout, one list more than SMs, launches of fewer."""
import pytest
import torch

pytestmark = pytest.mark.gpu

SHAPES = [  # layers, anchors every, seqs, lo, hi, heads, kv_heads, block, draft, tree, keep, max_sel
    (10, 2, 2, 6000, 7000, 32, 8, 64, 8, False, 100, 110),    # 32 rows
    (20, 1, 3, 1, 700, 8, 8, 64, 1, False, 9, 9),             # one row, 480 lists of 1 to 9 blocks
    (149, 4, 1, 2000, 2011, 4, 1, 64, 5, True, 20, 20),       # one list more than SMs
    (9, 1, 3, 1500, 4000, 64, 8, 64, 7, True, 50, 60),        # 56 rows
    (8, 3, 3, 2000, 5001, 64, 8, 128, 16, True, 30, 40),      # 128 rows, blocks of 128
    (8, 2, 4, 700, 2000, 16, 16, 64, 40, True, 20, 30),       # more than 32 draft tokens, 40 rows
    (12, 1, 5, 900, 2500, 28, 4, 64, 12, True, 33, 40),       # 84 rows (7 query heads per KV head)
    (10, 2, 6, 1500, 4000, 8, 4, 64, 60, True, 50, 60),       # 120 rows
    (4, 1, 6, 1000, 2500, 32, 8, 64, 60, True, 30, 40),       # two row tiles
    (5, 3, 7, 2000, 4500, 40, 8, 128, 26, False, 20, 30),     # two row tiles of 125 and 5 rows, blocks of 128
    (3, 1, 100, 1, 200, 32, 8, 64, 3, False, 3, 5),           # lists of no more than four blocks
]


@pytest.mark.parametrize("shape", SHAPES)
def test_lists_handed_out_equal_layer_by_layer(shape):
    import paper_2512_21911_b200 as sv
    from paper_2512_21911_b200 import binding
    L, every, S, lo, hi, Hq, Hkv, B, T, tree, keep, max_sel = shape
    g = torch.Generator().manual_seed(L + T)
    gg = torch.Generator(device="cuda").manual_seed(7)
    lens = torch.randint(lo, hi + 1, (S,), generator=g, dtype=torch.int32)
    lens[0] = hi
    NB = -(-hi // B)
    n_pages = 131   # (sequences may share pages: nothing is written to them)
    table = torch.randint(0, n_pages, (S, NB), generator=g, dtype=torch.int32)
    parent = None
    if tree:
        parent = torch.full((S, T), -1, dtype=torch.int32)
        for i in range(1, T):
            parent[:, i] = torch.randint(0, i, (S,), generator=g, dtype=torch.int32)
        parent = parent.cuda()
    budget = torch.randint(2, keep + 1, (S,), generator=g, dtype=torch.int32)
    budget[-1] = keep
    eng = sv.SparseVerifier(n_seq=S, n_q_heads=Hq, n_kv_heads=Hkv, head_dim=128, block_size=B, max_blocks=NB, n_draft=T, n_layers=L,
                            block_table=table.cuda(), seq_lens=lens.cuda(), budget_blocks=budget.cuda(), max_sel=max_sel,
                            anchors=[l % every == 0 for l in range(L)], parent=parent)
    rnd = lambda *s: torch.randn(s, generator=gg, device="cuda").to(torch.bfloat16)
    eng.set_kv_stack(rnd(L, n_pages, Hkv, B, 128), rnd(L, n_pages, Hkv, B, 128))
    for l in range(L):
        eng.build_reps(l)
    q, dk, dv = 2 * rnd(L, S, T, Hq, 128), rnd(L, S, T, Hkv, 128), rnd(L, S, T, Hkv, 128)
    out, want = torch.full_like(q, float("nan")), torch.full_like(q, float("nan"))

    def check():
        a, b = want.float(), out.float()
        assert torch.isfinite(b).all()
        assert (b - a).norm() <= 5e-3 * a.norm() and (b - a).abs().max() <= 0.03 * a.abs().max()
        assert ((b - a).norm(dim=-1) <= 1e-2 * a.norm(dim=-1)).all()

    handed = Hq // Hkv * T <= 64   # (128-row tiles are left to a CTA per list)
    assert L * S * Hkv > 148 and (binding._native.workspace_bytes_layers(eng.geom, L, max_sel) == 256) == handed
    for _ in range(2):   # (the counter of the launch before must not matter)
        eng.verify_step(q, dk, dv, out)
    for l in range(L):
        eng.verify_layer(l, q[l], dk[l], dv[l], want[l])
    check()
    # the same bits whichever layers a launch covers
    again = torch.full_like(q, float("nan"))
    for c0, c1 in ((0, 1), (1, L - 1), (L - 1, L)):
        assert eng._run_layers(c0, c1, q, dk, dv, again)
    assert torch.equal(again, out)
    out.fill_(float("nan")), want.fill_(float("nan"))
    eng.dense_step(q, dk, dv, out)
    for l in range(L):
        eng.dense_layer(l, q[l], dk[l], dv[l], want[l])
    check()
    assert not handed or int(eng._stack_workspace[0].max()) == 0, "the launches left their counter behind"
    eng.check_status()
