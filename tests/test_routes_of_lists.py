"""Every way a layer's lists are taken, each asserted by its launches and by what it leaves in the workspace, over lists of their own for every
(sequence, KV head), of no block up to all: merged in clusters, by the merge kernel (both of its forms), whole with a rest in clusters, by
turns.  Against plain fp32 attention (bounds of test_wide_tiles); sv_verify_attn_noalloc and sv_verify_attn_reused against sv_verify_attn."""
import pytest
import torch

pytestmark = pytest.mark.gpu

ROUTES = [  # seqs, heads, kv_heads, block, draft, tree, kept blocks, splits, launches
    (1, 8, 2, 64, 4, False, 16, 16, 1),      # clusters of eight
    (4, 32, 8, 64, 8, True, 32, 4, 1),       # ... of four
    (6, 32, 8, 64, 7, False, 20, 3, 1),      # ... of two or three
    (4, 64, 8, 128, 16, True, 12, 4, 1),     # 128 rows, cut at units
    (2, 32, 8, 64, 60, True, 16, 4, 1),      # two row tiles
    (5, 8, 8, 64, 40, True, 12, 3, 2),       # merged by the kernel that loads four splits at a time
    (1, 8, 8, 64, 40, True, 13, 13, 2),      # ... twenty at a time
    (2, 8, 8, 128, 33, False, 24, 8, 2),
    (1, 16, 2, 64, 8, False, 200, 67, 2),    # (more splits than that)
    (19, 32, 8, 64, 5, True, 15, 1, 2),      # 144 lists whole, 8 in clusters
    (20, 64, 8, 64, 16, False, 16, 1, 2),    # ... of 128 rows
    (149, 3, 1, 64, 3, True, 14, 1, 2),      # 148 and one
    (31, 32, 8, 64, 8, False, 5, 1, 1),      # 248 lists by turns
    (40, 8, 8, 64, 40, True, 6, 1, 1),       # 320 of them, of more than 32 draft tokens
]


def _plain(q, k, v, dk, dv, table, lens, parent, idx, cnt, block):
    S, T, Hq, D = q.shape
    Hkv = dk.shape[2]
    G = Hq // Hkv
    out = torch.zeros_like(q, dtype=torch.float32)
    for s in range(S):
        sees = torch.zeros((T, T), dtype=torch.bool)
        for i in range(T):
            j = i
            while j >= 0:
                sees[i, j] = True
                j = int(parent[s, j])
        sees = sees.to(q.device)
        for h in range(Hkv):
            blocks = idx[s, h, :int(cnt[s, h])].long()
            at = (blocks[:, None] * block + torch.arange(block, device=q.device)).flatten() < int(lens[s])
            rows = lambda pool, own: torch.cat([pool[table[s, blocks].long(), h].reshape(-1, D)[at].float(), own[s, :, h].float()])
            logits = torch.einsum("tgd,nd->tgn", q[s, :, h * G:(h + 1) * G].float(), rows(k, dk)) * D ** -0.5
            logits[:, :, int(at.sum()):].masked_fill_(~sees[:, None], -torch.inf)
            out[s, :, h * G:(h + 1) * G] = torch.einsum("tgn,nd->tgd", torch.softmax(logits, -1), rows(v, dv))
    return out


@pytest.mark.parametrize("route", ROUTES)
def test_lists_of_their_own_on_every_route(route):
    import paper_2512_21911_b200 as sv
    S, Hq, Hkv, B, T, tree, keep, splits, launches = route
    g = torch.Generator().manual_seed(S * T + keep)
    gg = torch.Generator(device="cuda").manual_seed(T)
    NB = keep + 3
    lens = torch.tensor([NB * B - (s * 13) % B for s in range(S)], dtype=torch.int32)
    rnd = lambda *s: (torch.randn(s, generator=gg, device="cuda") * 1.5).to(torch.bfloat16)
    k, v, q = rnd(S * NB, Hkv, B, 128), rnd(S * NB, Hkv, B, 128), rnd(S, T, Hq, 128)
    dk, dv = rnd(S, T, Hkv, 128), rnd(S, T, Hkv, 128)
    table = torch.randperm(S * NB, generator=g, dtype=torch.int32).view(S, NB).cuda()
    parent = torch.arange(-1, T - 1, dtype=torch.int32).repeat(S, 1)
    if tree:
        for i in range(1, T):
            parent[:, i] = torch.randint(0, i, (S,), generator=g, dtype=torch.int32)
    idx, cnt = torch.zeros((S, Hkv, keep), dtype=torch.int32), torch.zeros((S, Hkv), dtype=torch.int32)
    for n, (s, h) in enumerate((s, h) for s in range(S) for h in range(Hkv)):
        cnt[s, h] = c = (keep, 0, 1, keep // 2, keep - 1, 2, 5, keep)[(n + n // 8) % 8]
        idx[s, h, :c] = torch.randperm(NB, generator=g)[:c].sort().values.int()
    idx, cnt, lens_d, parent_d = idx.cuda(), cnt.cuda(), lens.cuda(), parent.cuda() if tree else None
    geom = sv.make_geom(S, Hq, Hkv, 128, B, NB, T)
    assert sv.sv_verify_attn_splits(geom, keep) == splits and sv.sv_verify_attn_launches(geom, keep) == launches
    n = sv.sv_workspace_bytes(geom, keep)
    workspace = torch.full((max(16, n),), 0x5A, dtype=torch.uint8, device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    kv = sv.make_kv(k, v, table, lens_d)
    fresh = lambda: (torch.full_like(q, float("nan")), torch.full((S, T, Hq), float("nan"), device="cuda"))
    out, lse = fresh()
    sv.sv_verify_attn(geom, q, kv, dk, dv, parent_d, idx, cnt, out, lse=lse, workspace=workspace, status_word=status)
    assert bool((workspace == 0x5A).all()) == (splits == 1 or launches == 1)   # (only the merge kernel's partials go there)
    want = _plain(q, k, v, dk, dv, table, lens, parent, idx, cnt, B)
    rows = (out.float() - want).norm(dim=-1) / want.norm(dim=-1)
    assert int(status) == 0 and bool(torch.isfinite(lse).all())
    assert float((out.float() - want).norm() / want.norm()) < 2.8e-3 and float(rows.max()) < 8.5e-3, float(rows.max())
    # lists that sv_verify_attn does not hand out or take in two launches are taken the same way by the other calls
    other, other_lse = fresh()
    sv.sv_verify_attn_reused(geom, q, kv, dk, dv, parent_d, idx, cnt, other, lse=other_lse, workspace=workspace, status_word=status)
    if splits > 1:
        assert torch.equal(other, out) and torch.equal(other_lse, lse)
    rows = (other.float() - want).norm(dim=-1) / want.norm(dim=-1)
    assert float((other.float() - want).norm() / want.norm()) < 2.8e-3 and float(rows.max()) < 8.5e-3, float(rows.max())
    for _ in range(2 if n <= sv.SV_NOALLOC_SCRATCH_BYTES else 0):   # (the built-in scratch holds what the last call left there)
        other, other_lse = fresh()
        sv.sv_verify_attn_noalloc(geom, q, kv, dk, dv, parent_d, idx, cnt, other, lse=other_lse, status_word=status)
        assert torch.equal(other, out) and torch.equal(other_lse, lse)
    assert int(status) == 0
