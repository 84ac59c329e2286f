"""Attention with 65 to 128 query rows per tile and with pairs of tiles, over lists of zero to a dozen units: with fewer units than
warpgroups, odd and even numbers of them, a pair whose second tile does not exist, lists that end inside a block.  Against plain fp32
attention; probabilities and outputs are rounded to bfloat16 (2^-9 each, of values that add up with random signs: a relative error of
2^-9 * sqrt(2) = 2.8e-3 in the 2-norm at most)."""
import pytest
import torch

pytestmark = pytest.mark.gpu

SHAPES = [  # seqs, heads, kv_heads, block, draft, tree
    (14, 64, 8, 64, 16, True),     # 128 rows
    (14, 64, 8, 128, 16, False),   # 128 rows, blocks of 128: slices cut at units
    (5, 28, 4, 64, 10, True),      # 70 rows
    (3, 8, 4, 64, 60, True),       # 120 rows, more than 32 draft tokens
    (14, 32, 8, 64, 60, True),     # two tiles of 128 and 112 rows, in pairs
    (14, 32, 8, 128, 33, True),    # two tiles of 128 and 4 rows, in pairs
    (2, 32, 8, 64, 60, True),      # two tiles, on CTAs of their own
    (37, 16, 2, 64, 40, True),     # three tiles: a pair and one by itself
    (37, 16, 2, 128, 33, False),   # ... of one draft token
]


def _reference(q, k, v, dk, dv, table, lens, parent, block):
    S, T, Hq, D = q.shape
    Hkv = dk.shape[2]
    out = torch.zeros_like(q, dtype=torch.float32)
    for s in range(S):
        n = int(lens[s])
        pages = table[s, :-(-n // block)].long()
        rows = lambda pool: pool[pages].permute(1, 0, 2, 3).reshape(Hkv, -1, D)[:, :n].float()
        keys = torch.cat([rows(k), dk[s].permute(1, 0, 2).float()], 1).repeat_interleave(Hq // Hkv, 0)
        vals = torch.cat([rows(v), dv[s].permute(1, 0, 2).float()], 1).repeat_interleave(Hq // Hkv, 0)
        sees = torch.zeros((T, T), dtype=torch.bool, device=q.device)
        for i in range(T):
            j = i
            while j >= 0:
                sees[i, j] = True
                j = int(parent[s, j])
        logits = torch.einsum("thd,hnd->htn", q[s].float(), keys) * D ** -0.5
        logits[:, :, n:].masked_fill_(~sees, -torch.inf)
        out[s] = torch.einsum("htn,hnd->thd", torch.softmax(logits, -1), vals)
    return out


@pytest.mark.parametrize("shape", SHAPES)
def test_wide_tiles_against_plain_attention(shape):
    import paper_2512_21911_b200 as sv
    S, Hq, Hkv, B, T, tree = shape
    g = torch.Generator().manual_seed(S * T)
    gg = torch.Generator(device="cuda").manual_seed(T)
    NB = 12 * 64 // B
    lens = torch.tensor([(0, 1, 63, 64, 65, 128, 191, 256, 300, 449, 575, 640, 700, 768)[s % 14] for s in range(S)], dtype=torch.int32)
    table = torch.randperm(S * NB, generator=g, dtype=torch.int32).view(S, NB)
    parent = torch.arange(-1, T - 1, dtype=torch.int32).repeat(S, 1)
    if tree:
        for i in range(1, T):
            parent[:, i] = torch.randint(0, i, (S,), generator=g, dtype=torch.int32)
    rnd = lambda *s: (torch.randn(s, generator=gg, device="cuda") * 1.5).to(torch.bfloat16)
    k, v, q = rnd(S * NB, Hkv, B, 128), rnd(S * NB, Hkv, B, 128), rnd(S, T, Hq, 128)
    dk, dv = rnd(S, T, Hkv, 128), rnd(S, T, Hkv, 128)
    geom = sv.make_geom(S, Hq, Hkv, 128, B, NB, T)
    table_d, lens_d, parent_d = table.cuda(), lens.cuda(), parent.cuda() if tree else None
    workspace = torch.empty(max(16, sv.sv_workspace_bytes(geom, NB)), dtype=torch.uint8, device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    out = torch.full_like(q, float("nan"))
    sv.sv_verify_attn(geom, q, sv.make_kv(k, v, table_d, lens_d), dk, dv, parent_d, None, None, out, workspace=workspace, status_word=status)
    want = _reference(q, k, v, dk, dv, table_d, lens, parent, B)
    assert int(status) == 0
    assert float((out.float() - want).norm() / want.norm()) < 2.8e-3
    for s in range(S):   # no sequence hides behind the others: three times the bound for one row's 128 values
        err = (out[s].float() - want[s]).norm(dim=-1) / want[s].norm(dim=-1)
        assert float(err.max()) < 8.5e-3, (s, int(lens[s]), float(err.max()))
