"""Several layers of a stack in one launch: selections, attention and commits must equal the layer-by-layer calls, which the
other tests compare with the oracle.  Sizes at the edges: one layer and more layers than a wave of CTAs, one sequence and
ragged ones that end inside a block, lists that are split over CTAs and lists that are not, row tiles of 16 to 128 rows
and several of them, layers that reuse lists, pools in one allocation and of their own."""
import pytest
import torch

pytestmark = pytest.mark.gpu

SHAPES = [  # layers, anchors every, seqs, lo, hi, heads, kv_heads, block, keep, draft, tree, one allocation
    (1, 1, 1, 64, 64, 8, 2, 64, 4, 1, False, True),
    (5, 2, 1, 1000, 1000, 8, 2, 64, 6, 4, False, False),
    (3, 1, 3, 65, 1500, 16, 16, 64, 7, 5, True, False),
    (24, 3, 2, 300, 2200, 32, 8, 64, 9, 8, False, True),
    (4, 4, 2, 129, 3000, 64, 8, 128, 8, 16, True, True),
    (2, 1, 2, 700, 2500, 32, 8, 64, 12, 60, True, False),
    (3, 2, 5, 20, 900, 28, 4, 128, 5, 3, False, True),
]


def _engine(sv, shape, seed):
    L, every, S, lo, hi, Hq, Hkv, B, keep, T, tree, stack = shape
    g = torch.Generator().manual_seed(seed)
    lens = torch.randint(lo, hi + 1, (S,), generator=g, dtype=torch.int32)
    lens[0] = hi
    NB = -(-(hi + T) // B)
    n_pages = S * NB
    table = torch.randperm(n_pages, generator=g, dtype=torch.int32).view(S, NB)
    parent = None
    if tree:
        parent = torch.full((S, T), -1, dtype=torch.int32)
        for i in range(1, T):
            parent[:, i] = torch.randint(0, i, (S,), generator=g, dtype=torch.int32)
        parent = parent.cuda()
    keep = min(keep, NB)
    eng = sv.SparseVerifier(n_seq=S, n_q_heads=Hq, n_kv_heads=Hkv, head_dim=128, block_size=B, max_blocks=NB, n_draft=T, n_layers=L,
                            block_table=table.cuda(), seq_lens=lens.cuda(), max_sel=keep,
                            budget_blocks=torch.full((S,), keep, dtype=torch.int32).cuda(),
                            anchors=[l % every == 0 for l in range(L)], parent=parent)
    rnd = lambda *s: torch.randn(s, generator=g).to(torch.bfloat16).cuda()
    k, v = rnd(L, n_pages, Hkv, B, 128), rnd(L, n_pages, Hkv, B, 128)
    if stack:
        eng.set_kv_stack(k, v)
    else:
        for l in range(L):
            eng.set_layer_kv(l, k[l].clone(), v[l].clone())
    for l in range(L):
        eng.build_reps(l)
    return eng, rnd(L, S, T, Hq, 128), rnd(L, S, T, Hkv, 128), rnd(L, S, T, Hkv, 128)


def _close(a, b):
    a, b = a.float(), b.float()
    assert (a - b).norm() <= 5e-3 * b.norm() and (a - b).abs().max() <= 0.03 * b.abs().max(), (a - b).abs().max()


@pytest.mark.parametrize("shape", SHAPES)
def test_step_equals_layer_by_layer(shape):
    import paper_2512_21911_b200 as sv
    eng, q, dk, dv = _engine(sv, shape, 3)
    out, want = torch.full_like(q, float("nan")), torch.full_like(q, float("nan"))
    eng.verify_step(q, dk, dv, out)
    lists = eng._lists_idx.clone(), eng._lists_cnt.clone()
    a = -1
    for l in range(eng.n_layers):
        eng.verify_layer(l, q[l], dk[l], dv[l], want[l])
        a += eng.anchors[l]
        assert torch.equal(eng.sel_idx, lists[0][a]) and torch.equal(eng.sel_cnt, lists[1][a]), l
    _close(out, want)
    eng.dense_step(q, dk, dv, out)
    for l in range(eng.n_layers):
        eng.dense_layer(l, q[l], dk[l], dv[l], want[l])
    _close(out, want)
    # per-layer tensors in a list: the calls go layer by layer
    outs = [torch.empty_like(q[0]) for _ in range(eng.n_layers)]
    eng.verify_step(list(q), list(dk), list(dv), outs)
    eng.verify_step(q, dk, dv, out)
    _close(torch.stack(outs), out)
    eng.check_status()


@pytest.mark.parametrize("shape", SHAPES)
def test_commit_equals_append_per_layer(shape):
    import paper_2512_21911_b200 as sv
    eng, q, dk, dv = _engine(sv, shape, 5)
    L, S, T = eng.n_layers, q.shape[1], q.shape[2]
    g = torch.Generator().manual_seed(6)
    for _ in range(3):   # the counters have to come back to zero behind every commit
        path = torch.stack([torch.randperm(T, generator=g) for _ in range(S)]).to(torch.int32).cuda()
        n_path = torch.randint(0, T + 1, (S,), generator=g, dtype=torch.int32).cuda()
        pools = [(k.clone(), v.clone()) for k, v in eng._pools]
        reps, lens, new = eng.reps.clone(), eng.seq_lens.clone(), torch.empty_like(eng.seq_lens)
        for l in range(L):
            sv.sv_kv_append(eng.geom, *pools[l], eng.block_table, lens, dk[l], dv[l], path, n_path, new, reps[l])
        eng.commit(dk, dv, path, n_path)
        assert torch.equal(eng.seq_lens, new) and torch.equal(eng.reps, reps)
        for (k, v), (k2, v2) in zip(pools, eng._pools):
            assert torch.equal(k, k2) and torch.equal(v, v2)
    before = eng.reps.clone()
    eng.reps.fill_(7.0)
    eng.refresh_tail_all()
    tail = (eng.seq_lens.long() - 1) // eng.geom.block_size
    for s in range(S):
        assert torch.equal(eng.reps[:, s, :, tail[s]], before[:, s, :, tail[s]])
