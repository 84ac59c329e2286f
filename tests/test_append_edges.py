"""Commit of up to 64 rows at the edges of blocks: the appended rows are summed from shared memory, the rows that the block held from the
pool, and both together have to give the bits of a full rebuild; one layer by itself and several in one launch."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("block", [64, 128])
@pytest.mark.parametrize("draft", [1, 9, 64])
def test_append_at_the_edges_of_blocks(block, draft):
    import paper_2512_21911_b200 as sv
    from paper_2512_21911_b200.engine import SparseVerifier
    B, T, Hkv, L, NB = block, draft, 2, 3, 4
    starts = [0, 1, B - T, B - 1, B, B + 1, 2 * B - T // 2, 2 * B - 1, 3 * B, 4 * B - T, 4 * B - 1, 4 * B]   # the table ends at 4 B
    cases = [(max(0, x), n) for x in starts for n in sorted({0, 1, T // 2, T})]
    S = len(cases)
    g = np.random.default_rng(block + draft)
    lens = np.array([x for x, _ in cases], np.int32)
    n_acc = np.array([n for _, n in cases], np.int32)
    rows = np.stack([np.sort(g.choice(T, size=T, replace=False)) for _ in range(S)]).astype(np.int32)
    table = g.permutation(S * NB).astype(np.int32).reshape(S, NB)
    gen = torch.Generator(device="cuda").manual_seed(1)
    normal = lambda *shape: torch.empty(shape, dtype=torch.bfloat16, device="cuda").normal_(generator=gen)
    k, v = normal(L, S * NB, Hkv, B, 128), normal(L, S * NB, Hkv, B, 128)
    dk, dv = normal(L, S, T, Hkv, 128), normal(L, S, T, Hkv, 128)
    dev = lambda a: torch.from_numpy(a).cuda()
    want_k, want_v = k.clone(), v.clone()
    new = np.minimum(lens + n_acc, NB * B).astype(np.int32)
    for s in range(S):
        for a in range(new[s] - lens[s]):
            t = int(lens[s]) + a
            want_k[:, table[s, t // B], :, t % B] = dk[:, s, rows[s, a]]
            want_v[:, table[s, t // B], :, t % B] = dv[:, s, rows[s, a]]
    geom = sv.make_geom(S, 2, Hkv, 128, B, NB, T)
    table_d, rows_d, n_d = dev(table), dev(rows), dev(n_acc)
    want_reps = torch.zeros((L, S, Hkv, NB, 128), device="cuda")
    before = torch.zeros_like(want_reps)
    for l in range(L):
        sv.sv_block_reps(geom, sv.make_kv(want_k[l], want_v[l], table_d, dev(new)), want_reps[l])
        sv.sv_block_reps(geom, sv.make_kv(k[l], v[l], table_d, dev(lens)), before[l])
    k1, v1, reps1, len1 = k[0].clone(), v[0].clone(), before[0].clone(), torch.zeros(S, dtype=torch.int32, device="cuda")
    sv.sv_kv_append(geom, k1, v1, table_d, dev(lens), dk[0], dv[0], rows_d, n_d, len1, reps1)
    assert torch.equal(len1, dev(new)) and torch.equal(k1, want_k[0]) and torch.equal(v1, want_v[0]) and torch.equal(reps1, want_reps[0])
    eng = SparseVerifier(n_seq=S, n_q_heads=2, n_kv_heads=Hkv, head_dim=128, block_size=B, max_blocks=NB, n_draft=T, n_layers=L,
                         block_table=table_d, seq_lens=dev(lens), budget_blocks=torch.full((S,), NB, dtype=torch.int32, device="cuda"), max_sel=NB)
    eng.set_kv_stack(k, v)
    eng.reps.copy_(before)
    eng.commit(dk, dv, rows_d, n_d)
    assert torch.equal(eng.seq_lens, dev(new)) and torch.equal(k, want_k) and torch.equal(v, want_v) and torch.equal(eng.reps, want_reps)
    assert int(eng._counters[:S].abs().max()) == 0   # ready for the next launch
