"""The steps of a stack against the fp64 oracle: taken layer by layer, the way a model reaches its layers and the benchmark times them
(verify_layer with behind_own_layer in a CUDA graph, layers that select and layers that reuse), and all at once with the lists
handed out to resident CTAs, sparse and dense.  Bars as in test_gpu_parity: lists exact, rows within 1e-2 relative L2."""
import numpy as np
import pytest
import torch

import oracle
import sv_inputs as si

pytestmark = pytest.mark.gpu


def _dev(a):
    return torch.from_numpy(a.view(np.int16)).view(torch.bfloat16).cuda()


def _stack(w, every):
    import paper_2512_21911_b200 as sv
    geom = si.make_geometry(w)
    layers = [si.make_layer(geom, layer=l, sharp=bool(l & 1)) for l in range(w.n_layers)]
    parent = None if geom["parent"] is None else torch.from_numpy(geom["parent"]).cuda()
    eng = sv.SparseVerifier(n_seq=w.n_seq, n_q_heads=w.n_q_heads, n_kv_heads=w.n_kv_heads, head_dim=128, block_size=w.block_size,
                            max_blocks=geom["max_blocks"], n_draft=w.n_draft, n_layers=w.n_layers,
                            block_table=torch.from_numpy(geom["block_table"]).cuda(), seq_lens=torch.from_numpy(geom["seq_lens"]).cuda(),
                            budget_blocks=torch.from_numpy(geom["budget"]).cuda(), max_sel=geom["max_sel"], n_sink=w.n_sink,
                            n_local=w.n_local, anchors=[l % every == 0 for l in range(w.n_layers)], parent=parent)
    pools = [torch.stack([_dev(c[x]) for c in layers]) for x in ("k_pool", "v_pool")]
    eng.set_kv_stack(*pools)
    for l in range(w.n_layers):
        eng.build_reps(l)
    return geom, layers, eng, [torch.stack([_dev(c[x]) for c in layers]) for x in ("q", "draft_k", "draft_v")]


def _check(layer, c, got, lists, n_rows, g):
    w = c["workload"]
    smp = np.stack([g.integers(0, n, n_rows) for n in (w.n_seq, w.n_draft, w.n_q_heads)], axis=1).astype(np.int32)
    args = c["q"], c["k_pool"], c["v_pool"], c["block_table"], c["seq_lens"], c["draft_k"], c["draft_v"], c["parent"]
    want, _ = oracle.dense_verify_attn(*args, samples=smp) if lists is None else oracle.verify_attn(*args, *lists, samples=smp)
    o = si.bf16_bits_to_f64(got.cpu().view(torch.int16).numpy().view(np.uint16))
    assert np.isfinite(o).all()
    o = np.stack([o[s, i, h] for s, i, h in smp])
    rel = np.linalg.norm(o - want, axis=-1) / np.linalg.norm(want, axis=-1)
    assert rel.max() <= 1e-2 and np.abs(o - want).max() <= 1e-2 * max(1.0, np.abs(want).max()), (layer, rel.max())


@pytest.mark.parametrize("every", [1, 2, 3])
def test_step_layer_by_layer_in_a_graph(every):
    w = si.shrink(si.WORKLOADS["cfg1"], n_layers=3)
    geom, layers, eng, (q, dk, dv) = _stack(w, every)
    out = torch.full_like(q, float("nan"))
    lists = [(torch.empty_like(eng.sel_idx), torch.empty_like(eng.sel_cnt)) for _ in layers]

    def step(keep_lists):
        eng.refresh_tail_all()
        for l in range(w.n_layers):
            eng.verify_layer(l, q[l], dk[l], dv[l], out[l], behind_own_layer=l > 0 and not keep_lists)
            if keep_lists:
                lists[l][0].copy_(eng.sel_idx), lists[l][1].copy_(eng.sel_cnt)

    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        step(True)
        stream.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            step(False)
        out.fill_(float("nan"))
        for _ in range(3):
            graph.replay()
        stream.synchronize()
    eng.check_status()
    g = np.random.default_rng(every)
    for l, c in enumerate(layers):
        a = layers[l - l % every]
        idx, cnt, _ = oracle.select_blocks(a["q"], a["k_pool"], a["block_table"], a["seq_lens"], a["budget"], w.n_sink, w.n_local,
                                           geom["max_sel"])
        np.testing.assert_array_equal(lists[l][1].cpu().numpy(), cnt)
        np.testing.assert_array_equal(lists[l][0].cpu().numpy(), idx)
        _check(l, c, out[l], (idx, cnt), 24, g)


@pytest.mark.parametrize("layers, seqs, lo, hi, heads, kv_heads, block, keep, draft, tree", [
    (20, 1, 1500, 1500, 32, 8, 64, 12, 8, False),    # 32 rows
    (7, 3, 400, 1900, 64, 8, 64, 9, 7, True),        # 56 rows, lengths that end inside a block
    (14, 2, 1025, 2200, 16, 16, 128, 7, 40, True),   # more than 32 draft tokens, blocks of 128
    (152, 1, 300, 300, 4, 1, 64, 3, 1, False),       # one row, a few lists more than SMs
])
def test_lists_handed_out_against_the_oracle(layers, seqs, lo, hi, heads, kv_heads, block, keep, draft, tree):
    w = si.Workload("stack", seqs, (lo, hi), heads, kv_heads, 128, block, keep, draft, tree, layers, 0.1, 77)
    geom, cases, eng, (q, dk, dv) = _stack(w, 3)
    import paper_2512_21911_b200 as sv
    handed = [sv.binding._native.workspace_bytes_layers(eng.geom, layers, n) == sv.binding.SV_STACK_STATE_BYTES
              for n in (geom["max_sel"], geom["max_blocks"])]
    assert all(handed)
    out, dense = torch.full_like(q, float("nan")), torch.full_like(q, float("nan"))
    eng.verify_step(q, dk, dv, out, refresh_tail=True)
    eng.dense_step(q, dk, dv, dense)
    eng.check_status()
    g = np.random.default_rng(layers)
    for l in sorted({0, 1, layers // 2, layers - 2, layers - 1}):
        a = cases[l - l % 3]
        idx, cnt, _ = oracle.select_blocks(a["q"], a["k_pool"], a["block_table"], a["seq_lens"], a["budget"], w.n_sink, w.n_local,
                                           geom["max_sel"])
        np.testing.assert_array_equal(eng._lists_cnt[l // 3].cpu().numpy(), cnt)
        for s in range(seqs):
            for h in range(kv_heads):
                np.testing.assert_array_equal(eng._lists_idx[l // 3, s, h, :cnt[s, h]].cpu().numpy(), idx[s, h, :cnt[s, h]])
        _check(l, cases[l], out[l], (idx, cnt), 64, g)
        _check(l, cases[l], dense[l], None, 64, g)
