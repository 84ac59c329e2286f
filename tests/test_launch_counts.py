"""sv_verify_attn_launches and SparseVerifier.launches_per_step against the kernels that a capture of the calls holds, for every route of a layer's
lists: whole, merged in a cluster, merged by the merge kernel, whole with a rest in clusters, handed out by turns; and for reused and dense lists."""
import pytest
import torch

pytestmark = pytest.mark.gpu


def _kernels(call):
    from cuda.bindings import runtime as rt
    call()   # (what is only set up once is not part of a step)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(graph):
        call()
    raw = graph.raw_cuda_graph()
    err, _, n = rt.cudaGraphGetNodes(raw)
    assert err == rt.cudaError_t.cudaSuccess
    err, nodes, n = rt.cudaGraphGetNodes(raw, n)
    kinds = [rt.cudaGraphNodeGetType(node)[1] for node in nodes]
    assert len(kinds) == n and all(k == rt.cudaGraphNodeType.cudaGraphNodeTypeKernel for k in kinds)
    return n


ROUTES = [  # seqs, heads, kv_heads, block, draft, kept blocks, splits > 1, launches
    (8, 32, 8, 64, 5, 4, False, 1),      # a CTA a list
    (1, 8, 2, 64, 4, 16, True, 1),       # a cluster
    (4, 64, 8, 64, 16, 32, True, 1),     # ... of 128-row tiles
    (1, 32, 8, 64, 8, 300, True, 2),     # the merge kernel
    (2, 8, 8, 64, 40, 24, True, 2),      # ... behind few rows of many draft tokens
    (19, 32, 8, 64, 5, 15, False, 2),    # 144 lists whole, 8 in clusters
    (20, 64, 8, 64, 16, 16, False, 2),   # ... of 128 rows
    (31, 32, 8, 64, 8, 5, False, 1),     # by turns
]


@pytest.mark.parametrize("route", ROUTES)
def test_launches_are_counted_as_they_are_made(route):
    import paper_2512_21911_b200 as sv
    S, Hq, Hkv, B, T, keep, split, launches = route
    layers, NB = 4, keep + 2
    rnd = lambda *s: torch.randn(s, device="cuda").to(torch.bfloat16)
    lens = torch.full((S,), NB * B - 9, dtype=torch.int32, device="cuda")
    table = torch.arange(S * NB, dtype=torch.int32, device="cuda").view(S, NB)
    eng = sv.SparseVerifier(n_seq=S, n_q_heads=Hq, n_kv_heads=Hkv, head_dim=128, block_size=B, max_blocks=NB, n_draft=T, n_layers=layers,
                            block_table=table, seq_lens=lens, max_sel=keep, budget_blocks=torch.full_like(lens, keep),
                            anchors=[True, False, True, False])
    k, v = rnd(S * NB, Hkv, B, 128), rnd(S * NB, Hkv, B, 128)
    for l in range(layers):
        eng.set_layer_kv(l, k, v)
        eng.build_reps(l)
    q, dk, dv = rnd(S, T, Hq, 128), rnd(S, T, Hkv, 128), rnd(S, T, Hkv, 128)
    out = torch.empty_like(q)
    assert (sv.sv_verify_attn_splits(eng.geom, keep) > 1) == split
    assert sv.sv_verify_attn_launches(eng.geom, keep) == launches
    attend = lambda entry, lists: entry(eng.geom, q, eng.kv[0], dk, dv, None, *lists, out, workspace=eng.workspace)
    eng.verify_layer(0, q, dk, dv, out)
    lists = (eng.sel_idx, eng.sel_cnt)
    assert _kernels(lambda: attend(sv.sv_verify_attn, lists)) == launches
    assert _kernels(lambda: attend(sv.sv_verify_attn_reused, lists)) == (launches if split else 1)
    step = lambda: [eng.verify_layer(l, q, dk, dv, out, behind_own_layer=l > 0) for l in range(layers)]
    assert _kernels(step) == eng.launches_per_step() <= eng.kernels_per_step()

    def with_tail():
        eng.refresh_tail_all()
        step()
    assert _kernels(with_tail) == eng.launches_per_step(refresh_tail=True)
    dense = sv.sv_verify_attn_splits(eng.geom, NB)
    want = sv.sv_verify_attn_launches(eng.geom, NB) if dense > 1 else 1
    assert _kernels(lambda: eng.dense_layer(0, q, dk, dv, out)) == want
