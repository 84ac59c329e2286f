"""The host-fed step in one library call: pinned tensors (first upload and last download by a kernel), slices of larger pinned
tensors, pageable ones (copies only), and every chunking must give the bits of the step on device tensors."""
import pytest
import torch

pytestmark = pytest.mark.gpu


def _step(layers, seqs, draft):
    import paper_2512_21911_b200 as sv
    g = torch.Generator(device="cuda").manual_seed(layers + seqs)
    rnd = lambda *s: torch.randn(s, generator=g, device="cuda").to(torch.bfloat16)
    lens = torch.arange(700, 700 + 131 * seqs, 131, dtype=torch.int32).cuda()
    NB = -(-(700 + 131 * seqs) // 64)
    eng = sv.SparseVerifier(n_seq=seqs, n_q_heads=8, n_kv_heads=2, head_dim=128, block_size=64, max_blocks=NB, n_draft=draft, n_layers=layers,
                            block_table=torch.arange(seqs * NB, dtype=torch.int32).view(seqs, NB).cuda(), seq_lens=lens, max_sel=7,
                            budget_blocks=torch.full((seqs,), 7, dtype=torch.int32).cuda(), anchors=[l % 2 == 0 for l in range(layers)])
    eng.set_kv_stack(rnd(layers, seqs * NB, 2, 64, 128), rnd(layers, seqs * NB, 2, 64, 128))
    for l in range(layers):
        eng.build_reps(l)
    return eng, rnd(layers, seqs, draft, 8, 128), rnd(layers, seqs, draft, 2, 128), rnd(layers, seqs, draft, 2, 128)


@pytest.mark.parametrize("layers, seqs, draft", [(1, 1, 1), (4, 2, 3), (9, 1, 33), (20, 3, 8)])
@pytest.mark.parametrize("memory", ["pinned", "slice", "pageable"])
@pytest.mark.parametrize("chunks", [None, 1, [1, 2]])
def test_host_fed_step_equals_device_step(layers, seqs, draft, memory, chunks):
    eng, q, dk, dv = _step(layers, seqs, draft)
    want = torch.full_like(q, float("nan"))
    eng.verify_step(q, dk, dv, want, refresh_tail=True)

    def host(t):
        h = torch.zeros((t.shape[0] + 2,) + t.shape[1:], dtype=t.dtype, pin_memory=memory != "pageable")
        h = h[1:-1] if memory == "slice" else h[:-2]
        h.copy_(t)
        return h

    ins, dev = [host(t) for t in (q, dk, dv)], [torch.full_like(t, float("nan")) for t in (q, dk, dv)]
    out, out_h = torch.full_like(q, float("nan")), host(torch.zeros_like(q))
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        for _ in range(2):
            eng.verify_step_from_host(*ins, *dev, out, out_h, layers_per_chunk=chunks, refresh_tail=True)
    side.synchronize()
    assert torch.equal(out_h, want.cpu())
    assert all(torch.equal(d, t) for d, t in zip(dev, (q, dk, dv)))
    eng.check_status()


@pytest.mark.parametrize("layers, seqs, heads, kv_heads, block, draft, keep", [
    (32, 1, 32, 8, 64, 8, 64),      # lists handed out as a stack; 8 lists of 64 units a layer
    (19, 2, 16, 4, 128, 33, 9),     # ... of more than 32 draft tokens, blocks of 128: 9 blocks are 18 units
    (7, 3, 64, 8, 64, 16, 21),      # 128 rows, one CTA a list as a stack
    (4, 1, 32, 8, 64, 8, 33),       # split as a stack already, further as a chunk
    (10, 1, 32, 8, 64, 60, 25),     # two row tiles, which pair up in some of the launches
    (38, 1, 8, 4, 64, 3, 9),        # slices of nine units; eight are left alone
])
def test_chunks_of_few_lists_are_split_for_themselves(layers, seqs, heads, kv_heads, block, draft, keep):
    """... and give the step's outputs to bf16 rounding; with a workspace that has no room for it, bit for bit.  What the launches
    of the whole stack keep in their workspace survives it."""
    import paper_2512_21911_b200 as sv
    g = torch.Generator(device="cuda").manual_seed(layers)
    rnd = lambda *s: torch.randn(s, generator=g, device="cuda").to(torch.bfloat16)
    NB = keep + 5
    lens = torch.tensor([NB * block - 37 * s for s in range(seqs)], dtype=torch.int32).cuda()
    eng = sv.SparseVerifier(n_seq=seqs, n_q_heads=heads, n_kv_heads=kv_heads, head_dim=128, block_size=block, max_blocks=NB, n_draft=draft,
                            n_layers=layers, block_table=torch.arange(seqs * NB, dtype=torch.int32).view(seqs, NB).cuda(), seq_lens=lens,
                            max_sel=keep, budget_blocks=torch.full((seqs,), keep, dtype=torch.int32).cuda(),
                            anchors=[l % 3 == 0 for l in range(layers)])
    eng.set_kv_stack(rnd(layers, seqs * NB, kv_heads, block, 128), rnd(layers, seqs * NB, kv_heads, block, 128))
    for l in range(layers):
        eng.build_reps(l)
    ins = 2 * rnd(layers, seqs, draft, heads, 128), rnd(layers, seqs, draft, kv_heads, 128), rnd(layers, seqs, draft, kv_heads, 128)
    host = [t.cpu().pin_memory() for t in ins]
    want, out, out_h = torch.empty_like(ins[0]), torch.empty_like(ins[0]), torch.empty_like(host[0]).pin_memory()
    eng.verify_step(*ins, want)
    a = want.float()

    def step(chunks):
        out.fill_(float("nan")), out_h.fill_(float("nan"))
        eng.verify_step_from_host(*host, *ins, out, out_h, layers_per_chunk=chunks)
        torch.cuda.synchronize()
        return out_h.cuda().float()

    for chunks in (1, 2, [1, layers - 2, 1], None, layers):
        b = step(chunks)
        assert (b - a).norm() <= 5e-3 * a.norm() and (b - a).abs().max() <= 0.03 * a.abs().max(), chunks
        assert ((b - a).norm(dim=-1) <= 1e-2 * a.norm(dim=-1)).all(), chunks
        eng.verify_step(*ins, out)
        assert torch.equal(out, want)
    room = eng._workspace_of_stack(False)
    stack = sv.binding._native.workspace_bytes_layers(eng.geom, layers, keep)
    assert room.nbytes == sv.binding._native.workspace_bytes_host_step(eng.geom, layers, keep) > stack
    eng._stack_workspace[0] = room[:max(16, stack)]
    assert torch.equal(step(1), a)
    eng.check_status()
