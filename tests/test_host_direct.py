"""The host-fed step without chunks, whose attention launch reads and writes pinned memory itself: the bits of the step on device tensors, in
out and in out_host, and the inputs in the device tensors, for every form of the handed-out kernel (up to 32 and 64 query rows, more than 32
draft tokens), row counts that are no multiple of anything, lists of no unit and of many; memory it cannot take goes in chunks as ever."""
import pytest
import torch

pytestmark = pytest.mark.gpu


def _stack(layers, seqs, heads, kv_heads, block, draft, keep, tree):
    import paper_2512_21911_b200 as sv
    gen = torch.Generator(device="cuda").manual_seed(layers + draft)
    cpu = torch.Generator().manual_seed(layers)
    rnd = lambda *s: torch.randn(s, generator=gen, device="cuda").to(torch.bfloat16)
    NB = keep + 9
    lens = torch.tensor([max(1, NB * block - 3 - (s * 7 * block) // 2) if s != 1 else 5 for s in range(seqs)], dtype=torch.int32)
    parent = torch.arange(-1, draft - 1, dtype=torch.int32).repeat(seqs, 1)
    for i in range(1, draft):
        parent[:, i] = torch.randint(0, i, (seqs,), generator=cpu, dtype=torch.int32)
    eng = sv.SparseVerifier(n_seq=seqs, n_q_heads=heads, n_kv_heads=kv_heads, head_dim=128, block_size=block, max_blocks=NB, n_draft=draft,
                            n_layers=layers, block_table=torch.randperm(seqs * NB, generator=cpu, dtype=torch.int32).view(seqs, NB).cuda(),
                            seq_lens=lens.cuda(), max_sel=keep, budget_blocks=torch.full((seqs,), keep, dtype=torch.int32).cuda(),
                            anchors=[l % 3 == 0 for l in range(layers)], parent=parent.cuda() if tree else None)
    eng.set_kv_stack(rnd(layers, seqs * NB, kv_heads, block, 128), rnd(layers, seqs * NB, kv_heads, block, 128))
    for l in range(layers):
        eng.build_reps(l)
    return eng, [rnd(layers, seqs, draft, heads, 128), rnd(layers, seqs, draft, kv_heads, 128), rnd(layers, seqs, draft, kv_heads, 128)]


def _pinned(t, offset=0):
    h = torch.zeros(t.numel() + offset, dtype=t.dtype).pin_memory()[offset:].view(t.shape)
    h.copy_(t)
    return h


@pytest.mark.parametrize("layers, seqs, heads, kv_heads, block, draft, keep, tree", [
    (20, 1, 32, 8, 64, 8, 12, False),    # 32 rows
    (38, 2, 8, 2, 64, 3, 7, True),       # 12 rows
    (11, 4, 28, 4, 64, 1, 5, False),     # 7 rows, one draft token
    (19, 2, 28, 4, 128, 9, 6, True),     # 63 rows
    (10, 2, 8, 8, 64, 40, 9, True),      # 40 rows of 40 draft tokens
    (5, 8, 64, 8, 64, 8, 4, False),      # 64 rows, lists of four units
])
def test_direct_step_equals_device_step(layers, seqs, heads, kv_heads, block, draft, keep, tree):
    eng, ins = _stack(layers, seqs, heads, kv_heads, block, draft, keep, tree)
    assert eng._direct
    want = torch.empty_like(ins[0])
    eng.verify_step(*ins, want, refresh_tail=True)
    host, dev = [_pinned(t) for t in ins], [torch.full_like(t, float("nan")) for t in ins]
    out, out_h = torch.full_like(want, float("nan")), _pinned(torch.zeros_like(want))
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        for _ in range(2):
            eng.verify_step_from_host(*host, *dev, out, out_h, refresh_tail=True)
    side.synchronize()
    assert eng._copy_streams is None   # (no chunks, no side streams)
    assert torch.equal(out_h, want.cpu()) and torch.equal(out, want)
    assert all(torch.equal(d, t) for d, t in zip(dev, ins))
    # captured, and replayed on what host memory holds by then
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        eng.verify_step_from_host(*host, *dev, out, out_h)
    for h, t in zip(host, ins):
        h.copy_(t.flip(-1).cpu()), t.copy_(t.flip(-1))
    graph.replay()
    eng.verify_step(*ins, want)
    torch.cuda.synchronize()
    assert torch.equal(out_h, want.cpu()) and all(torch.equal(d, t) for d, t in zip(dev, ins))
    eng.check_status()


def test_memory_that_cannot_be_read_directly_goes_in_chunks():
    eng, ins = _stack(20, 1, 32, 8, 64, 8, 12, False)
    want = torch.empty_like(ins[0])
    eng.verify_step(*ins, want)
    for host, out_h in (([_pinned(t, 1) for t in ins], _pinned(want, 3)),                         # not 16-byte aligned
                        ([t.cpu() for t in ins], torch.zeros_like(want, device="cpu")),           # pageable
                        ([_pinned(ins[0])] + [t.cpu() for t in ins[1:]], _pinned(want))):
        dev, out = [torch.full_like(t, float("nan")) for t in ins], torch.full_like(want, float("nan"))
        out_h.zero_()
        eng.verify_step_from_host(*host, *dev, out, out_h)
        torch.cuda.synchronize()
        assert eng._copy_streams is not None
        assert (out_h.cuda().float() - want.float()).norm() <= 5e-3 * want.float().norm()
        assert all(torch.equal(d, t) for d, t in zip(dev, ins))
