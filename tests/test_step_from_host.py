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
