"""An engine whose first step is captured into a CUDA graph, so that nothing the capture allocates has been written when the next
call runs eagerly: the words a stack's launches keep between calls must not be among it.  Stacks of more lists than SMs, where the
lists are handed out through a counter: sparse, dense, and fed from the host."""
import pytest
import torch

pytestmark = pytest.mark.gpu


def _engine(sv):
    L, S, Hq, Hkv, B, T, L0 = 20, 2, 16, 4, 64, 5, 700
    gen = torch.Generator(device="cuda").manual_seed(1)
    rnd = lambda *s: torch.randn(s, generator=gen, device="cuda").to(torch.bfloat16)
    NB = -(-L0 // B)
    eng = sv.SparseVerifier(n_seq=S, n_q_heads=Hq, n_kv_heads=Hkv, head_dim=128, block_size=B, max_blocks=NB, n_draft=T, n_layers=L,
                            block_table=torch.arange(S * NB, dtype=torch.int32).view(S, NB).cuda(), max_sel=6,
                            seq_lens=torch.tensor([L0, L0 - 77], dtype=torch.int32).cuda(),
                            budget_blocks=torch.full((S,), 6, dtype=torch.int32).cuda(), anchors=[l % 2 == 0 for l in range(L)])
    eng.set_kv_stack(rnd(L, S * NB, Hkv, B, 128), rnd(L, S * NB, Hkv, B, 128))
    for l in range(L):
        eng.build_reps(l)
    assert L * S * Hkv > 148
    return eng, 2 * rnd(L, S, T, Hq, 128), rnd(L, S, T, Hkv, 128), rnd(L, S, T, Hkv, 128)


@pytest.mark.parametrize("form", ["sparse", "dense", "host"])
def test_eager_step_between_capture_and_first_replay(form):
    import paper_2512_21911_b200 as sv
    eng, q, dk, dv = _engine(sv)
    want = torch.full_like(q, float("nan"))
    for l in range(eng.n_layers):
        (eng.dense_layer if form == "dense" else eng.verify_layer)(l, q[l], dk[l], dv[l], want[l])
    out = torch.full_like(q, float("nan"))
    host = [t.cpu().pin_memory() for t in (q, dk, dv, out)]

    def step():
        if form == "host":
            eng.verify_step_from_host(host[0], host[1], host[2], q, dk, dv, out, host[3], layers_per_chunk=eng.n_layers)
        else:
            (eng.dense_step if form == "dense" else eng.verify_step)(q, dk, dv, out)

    # a pool for captures whose memory holds large numbers where a capture that follows allocates
    pool = torch.cuda.graph_pool_handle()
    other, stream = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    flag = torch.zeros(1, device="cuda")
    torch.cuda.synchronize()
    with torch.cuda.graph(other, pool=pool, stream=stream):
        flag.add_(1)
        junk = [torch.empty(256, dtype=torch.uint8, device="cuda") for _ in range(64)] + [torch.empty(8 << 20, dtype=torch.uint8, device="cuda")]
    for j in junk:
        j.fill_(0x7f)
    torch.cuda.synchronize()
    del junk, j
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, pool=pool, stream=stream):
        step()
    torch.cuda.synchronize()

    def check():
        torch.cuda.synchronize()
        got = (host[3] if form == "host" else out).cuda().float()
        assert torch.isfinite(got).all(), "rows were never written"
        assert (got - want.float()).norm() <= 5e-3 * want.float().norm()
        eng.check_status()

    for _ in range(2):
        out.fill_(float("nan")), host[3].fill_(float("nan"))
        step()
        check()
    for _ in range(2):
        out.fill_(float("nan")), host[3].fill_(float("nan"))
        graph.replay()
        check()
