"""Entry points release the interpreter lock while they are in the library: a launch that waits for room in a full queue stops
its own thread only, not the threads that drive other devices."""
import threading
import time

import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("call", ["layer", "step"])
def test_other_threads_run_while_a_launch_waits(call):
    import paper_2512_21911_b200 as sv
    L, S, Hq, Hkv, B, T, NB = 2, 1, 8, 2, 64, 4, 8
    rnd = lambda *s: torch.randn(s, device="cuda").to(torch.bfloat16)
    eng = sv.SparseVerifier(n_seq=S, n_q_heads=Hq, n_kv_heads=Hkv, head_dim=128, block_size=B, max_blocks=NB, n_draft=T, n_layers=L,
                            block_table=torch.arange(NB, dtype=torch.int32).view(S, NB).cuda(), max_sel=6,
                            seq_lens=torch.tensor([NB * B], dtype=torch.int32).cuda(),
                            budget_blocks=torch.full((S,), 6, dtype=torch.int32).cuda())
    eng.set_kv_stack(rnd(L, NB, Hkv, B, 128), rnd(L, NB, Hkv, B, 128))
    for l in range(L):
        eng.build_reps(l)
    q, dk, dv = rnd(L, S, T, Hq, 128), rnd(L, S, T, Hkv, 128), rnd(L, S, T, Hkv, 128)
    out = torch.empty_like(q)

    def run():
        if call == "layer":
            eng.verify_layer(0, q[0], dk[0], dv[0], out[0])
        else:
            eng.verify_step(q, dk, dv, out)

    run()
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    torch.cuda._sleep(100_000_000)
    torch.cuda.synchronize()
    per_cycle = (time.perf_counter() - t0) / 1e8
    done = threading.Event()

    def fill_the_queue():
        for _ in range(3000):
            run()
        done.set()

    torch.cuda._sleep(int(1.0 / per_cycle))   # a second of work ahead of the launches: they fill the queue and wait
    worker = threading.Thread(target=fill_the_queue)
    t0 = last = time.perf_counter()
    worker.start()
    longest = 0.0
    while not done.is_set():
        time.sleep(0.001)
        now = time.perf_counter()
        longest, last = max(longest, now - last), now
    worker.join()
    torch.cuda.synchronize()
    waited = last - t0
    if waited < 0.5:
        pytest.skip("the launches found room in the queue")
    assert longest < 0.25, (longest, waited)
    eng.check_status()
