"""A bad argument of the host-fed step without chunks is refused before anything is launched: the device tensors, the lists and the
representatives stay as they were, whichever of its launches would have refused it."""
import pytest
import torch

from test_host_direct import _pinned, _stack

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bad, status", [("workspace", 5), ("budget", 4), ("sinks", 4), ("out", 3), ("draft", 3), ("reps", 3)])
def test_refused_before_the_first_launch(bad, status):
    import paper_2512_21911_b200 as sv
    eng, ins = _stack(20, 1, 32, 8, 64, 8, 12, False)
    dev = [torch.full_like(t, 7.0) for t in ins]
    out, out_h = torch.full_like(ins[0], 7.0), _pinned(torch.full_like(ins[0], 7.0))
    odd = lambda t: torch.full((t.numel() + 1,), 7.0, dtype=t.dtype, device="cuda")[1:].view(t.shape)   # contiguous, not 16-byte aligned
    if bad == "workspace":
        eng._stack_workspace[0] = torch.zeros(16, dtype=torch.uint8, device="cuda")
    elif bad == "budget":
        eng.n_local = eng.max_sel + 1
    elif bad == "sinks":
        eng.n_sink = eng.n_local = 1 << 30
    elif bad == "out":
        out = odd(out)
    elif bad == "draft":
        dev[2] = odd(dev[2])
    else:
        eng.reps = odd(eng.reps)
    lists = eng._lists_idx.fill_(-3), eng._lists_cnt.fill_(-3)
    reps = eng.reps.fill_(2.0)
    with pytest.raises(sv.SvError) as e:
        eng._from_host(None, *[_pinned(t) for t in ins], *dev, out, out_h, True)
    torch.cuda.synchronize()
    assert e.value.status == status
    assert all(bool((t == 7.0).all()) for t in (*dev, out, out_h))
    assert all(bool((t == -3).all()) for t in lists) and bool((reps == 2.0).all())
