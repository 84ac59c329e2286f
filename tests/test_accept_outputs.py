"""The three outputs of SparseVerifier.accept share an allocation: they must not overlap, and behave like tensors of their own."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("S,T", [(1, 1), (1, 8), (3, 43), (128, 1), (2, 64), (130, 5)])
def test_outputs_of_accept_do_not_overlap(S, T):
    from paper_2512_21911_b200 import binding as sv
    V = 64
    g = torch.Generator(device="cuda").manual_seed(S)
    p = torch.softmax(torch.randn((S, T, V), generator=g, device="cuda"), -1)
    tokens = torch.zeros((S, T), dtype=torch.int32, device="cuda")
    u = torch.rand((S, T), generator=g, device="cuda")
    args = (p, p, tokens, None, u, u[:, 0].contiguous())
    want = [torch.empty(shape, dtype=torch.int32, device="cuda") for shape in ((S, T), (S,), (S,))]
    sv.sv_accept(*args, *want)
    got = sv._native.accept_new(*args, S, T)
    for w, x in zip(want, got):
        assert x.shape == w.shape and x.is_contiguous() and x.dtype == torch.int32 and x.data_ptr() % 512 == 0 and not x._is_view()
    n = want[1]
    assert torch.equal(got[1], n) and torch.equal(got[2], want[2])
    for s in range(S):   # (rows past the kept path are unspecified)
        assert torch.equal(got[0][s, :int(n[s])], want[0][s, :int(n[s])])
    for i, x in enumerate(got):
        x.fill_(1000 + i)
    for i, x in enumerate(got):
        assert bool((x == 1000 + i).all())
