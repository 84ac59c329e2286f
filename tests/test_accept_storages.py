"""The three outputs of SparseVerifier.accept are tensors of their own: each can grow, be saved and be dropped without the others noticing."""
import io

import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("S,T", [(1, 1), (3, 43), (130, 5)])
def test_every_output_has_its_own_storage(S, T):
    import paper_2512_21911_b200 as sv
    p = torch.full((S, T, 64), 1 / 64, device="cuda")
    tokens, u = torch.zeros((S, T), dtype=torch.int32, device="cuda"), torch.full((S, T), 0.5, device="cuda")
    args = (p, p, tokens, None, u, u[:, 0].contiguous(), S, T)
    outputs = sv.binding._native.accept_new(*args)
    for i in range(3):
        got = list(sv.binding._native.accept_new(*args))
        assert got[i].storage_offset() == 0 and got[i].untyped_storage().nbytes() == 4 * got[i].numel()
        others = [(x, x.clone()) for j, x in enumerate(got) if j != i]
        got[i].resize_(got[i].numel() + 4096).fill_(-5)
        assert all(torch.equal(x, before) for x, before in others)
    sizes = []
    for x in outputs:
        f = io.BytesIO()
        torch.save(x, f)
        sizes.append(f.tell())
    alone = io.BytesIO()
    torch.save(torch.zeros(S, dtype=torch.int32, device="cuda"), alone)
    assert sizes[1] == sizes[2] == alone.tell()
    path = outputs[0]
    want = path.clone()
    del outputs
    torch.full((S, T), 9, dtype=torch.int32, device="cuda")
    assert torch.equal(path, want)

