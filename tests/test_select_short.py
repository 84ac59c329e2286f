"""Selection over short tables, around the lengths at which it changes its way (an eighth, three sixteenths of a CTA's 512 or 256 threads): scores
that are exact small integers, so that most of them are tied, and both signs of zero; against a stable sort."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("seqs", [40, 320])   # CTAs of 512 threads, of 256
@pytest.mark.parametrize("spread", [1, 3, 1000])
def test_short_tables_against_a_stable_sort(seqs, spread):
    import paper_2512_21911_b200 as sv
    g = torch.Generator().manual_seed(seqs + spread)
    edges = (1, 2, 3, 4, 5, 7, 8, 31, 32, 33, 47, 48, 49, 63, 64, 65, 66, 67, 95, 96, 97, 98, 127, 129)
    NB, keep, n_sink, n_local = 130, 40, 1, 2
    nbs = torch.tensor([edges[s % len(edges)] for s in range(seqs)])
    scores = torch.randint(-spread, spread + 1, (seqs, NB), generator=g).float() * torch.where(torch.rand((seqs, NB), generator=g) < 0.5, 1.0, -1.0)
    budget = torch.tensor([(3, 4, 9, 30, 40)[(s // len(edges) + s) % 5] for s in range(seqs)], dtype=torch.int32)
    reps = torch.zeros((seqs, 1, NB, 128))
    reps[:, 0, :, 0] = scores
    for s in range(seqs):
        reps[s, 0, int(nbs[s]):] = float("nan")   # what is past the end is never looked at
    q = torch.zeros((seqs, 1, 1, 128))
    q[..., 0] = 1.0
    idx, cnt = torch.full((seqs, 1, keep), -7, dtype=torch.int32, device="cuda"), torch.zeros((seqs, 1), dtype=torch.int32, device="cuda")
    sv.sv_select_blocks(sv.make_geom(seqs, 1, 1, 128, 64, NB, 1), q.bfloat16().cuda(), reps.cuda(), (nbs * 64).int().cuda(), budget.cuda(), n_sink,
                        n_local, idx, cnt)
    for s in range(seqs):
        nb, n = int(nbs[s]), int(budget[s])
        forced = set(range(min(n_sink, nb))) | set(range(max(0, nb - n_local), nb))
        n = min(max(n, len(forced)), nb)
        rest = sorted((b for b in range(nb) if b not in forced), key=lambda b: (-float(scores[s, b]), b))
        want = sorted(forced | set(rest[:n - len(forced)]))
        assert int(cnt[s]) == n and idx[s, 0, :n].tolist() == want, (s, nb, n)
