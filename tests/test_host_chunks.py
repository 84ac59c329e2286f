"""The schedule of the host-fed step: whatever the stack, the chunks cover every layer once, in order; a step of few bytes is one chunk, one
that gathers as long as it copies is not; and no schedule is picked that the reckoning does not put ahead of the usual one."""
from types import SimpleNamespace

import pytest

from paper_2512_21911_b200.engine import SparseVerifier, host_step_schedule, host_step_us


@pytest.mark.parametrize("lists", [1, 8, 300])
@pytest.mark.parametrize("upload, download, gathered", [(1e3, 1e3, 1e5), (1e5, 7e4, 5e6), (1e6, 7e5, 1e7), (1e5, 7e4, 2e8), (1, 1, 1e9)])
def test_schedule_covers_the_layers(upload, download, gathered, lists):
    for n in list(range(1, 40)) + [127, 128]:
        sizes = host_step_schedule(n, upload, download, gathered, lists)
        assert all(x > 0 for x in sizes) and sum(sizes) == n
        chunks = SparseVerifier._chunks(SimpleNamespace(n_layers=n, _schedule=sizes), None)
        assert chunks[0][0] == 0 and chunks[-1][1] == n
        assert all(a < b for a, b in chunks) and all(x[1] == y[0] for x, y in zip(chunks, chunks[1:]))
        first = max(1, n * 7 // 16)
        usual = [first, n - first] if n > 1 else [n]
        assert host_step_us(sizes, upload, download, gathered, lists) <= host_step_us(usual, upload, download, gathered, lists)


def test_few_bytes_go_in_one_chunk_and_many_do_not():
    assert host_step_schedule(12, 16e3, 12e3, 1.5e6, 2) == [12]
    assert len(host_step_schedule(24, 600e3, 400e3, 6e6, 24)) == 3
    assert len(host_step_schedule(6, 300e3, 200e3, 120e6, 32)) > 1
