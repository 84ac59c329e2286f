"""The schedule of the host-fed step: the chunks cover every layer once, in order, whatever the stack; a step of few bytes is one chunk."""
from types import SimpleNamespace

import pytest

from paper_2512_21911_b200.engine import ONE_CHUNK_BYTES, SparseVerifier


@pytest.mark.parametrize("seqs", [1, 2, 9])
@pytest.mark.parametrize("draft", [1, 5, 64])
@pytest.mark.parametrize("heads, kv_heads", [(8, 2), (32, 8), (16, 16)])
def test_default_schedule(seqs, draft, heads, kv_heads):
    for layers in list(range(1, 34)) + [127, 128]:
        geom = SimpleNamespace(n_seq=seqs, n_draft=draft, n_q_heads=heads, n_kv_heads=kv_heads, head_dim=128)
        chunks = SparseVerifier._chunks(SimpleNamespace(n_layers=layers, geom=geom), None)
        assert chunks[0][0] == 0 and chunks[-1][1] == layers
        assert all(a < b for a, b in chunks) and all(x[1] == y[0] for x, y in zip(chunks, chunks[1:]))
        few = layers * seqs * draft * (heads + 2 * kv_heads) * 256 <= ONE_CHUNK_BYTES
        assert (len(chunks) == 1) == (few or layers < 4)
