"""The schedule of the host-fed step against measured steps: for stacks on which a split that reckoned well was measured to be slow (and some
that another one serves best) what is picked is no slower than the usual split and near the best of those measured."""
import pytest

from paper_2512_21911_b200.engine import host_step_schedule

# layers, sequences, cached tokens, query heads, KV heads, block, kept blocks, draft tokens, a selecting layer every n; us per step by
# layers per chunk.  All of one machine per stack, schedules timed in turn.
MEASURED = [
    ((32, 1, 32768, 32, 8, 64, 64, 8, 1), {(14, 18): 178.8, (16, 16): 178.1, (32,): 216.2, (10, 14, 8): 182.7}),
    ((32, 1, 32768, 32, 8, 64, 64, 8, 2), {(14, 18): 175.5, (16, 16): 173.5, (32,): 211.7, (10, 14, 8): 177.8}),
    ((32, 1, 32768, 64, 8, 64, 64, 8, 1), {(14, 18): 252.3, (16, 16): 230.8, (32,): 306.6, (10, 14, 8): 227.4}),
    ((31, 5, 7449, 28, 4, 128, 7, 10, 4), {(13, 18): 501.3, (15, 16): 514.1, (31,): 587.0, (9, 15, 7): 460.3}),
    ((19, 1, 18954, 32, 8, 128, 35, 1, 1), {(8, 11): 110.5, (9, 10): 112.2, (19,): 124.9, (5, 10, 4): 126.7}),
    ((13, 1, 56830, 8, 2, 64, 65, 3, 1), {(5, 8): 53.2, (6, 7): 52.7, (13,): 37.3, (4, 6, 3): 67.8}),
    ((8, 2, 50076, 32, 8, 64, 176, 13, 1), {(3, 5): 212.0, (4, 4): 246.0, (8,): 241.5, (2, 4, 2): 225.7}),
    # two and three layers: the usual is one chunk
    ((3, 8, 32768, 32, 8, 64, 128, 16, 1), {(1, 2): 271.8, (3,): 326.5}),
    ((3, 6, 11213, 32, 8, 64, 6, 11, 1), {(1, 2): 122.3, (3,): 108.4}),
    ((3, 4, 29931, 28, 4, 64, 78, 26, 1), {(1, 2): 179.2, (3,): 163.2}),
    ((2, 7, 2036, 32, 8, 64, 5, 11, 1), {(1, 1): 102.1, (2,): 87.9}),
    ((2, 2, 8192, 32, 8, 64, 40, 60, 1), {(1, 1): 144.7, (2,): 135.2}),
]


@pytest.mark.parametrize("stack, us", MEASURED)
def test_picked_schedule_is_not_slower_than_the_usual_one(stack, us):
    layers, seqs, tokens, heads, kv_heads, block, keep, draft, every = stack
    blocks, anchors = -(-(tokens + draft) // block), -(-layers // every)
    rows, pairs = seqs * draft * 256, seqs * kv_heads
    sizes = host_step_schedule(layers, rows * (heads + 2 * kv_heads), rows * heads, pairs * 512 * (keep * block + blocks * anchors / layers), pairs)
    first = layers * 7 // 16
    usual = (layers,) if layers < 4 else (first, layers - first)
    assert us[tuple(sizes)] <= 1.01 * us[usual]
    assert us[tuple(sizes)] <= 1.02 * min(us.values())
