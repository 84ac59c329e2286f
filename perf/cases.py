"""Performance cases of the sparse verification path, called the way a decoding loop calls it: through SparseVerifier.

A case is one call (or, for "decode" and "finish", the calls that close a decoding step) on one shape:

  layer   one layer of a verification step: block selection, then attention over the kept blocks and the draft
  dense   dense verification attention of one layer (short caches, layers kept dense, the comparison run)
  step    a whole verification step of a stack of layers, tail blocks refreshed first
  host    the same with the step's inputs in pinned host memory and its outputs wanted there
  reps    the block representatives of one layer's whole cache (what follows a prefill)
  finish  what follows a verification step: acceptance of the draft, commit of the kept rows to every layer's cache
  decode  a whole decoding step: verification of the stack, acceptance, commit

Keys of a case: seqs, lo, hi (cached tokens of a sequence, uniform in lo..hi), heads (query), kv_heads, block (tokens),
keep (blocks kept per KV head), draft (rows verified per sequence), tree (a draft tree, else a chain), layers,
anchor_every (layers that select for themselves; the others reuse the list of the layer before), vocab.

Inputs are random with the shape of the real thing: attention logits with a standard deviation of about 3, block scores
that are a continuous bulk with a heavy upper tail, pages in random order, distributions over the vocabulary that keep
the entries within a factor of 50 of the likeliest (what sampling leaves of a language model's logits), draft
tokens drawn from the draft distribution.  Which blocks are kept is decided by comparing fp32 sums, so the kept and the
evicted scores of every list are moved a twentieth of the bulk's standard deviation apart: far more than the rounding
of the keys, too little for the scores to look different.
"""
import math

import torch

from paper_2512_21911_b200 import engine

HEAD_DIM = 128
SINK, LOCAL = 1, 1           # blocks kept at the two ends of every list
SIGMA = math.sqrt(3.0)       # of queries and keys: logits q.k / sqrt(128) then have a standard deviation of 3
GIB = 1 << 30


def _case(op, seqs, lo, hi, heads, kv_heads, block, keep, draft, tree=False, layers=1, anchor_every=1, vocab=0):
    return dict(op=op, seqs=seqs, lo=lo, hi=hi, heads=heads, kv_heads=kv_heads, block=block, keep=keep, draft=draft,
                tree=tree, layers=layers, anchor_every=anchor_every, vocab=vocab)


def listed():
    return [
        # the smallest call: one short sequence on a small model, where launches and host work are everything
        dict(_case("layer", 1, 4096, 4096, 8, 2, 64, 16, 4), name="layer_4k_small_model"),
        # a serving batch: 16 requests of different lengths, chains of five
        dict(_case("layer", 16, 4096, 16384, 32, 8, 64, 32, 5), name="layer_batch16_ragged"),
        # long documents with a draft tree, eight query heads per KV head, blocks of 128 tokens
        dict(_case("layer", 4, 131072, 131072, 64, 8, 128, 32, 16, tree=True), name="layer_4x128k_tree16"),
        # one request verified with a wide tree (60 rows, 240 query rows per KV head)
        dict(_case("layer", 1, 32768, 32768, 32, 8, 64, 109, 60, tree=True), name="layer_32k_tree60"),
        # the same for a batch of shorter requests, odd lengths
        dict(_case("layer", 12, 6001, 9999, 32, 8, 64, 74, 60, tree=True), name="layer_batch12_tree60"),
        # the headline: one 32K request through a stack of 32 layers, every layer selecting
        dict(_case("step", 1, 32768, 32768, 32, 8, 64, 64, 8, layers=32), name="step_32k_32_layers"),
        # the same stack with every second layer reusing the list before it, fed from and read back to the host
        dict(_case("host", 1, 32768, 32768, 32, 8, 64, 64, 8, layers=32, anchor_every=2), name="host_step_32k_reuse"),
        # dense verification of one layer of that request, and of the long batch (the largest case: 2 GiB of cache)
        dict(_case("dense", 1, 32768, 32768, 32, 8, 64, 512, 8), name="dense_32k_chain8"),
        dict(_case("dense", 4, 131072, 131072, 64, 8, 128, 1024, 16, tree=True), name="dense_4x128k_tree16"),
        # representatives after the prefill of a ragged batch
        dict(_case("reps", 16, 4096, 16384, 32, 8, 64, 32, 5), name="reps_batch16_ragged"),
        # the end of a step for a single request on a 32-layer stack, vocabulary of 128256
        dict(_case("finish", 1, 32768, 32768, 32, 8, 64, 64, 8, layers=32, vocab=128256), name="finish_32k_32_layers"),
        # a whole decoding step of a small batch with odd lengths, every fourth layer selecting
        dict(_case("decode", 4, 7001, 16001, 32, 8, 64, 48, 6, layers=16, anchor_every=4, vocab=128256),
             name="decode_batch4_16_layers"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    while True:
        op = rng.choice(["layer", "layer", "layer", "dense", "step", "host", "reps", "finish", "decode"])
        heads, kv_heads = rng.choice([(8, 2), (32, 8), (32, 8), (64, 8), (28, 4), (40, 8), (16, 16)])
        stack = op in ("step", "host", "finish", "decode")
        block = rng.choice([64, 64, 128])
        hi = _log(rng, 1024, 131072)
        lo = hi if rng.random() < 0.4 else rng.randint(hi // 3, hi)
        seqs = _log(rng, 1, 8 if stack else 32)
        layers = _log(rng, 4, 32) if stack else 1
        tree = rng.random() < 0.4
        draft = rng.randint(1, 16) if stack or not tree or rng.random() < 0.5 else rng.randint(17, 60)
        keep = max(SINK + LOCAL + 2, int(-(-hi // block) * math.exp(rng.uniform(math.log(1 / 32), math.log(1 / 4)))))
        case = _case(op, seqs, lo, hi, heads, kv_heads, block, keep, draft, tree, layers,
                     rng.choice([1, 1, 2, 4]) if stack else 1, rng.choice([32000, 128256, 151936]) if op in ("finish", "decode") else 0)
        pool = 2 * layers * seqs * hi * kv_heads * HEAD_DIM * 2
        w = work(case)
        if pool <= 4.3 * GIB and w["bytes"] <= 2.1 * GIB and w["flops"] <= 2.6e11:
            return case


# ------------------------------------------------------------------------------------------------ inputs


def _normal(gen, *shape, sigma=1.0):
    return torch.empty(shape, dtype=torch.bfloat16, device="cuda").normal_(0.0, sigma, generator=gen)


def _shape_keys(gen, k_pool, q, table, lens, n_blocks, case):
    """Moves every block's mean key along the retrieval query so that the block scores follow a continuous bulk with a
    heavy upper tail, and the kept and the evicted ones are apart."""
    S, H, B = case["seqs"], case["kv_heads"], case["block"]
    qbar = q[:, 0].float().view(S, H, case["heads"] // H, HEAD_DIM).mean(2)
    u = qbar / qbar.norm(dim=-1, keepdim=True)
    nb_max = int(n_blocks.max())
    sd = SIGMA / math.sqrt(B)
    b = torch.arange(nb_max, device="cuda")
    exists = b < n_blocks[:, None]
    free = exists & (b >= SINK) & (b < n_blocks[:, None] - LOCAL)
    bulk = torch.randn((S, H, nb_max), generator=gen, device="cuda")
    tail = torch.empty((S, H, nb_max), device="cuda").exponential_(1.0, generator=gen) * 2.0
    tail *= torch.rand((S, H, nb_max), generator=gen, device="cuda") < 0.1
    want = (bulk + tail).masked_fill(~free[:, None], -math.inf)
    rank = want.argsort(dim=-1, descending=True).argsort(dim=-1)
    n_free = (torch.full_like(n_blocks, case["keep"]).minimum(n_blocks) - SINK - LOCAL).clamp(min=0)
    want = want + 0.05 * (rank < n_free[:, None, None])
    for s in range(S):
        nb = int(n_blocks[s])
        for c in range(0, nb, 1024):
            pages = table[s, c:min(nb, c + 1024)].long()
            k = k_pool[pages].float()                                             # [blocks][H][B][D]
            at = torch.arange(c, c + k.shape[0], device="cuda")
            held = (lens[s] - at * B).clamp(max=B)
            along = torch.einsum("nhbd,hd->nhb", k, u[s])
            valid = torch.arange(B, device="cuda") < held[:, None, None]
            mean = (along * valid).sum(-1) / held[:, None]
            goal = want[s, :, c:c + k.shape[0]].T * sd
            shift = torch.where(torch.isfinite(goal), goal - mean, torch.zeros_like(mean))
            k_pool[pages] = (k + shift[:, :, None, None] * u[s][None, :, None, :]).to(torch.bfloat16)


def _distributions(gen, case):
    S, T, V = case["seqs"], case["draft"], case["vocab"]

    def dist(logits):
        logits = logits.masked_fill(logits < logits.amax(-1, keepdim=True) - math.log(50.0), -math.inf)
        return torch.softmax(logits, dim=-1)

    target = torch.randn((S, T, V), generator=gen, device="cuda") / 0.35
    draft = target + 0.2 / 0.35 * torch.randn((S, T, V), generator=gen, device="cuda")
    return dist(target), dist(draft)


def prepare(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    cpu = torch.Generator().manual_seed(seed)
    S, T, L, B = case["seqs"], case["draft"], case["layers"], case["block"]
    Hq, Hkv, op = case["heads"], case["kv_heads"], case["op"]
    lens = torch.randint(case["lo"], case["hi"] + 1, (S,), generator=cpu, dtype=torch.int32)
    room = (lens + T + B - 1) // B                       # blocks the sequence holds once a whole draft was accepted
    max_blocks = -(-(case["hi"] + T) // B)
    n_pages = S * max_blocks
    pages = torch.randperm(n_pages, generator=cpu, dtype=torch.int32)
    table = torch.full((S, max_blocks), -1, dtype=torch.int32)
    at = 0
    for s in range(S):
        n = int(room[s])
        table[s, :n] = pages[at:at + n]
        at += n
    table, lens = table.cuda(), lens.cuda()
    n_blocks = (lens + B - 1) // B
    parent = torch.arange(-1, T - 1, dtype=torch.int32).repeat(S, 1)
    if case["tree"]:
        for i in range(1, T):
            parent[:, i] = torch.randint(0, i, (S,), generator=cpu, dtype=torch.int32)
    keep = min(case["keep"], max_blocks)
    verifier = engine.SparseVerifier(
        n_seq=S, n_q_heads=Hq, n_kv_heads=Hkv, head_dim=HEAD_DIM, block_size=B, max_blocks=max_blocks, n_draft=T, n_layers=L,
        block_table=table, seq_lens=lens.clone(), budget_blocks=torch.full((S,), keep, dtype=torch.int32, device="cuda"),
        max_sel=keep, n_sink=SINK, n_local=LOCAL, anchors=[l % case["anchor_every"] == 0 for l in range(L)],
        parent=parent.cuda() if case["tree"] else None)
    st = dict(op=op, verifier=verifier, lens=lens)
    st["k"] = _normal(gen, L, n_pages, Hkv, B, HEAD_DIM, sigma=SIGMA)
    st["v"] = _normal(gen, L, n_pages, Hkv, B, HEAD_DIM)
    st["q"] = _normal(gen, L, S, T, Hq, HEAD_DIM, sigma=SIGMA)
    st["draft_k"] = _normal(gen, L, S, T, Hkv, HEAD_DIM, sigma=SIGMA)
    st["draft_v"] = _normal(gen, L, S, T, Hkv, HEAD_DIM)
    st["out"] = torch.zeros_like(st["q"])
    if op in ("layer", "step", "host", "decode"):
        for l in range(L):
            _shape_keys(gen, st["k"][l], st["q"][l], table, lens, n_blocks, case)
    if op in ("step", "host"):
        verifier.set_kv_stack(st["k"], st["v"])          # one allocation for all layers
    else:
        for l in range(L):
            verifier.set_layer_kv(l, st["k"][l], st["v"][l])
    if op != "reps":
        for l in range(L):
            verifier.build_reps(l)
    if op == "host":
        for name in ("q", "draft_k", "draft_v", "out"):
            st[name + "_host"] = st[name].cpu().pin_memory()
    if op in ("finish", "decode"):
        st["p_target"], st["p_draft"] = _distributions(gen, case)
        tokens = torch.zeros((S, T), dtype=torch.int32, device="cuda")
        for s in range(S):
            for i in range(1, T):
                tokens[s, i] = torch.multinomial(st["p_draft"][s, parent[s, i]], 1, generator=gen)[0]
        st["tokens"] = tokens
        st["u_accept"] = torch.rand((S, T), generator=gen, device="cuda")
        st["u_next"] = torch.rand((S,), generator=gen, device="cuda")
    return st


# ------------------------------------------------------------------------------------------------ one pass


def _finish(st):
    v = st["verifier"]
    path, n_path, next_token = v.accept(st["p_target"], st["p_draft"], st["tokens"], st["u_accept"], st["u_next"])
    v.commit(st["draft_k"], st["draft_v"], path, n_path)
    return dict(path=path, n_path=n_path, next_token=next_token, seq_lens=v.seq_lens, reps=v.reps, k=st["k"], v=st["v"])


def run(st):
    v, op = st["verifier"], st["op"]
    if op == "layer":
        v.verify_layer(0, st["q"][0], st["draft_k"][0], st["draft_v"][0], st["out"][0])
        return dict(out=st["out"], idx=v.sel_idx, cnt=v.sel_cnt)
    if op == "dense":
        v.dense_layer(0, st["q"][0], st["draft_k"][0], st["draft_v"][0], st["out"][0])
        return st["out"]
    if op == "step":
        v.verify_step(st["q"], st["draft_k"], st["draft_v"], st["out"], refresh_tail=True)
        return dict(out=st["out"], reps=v.reps)
    if op == "host":
        v.verify_step_from_host(st["q_host"], st["draft_k_host"], st["draft_v_host"], st["q"], st["draft_k"], st["draft_v"],
                                st["out"], st["out_host"], refresh_tail=True)
        return dict(out=st["out_host"], reps=v.reps)
    if op == "reps":
        v.build_reps(0)
        return v.reps
    v.seq_lens.copy_(st["lens"])     # the tokens of the pass before are retracted: every pass is the same decoding step
    if op == "finish":
        return _finish(st)
    v.verify_step(st["q"], st["draft_k"], st["draft_v"], st["out"])
    return dict(_finish(st), out=st["out"])


# ------------------------------------------------------------------------------------------------ what a pass needs


def work(case):
    """Bytes and operations of one pass: every input read once, every output written once."""
    S, T, L, B = case["seqs"], case["draft"], case["layers"], case["block"]
    Hq, Hkv, op = case["heads"], case["kv_heads"], case["op"]
    tokens = (case["lo"] + case["hi"]) / 2
    blocks = tokens / B
    anchors = -(-L // case["anchor_every"])
    rows = S * T * Hq
    io = L * (2 * rows + 2 * S * T * Hkv) * HEAD_DIM * 2                       # Q and output, the draft's K and V
    select = anchors * S * Hkv * (blocks * HEAD_DIM * 4 + min(case["keep"], blocks) * 4)
    tail = L * S * Hkv * HEAD_DIM * (B / 2 * 2 + 4)                            # half a block read, its mean written

    def attention(kept):
        return dict(bytes=io + L * S * Hkv * kept * HEAD_DIM * 4, flops=L * rows * (kept + T / 2) * HEAD_DIM * 4)

    sparse = attention(min(case["keep"] * B, tokens))
    scores = anchors * S * Hkv * blocks * HEAD_DIM * 2
    accept = S * case["vocab"] * 4 * 2                                         # a row of either distribution
    commit = tail + L * S * Hkv * HEAD_DIM * 2 * 2 * 2 * min(T, 3)             # K and V of the kept rows, read and written
    if op == "layer":
        return dict(bytes=sparse["bytes"] + select, flops=sparse["flops"] + scores)
    if op == "dense":
        return attention(tokens)
    if op in ("step", "host"):
        return dict(bytes=sparse["bytes"] + select + tail, flops=sparse["flops"] + scores)
    if op == "reps":
        return dict(bytes=L * S * Hkv * HEAD_DIM * (tokens * 2 + blocks * 4), flops=L * S * Hkv * HEAD_DIM * tokens)
    if op == "finish":
        return dict(bytes=accept + commit, flops=S * case["vocab"] * 4)
    return dict(bytes=sparse["bytes"] + select + accept + commit, flops=sparse["flops"] + scores + S * case["vocab"] * 4)


def tolerance(case):
    """Lists, tokens, lengths and cache rows are whole values or copies; representatives are fp32 means; attention rounds
    its probabilities and its outputs to bf16."""
    if case["op"] in ("reps", "finish"):
        return {"rel": 1e-5, "max": 1e-4, "differ": 0.0}
    return {"rel": 5e-3, "max": 0.05, "differ": 0.0}
