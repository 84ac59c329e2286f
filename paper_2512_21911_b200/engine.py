"""SparseVerifier: runs block selection and sparse verification attention for a stack of layers.

A thin driver over the C-ABI calls: it owns the per-layer representatives, the block lists,
the split-KV workspace and the outputs.  ``verify_layer`` enqueues one layer: ``sv_select_blocks`` (anchor
layers) or the reuse of the previous layer's list (Eq. 9), then ``sv_verify_attn``.  ``verify_step`` is handed the inputs
of all layers at once; but for the lists they reuse the layers are then independent problems, so it runs all
selections in one launch and all attention in another.  After verification,
``accept`` (Eq. 2-3) and ``commit`` (append the kept rows to the cache) close the decoding step.  All compute
is in the library's kernels; this class only holds buffers and calls them in order.
"""
from __future__ import annotations

from typing import List, Optional, Sequence

import torch

from . import binding as sv


DIRECT_BYTES = 24 << 20   # what a host-fed step may upload and still go without chunks (SparseVerifier._direct)
# What the schedule of a host-fed step reckons with: bytes per microsecond up, down, from HBM and by one CTA alone, microseconds per
# chunk (its launches; the copies of a further one).  Fitted to the differences between the schedules of 184 stacks on two
# machines (the sums come out 4 % high on average): a B200 on a PCIe 5 link, of which only the proportions matter here.
UP_RATE, DOWN_RATE, HBM_RATE, CTA_RATE, LAUNCH_US, COPY_US = 36e3, 57e3, 6.4e6, 76e3, 18.0, 18.0


def host_step_us(sizes: Sequence[int], upload: float, download: float, gathered: float, lists: int, sms: int = 148) -> float:
    """What a host-fed step in chunks of these sizes takes, by bytes and lists per layer: uploads one after the other, a chunk's
    kernels behind its upload and the chunk before, its download behind them.  A chunk is taken to gather at the rate of HBM however
    few its lists are (few are split over the SMs); where there are more lists than SMs, the last of them run on a part of the SMs
    (32 layers of 8 lists in chunks of 14 + 18 layers: 178 us, of 12 + 20 layers, 160 lists: 213)."""
    up = computed = down = 0.0
    for i, n in enumerate(sizes):
        up += n * upload / UP_RATE + (COPY_US if i else 0.0)
        computed = max(up, computed) + LAUNCH_US + n * gathered / HBM_RATE
        if n * lists > sms:
            computed += gathered / lists / CTA_RATE * (-n * lists % sms) / sms
        down = max(computed, down) + n * download / DOWN_RATE
    return down


def host_step_schedule(n: int, upload: float, download: float, gathered: float, lists: int, sms: int = 148) -> List[int]:
    """Layers per chunk of a host-fed step of n layers.  Nothing hides the first upload and the last download, and every chunk costs
    launches and copies: a step of few bytes is one chunk, one with much to move and to compute ends soonest with a short last
    chunk.  7/16 and 9/16 of the layers (fewer than four: all at once) unless another split is reckoned to be 2 % faster.

    Over 331 timings of stacks on three machines (2 to 32 layers, 1 to 8 sequences of 1K to 131K tokens, 1 to 60 draft tokens), the 147 of
    one machine not part of the fit, what this picks takes 0.938 of the time of that usual split in the geometric mean, more than 1.01 of it for ten of them
    and 1.05 at worst (7.7 MB up and 34 MB gathered, in three chunks), and 1.006 of the best of these four: 13 layers x 57K 53 -> 37
    us, 31 layers x 5 sequences 501 -> 460, 3 x 8 sequences of 32K 327 -> 272; 32 layers of a 32K context 178 (183 in 10 + 14 + 8)."""
    if n == 1:
        return [1]
    first = max(1, n * 7 // 16)
    splits = [[first, n - first], [n], [n // 2, n - n // 2]]
    if n >= 4:
        third = max(1, n * 5 // 16)
        splits.append([third, n - third - n // 4, n // 4])
    usual = splits[0] if n >= 4 else splits[1]
    reckon = lambda sizes: host_step_us(sizes, upload, download, gathered, lists, sms)
    best = min(splits, key=reckon)
    return best if reckon(best) < 0.98 * reckon(usual) else usual


class SparseVerifier:
    def __init__(self, *, n_seq: int, n_q_heads: int, n_kv_heads: int, head_dim: int, block_size: int,
                 max_blocks: int, n_draft: int, n_layers: int, block_table: torch.Tensor, seq_lens: torch.Tensor,
                 budget_blocks: torch.Tensor, max_sel: int, n_sink: int = 1, n_local: int = 1,
                 anchors: Optional[Sequence[bool]] = None, parent: Optional[torch.Tensor] = None,
                 device: str = "cuda"):
        self.geom = sv.make_geom(n_seq, n_q_heads, n_kv_heads, head_dim, block_size, max_blocks, n_draft)
        self.n_layers = n_layers
        self.block_table, self.seq_lens, self.budget, self.parent = block_table, seq_lens, budget_blocks, parent
        self.n_sink, self.n_local, self.max_sel = n_sink, n_local, max_sel
        self.anchors = list(anchors) if anchors is not None else [True] * n_layers
        assert self.anchors[0], "layer 0 has no preceding layer to reuse"
        dev = torch.device(device)
        self.reps = torch.zeros((n_layers, n_seq, n_kv_heads, max_blocks, head_dim), dtype=torch.float32, device=dev)
        self._make_lists(bytes(map(bool, self.anchors)), dev)
        self.workspace = torch.empty(max(16, sv.sv_workspace_bytes(self.geom, max_sel)), dtype=torch.uint8, device=dev)
        self.dense_workspace = None
        self.status = torch.zeros(1, dtype=torch.int32, device=dev)
        self.kv: List[Optional[sv.sv_kv]] = [None] * n_layers
        self._pools = [None] * n_layers   # keep the tensors alive
        self._one_allocation = False
        self._copy_streams = None
        self._host_step = None
        rows, pairs = n_seq * n_draft * head_dim * 2, n_seq * n_kv_heads
        self._schedule = host_step_schedule(
            n_layers, rows * (n_q_heads + 2 * n_kv_heads), rows * n_q_heads,
            pairs * head_dim * 4 * (min(max_sel, max_blocks) * block_size + max_blocks * sum(map(bool, self.anchors)) / n_layers), pairs,
            torch.cuda.get_device_properties(dev).multi_processor_count)
        self._counters = torch.zeros(2 * n_seq, dtype=torch.int32, device=dev)   # see sv_kv_append_layers
        # what the layers' kernels look up when several layers run in one launch (a row is valid once its layer has pools)
        stackable = n_layers <= sv.SV_MAX_LAYERS and n_layers * n_seq <= 65535
        row = sv._lib.sv_layer_table_bytes(1)
        self._table = torch.zeros((n_layers, row), dtype=torch.uint8, device=dev) if stackable else None
        self._rows_missing = n_layers
        # Of a stack's workspaces (sparse, dense) those in which the launches keep something between calls are made and zeroed
        # here: a fill in the first step would be a node of a graph, and not have run, when that step is captured.  The others
        # are scratch of many megabytes, written before they are read: made when they are needed.
        need = [sv._native.workspace_bytes_layers(self.geom, n_layers, n) if stackable else 0 for n in (max_sel, self.geom.max_blocks)]
        keeps = [n == sv.SV_STACK_STATE_BYTES for n in need]
        # A host-fed step of a stack whose lists go to resident CTAs needs no chunks.  90 such stacks (4 to 30 layers, 1 to 8 sequences of
        # 1K to 42K tokens, 1 to 16 draft tokens) take 0.81 of the time of the schedule above in the geometric mean, 1.01 or more only one
        # of them, with 33 MB to read: there the bus is all that counts, and the copy engine has a few percent more of it.
        self._direct = keeps[0] and n_layers * rows * (n_q_heads + 2 * n_kv_heads) <= DIRECT_BYTES
        self._stack_bytes = [sv._native.workspace_bytes_host_step(self.geom, n_layers, max_sel) if stackable else 0, need[1]]
        self._stack_workspace = [torch.zeros(n, dtype=torch.uint8, device=dev) if k else None for n, k in zip(self._stack_bytes, keeps)]

    def _make_lists(self, flags: bytes, dev) -> None:
        """One block list per anchor layer; sel_idx / sel_cnt is the last one, which is also what verify_layer keeps its
        current list in."""
        g, n = self.geom, max(1, sum(flags))
        self._flags = flags
        self._lists_idx = torch.zeros((n, g.n_seq, g.n_kv_heads, self.max_sel), dtype=torch.int32, device=dev)
        self._lists_cnt = torch.zeros((n, g.n_seq, g.n_kv_heads), dtype=torch.int32, device=dev)
        self.sel_idx, self.sel_cnt = self._lists_idx[-1], self._lists_cnt[-1]

    def set_layer_kv(self, layer: int, k_pool: torch.Tensor, v_pool: torch.Tensor) -> None:
        new = self.kv[layer] is None
        self._pools[layer] = (k_pool, v_pool)
        self.kv[layer] = sv.make_kv(k_pool, v_pool, self.block_table, self.seq_lens)
        if self._table is not None:
            row = sv._native.layer_row(self.geom, self.kv[layer])
            if isinstance(row, int):
                self._table = None   # not a cache the kernels take: the call that uses it says so
            else:
                self._table[layer].copy_(torch.frombuffer(bytearray(row), dtype=torch.uint8))
        self._rows_missing -= new

    def set_kv_stack(self, k_all: torch.Tensor, v_all: torch.Tensor) -> None:
        """All layers' pools in one allocation, bf16 [layers][n_pages][Hkv][B][D]."""
        n_layers = int(k_all.shape[0])
        assert n_layers == self.n_layers and k_all.is_contiguous() and v_all.is_contiguous()
        for l in range(n_layers):
            self.set_layer_kv(l, k_all[l], v_all[l])
        self._one_allocation = True

    def sync_block_table(self) -> None:
        """Kept for callers that announce newly assigned pages: every launch reads block_table itself, so there is nothing
        to rebuild."""

    def _stacked(self) -> bool:
        """Whether launches may cover several layers: every layer has its pools, over the same page table and lengths."""
        return self._table is not None and self._rows_missing == 0

    def refresh_tail_all(self) -> None:
        """Recompute the representative of every sequence's last block in all layers (one launch)."""
        self._refresh_tail(None)

    def _refresh_tail(self, which: Optional[bytes]) -> None:
        if self._stacked():
            sv._check(sv._native.block_reps_layers(self.geom, self._table, self.kv[0], which, sv.SV_TAIL_BLOCK, -1, self.reps),
                      "sv_block_reps_layers")
            return
        for l in range(self.n_layers):
            if which is None or which[l]:
                sv.sv_block_reps(self.geom, self.kv[l], self.reps[l], sv.SV_TAIL_BLOCK)

    def _anchor_flags(self) -> bytes:
        flags = bytes(map(bool, self.anchors))
        if flags != self._flags:
            self._make_lists(flags, self.workspace.device)
        return flags

    def _workspace_of_stack(self, dense: bool) -> torch.Tensor:
        if self._stack_workspace[dense] is None:
            self._stack_workspace[dense] = torch.empty(max(16, self._stack_bytes[dense]), dtype=torch.uint8, device=self.workspace.device)
        return self._stack_workspace[dense]

    def _run_layers(self, first: int, end: int, q, draft_k, draft_v, out, dense: bool = False) -> bool:
        """Layers first .. end - 1 in two launches (dense: one; three when the splits have to be merged).  False when the
        inputs are not stacked tensors: the caller then goes layer by layer."""
        if not self._stacked():
            return False
        flags = self._anchor_flags()
        failed = sv._native.verify_layers(self.geom, self._table, self.kv[0], first, end, flags, q, draft_k, draft_v, self.parent, out,
                                          self.reps, self.budget, self.n_sink, self.n_local, None if dense else self._lists_idx,
                                          None if dense else self._lists_cnt, self._workspace_of_stack(dense), self.status)
        if failed is False:
            return False
        if failed:
            raise sv.SvError(failed[0], "sv_select_blocks_layers" if failed[1] else "sv_verify_attn_layers")
        return True

    def build_reps(self, layer: int, block_begin: int = 0, block_end: int = -1) -> None:
        """(Re)compute block representatives of a layer; a decoding loop only refreshes the tail block."""
        sv.sv_block_reps(self.geom, self.kv[layer], self.reps[layer], block_begin, block_end)

    def verify_layer(self, layer: int, q, draft_k, draft_v, out, lse=None, behind_own_layer: bool = False) -> None:
        """select (anchor) or reuse (non-anchor), then sparse verification attention, on the current stream.

        behind_own_layer: the kernel just before this call in the stream is the preceding layer's attention / merge
        (as inside verify_step), which writes neither the block list nor the cache: a layer that reuses the list
        then starts its gather while that kernel drains (sv_verify_attn_reused)."""
        # a layer that reuses (Eq. 9) finds the preceding layer's list in place, so nothing is launched for it
        failed = sv._native.verify_layer(self.geom, self.kv[layer], q, self.reps, layer, self.seq_lens, self.budget, self.n_sink,
                                         self.n_local, self.sel_idx, self.sel_cnt, draft_k, draft_v, self.parent, out, lse,
                                         self.workspace, self.status, self.anchors[layer], behind_own_layer)
        if failed:
            raise sv.SvError(failed[0], "sv_select_blocks" if failed[1] else "sv_verify_attn")

    def dense_layer(self, layer: int, q, draft_k, draft_v, out, lse=None) -> None:
        """Dense ("strict") verification attention over every cached block, for comparison."""
        if self.dense_workspace is None:
            n = max(16, sv.sv_workspace_bytes(self.geom, self.geom.max_blocks))
            self.dense_workspace = torch.empty(n, dtype=torch.uint8, device=self.workspace.device)
        sv.sv_verify_attn(self.geom, q, self.kv[layer], draft_k, draft_v, self.parent, None, None, out, lse=lse,
                          workspace=self.dense_workspace, status_word=self.status)

    def verify_step(self, q, draft_k, draft_v, out, refresh_tail: bool = False) -> None:
        """One verification step of the whole stack.  q/out: [layers][S][T][Hq][D]; draft_k/v: [layers][S][T][Hkv][D].

        refresh_tail: first recompute the representative of every sequence's last block (the block that
        grew when the previous step's accepted tokens were appended), in one launch: of all layers when the pools were
        given with set_kv_stack, else of the anchor layers.

        All layers' selections are one launch and all their attention another (32 layers of a 32K context: about 110 us
        instead of 440 layer by layer, where every layer pays the latency chain of its kernels).  A model whose layers
        wait for one another calls verify_layer."""
        if refresh_tail:
            self._refresh_tail(None if self._one_allocation else self._anchor_flags())
        if self._run_layers(0, self.n_layers, q, draft_k, draft_v, out):
            return
        for l in range(self.n_layers):
            self.verify_layer(l, q[l], draft_k[l], draft_v[l], out[l], behind_own_layer=l > 0)

    def verify_step_from_host(self, q_host, draft_k_host, draft_v_host, q, draft_k, draft_v, out, out_host,
                              layers_per_chunk=None, refresh_tail: bool = False) -> None:
        """verify_step with the step's inputs in pinned host memory and its outputs wanted there.  q/draft_k/draft_v/out are the
        device staging tensors (shapes as for verify_step); the *_host tensors the pinned ones.  Returns with everything enqueued; the
        current stream ends behind the last byte that is brought back.  Capturable in a CUDA graph.

        Where the stack's lists are handed out to resident CTAs (more lists than SMs, at most 64 query rows a KV head), the step
        uploads no more than DIRECT_BYTES, the memory is pinned and 16-byte aligned and no chunks are asked for, there are none: the
        attention launch itself reads a list's rows from host memory when a CTA takes the list and writes its outputs there, and the
        outputs are those of verify_step bit for bit.

        Else the copies go in chunks of a few layers (layers_per_chunk: one size, or a list of sizes) on two side streams, which fork
        from and join the current one: a chunk's layers start as soon as its inputs have arrived, its outputs leave while the next
        chunk computes, so only the first upload and the last download are not hidden behind kernels.  A chunk of few lists is
        split over the SMs for itself, so the outputs are those of verify_step to bf16 rounding.  Large chunks are faster: each is a
        launch of its own that the next one waits for.

        32 layers of a 32K context that all select, on one machine: 142 us without chunks, 176 in two, 184 in chunks of eight layers,
        224 of four, 550 of one."""
        if layers_per_chunk is None and self._direct and self._stacked() and \
                self._from_host(None, q_host, draft_k_host, draft_v_host, q, draft_k, draft_v, out, out_host, refresh_tail):
            return
        chunks = self._chunks(layers_per_chunk)
        if self._copy_streams is None:
            self._copy_streams = (torch.cuda.Stream(device=q.device), torch.cuda.Stream(device=q.device))
        if self._stacked() and self._from_host(chunks, q_host, draft_k_host, draft_v_host, q, draft_k, draft_v, out, out_host, refresh_tail):
            return
        main = torch.cuda.current_stream()
        s_in, s_out = self._copy_streams
        s_in.wait_stream(main)
        s_out.wait_stream(main)
        arrived = []
        with torch.cuda.stream(s_in):
            for c0, c1 in chunks:
                q[c0:c1].copy_(q_host[c0:c1], non_blocking=True)
                draft_k[c0:c1].copy_(draft_k_host[c0:c1], non_blocking=True)
                draft_v[c0:c1].copy_(draft_v_host[c0:c1], non_blocking=True)
                ev = torch.cuda.Event()
                ev.record(s_in)
                arrived.append(ev)
        if refresh_tail:
            self._refresh_tail(None if self._one_allocation else self._anchor_flags())
        for (c0, c1), ev in zip(chunks, arrived):
            main.wait_event(ev)
            if not self._run_layers(c0, c1, q, draft_k, draft_v, out):
                for l in range(c0, c1):
                    # the kernel before a chunk's first layer is not this stream's previous layer alone (the upload joins there)
                    self.verify_layer(l, q[l], draft_k[l], draft_v[l], out[l], behind_own_layer=l > c0)
            done = torch.cuda.Event()
            done.record(main)
            s_out.wait_event(done)
            with torch.cuda.stream(s_out):
                out_host[c0:c1].copy_(out[c0:c1], non_blocking=True)
        main.wait_stream(s_in)
        main.wait_stream(s_out)

    def _chunks(self, layers_per_chunk):
        if layers_per_chunk is None:
            layers_per_chunk = self._schedule
        if isinstance(layers_per_chunk, int):
            sizes = [layers_per_chunk] * -(-self.n_layers // layers_per_chunk)
        else:   # a schedule: e.g. a small first and last chunk (their copies are the ones nothing hides), large ones between
            sizes = list(layers_per_chunk)
        chunks, c0 = [], 0
        for n in sizes:
            if c0 < self.n_layers and n > 0:
                chunks.append((c0, min(c0 + n, self.n_layers)))
                c0 += n
        if c0 < self.n_layers:
            chunks.append((c0, self.n_layers))
        return chunks

    def _from_host(self, chunks, q_host, draft_k_host, draft_v_host, q, draft_k, draft_v, out, out_host, refresh_tail) -> bool:
        """verify_step_from_host in one call of the library.  False when the tensors are not stacked ones."""
        flags = self._anchor_flags()
        if chunks is not None and self._host_step is None:
            self._host_step = sv._native.host_step()
            if isinstance(self._host_step, int):
                raise sv.SvError(self._host_step, "sv_host_step_create")
        st = sv._native.verify_step_from_host(
            self._host_step, self.geom, self._table, self.kv[0], flags, chunks and [c1 for _, c1 in chunks], q_host, draft_k_host, draft_v_host, q,
            draft_k, draft_v, self.parent, self.reps, self.budget, self.n_sink, self.n_local, self._lists_idx, self._lists_cnt, out,
            out_host, self._workspace_of_stack(False), self.status, refresh_tail, None if self._one_allocation else flags,
            *(self._copy_streams if chunks else (None, None)))
        if st is False:
            return False
        sv._check(st, "sv_verify_step_from_host")
        return True

    def accept(self, p_target, p_draft, tokens, u_accept, u_next):
        """Acceptance of the step's draft tokens (Eq. 2-3).  Returns (path [S][T], n_path [S], next_token [S]):
        the rows whose K/V enter the cache (root first) and the token drawn after the kept path."""
        got = sv._native.accept_new(p_target, p_draft, tokens, self.parent, u_accept, u_next, self.geom.n_seq, self.geom.n_draft)
        if isinstance(got, int):
            raise sv.SvError(got, "sv_accept")
        return got

    def commit(self, draft_k, draft_v, path, n_path) -> None:
        """Append the kept rows' K/V of every layer to the paged cache (sv_kv_append, which also refreshes the
        representatives of the blocks that grew, in one launch for all layers) and advance the sequence lengths.  The
        block table must already hold pages for the blocks the sequences grow into.  draft_k/v: [layers][S][T][Hkv][D]."""
        if self._stacked():
            st = sv._native.kv_append_layers(self.geom, self._table, self.kv[0], draft_k, draft_v, path, n_path, self.seq_lens,
                                             self._counters, self.reps)
            if st is not False:
                sv._check(st, "sv_kv_append_layers")
                return
        new_len = torch.empty_like(self.seq_lens)
        for l in range(self.n_layers):
            k_pool, v_pool = self._pools[l]
            sv.sv_kv_append(self.geom, k_pool, v_pool, self.block_table, self.seq_lens, draft_k[l], draft_v[l], path,
                            n_path, new_len, self.reps[l])
        self.seq_lens.copy_(new_len)          # every layer has read the old lengths by now (same stream)

    def check_status(self) -> None:
        """Read the device status word back (this synchronises with the stream) and raise if a kernel gave up
        on a bounded wait, clamped a block index or page id, or met a list that block selection marked invalid
        (count -1).  The outputs written since the word was last zero are then invalid."""
        st = sv.sv_status_word_check(int(self.status.item()))
        if st == sv.SV_OK and int(self._lists_cnt.min().item()) < 0:
            st = 9   # SV_ERR_INDEX: a list marked invalid that no attention call has consumed yet
        if st != sv.SV_OK:
            raise sv.SvError(st, "SparseVerifier.check_status")

    def dense_step(self, q, draft_k, draft_v, out) -> None:
        if self._run_layers(0, self.n_layers, q, draft_k, draft_v, out, dense=True):
            return
        for l in range(self.n_layers):
            self.dense_layer(l, q[l], draft_k[l], draft_v[l], out[l])

    def kernels_per_step(self, refresh_tail: bool = False, dense: bool = False) -> int:
        """An upper bound for the kernel launches of one step taken layer by layer (verify_layer, the order in which a model reaches
        its layers): tail refresh, select per anchor layer, attention per layer and, where lists are split, a merge kernel, which the
        splits that a cluster merges do not have; two launches where the rest of a batch goes by itself.  A sparse step's own number
        is launches_per_step."""
        splits = sv.sv_verify_attn_splits(self.geom, self.geom.max_blocks if dense else self.max_sel)
        attn = self.n_layers * (2 if splits > 1 else 1)
        if dense:
            return attn
        attn = max(attn, self.n_layers * sv.sv_verify_attn_launches(self.geom, self.max_sel))
        refresh = 0 if not refresh_tail else (1 if self._stacked() else sum(self.anchors))
        return refresh + sum(self.anchors) + attn

    def launches_per_step(self, refresh_tail: bool = False) -> int:
        """Kernel launches of one sparse step taken layer by layer, each behind its own preceding layer (verify_layer with
        behind_own_layer, as in verify_step), as they are made on this device."""
        refresh = 0 if not refresh_tail else (1 if self._stacked() else sum(self.anchors))
        selecting = sv.sv_verify_attn_launches(self.geom, self.max_sel)
        # (a reused list of more lists than SMs has no second launch for the rest, see sv_verify_attn_launches)
        reusing = 1 if sv.sv_verify_attn_splits(self.geom, self.max_sel) == 1 else selecting
        n = sum(map(bool, self.anchors))
        return refresh + n + n * selecting + (self.n_layers - n) * reusing
