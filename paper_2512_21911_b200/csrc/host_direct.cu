// sv_verify_step_from_host_direct: a verification step whose inputs are in pinned host memory and whose outputs are wanted there, as four
// launches: tail blocks, the queries that select, selection, attention.  The attention kernel reads a list's rows from host memory when a
// CTA takes the list and writes its outputs there when it is through (kHost in verify_attn_tc.cu); there are no copies ahead of it or
// behind it, no side streams and no chunks whose launches wait for one another.  Bound by what the K/V take from HBM, by the bus where the
// queries are many.  32 layers of 8 lists of 64 units, 3 MiB up, 2 MiB down, all
// selecting: 176 us in two chunks, 142 this way (100 with everything on the device); every second one selecting 174 and 132 to 137.  On
// another machine 24 layers x 16 lists of 16 units 139 -> 107, 16 layers x 32 lists x 48 units 257 -> 202.
#include <cuda_runtime.h>

#include "sv.h"
#include "sv_host.h"
#include "sv_ptx.cuh"

namespace {

// The first draft token's query rows of the selecting layers, which selection reads, to their place in the device tensor.  Bound by the
// bus: 128 KB of 16 layers, 3 us and a round trip.
struct FirstRows {
    const uint4 *from;
    uint4 *to;
    int32_t words, pitch, S, total;   // 16-byte words of a row (all query heads), from one sequence's to the next one's; sequences; all words
    uint8_t layer_of[SV_MAX_LAYERS];
};
constexpr int kThreads = 256;
__global__ void __launch_bounds__(kThreads) first_rows_kernel(const FirstRows p)
{
    svk::grid_dependency_wait();
    svk::grid_launch_dependents();
    const int i = blockIdx.x * kThreads + threadIdx.x;
    if (i >= p.total) return;
    const int row = i / p.words, a = row / p.S, s = row - a * p.S;
    const size_t at = ((size_t)p.layer_of[a] * p.S + s) * p.pitch + (i - row * p.words);
    p.to[at] = __ldcv(p.from + at);
}

}  // namespace

extern "C" sv_status sv_verify_step_from_host_direct(const sv_geom *geom, const sv_layers *layers, const uint8_t *anchors, const void *q_host,
                                                     const void *draft_k_host, const void *draft_v_host, void *q, void *draft_k,
                                                     void *draft_v, const int32_t *parent, float *reps, const int32_t *budget_blocks,
                                                     int32_t n_sink, int32_t n_local, int32_t *idx, int32_t *cnt, int32_t max_sel, void *out,
                                                     void *out_host, void *workspace, size_t workspace_bytes, int32_t *status_word,
                                                     int32_t refresh_tail, const uint8_t *refresh_which, void *stream)
{
    if (!q_host || !draft_k_host || !draft_v_host || !out_host || !q || !draft_k || !draft_v || !out || !anchors) return SV_ERR_NULL;
    sv_status st = svh::check_layers(geom, layers, 0, layers ? layers->n_layers : 1);
    if (st != SV_OK) return st;
    if (!svh::lists_handed_out(geom, layers, max_sel)) return SV_ERR_UNSUPPORTED;
    const svh::HostTensors host = {svh::mapped(q_host), svh::mapped(draft_k_host), svh::mapped(draft_v_host), svh::mapped(out_host)};
    for (const void *p : {host.q, host.draft_k, host.draft_v, static_cast<const void *>(host.out)})
        if (!p || !svh::aligned(p, 16)) return SV_ERR_UNSUPPORTED;
    // everything that a later launch would refuse, ahead of the first one
    const auto attend = [&](bool check_only) {
        return svh::verify_attn_from_host(geom, layers, anchors, host, q, draft_k, draft_v, parent, idx, cnt, max_sel, out, workspace,
                                          workspace_bytes, status_word, stream, check_only);
    };
    st = svh::check_select_layers(geom, anchors, q, reps, budget_blocks, n_sink, n_local, idx, cnt, max_sel);
    if (st == SV_OK) st = attend(true);
    if (st != SV_OK) return st;
    FirstRows rows;
    rows.from = static_cast<const uint4 *>(host.q), rows.to = static_cast<uint4 *>(q);
    rows.words = geom->n_q_heads * 16, rows.pitch = geom->n_draft * geom->n_q_heads * 16, rows.S = geom->n_seq;
    int n = 0;
    for (int l = 0; l < layers->n_layers; ++l)
        if (anchors[l]) rows.layer_of[n++] = (uint8_t)l;
    const long long total = (long long)n * geom->n_seq * rows.words;
    if (total >= 1ll << 31 || (long long)rows.pitch * geom->n_seq >= 1ll << 31) return SV_ERR_UNSUPPORTED;
    rows.total = (int32_t)total;
    if (refresh_tail) {
        st = sv_block_reps_layers(geom, layers, refresh_which, SV_TAIL_BLOCK, -1, reps, stream);
        if (st != SV_OK) return st;
    }
    if (total > 0) {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3((unsigned)((total + kThreads - 1) / kThreads));
        cfg.blockDim = dim3(kThreads);
        cfg.stream = static_cast<cudaStream_t>(stream);
        cudaLaunchAttribute attr[1];
        svh::pdl_attribute(attr);
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        if (cudaLaunchKernelEx(&cfg, first_rows_kernel, rows) != cudaSuccess) return SV_ERR_CUDA;
    }
    st = sv_select_blocks_layers(geom, layers, 0, layers->n_layers, anchors, q, reps, budget_blocks, n_sink, n_local, idx, cnt, max_sel, stream);
    if (st != SV_OK) return st;
    return attend(false);
}
