// sv_verify_step_from_host: a verification step whose inputs are in pinned host memory and whose outputs are wanted there.
// The layers go in chunks: a chunk's inputs are uploaded on one side stream while the chunk before it computes, its
// outputs leave on another while the chunk behind it computes, so only the first upload and the last download are not
// hidden.  (Stacks whose lists are handed out have a form without chunks: host_direct.cu.)  Bound by PCIe for those two and by the launches between them (32 layers of a 32K context, 3 MiB up, 2 MiB down, two
// halves: 178 us, of which the layers' kernels 113 and the two bare transfers 51).  Everything is enqueued here, in one
// call: the same sequence of copies, launches and events from Python took about 5 us each, and the step waited for it
// (245 us).
#include <cuda_runtime.h>

#include <new>

#include "sv.h"
#include "sv_host.h"
#include "sv_ptx.cuh"

namespace {

// The first upload and the last download, which nothing hides, go through a kernel on the step's own stream: pinned memory is
// read and written directly, all tensors in one launch, and neither a copy's 4 us of latency nor a hop between streams
// comes on top of the bytes (181 against 189 us for the step; PCIe is full from four CTAs on, 46 GB/s).
struct Parts {
    uint4 *to[3];
    const uint4 *from[3];
    unsigned end[3];   // running sums of 16-byte words
};
constexpr int kCopyThreads = 256, kCopyCtas = 32, kCopyDepth = 8;
__global__ void __launch_bounds__(kCopyThreads) copy_parts_kernel(const Parts p)
{
    svk::grid_dependency_wait();
    svk::grid_launch_dependents();
    for (unsigned i0 = blockIdx.x * kCopyThreads * kCopyDepth + threadIdx.x; i0 < p.end[2]; i0 += gridDim.x * kCopyThreads * kCopyDepth) {
        uint4 v[kCopyDepth];
#pragma unroll
        for (int u = 0; u < kCopyDepth; ++u) {
            const unsigned i = i0 + u * kCopyThreads;
            if (i < p.end[2]) v[u] = __ldcv(i < p.end[0] ? p.from[0] + i : i < p.end[1] ? p.from[1] + (i - p.end[0]) : p.from[2] + (i - p.end[1]));
        }
#pragma unroll
        for (int u = 0; u < kCopyDepth; ++u) {
            const unsigned i = i0 + u * kCopyThreads;
            if (i < p.end[2]) *(i < p.end[0] ? p.to[0] + i : i < p.end[1] ? p.to[1] + (i - p.end[0]) : p.to[2] + (i - p.end[1])) = v[u];
        }
    }
}

}  // namespace

// Events are kept: creating and destroying them costs as much as a launch each.
struct sv_host_step {
    cudaEvent_t fork = nullptr, joined = nullptr;
    cudaEvent_t arrived[SV_MAX_HOST_CHUNKS] = {}, done[SV_MAX_HOST_CHUNKS] = {};
};

extern "C" sv_host_step *sv_host_step_create(void)
{
    sv_host_step *h = new (std::nothrow) sv_host_step;
    if (!h) return nullptr;
    bool ok = true;
    auto event = [&](cudaEvent_t &e) { ok = ok && cudaEventCreateWithFlags(&e, cudaEventDisableTiming) == cudaSuccess; };
    event(h->fork), event(h->joined);
    for (int c = 0; c < SV_MAX_HOST_CHUNKS; ++c) event(h->arrived[c]), event(h->done[c]);
    if (ok) return h;
    (void)cudaGetLastError();
    sv_host_step_destroy(h);
    return nullptr;
}

extern "C" void sv_host_step_destroy(sv_host_step *h)
{
    if (!h) return;
    auto event = [](cudaEvent_t e) {
        if (e) cudaEventDestroy(e);
    };
    event(h->fork), event(h->joined);
    for (int c = 0; c < SV_MAX_HOST_CHUNKS; ++c) event(h->arrived[c]), event(h->done[c]);
    delete h;
}

extern "C" sv_status sv_verify_step_from_host(sv_host_step *step, const sv_geom *geom, const sv_layers *layers, const uint8_t *anchors,
                                              const int32_t *chunk_end, int32_t n_chunks, const void *q_host, const void *draft_k_host,
                                              const void *draft_v_host, void *q, void *draft_k, void *draft_v,
                                              const int32_t *parent, float *reps, const int32_t *budget_blocks, int32_t n_sink,
                                              int32_t n_local, int32_t *idx, int32_t *cnt, int32_t max_sel, void *out, void *out_host,
                                              void *workspace, size_t workspace_bytes, int32_t *status_word, int32_t refresh_tail,
                                              const uint8_t *refresh_which, void *stream_in, void *stream_out, void *stream)
{
    if (!step || !chunk_end || !q_host || !draft_k_host || !draft_v_host || !out_host || !q || !draft_k || !draft_v || !out)
        return SV_ERR_NULL;
    sv_status st = svh::check_layers(geom, layers, 0, layers ? layers->n_layers : 1);
    if (st != SV_OK) return st;
    if (n_chunks < 1 || n_chunks > SV_MAX_HOST_CHUNKS || chunk_end[n_chunks - 1] != layers->n_layers) return SV_ERR_SHAPE;
    for (int c = 0; c < n_chunks; ++c)
        if (chunk_end[c] <= (c ? chunk_end[c - 1] : 0)) return SV_ERR_SHAPE;
    cudaStream_t main = static_cast<cudaStream_t>(stream), in = static_cast<cudaStream_t>(stream_in), back = static_cast<cudaStream_t>(stream_out);
    bool ok = true;
    auto cuda = [&](cudaError_t e) { ok = ok && e == cudaSuccess; };
    // `to` goes on behind what is on `from` by now; whether it does
    auto order = [&](cudaEvent_t e, cudaStream_t from, cudaStream_t to) {
        const bool done = cudaEventRecord(e, from) == cudaSuccess && cudaStreamWaitEvent(to, e, 0) == cudaSuccess;
        ok = ok && done;
        return done;
    };
    const size_t q_layer = (size_t)geom->n_seq * geom->n_draft * geom->n_q_heads * 256, kv_layer = (size_t)geom->n_seq * geom->n_draft * geom->n_kv_heads * 256;
    auto part = [&](void *to, const void *from, size_t layer, int c, cudaMemcpyKind kind, cudaStream_t s) {
        const size_t l0 = c ? chunk_end[c - 1] : 0, l1 = chunk_end[c];
        cuda(cudaMemcpyAsync(static_cast<char *>(to) + l0 * layer, static_cast<const char *>(from) + l0 * layer, (l1 - l0) * layer, kind, s));
    };
    auto upload = [&](int c) {
        part(q, q_host, q_layer, c, cudaMemcpyHostToDevice, in);
        part(draft_k, draft_k_host, kv_layer, c, cudaMemcpyHostToDevice, in);
        part(draft_v, draft_v_host, kv_layer, c, cudaMemcpyHostToDevice, in);
        cuda(cudaEventRecord(step->arrived[c], in));
    };
    auto copy_parts = [&](const Parts &p) {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(kCopyCtas);
        cfg.blockDim = dim3(kCopyThreads);
        cfg.stream = main;
        cudaLaunchAttribute attr[1];
        svh::pdl_attribute(attr);
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        cuda(cudaLaunchKernelEx(&cfg, copy_parts_kernel, p));
    };
    const void *q_map = svh::mapped(q_host), *k_map = svh::mapped(draft_k_host), *v_map = svh::mapped(draft_v_host);
    void *out_map = svh::mapped(out_host);
    auto words = [&](size_t layer, int c) { return (chunk_end[c] - (c ? chunk_end[c - 1] : 0)) * layer / 16; };
    const bool direct_in = q_map && k_map && v_map && words(q_layer + 2 * kv_layer, 0) < 1u << 31 && svh::aligned(q_map, 16) &&
                           svh::aligned(k_map, 16) && svh::aligned(v_map, 16);
    const bool direct_out = out_map && words(q_layer, n_chunks - 1) < 1u << 31 && svh::aligned(out_map, 16);
    if (direct_in) {
        const unsigned nq = (unsigned)words(q_layer, 0), nk = (unsigned)words(kv_layer, 0);
        copy_parts({{static_cast<uint4 *>(q), static_cast<uint4 *>(draft_k), static_cast<uint4 *>(draft_v)},
                    {static_cast<const uint4 *>(q_map), static_cast<const uint4 *>(k_map), static_cast<const uint4 *>(v_map)},
                    {nq, nq + nk, nq + 2 * nk}});
    }
    // (the uploads of later chunks would only take bandwidth from the first one's)
    const bool in_forked = order(step->fork, main, in);
    bool back_forked = false;
    if (!direct_in && ok) upload(0);
    if (refresh_tail && ok) {
        st = sv_block_reps_layers(geom, layers, refresh_which, SV_TAIL_BLOCK, -1, reps, stream);
        ok = st == SV_OK;
    }
    // (a chunk's launches are issued ahead of the uploads that it does not need)
    for (int c = 0; c < n_chunks && ok; ++c) {
        if (c + 1 < n_chunks) upload(c + 1);
        if (c > 0 || !direct_in) cuda(cudaStreamWaitEvent(main, step->arrived[c], 0));
        if (!ok) break;
        const int first = c ? chunk_end[c - 1] : 0, end = chunk_end[c];
        st = sv_select_blocks_layers(geom, layers, first, end, anchors, q, reps, budget_blocks, n_sink, n_local, idx, cnt, max_sel, stream);
        if (st == SV_OK)
            st = svh::verify_attn_layers(geom, layers, first, end, anchors, q, draft_k, draft_v, parent, idx, cnt, max_sel, 0.f, out,
                                         workspace, workspace_bytes, status_word, stream, true);
        if (st != SV_OK) break;
        if (c == n_chunks - 1 && direct_out) {
            const size_t at = (c ? chunk_end[c - 1] : 0) * q_layer;
            const unsigned n = (unsigned)words(q_layer, c);
            copy_parts({{reinterpret_cast<uint4 *>(static_cast<char *>(out_map) + at)},
                        {reinterpret_cast<const uint4 *>(static_cast<const char *>(out) + at)},
                        {n, n, n}});
            continue;
        }
        if (!order(step->done[c], main, back)) break;
        back_forked = true;
        part(out_host, out, q_layer, c, cudaMemcpyDeviceToHost, back);
    }
    // The side streams that were forked join whatever happened: their copies still use the caller's memory, and a captured stream
    // may not be left forked.
    if (in_forked) order(step->joined, in, main);
    if (back_forked) order(step->joined, back, main);
    if (st != SV_OK) return st;
    return ok ? SV_OK : SV_ERR_CUDA;
}
