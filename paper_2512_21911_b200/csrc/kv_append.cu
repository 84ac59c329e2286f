// sv_kv_append: commit the accepted draft tokens of a verification step to the paged KV cache and refresh
// the representatives (block means, Eq. 5) of the blocks that grew -- the step on either side of the
// verification attention (Section 2.1: the accepted prefix of the draft is kept; Section 3.1: blocks are cut
// from the current cache).
//
// One CTA per (KV head, sequence).  At most 64 tokens are appended per sequence, so at most two blocks are
// touched: the rows are copied with 128-bit loads/stores (K and V), then the one or two affected block
// means are recomputed exactly as sv_block_reps does (fp32 sums in a fixed order), which keeps
// them bit-identical to a full rebuild.  Page ids are checked against the pool size before anything is
// written: a table entry that is not a page of the pool ends the table (the rows are dropped).  Traffic: n*512 bytes copied + at
// most B*256 bytes read per (sequence, KV head): latency-bound, not bandwidth-bound.  Three trips to memory, each needing
// the one before: length, count and kept rows' numbers; page ids and draft rows; the rows that the block held already.  The appended
// rows are summed from shared memory, and the length is advanced by a warp of its own, whose fences and atomics would
// otherwise hold up the copy (32 layers of one sequence: 3.9 us behind the acceptance, 5 before, when rows were written, read back
// and waited for the atomics).
#include <cuda_bf16.h>

#include "attn_common.cuh"
#include "sv_host.h"
#include "sv_ptx.cuh"

namespace {

constexpr int kThreads = 256;       // that copy and sum; one more warp advances the length
constexpr int kRowGroups = kThreads / 16;
constexpr int kMaxAppended = 64;    // rows per sequence (svh::kMaxDraft)

template <int B>
__global__ void __launch_bounds__(kThreads + 32) kv_append_kernel(uint4 *__restrict__ k_pool, uint4 *__restrict__ v_pool,
                                                             const int32_t *__restrict__ block_table,
                                                             const int32_t *seq_lens,
                                                             const uint4 *__restrict__ draft_k,
                                                             const uint4 *__restrict__ draft_v,
                                                             const int32_t *__restrict__ accept_idx,
                                                             const int32_t *__restrict__ n_accept, int max_accept,
                                                             int32_t *seq_lens_out, float *__restrict__ reps,
                                                             int T, int Hkv, int NBmax, int n_pages,
                                                             const svk::LayerRow *layers, uint32_t *readers)
{
    __shared__ uint4 fresh[kMaxAppended * 16];   // the appended K rows
    __shared__ float part[kRowGroups][128];
    const int h = blockIdx.x, s = blockIdx.y, tid = threadIdx.x;
    int bz = s;   // batch index of what the layer owns (draft K/V, representatives)
    if (layers) {
        const svk::LayerRow *row = layers + blockIdx.z;
        bz += blockIdx.z * gridDim.y;
        k_pool = static_cast<uint4 *>(row->k_pool), v_pool = static_cast<uint4 *>(row->v_pool);
        n_pages = row->n_pages;
    }
    svk::grid_dependency_wait();
    svk::grid_launch_dependents();
    // first trip: length, number of rows, and (thread: 32 per row, K and V) the draft row that is kept
    const int which = (tid >> 4) & 1, c = tid & 15;
    const auto kept = [&](int a) { return a < max_accept ? accept_idx[(size_t)s * max_accept + a] : 0; };
    const auto draft_row = [&](int j) {
        const size_t src = (((size_t)bz * T + min(max(j, 0), T - 1)) * Hkv + h) * 16 + c;
        return __ldg((which ? draft_v : draft_k) + src);
    };
    const int L = seq_lens[s];
    int n = n_accept[s];
    const int j_first = kept(tid >> 5);
    // second trip: the page or pages, and the draft row
    const int *pages = block_table + (size_t)s * NBmax;
    const int b0 = L < 0 ? 0 : L / B;
    const int page0 = b0 < NBmax ? pages[b0] : -1, page1 = b0 + 1 < NBmax ? pages[b0 + 1] : -1;
    const uint4 first = draft_row(j_first);
    n = min(max(n, 0), max_accept);
    n = L < 0 ? 0 : max(0, min(n, NBmax * B - L));   // never past the last page of the table (nothing if L is already there)
    // A block whose table entry is not a page of the pool (not assigned yet: -1, or stale) ends the table: no row
    // enters it.  n <= 64 <= B, so the rows touch at most the blocks L / B and L / B + 1.
    if (page0 < 0 || page0 >= n_pages) n = 0;
    if (page1 < 0 || page1 >= n_pages) n = min(n, (b0 + 1) * B - L);
    const int Ln = L + n;
    if (readers) {
        // The lengths are advanced in place, by the last CTA of the sequence to have read the old one; the counter wraps to
        // zero behind it.  readers[S + s]: the new length on its way there (of the last layer, should the layers' pools
        // hold different numbers of pages).  Fences and atomics take as long as the rest of the kernel, so a warp of its own
        // does this.
        if (tid >= kThreads) {
            svk::named_bar_sync(1, kThreads + 32);   // every thread of this CTA holds the old length
            if (tid == kThreads) {
                int *fresh_len = reinterpret_cast<int *>(readers) + gridDim.y + s;
                if (h == 0 && blockIdx.z == gridDim.z - 1) atomicExch(fresh_len, Ln);
                __threadfence();
                if (atomicInc(readers + s, gridDim.x * gridDim.z - 1) == gridDim.x * gridDim.z - 1) {
                    __threadfence();
                    seq_lens_out[s] = atomicAdd(fresh_len, 0);
                }
            }
            return;
        }
        svk::named_bar_arrive(1, kThreads + 32);
    } else {
        if (tid >= kThreads) return;
        if (h == 0 && tid == 0) seq_lens_out[s] = Ln;
    }
    if (n <= 0) return;

    // third trip: the rows that the first block held already
    constexpr int kIter = B / kRowGroups;
    const int chunk = tid & 15, rg = tid >> 4;
    uint4 v[kIter];
    if (reps) {
        const uint4 *tile = k_pool + ((size_t)page0 * Hkv + h) * (B * 16);
#pragma unroll
        for (int i = 0; i < kIter; ++i) {
            const int row = rg + i * kRowGroups;
            v[i] = b0 * B + row < L ? tile[row * 16 + chunk] : make_uint4(0u, 0u, 0u, 0u);
        }
    }
    // copy the accepted rows: 16 threads per 256-byte row, K and V
    for (int a = tid >> 5; a < n; a += kThreads / 32) {
        const uint4 row = a == tid >> 5 ? first : draft_row(kept(a));
        const int t = L + a;
        const size_t dst = (((size_t)(t / B == b0 ? page0 : page1) * Hkv + h) * B + (t % B)) * 16 + c;
        (which ? v_pool : k_pool)[dst] = row;
        if (!which) fresh[a * 16 + c] = row;
    }
    if (!reps) return;
    svk::named_bar_sync(2, kThreads);

    // the means of the one or two blocks that grew (a second one holds appended rows only)
    for (int b = b0; b <= (Ln - 1) / B; ++b) {
        const int cnt = min(B, Ln - b * B);
        float acc[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int i = 0; i < kIter; ++i) {
            const int row = rg + i * kRowGroups, t = b * B + row;
            uint4 x = b == b0 ? v[i] : make_uint4(0u, 0u, 0u, 0u);
            if (t >= L && row < cnt) x = fresh[(t - L) * 16 + chunk];
            const __nv_bfloat162 *p2 = reinterpret_cast<const __nv_bfloat162 *>(&x);
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const float2 f = __bfloat1622float2(p2[j]);
                acc[2 * j] += f.x;
                acc[2 * j + 1] += f.y;
            }
        }
#pragma unroll
        for (int j = 0; j < 8; ++j) part[rg][chunk * 8 + j] = acc[j];
        svk::named_bar_sync(2, kThreads);
        if (tid < 128) {
            float sum = 0.f;
#pragma unroll
            for (int g = 0; g < kRowGroups; ++g) sum += part[g][tid];
            reps[(((size_t)bz * Hkv + h) * NBmax + b) * 128 + tid] = sum / (float)cnt;
        }
        svk::named_bar_sync(2, kThreads);
    }
}

}  // namespace

extern "C" sv_status sv_kv_append(const sv_geom *geom, void *k_pool, void *v_pool, int32_t n_pages,
                                  const int32_t *block_table, const int32_t *seq_lens, const void *draft_k,
                                  const void *draft_v, const int32_t *accept_idx, const int32_t *n_accept,
                                  int32_t max_accept, int32_t *seq_lens_out, float *reps, void *stream)
{
    sv_status st = svh::check_geom(geom);
    if (st != SV_OK) return st;
    if (!k_pool || !v_pool || !block_table || !seq_lens || !draft_k || !draft_v || !accept_idx || !n_accept || !seq_lens_out)
        return SV_ERR_NULL;
    if (n_pages < 1 || max_accept < 1 || max_accept > geom->n_draft) return SV_ERR_SHAPE;
    if (seq_lens_out == seq_lens) return SV_ERR_SHAPE;   // CTAs of the other KV heads still read the old length
    if (!svh::aligned(k_pool, 128) || !svh::aligned(v_pool, 128) || !svh::aligned(draft_k, 16) ||
        !svh::aligned(draft_v, 16) || (reps && !svh::aligned(reps, 16)))
        return SV_ERR_ALIGN;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(geom->n_kv_heads, geom->n_seq);
    cfg.blockDim = dim3(kThreads + 32);
    cfg.stream = static_cast<cudaStream_t>(stream);
    cudaLaunchAttribute attr[1];
    svh::pdl_attribute(attr);
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    uint4 *kp = static_cast<uint4 *>(k_pool), *vp = static_cast<uint4 *>(v_pool);
    const uint4 *dk = static_cast<const uint4 *>(draft_k), *dv = static_cast<const uint4 *>(draft_v);
    const cudaError_t e =
        geom->block_size == 64
            ? cudaLaunchKernelEx(&cfg, kv_append_kernel<64>, kp, vp, block_table, seq_lens, dk, dv, accept_idx, n_accept,
                                 (int)max_accept, seq_lens_out, reps, (int)geom->n_draft, (int)geom->n_kv_heads,
                                 (int)geom->max_blocks, (int)n_pages, nullptr, nullptr)
            : cudaLaunchKernelEx(&cfg, kv_append_kernel<128>, kp, vp, block_table, seq_lens, dk, dv, accept_idx, n_accept,
                                 (int)max_accept, seq_lens_out, reps, (int)geom->n_draft, (int)geom->n_kv_heads,
                                 (int)geom->max_blocks, (int)n_pages, nullptr, nullptr);
    return e == cudaSuccess ? svh::launch_status() : SV_ERR_CUDA;
}

extern "C" sv_status sv_kv_append_layers(const sv_geom *geom, const sv_layers *layers, const void *draft_k, const void *draft_v,
                                         const int32_t *accept_idx, const int32_t *n_accept, int32_t max_accept,
                                         int32_t *seq_lens, uint32_t *counters, float *reps, void *stream)
{
    const sv_status st = svh::check_layers(geom, layers, 0, layers ? layers->n_layers : 1);
    if (st != SV_OK) return st;
    if (!draft_k || !draft_v || !accept_idx || !n_accept || !seq_lens || !counters) return SV_ERR_NULL;
    if (max_accept < 1 || max_accept > geom->n_draft) return SV_ERR_SHAPE;
    if (seq_lens != layers->seq_lens) return SV_ERR_SHAPE;
    if (!svh::aligned(draft_k, 16) || !svh::aligned(draft_v, 16) || !svh::aligned(counters, 4) || (reps && !svh::aligned(reps, 16)))
        return SV_ERR_ALIGN;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(geom->n_kv_heads, geom->n_seq, layers->n_layers);
    cfg.blockDim = dim3(kThreads + 32);
    cfg.stream = static_cast<cudaStream_t>(stream);
    cudaLaunchAttribute attr[1];
    svh::pdl_attribute(attr);
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    const auto kernel = geom->block_size == 64 ? kv_append_kernel<64> : kv_append_kernel<128>;
    const cudaError_t e = cudaLaunchKernelEx(
        &cfg, kernel, (uint4 *)nullptr, (uint4 *)nullptr, layers->block_table, (const int32_t *)seq_lens,
        static_cast<const uint4 *>(draft_k), static_cast<const uint4 *>(draft_v), accept_idx, n_accept, (int)max_accept, seq_lens, reps,
        (int)geom->n_draft, (int)geom->n_kv_heads, (int)geom->max_blocks, 0, static_cast<const svk::LayerRow *>(layers->table), counters);
    return e == cudaSuccess ? svh::launch_status() : SV_ERR_CUDA;
}
