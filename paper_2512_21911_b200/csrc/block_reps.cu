// sv_block_reps: mean key of every KV block (the block representative implied by Eq. 5).
//
// Pure streaming reduction, bound by HBM bandwidth: one CTA per (block, KV head,
// sequence) reads the contiguous B x 128 bf16 tile of the block with 128-bit loads
// (all of a thread's loads are issued before the first use), accumulates in fp32 in a
// fixed order and writes 128 fp32 values.  Algorithmic traffic: B*256 bytes read +
// 512 bytes written per block.
#include <cuda_bf16.h>

#include <type_traits>

#include "attn_common.cuh"
#include "sv_host.h"
#include "sv_ptx.cuh"

namespace {

constexpr int kThreads = 256;
constexpr int kRowGroups = kThreads / 16;   // 16 threads cover one 256-byte key row

// Several layers in one launch: grid.z = layers x sequences, the pool is the layer's.  A kernel of its own: with 30000
// short CTAs even 270 bytes more of arguments and a branch cost a launch over one layer 10 %.
struct OneLayer {};
struct StackParams {
    const svk::LayerRow *layers;
    int S;
    uint8_t layer_of[SV_MAX_LAYERS];
};

// OutT: float (the default representatives) or __nv_bfloat16 (storage variant: the fp32 mean rounded once).
template <int B, typename OutT, class Stack>
__global__ void __launch_bounds__(kThreads) block_reps_kernel(const uint4 *__restrict__ k_pool,
                                                              const int32_t *__restrict__ block_table,
                                                              const int32_t *__restrict__ seq_lens,
                                                              OutT *__restrict__ reps, int Hkv, int NBmax,
                                                              int block_begin, int block_end, const Stack stack)
{
    const int h = blockIdx.y, z = blockIdx.z;
    int s = z, bz = z;   // sequence (table, length); batch index of the representatives
    if constexpr (std::is_same_v<Stack, StackParams>) {
        const int l = z / stack.S;
        s = z - l * stack.S;
        bz = stack.layer_of[l] * stack.S + s;
        k_pool = static_cast<const uint4 *>(stack.layers[stack.layer_of[l]].k_pool);
    }
    svk::grid_dependency_wait();      // the keys may come from the kernel just before (a cache append)
    svk::grid_launch_dependents();
    const int L = seq_lens[s];
    const int nb = min((L + B - 1) / B, NBmax);
    const int b = block_begin < 0 ? nb - 1 : block_begin + blockIdx.x;   // block_begin < 0: the tail block
    if (b < 0 || b >= nb || (block_begin >= 0 && block_end >= 0 && b >= block_end)) return;
    const int cnt = min(B, L - b * B);
    const int page = block_table[(size_t)s * NBmax + b];
    const uint4 *tile = k_pool + ((size_t)page * Hkv + h) * (B * 16);

    const int chunk = threadIdx.x & 15;     // 8 dims = one 16-byte chunk of the row
    const int rg = threadIdx.x >> 4;
    constexpr int kIter = B / kRowGroups;
    uint4 v[kIter];
#pragma unroll
    for (int i = 0; i < kIter; ++i) {
        const int row = rg + i * kRowGroups;
        v[i] = row < cnt ? __ldg(tile + row * 16 + chunk) : make_uint4(0u, 0u, 0u, 0u);
    }
    float acc[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int i = 0; i < kIter; ++i) {
        const __nv_bfloat162 *p = reinterpret_cast<const __nv_bfloat162 *>(&v[i]);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const float2 f = __bfloat1622float2(p[j]);
            acc[2 * j] += f.x;
            acc[2 * j + 1] += f.y;
        }
    }
    __shared__ float part[kRowGroups][128];
#pragma unroll
    for (int j = 0; j < 8; ++j) part[rg][chunk * 8 + j] = acc[j];
    __syncthreads();
    if (threadIdx.x < 128) {
        float sum = 0.f;
#pragma unroll
        for (int g = 0; g < kRowGroups; ++g) sum += part[g][threadIdx.x];
        reps[(((size_t)bz * Hkv + h) * NBmax + b) * 128 + threadIdx.x] = static_cast<OutT>(sum / (float)cnt);
    }
}

}  // namespace

// `n_batch`: sequences, or (layer, sequence) pairs of a stack.
template <typename OutT, class Stack>
static sv_status launch_block_reps(const sv_geom *geom, const void *k_pool, const int32_t *block_table, const int32_t *seq_lens,
                                   const Stack &stack, int n_batch, int32_t block_begin, int32_t block_end, OutT *reps,
                                   void *stream)
{
    if (!reps) return SV_ERR_NULL;
    if (!svh::aligned(reps, 16)) return SV_ERR_ALIGN;
    if (block_begin < 0 && block_begin != SV_TAIL_BLOCK) return SV_ERR_SHAPE;
    const int hi = (block_end < 0 || block_end > geom->max_blocks) ? geom->max_blocks : block_end;
    if (block_begin >= 0 && hi <= block_begin) return SV_OK;   // empty range: nothing to do
    dim3 grid(block_begin < 0 ? 1 : hi - block_begin, geom->n_kv_heads, n_batch);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(kThreads);
    cfg.stream = static_cast<cudaStream_t>(stream);
    cudaLaunchAttribute attr[1];
    svh::pdl_attribute(attr);
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    const uint4 *pool = static_cast<const uint4 *>(k_pool);
    const auto kernel = geom->block_size == 64 ? block_reps_kernel<64, OutT, Stack> : block_reps_kernel<128, OutT, Stack>;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, pool, block_table, seq_lens, reps, (int)geom->n_kv_heads,
                                             (int)geom->max_blocks, (int)block_begin, (int)block_end, stack);
    return e == cudaSuccess ? svh::launch_status() : SV_ERR_CUDA;
}

template <typename OutT>
static sv_status block_reps_impl(const sv_geom *geom, const sv_kv *kv, int32_t block_begin, int32_t block_end, OutT *reps,
                                 void *stream)
{
    sv_status st = svh::check_geom(geom);
    if (st != SV_OK) return st;
    st = svh::check_kv(geom, kv, false);
    if (st != SV_OK) return st;
    return launch_block_reps(geom, kv->k_pool, kv->block_table, kv->seq_lens, OneLayer{}, geom->n_seq, block_begin, block_end, reps, stream);
}

extern "C" sv_status sv_block_reps(const sv_geom *geom, const sv_kv *kv, int32_t block_begin, int32_t block_end,
                                   float *reps, void *stream)
{
    return block_reps_impl<float>(geom, kv, block_begin, block_end, reps, stream);
}

extern "C" sv_status sv_block_reps_bf16(const sv_geom *geom, const sv_kv *kv, int32_t block_begin, int32_t block_end,
                                        void *reps_bf16, void *stream)
{
    return block_reps_impl<__nv_bfloat16>(geom, kv, block_begin, block_end, static_cast<__nv_bfloat16 *>(reps_bf16), stream);
}

extern "C" sv_status sv_block_reps_layers(const sv_geom *geom, const sv_layers *layers, const uint8_t *which, int32_t block_begin,
                                          int32_t block_end, float *reps, void *stream)
{
    const sv_status st = svh::check_layers(geom, layers, 0, layers ? layers->n_layers : 1);
    if (st != SV_OK) return st;
    StackParams stack;
    stack.layers = static_cast<const svk::LayerRow *>(layers->table);
    stack.S = geom->n_seq;
    int n = 0;
    for (int l = 0; l < layers->n_layers; ++l)
        if (!which || which[l]) stack.layer_of[n++] = (uint8_t)l;
    if (n == 0) return SV_OK;
    return launch_block_reps(geom, nullptr, layers->block_table, layers->seq_lens, stack, n * geom->n_seq, block_begin, block_end, reps,
                             stream);
}
