// Launch parameters of the attention kernel and the split merge, shared by the two files that hold them.
#pragma once
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "sv.h"
#include "sv_ptx.cuh"

namespace svk {

// Bits of the optional device status word (the values documented in sv.h).
constexpr int kStatusIndex = SV_STATUS_INDEX;   // a block index or page id outside its table was clamped
constexpr int kStatusNoList = SV_STATUS_NO_LIST;  // a selection count was negative (block selection gave up on that list)

// One layer of a layer table (sv_layer_table): what differs between the layers of a stack on the cache side.
struct alignas(64) LayerRow {
    CUtensorMap k_map, v_map;   // over the layer's pools, see pool_tensor_map
    void *k_pool, *v_pool;
    int32_t n_pages;
    int32_t pad[11];
};
static_assert(sizeof(LayerRow) == 320, "rows stay 64-byte aligned, as tensor maps have to be");

struct AttnParams {
    const __nv_bfloat16 *q;
    const __nv_bfloat16 *draft_k;
    const __nv_bfloat16 *draft_v;
    const int32_t *parent;
    const int32_t *block_table;
    const int32_t *seq_lens;
    const int32_t *sel_idx;
    const int32_t *sel_cnt;
    __nv_bfloat16 *out;
    float *lse;
    float *ws_o;    // [S][Hkv][splits][rows][128]
    float *ws_ml;   // [S][Hkv][splits][rows][2]
    int32_t *status;
    int T, Hq, Hkv, G, B, NBmax, max_sel, splits;
    float scale_log2;
    int Tt, tiles;   // draft tokens per row tile (G * Tt <= 128 query rows) and number of row tiles
    int pair;        // 1: a CTA serves two row tiles (grid.x = splits x ceil(tiles / 2)); 0: one (grid.x = splits x tiles)
    int n_pages;     // pages in each pool: page ids from the block table are clamped to it
    int n_claims;       // > 0: that many lists are handed out to one CTA per SM (splits = 1)
    uint32_t *claims;   // ... through these two words (list_claims.h), zero before and after the launch; null: by turns
    int cluster;     // 1: the splits of a (sequence, KV head) are a cluster that merges them itself (no partials, no merge kernel)
    int early_gather;   // 1: nothing the gather reads comes from the kernel just before; it starts ahead of the dependency wait
};

// Several layers in one launch: grid.z = layers x sequences, layer-major.  What a layer owns (q, out, draft K/V, partials)
// is numbered like the grid; tables, lengths and parents are those of the sequence, block lists of the layer's anchor.
struct StackAttnParams : AttnParams {
    const LayerRow *layers;           // device layer table, from the launch's first layer on
    int S;                            // sequences of a layer
    uint8_t list_of[SV_MAX_LAYERS];   // block list of a layer: the ordinal of the last anchor up to it
    // Not null: queries and draft K/V are read from these (pinned host memory), and copied to q, draft_k and draft_v on the way; the
    // outputs go to out_host as well.
    const __nv_bfloat16 *q_host = nullptr, *draft_k_host = nullptr, *draft_v_host = nullptr;
    __nv_bfloat16 *out_host = nullptr;
};

// The sum over the splits of a row, four output dims: o = sum_j 2^(m_j - m) o_j / sum_j 2^(m_j - m) l_j, a batch of splits at a time.
struct SplitSum {
    float M = -INFINITY, l = 0.f;
    float4 acc = {0.f, 0.f, 0.f, 0.f};
    template <int U>
    __device__ void add(const float2 (&ml)[U], const float4 (&o)[U])
    {
        float Mb = M;
#pragma unroll
        for (int u = 0; u < U; ++u) Mb = fmaxf(Mb, ml[u].x);
        const float M_use = (Mb == -INFINITY) ? 0.f : Mb;
        const float c = fast_exp2(M - M_use);   // rescale what earlier batches accumulated
        acc.x *= c, acc.y *= c, acc.z *= c, acc.w *= c;
        l *= c;
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const float w = fast_exp2(ml[u].x - M_use);
            acc.x += w * o[u].x, acc.y += w * o[u].y, acc.z += w * o[u].z, acc.w += w * o[u].w;
            l += w * ml[u].y;
        }
        M = Mb;
    }
    __device__ uint2 out() const
    {
        const float inv = 1.f / l;
        return make_uint2(pack_bf16(acc.x * inv, acc.y * inv), pack_bf16(acc.z * inv, acc.w * inv));
    }
    __device__ float lse() const { return (M + log2f(l)) * 0.69314718055994531f; }
};

constexpr int kMaxCluster = 8;   // CTAs of a cluster that merges its splits (the portable size)
// Whether a cluster of `splits` CTAs has room for each other's partials of `rows` query rows, and how many clusters of a size the
// device runs at once (0: none, or no device).
bool cluster_holds_partials(int splits, int rows);
int clusters_at_once(int size);

// tcgen05 / TMEM attention kernel (verify_attn_tc.cu): rows = G*T <= 128 packed as one M=128 tile.
cudaError_t launch_attn_tc(const CUtensorMap &tm_k, const CUtensorMap &tm_v, const AttnParams &p, dim3 grid,
                           cudaStream_t stream);
// the lists of a single layer, handed out (layers and claims null: CTA i takes lists i, i + CTAs, ...)
cudaError_t launch_attn_tc_handed(const CUtensorMap &tm_k, const CUtensorMap &tm_v, const StackAttnParams &p, dim3 grid, cudaStream_t stream);
cudaError_t launch_attn_tc_stack(const StackAttnParams &p, dim3 grid, cudaStream_t stream);

}  // namespace svk
